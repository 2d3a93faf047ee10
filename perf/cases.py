"""The work that users of gnnpre have it do, as cases that can be timed and compared.

Every case is one call (or, where a user makes them together, one short sequence of calls) of the public entry
points of ``paper_2207_12000_b200.binding``.  Graph and matrix sizes are those of this repository's own
workloads (``gnnpre_inputs.configs``); graphs are R-MAT or Erdos-Renyi draws of ``gnnpre_inputs.graphs``.

Kinds of case:

  propagate    the K hops of a resident feature matrix over a plan that is kept (features change, the graph does not)
  precompute   what a dataset costs once: plan from the CSR on the device, K hops, plan destroyed
  weighted     personalised-PageRank steps and their fixed-weight sum, hops not kept
  streamed     the K hops of a matrix in pinned host memory, results back in pinned host memory
  normalize    the values of the normalised adjacency, on the device
  lc           the first dense stage of a model over rows of the precomputed hops
"""
from __future__ import annotations

import math

import torch

from gnnpre_inputs import graphs
from paper_2207_12000_b200 import binding as B

GCN, SAGE, GIN = B.GNNPRE_OP_GCN_SYM, B.GNNPRE_OP_SAGE_MEAN, B.GNNPRE_OP_GIN_SUM
GIN_EPS = 0.1


def listed():
    return [
        # A small graph, two hops: launches and latency are what counts (the unit-test and toy-dataset size).
        {"name": "small_gcn_f64", "kind": "propagate", "graph": "er", "n": 4096, "m": 32768, "op": GCN, "F": 64, "K": 2, "b": 1},
        # A citation graph of 169 K papers at its own feature width, four edge blocks: the ordinary case.
        {"name": "citation_gcn_f128", "kind": "propagate", "graph": "rmat_directed", "n": 169343, "m": 1166243, "op": GCN,
         "F": 128, "K": 3, "b": 4},
        # The same graph with the mean operator at the narrowest width of the width sweep (reduced features).
        {"name": "citation_sage_f16", "kind": "propagate", "graph": "rmat_directed", "n": 169343, "m": 1166243, "op": SAGE,
         "F": 16, "K": 3, "b": 1},
        # ... and with the sum operator at twice its width.
        {"name": "citation_gin_f256", "kind": "propagate", "graph": "rmat_directed", "n": 169343, "m": 1166243, "op": GIN,
         "F": 256, "K": 3, "b": 8},
        # A co-purchase graph of 2.4 M products and 124 M directed edges: the largest resident workload.
        {"name": "products_sage_f100", "kind": "propagate", "graph": "rmat", "n": 2449029, "m": 61859140, "op": SAGE, "F": 100,
         "K": 3, "b": 32},
        # A dense social graph with rows of 602 features (wide, and not a multiple of four).
        {"name": "social_gcn_f602", "kind": "propagate", "graph": "rmat", "n": 232965, "m": 11606919, "op": GCN, "F": 602, "K": 2,
         "b": 0},
        # An image graph with 500 features, from its CSR to its hops: what is run once per dataset.
        {"name": "image_once_gcn_f500", "kind": "precompute", "graph": "rmat", "n": 89250, "m": 899756, "op": GCN, "F": 500,
         "K": 2, "b": 0},
        # Ten personalised-PageRank steps on hidden features of the citation graph, only their weighted sum wanted.
        {"name": "citation_ppr_f64", "kind": "weighted", "graph": "rmat_directed", "n": 169343, "m": 1166243, "op": GCN, "F": 64,
         "K": 10, "b": 0},
        # A 1/64 cut of the 111 M-node citation graph through pinned host memory, as the whole graph is run.
        {"name": "papers_streamed_f128", "kind": "streamed", "graph": "rmat", "n": 1735311, "m": 12622545, "op": GCN, "F": 128,
         "K": 2, "b": 0},
        # The normalised adjacency of a 1/32 cut of that graph, exported for another library.
        {"name": "papers_normalize", "kind": "normalize", "graph": "rmat", "n": 3470623, "m": 25245091, "op": GCN, "F": 128, "K": 0,
         "b": 0},
        # The first dense stage on a training mini-batch of 4096 rows of three hops, at the call's default precision.
        {"name": "batch_tf32_f128_h256", "kind": "lc", "n": 169343, "rows": 4096, "F": 128, "K": 3, "H": 256, "precision": "tf32"},
        # ... and over all rows of the products graph in random order (one epoch, or inference), fp32-class precision.
        {"name": "epoch_x3_f100_h256", "kind": "lc", "n": 2449029, "rows": 2449029, "F": 100, "K": 3, "H": 256,
         "precision": "tf32x3"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["propagate", "propagate", "propagate", "precompute", "weighted", "streamed", "normalize", "lc", "lc"])
    if kind == "lc":
        n = _log(rng, 10000, 2449029)
        F = _log(rng, 16, 602)
        K = rng.randint(1, 4)
        rows = _log(rng, 512, min(n, 7.5e8 / (K * (F + 256))))
        precision = rng.choice(["tf32", "tf32x3"])
        return {"kind": kind, "n": n, "rows": rows, "F": F, "K": K, "H": rng.choice([64, 128, 192, 256]), "precision": precision}
    op = rng.choice([GCN, SAGE, GIN])
    if kind == "streamed":
        n = _log(rng, 50000, 1735311)
        F = _log(rng, 32, 256)
        K = rng.randint(1, 3)
        F = max(32, min(F, int(6.6e8 / ((K + 1) * n))))
    else:
        n = _log(rng, 4096, 3470623 if kind == "normalize" else 2449029)
        F = _log(rng, 16, 602)
        K = 0 if kind == "normalize" else 10 if kind == "weighted" else rng.randint(1, 3)
        F = max(16, min(F, int(9.5e8 / ((min(K, 3) + 1) * n))))
    degree = math.exp(rng.uniform(math.log(8), math.log(100)))
    most = min(30e6, 1.8e10 / (max(K, 1) * F))
    m = max(n, int(min(n * degree / 2, most)))
    # (merged reciprocal edges make the size of a "rmat_directed" edge list depend on the seed)
    graph = "er" if n <= 16384 else "rmat" if kind == "normalize" else rng.choice(["rmat", "rmat_directed"])
    b = rng.choice([0, 1, 4, 32])
    if kind in ("streamed", "weighted", "precompute", "normalize"):
        b = 0
    return {"kind": kind, "graph": graph, "n": n, "m": m, "op": op, "F": F, "K": K, "b": b}


def _graph(case, seed):
    if case["graph"] == "er":
        return graphs.erdos_renyi(case["n"], case["m"], seed, device="cuda")
    return graphs.rmat(case["n"], case["m"], seed, directed_candidates=case["graph"] == "rmat_directed", device="cuda")


def _matrix(n, F, gen, scale=1.0):
    """Standard-normal features; rows padded to whole groups of four columns, as the library wants them."""
    buf = torch.zeros((n, (F + 3) // 4 * 4), device="cuda")
    buf[:, :F].normal_(generator=gen)
    return buf[:, :F].mul_(scale) if scale != 1.0 else buf[:, :F]


def _empty(n, F):
    return torch.empty((n, (F + 3) // 4 * 4), device="cuda")[:, :F]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, n, F, K = case["kind"], case["n"], case["F"], case["K"]
    s = {"case": case}
    if kind == "lc":
        H = case["H"]
        s["hops"] = [_matrix(n, F, gen) for _ in range(K)]
        s["Wt"] = _matrix(H, F, gen, 1.0 / math.sqrt(F))
        s["batch"] = torch.randperm(n, generator=gen, device="cuda", dtype=torch.int32)[:case["rows"]].contiguous()
        s["out"] = torch.empty((K, case["rows"], H), device="cuda")
        s["relu_mask"] = (1 << K) - 2  # every term but the first has another layer after it
        s["precision"] = B.GNNPRE_LC_TF32X3 if case["precision"] == "tf32x3" else B.GNNPRE_LC_TF32
        return s
    g = _graph(case, seed)
    host = kind == "streamed"
    if kind == "precompute":
        s["g"] = g
    else:
        s["plan"] = B.gnnpre_build_plan(g.rowptr, g.colidx, case["op"], F, gin_eps=GIN_EPS if case["op"] == GIN else 0.0,
                                        force_blocks=case["b"], teleport_alpha=0.1 if kind == "weighted" else 0.0,
                                        operands_mem=B.GNNPRE_MEM_HOST if host else B.GNNPRE_MEM_DEVICE)
    if kind == "normalize":
        s["vals"] = torch.empty(B.gnnpre_plan_info(s["plan"])["nnz_tilde"], device="cuda")
        return s
    s["X"] = _matrix(n, F, gen)
    if host:
        Fp = (F + 3) // 4 * 4
        X = torch.empty((n, Fp), pin_memory=True)[:, :F]
        X.copy_(s["X"])
        s["X"] = X
        s["out"] = [torch.empty((n, Fp), pin_memory=True)[:, :F] for _ in range(K)]
    elif kind == "weighted":
        s["gamma"] = [0.1 * 0.9 ** k for k in range(K)] + [0.9 ** K]
        two = [_empty(n, F) for _ in range(min(K, 2))]
        s["out"] = [two[k % 2] for k in range(K)]
        s["Z"] = _empty(n, F)
    else:
        s["out"] = [_empty(n, F) for _ in range(K)]
    return s


def run(s):
    case = s["case"]
    kind, K = case["kind"], case["K"]
    if kind == "lc":
        return B.gnnpre_lc_first_layer(s["hops"], s["batch"], s["Wt"], relu_mask=s["relu_mask"], precision=s["precision"],
                                       out=s["out"], check=False)
    if kind == "normalize":
        return B.gnnpre_normalize(s["plan"], s["vals"])
    if kind == "weighted":
        hops, Z = B.gnnpre_propagate_weighted(s["plan"], s["X"], s["gamma"], out=s["out"], Z=s["Z"])
        return {"last": hops[-2:], "Z": Z}
    if kind == "precompute":
        plan = B.gnnpre_build_plan(s["g"].rowptr, s["g"].colidx, case["op"], case["F"], gin_eps=GIN_EPS if case["op"] == GIN else 0.0)
        out, _ = B.gnnpre_propagate(plan, s["X"], K, out=s["out"])
        plan.close()
        return out
    out, _ = B.gnnpre_propagate(s["plan"], s["X"], K, out=s["out"])
    return out


def work(case):
    """Every input read once, every output written once (hops that a hop reads back are outputs); the graph is its CSR."""
    kind, n, F, K = case["kind"], case["n"], case["F"], case["K"]
    if kind == "lc":
        rows, H = case["rows"], case["H"]
        return {"bytes": 4 * K * rows * (F + H) + 4 * H * F + 4 * rows, "flops": 2 * K * rows * F * H}
    nnz = 2 * case["m"]
    E = nnz + (0 if case["op"] == SAGE else n)
    csr = 4 * nnz + 8 * (n + 1)
    if kind == "normalize":
        return {"bytes": csr + 4 * E, "flops": 2 * E}
    matrices = 4 if kind == "weighted" else K + 1
    return {"bytes": csr + 4 * n * F * matrices, "flops": 2 * E * F * K}


def tolerance(case):
    """About four times the error of one pass against the same sums in 64 bits."""
    kind = case["kind"]
    if kind == "normalize":
        return "exact"  # evaluated in fp64 and rounded once
    if kind == "lc":
        # tf32 operands: 7.7e-4 (largest single error 2.8e-3 of the output's size); split operands: 1.2e-6 (6e-6)
        return {"rel": 3e-3, "max": 1.2e-2} if case["precision"] == "tf32" else {"rel": 4e-6, "max": 4e-5}
    # compensated fp32 sums: 1e-8 .. 8e-8 (largest single error 2.8e-6)
    return {"rel": 4e-7, "max": 1.2e-5}
