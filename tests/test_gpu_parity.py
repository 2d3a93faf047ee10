"""GPU parity: the CUDA library, called through its C ABI, against the fp64 CPU oracle.

Integer outputs (degrees, the support's edge list, block tables, Eq. 12) must match bit for bit;
scale factors are fp64-computed and rounded once, so they match bit for bit too; propagated
features must stay within 1e-5 relative error per hop.
"""
import itertools

import numpy as np
import pytest
import torch

import gnnpre_inputs as gi
import oracle as orc
from parity_util import TOL, backward_error, check_all_hops, hop_error, single_hop_of, to_np

pytestmark = pytest.mark.gpu

OPS = (0, 1, 2)
EPS = 0.1


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_12000_b200 import binding
    return binding


def dev(g):
    return g.rowptr.cuda(), g.colidx.cuda()


def small_graphs():
    yield "er33", gi.erdos_renyi(33, 70, 5)
    yield "er1000", gi.erdos_renyi(1000, 6000, 6)
    yield "rmat3000", gi.rmat(3000, 20000, 7, directed_candidates=True)
    yield "star", gi.from_edge_list(700, [(0, j) for j in range(1, 650)])  # hub + isolated tail nodes
    yield "path2", gi.from_edge_list(2, [(0, 1)])
    yield "lonely", gi.from_edge_list(5, [])  # no edges at all


# ------------------------------------------------------------------ plan parity (bit-exact)

@pytest.mark.parametrize("name,g", list(small_graphs()) + [("c1", None)])
@pytest.mark.parametrize("op", OPS)
def test_plan_matches_oracle_bit_for_bit(B, name, g, op):
    if g is None:
        g = gi.make_graph(gi.WORKLOADS["c1"])
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    drp, dci = dev(g)
    deg = orc.degrees(rp)
    np.testing.assert_array_equal(to_np(B.gnnpre_degrees(drp, dci)), deg)
    rp_t, ci_t = orc.support(op, rp, ci)
    m = int(rp_t[-1])
    for b in sorted({1, 2, 3, 7, 64, m} - {0}):
        if b > m:
            continue
        plan = B.gnnpre_build_plan(drp, dci, op, 16, gin_eps=EPS, force_blocks=b, force_col_slabs=1, segment_edges=8)
        info = plan.info()
        assert (info["n"], info["nnz"], info["nnz_tilde"], info["b"], info["c"]) == (g.n, g.nnz, m, b, 1)
        assert info["B_S"] == 4 * m + 8 * (g.n + 1) and info["B_X"] == 4 * g.n * 16
        pdeg, r, c = B.gnnpre_plan_scales(plan)
        np.testing.assert_array_equal(pdeg.numpy(), deg)
        wr, wc = orc.scales_f32(op, deg)
        np.testing.assert_array_equal(r.numpy().view(np.uint32), wr.view(np.uint32))
        np.testing.assert_array_equal(c.numpy().view(np.uint32), wc.view(np.uint32))
        srp, sci = B.gnnpre_plan_support(plan)
        np.testing.assert_array_equal(srp.numpy(), rp_t)
        np.testing.assert_array_equal(sci.numpy(), ci_t)
        e_off = orc.block_offsets(m, b)
        row_lo, row_hi, fp, lp = orc.block_rows(rp_t, e_off)
        for l in range(b):
            blk = B.gnnpre_plan_block(plan, l)
            assert (blk["e_lo"], blk["e_hi"]) == (e_off[l], e_off[l + 1])
            assert (blk["row_lo"], blk["row_hi"]) == (row_lo[l], row_hi[l])
            assert (blk["first_row_partial"], blk["last_row_partial"]) == (fp[l], lp[l])
        plan.close()


def test_plan_with_caller_degrees_and_budget_search(B):
    g = gi.erdos_renyi(500, 3000, 8)
    drp, dci = dev(g)
    deg = B.gnnpre_degrees(drp, dci)
    F = 64
    m = g.nnz + g.n
    B_S, B_X, B_fixed = 4 * m + 8 * (g.n + 1), 4 * g.n * F, 16 * g.n
    for budget in (B_fixed + B_S + 2 * B_X, B_fixed + B_S // 3 + B_X, B_fixed + 2000 + B_X // 2):
        want = orc.solve_budget(B_S, B_X, B_fixed, 1, 2, budget, min(m, 1 << 20), F // 4)
        plan = B.gnnpre_build_plan(drp, dci, 0, F, degrees=deg, budget_bytes=budget)
        info = plan.info()
        assert (info["b"], info["c"]) == want
        assert info["slab_width"] == orc.slab_width(F, info["c"])
        plan.close()
    with pytest.raises(B.GnnpreError) as ei:
        B.gnnpre_build_plan(drp, dci, 0, F, budget_bytes=B_fixed + 100)
    assert ei.value.status == -6


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("nnz_half", [15, 16, 17, 127, 128, 129, 700])
def test_support_across_warp_boundaries_and_runs_of_empty_rows(B, op, nnz_half):
    """The support's edge list is built 256 edges to a warp, 32 at a time: edge counts around those sizes, a hub, runs of
    31 to 5,000 rows without edges, self-loops before, inside and behind a row's columns; and each kind of violation of
    the column contract is found wherever it sits."""
    n = 9000
    far = [40, 72, 105, 400, 5400, 8999]
    edges = [(far[i % 6] - i // 6 % 30 - 1, far[(i + 1 + i // 180) % 6] - i // 6 % 30 - 1) for i in range(nnz_half // 2)]
    edges += [(2000, 2001 + j) for j in range(nnz_half - len(edges))]
    g = gi.from_edge_list(n, edges)
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    rp_t, ci_t = orc.support(op, rp, ci)
    plan = B.gnnpre_build_plan(*dev(g), op, 16)
    srp, sci = B.gnnpre_plan_support(plan)
    np.testing.assert_array_equal(srp.numpy(), rp_t)
    np.testing.assert_array_equal(sci.numpy(), ci_t)
    plan.close()
    for at in (0, g.nnz // 2, g.nnz - 1):
        for value in (n, -1, int(np.searchsorted(rp, at, side="right")) - 1):  # out of range twice, on the diagonal
            bad = g.colidx.clone()
            bad[at] = value
            with pytest.raises(B.GnnpreError) as ei:
                B.gnnpre_build_plan(g.rowptr.cuda(), bad.cuda(), op, 16)
            assert ei.value.status == -2


# ------------------------------------------------------------------ propagation parity

def run_case(B, g, op, F, K, *, b=1, c=1, seg=0, flags=0, ldx=None, ldo=None, seed=1):
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    drp, dci = dev(g)
    ldx = ldx or F
    ldo = ldo or F
    Xbuf = torch.full((g.n, ldx), float("nan"), device="cuda")
    X = Xbuf[:, :F]
    X.copy_(gi.normal_matrix(g.n, F, seed, device="cuda"))
    obufs = [torch.full((g.n, ldo), -7.0, device="cuda") for _ in range(K)]
    outs = [o[:, :F] for o in obufs]
    plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, force_blocks=b, force_col_slabs=c, segment_edges=seg,
                               flags=flags)
    B.gnnpre_propagate(plan, X, K, outs)
    torch.cuda.synchronize()
    for o in obufs:
        assert bool((o[:, F:] == -7.0).all()), "padding columns were written"
    worst = check_all_hops(op, EPS, rp, ci, to_np(X), outs, single_hop=single_hop_of(B, plan))
    plan.close()
    return worst, outs


def test_config1_erdos_renyi_gcn(B):
    """Configuration 1: 4,096 nodes, 32,768 edges, F=64, K=2, GCN, a single edge block."""
    w = gi.WORKLOADS["c1"]
    g = gi.make_graph(w)
    assert (g.n, g.nnz) == (4096, 65536)
    run_case(B, g, w.op, w.feat_dim, w.hops, b=w.blocks, seed=w.seed)


@pytest.mark.parametrize("name,g", list(small_graphs()))
@pytest.mark.parametrize("op", OPS)
def test_small_graphs_all_shapes(B, name, g, op):
    m = orc.support_nnz(op, g.n, g.nnz)
    for F, seg in ((4, 8), (16, 4), (20, 32), (64, 8), (100, 16), (128, 0), (256, 8), (516, 32), (640, 16), (1040, 8)):
        for b in (1, 3):
            if b > m:
                continue
            run_case(B, g, op, F, 2, b=b, seg=seg)


@pytest.mark.parametrize("op", OPS)
def test_blocks_slabs_and_launch_modes_agree(B, op):
    """Different (b, c), segment sizes and launch groupings change only the rounding order."""
    g = gi.rmat(5000, 40000, 9, directed_candidates=True)
    F, K = 72, 3
    ref = None
    for b, c, seg, flags in ((1, 1, 0, 0), (4, 1, 64, 0), (64, 1, 16, 1), (7, 3, 32, 1), (1, 18, 1, 0), (5, 2, 0, 0)):
        _, outs = run_case(B, g, op, F, K, b=b, c=c, seg=seg, flags=flags, ldx=F + 4, ldo=F + 8)
        cur = [to_np(o).astype(np.float64) for o in outs]
        if ref is None:
            ref = cur
        else:
            for k in range(K):
                assert hop_error(cur[k], ref[k]) <= TOL


def test_hub_longer_than_many_segments_and_blocks(B):
    """A row far longer than a segment and a block: its parts are summed by the fix-up pass."""
    n = 40000
    edges = [(0, j) for j in range(1, n)] + [(j, j + 1) for j in range(1, 2000)]
    g = gi.from_edge_list(n, edges)
    for op in OPS:
        run_case(B, g, op, 32, 2, b=9, seg=32)
        run_case(B, g, op, 128, 2, b=1, seg=0)


def test_runs_are_bitwise_reproducible(B):
    g = gi.rmat(20000, 200000, 10, directed_candidates=True)
    drp, dci = dev(g)
    X = gi.normal_matrix(g.n, 128, 3, device="cuda")
    plan = B.gnnpre_build_plan(drp, dci, 0, 128, force_blocks=4)
    a, _ = B.gnnpre_propagate(plan, X, 3)
    b, _ = B.gnnpre_propagate(plan, X, 3)
    torch.cuda.synchronize()
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    plan.close()


def test_config2_rmat_gcn_four_blocks(B):
    """Configuration 2: 169,343 nodes, 1,166,243 directed R-MAT edges symmetrised, F=128, K=3, GCN, b=4."""
    w = gi.WORKLOADS["c2"]
    g = gi.make_graph(w, device="cuda").to("cpu")
    assert g.n == 169343
    run_case(B, g, w.op, w.feat_dim, w.hops, b=w.blocks, seed=w.seed)


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("F", [16, 64, 128, 256, 512])
def test_config3_operator_width_block_sweep(B, op, F):
    """Configuration 3: ops x widths x block counts {1, 8, 64} on the 169,343-node graph, K=3."""
    w = gi.WORKLOADS["c3"]
    g = gi.make_graph(w, device="cuda").to("cpu")
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    drp, dci = dev(g)
    X = gi.normal_matrix(g.n, F, w.seed, device="cuda")
    Xn = to_np(X)
    want = orc.propagate(op, w.gin_eps, rp, ci, Xn, w.hops)
    for b in w.sweep["blocks"]:
        plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=w.gin_eps, force_blocks=b)
        outs, _ = B.gnnpre_propagate(plan, X, w.hops)
        torch.cuda.synchronize()
        one_hop = single_hop_of(B, plan)
        for k in range(w.hops):
            gk = to_np(outs[k])
            assert hop_error(gk, want[k]) <= TOL
            rows = np.random.default_rng(k).integers(0, g.n, 4096)
            # floor-free check of one hop on an input both sides share: X_0, then the oracle's hops in fp32
            prev = Xn if k == 0 else np.ascontiguousarray(want[k - 1].astype(np.float32))
            assert backward_error(op, w.gin_eps, rp, ci, prev, gk if k == 0 else one_hop(prev), rows) <= TOL
        plan.close()


# ------------------------------------------------------------------ errors and edge cases

def test_invalid_inputs_are_rejected(B):
    g = gi.erdos_renyi(100, 300, 11)
    drp, dci = dev(g)

    def status(fn):
        with pytest.raises(B.GnnpreError) as ei:
            fn()
        return ei.value.status

    assert status(lambda: B.gnnpre_build_plan(drp, dci, 0, 0)) == -1           # F < 1
    assert status(lambda: B.gnnpre_build_plan(drp, dci, 5, 16)) == -1          # bad op
    assert status(lambda: B.gnnpre_build_plan(drp, dci, 1, 16, force_blocks=g.nnz + 1)) == -1  # empty block
    assert status(lambda: B.gnnpre_build_plan(drp, dci, 0, 16, force_col_slabs=5)) == -1
    bad = dci.clone()
    bad[3] = 10 ** 6
    assert status(lambda: B.gnnpre_build_plan(drp, bad, 0, 16)) == -2          # column out of range
    bad = dci.clone()
    bad[int(g.rowptr[5])] = 5
    assert status(lambda: B.gnnpre_build_plan(drp, bad, 0, 16)) == -2          # a diagonal entry or broken order
    bad = dci.clone()
    lo = int(g.rowptr[7])
    bad[lo + 1] = bad[lo]
    assert status(lambda: B.gnnpre_build_plan(drp, bad, 0, 16)) == -2          # duplicate column
    badrp = drp.clone()
    badrp[10] = badrp[11] + 1
    assert status(lambda: B.gnnpre_build_plan(badrp, dci, 0, 16)) == -2        # rowptr not monotone
    plan = B.gnnpre_build_plan(drp, dci, 0, 16)
    X = torch.zeros((100, 18), device="cuda")[:, :16]
    assert status(lambda: B.gnnpre_propagate(plan, X, 1)) == -3               # ldx % 4
    X = torch.zeros((100, 16), device="cuda")
    assert status(lambda: B.gnnpre_propagate(plan, X, 0, [])) == -1
    assert status(lambda: B.gnnpre_propagate(plan, X, 2, [X.clone(), X])) == -1  # out aliases X
    plan.close()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("fault", ["descending", "negative", "beyond", "short", "column", "diagonal", "order"])
def test_invalid_graphs_are_rejected_by_a_build_that_looks_once(B, op, fault):
    """Graphs of more than 1 MB of tables: the build launches everything before the host reads what the device found."""
    g = gi.rmat(60000, 400000, 47, directed_candidates=True)
    rp, ci = dev(g)
    row = int((g.rowptr[1:] - g.rowptr[:-1] >= 3).nonzero()[1000])
    lo = int(g.rowptr[row])
    if fault == "descending":
        rp[row + 1] = lo - 2
    elif fault == "negative":
        rp[row + 1] = -5
    elif fault == "beyond":
        rp[row + 1] = g.nnz + 7
    elif fault == "short":
        rp[-1] = g.nnz - 1
    else:
        ci[lo + 1] = {"column": g.n, "diagonal": row, "order": int(ci[lo])}[fault]
    with pytest.raises(B.GnnpreError) as ei:
        B.gnnpre_build_plan(rp, ci, op, 64)
    assert ei.value.status == -2
    plan = B.gnnpre_build_plan(*dev(g), op, 64, gin_eps=EPS)  # and the next one is as good as ever
    X = gi.normal_matrix(g.n, 64, 48)
    outs, _ = B.gnnpre_propagate(plan, X.cuda(), 1)
    check_all_hops(op, EPS, g.rowptr.numpy(), g.colidx.numpy(), X.numpy(), outs)
    plan.close()


def test_graph_without_edges(B):
    g = gi.from_edge_list(6, [])
    drp, dci = dev(g)
    X = gi.normal_matrix(6, 8, 1, device="cuda")
    for op, want in ((0, X), (1, torch.zeros_like(X)), (2, (1 + np.float32(EPS)) * X)):
        plan = B.gnnpre_build_plan(drp, dci, op, 8, gin_eps=EPS)
        outs, _ = B.gnnpre_propagate(plan, X, 2)
        torch.cuda.synchronize()
        torch.testing.assert_close(outs[0], want, rtol=1e-6, atol=0)
        plan.close()


# ------------------------------------------------------------------ streamed operands

@pytest.mark.parametrize("csr_on_host,x_on_host,out_on_host", [(False, True, True), (True, True, True),
                                                               (False, False, True), (True, True, False)])
@pytest.mark.parametrize("op", OPS)
def test_streamed_equals_resident_bitwise(B, op, csr_on_host, x_on_host, out_on_host):
    """Host-resident operands travel through the same kernels in the same order, so for the same
    (b, c) and segment size the result is bit-identical to the device-resident run."""
    g = gi.rmat(30000, 250000, 13, directed_candidates=True)
    F, K = 48, 3
    drp, dci = dev(g)
    X = gi.normal_matrix(g.n, F, 5, device="cuda")
    for b, c in ((1, 1), (5, 1), (3, 3), (2, 12)):
        ref_plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, force_blocks=b, force_col_slabs=c,
                                       segment_edges=64)
        ref, _ = B.gnnpre_propagate(ref_plan, X, K)
        torch.cuda.synchronize()
        pb_plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, force_blocks=b, force_col_slabs=c,
                                      segment_edges=64, flags=B.GNNPRE_FLAG_LAUNCH_PER_BLOCK)
        pb, _ = B.gnnpre_propagate(pb_plan, X, K)  # one launch per block: same bits as one launch per hop
        torch.cuda.synchronize()
        for k in range(K):
            assert torch.equal(pb[k], ref[k])
        pb_plan.close()
        rp, ci = (g.rowptr.pin_memory(), g.colidx.pin_memory()) if csr_on_host else (drp, dci)
        plan = B.gnnpre_build_plan(rp, ci, op, F, gin_eps=EPS, force_blocks=b, force_col_slabs=c, segment_edges=64,
                                   operands_mem=B.GNNPRE_MEM_HOST)
        assert plan.info()["structure_mem"] == (1 if csr_on_host else 0)
        Xin = X.cpu().pin_memory() if x_on_host else X
        ldo = F + 4
        if out_on_host:
            obuf = [torch.full((g.n, ldo), -3.0).pin_memory() for _ in range(K)]
        else:
            obuf = [torch.full((g.n, ldo), -3.0, device="cuda") for _ in range(K)]
        for rep in range(2):  # the second call reuses the plan's staging buffers
            outs, st = B.gnnpre_propagate(plan, Xin, K, [o[:, :F] for o in obuf], want_stats=True)
            torch.cuda.synchronize()
            for k in range(K):
                assert torch.equal(outs[k].cpu(), ref[k].cpu()), (b, c, k, rep)
                assert bool((obuf[k][:, F:] == -3.0).all())
            assert st.d2h_bytes == (4 * g.n * F * K if out_on_host else 0)
            assert st.h2d_bytes >= (4 * g.n * F if x_on_host else 0)
        plan.close()
        ref_plan.close()


def test_streamed_pageable_host_memory_and_check_against_oracle(B):
    g = gi.erdos_renyi(2000, 9000, 14)
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    X = gi.normal_matrix(g.n, 32, 6)  # ordinary pageable host tensors
    plan = B.gnnpre_build_plan(g.rowptr, g.colidx, 0, 32, force_blocks=3, force_col_slabs=2,
                               operands_mem=B.GNNPRE_MEM_HOST)
    outs = [torch.empty(g.n, 32) for _ in range(2)]
    B.gnnpre_propagate(plan, X, 2, outs)
    check_all_hops(0, 0.0, rp, ci, X.numpy(), outs)
    plan.close()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("F", [68, 100, 128, 300, 516])
def test_bulk_copy_kernel_matches_register_kernel_bitwise(B, op, F):
    """The mean operator's rows of 68..124 columns are staged through shared memory by the copy engine on large graphs, here
    asked for; wider ones are cut into equal tiles (300 = three of 100, 516 = five of at most 104).  The summation order is
    the register kernel's (plain sums over steps of 8 edges), so the two agree bit for bit and both agree with the oracle.
    The other operators and 128 columns take the register kernel either way."""
    g = gi.rmat(30000, 400000, 17, directed_candidates=True)
    drp, dci = dev(g)
    X = gi.normal_matrix(g.n, F, 9, device="cuda")
    for b, seg in ((1, 256), (3, 64), (2, 1000)):  # same segment length for both: same summation order
        res = []
        for flags in (B.GNNPRE_FLAG_BULK_COPY, B.GNNPRE_FLAG_NO_BULK_COPY):
            plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, force_blocks=b, segment_edges=seg, flags=flags)
            outs, st = B.gnnpre_propagate(plan, X, 2, want_stats=True)
            res.append(outs)
            plan.close()
        for k in range(2):
            assert torch.equal(res[0][k], res[1][k]), (b, seg, k)
        if F > 128:
            check_all_hops(op, EPS, g.rowptr.numpy(), g.colidx.numpy(), to_np(X), res[1])
            check_all_hops(op, EPS, g.rowptr.numpy(), g.colidx.numpy(), to_np(X), res[0])
    check_all_hops(op, EPS, g.rowptr.numpy(), g.colidx.numpy(), to_np(X), res[0])


@pytest.mark.parametrize("op,F", [(1, 92), (1, 100), (1, 124), (1, 200)])
def test_bulk_copy_kernel_on_a_dense_graph_far_larger_than_the_cache(B, op, F):
    """The copy engine takes over when X is more than four times the L2 and rows are long; same segments, same order of
    additions, so the register kernel must give the same bits."""
    g = gi.rmat(1500000, 25000000, 29, directed_candidates=False, device="cuda")
    X = gi.normal_matrix(g.n, F, 9, device="cuda")
    res = []
    for flags in (0, B.GNNPRE_FLAG_NO_BULK_COPY):
        plan = B.gnnpre_build_plan(g.rowptr, g.colidx, op, F, gin_eps=EPS, force_blocks=2, segment_edges=1000, flags=flags)
        res.append(B.gnnpre_propagate(plan, X, 1)[0][0])
        torch.cuda.synchronize()
        plan.close()
    assert torch.equal(res[0], res[1])


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("graph", ["hubs", "no hubs", "one row"])
@pytest.mark.parametrize("F,seg", [(128, 32), (200, 200)])
def test_segments_in_the_order_of_their_sources_give_the_same_bits(B, op, graph, F, seg):
    """A whole hop over a matrix beyond the L2 takes its segments in the order of their columns, hops launched block by block in
    that of the edge list: segments of one row, of several, empty ones, those of one row only (the star's centre)."""
    n = 300000
    g = {"hubs": lambda: gi.rmat(n, 900000, 41, directed_candidates=False, device="cuda"), "no hubs": lambda: gi.erdos_renyi(n, 700000, 42, device="cuda"),
         "one row": lambda: gi.from_edge_list(n, [(n - 1000, 700 * j) for j in range(1, 401)], device="cuda")}[graph]()
    X = gi.normal_matrix(n, F, 43, device="cuda")
    kw = dict(gin_eps=EPS, segment_edges=seg, force_blocks=1, force_col_slabs=1)
    a = B.gnnpre_build_plan(g.rowptr, g.colidx, op, F, **kw)
    b = B.gnnpre_build_plan(g.rowptr, g.colidx, op, F, flags=B.GNNPRE_FLAG_LAUNCH_PER_BLOCK, **kw)
    assert a.info()["num_segments"] == b.info()["num_segments"]
    ascending = [bool((first[1:] >= first[:-1]).all()) for first in map(B.gnnpre_plan_hop_order, (a, b))]
    # (self-loops: hardly any segment lies in one row; segments of 200: no row is cut, and the centre's is the last one)
    assert ascending == [graph == "no hubs" or (graph == "one row" and (op != 1 or seg == 200)), True]
    for x, y in zip(B.gnnpre_propagate(a, X, 2)[0], B.gnnpre_propagate(b, X, 2)[0]):
        assert torch.equal(x, y)
    a.close()
    b.close()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("seg", [32, 200])
@pytest.mark.parametrize("graph", ["hubs", "no hubs", "numbered"])
def test_segments_of_several_rows_stay_in_the_order_of_the_edge_list(B, op, graph, seg):
    """Over a matrix beyond the L2 a hop takes the segments inside one row first, by their middle columns, and the others as the
    edge list has them; all of them so where hardly any lies in one row (no hubs) or those that do read rows numbered like
    their own (hubs of their neighbours): a caller's numbering keeps its locality."""
    n, F = 300000, 128
    g = {"hubs": lambda: gi.rmat(n, 3000000, 41, directed_candidates=False, device="cuda"), "no hubs": lambda: gi.erdos_renyi(n, 700000, 42, device="cuda"),
         "numbered": lambda: gi.from_edge_list(n, [(i - i % 1000, i) for i in range(n) if i % 1000], device="cuda")}[graph]()
    plan = B.gnnpre_build_plan(g.rowptr, g.colidx, op, F, gin_eps=EPS, segment_edges=seg, force_blocks=1, force_col_slabs=1)
    order = B.gnnpre_plan_hop_order(plan).numpy()
    rp, ci = (t.numpy() for t in B.gnnpre_plan_support(plan))
    plan.close()
    lo = np.sort(order)
    if graph != "hubs":
        assert np.array_equal(order, lo)
        return
    hi = np.append(lo[1:], len(ci))
    row_of = lambda e: np.searchsorted(rp, e, side="right") - 1
    one_row = (hi > lo) & (hi < len(ci)) & (row_of(lo) == row_of(np.maximum(hi - 1, 0)))
    first = int(one_row.sum())
    assert len(lo) // 64 < first < len(lo)
    assert np.array_equal(order[first:], lo[~one_row])
    assert np.array_equal(np.sort(order[:first]), lo[one_row])
    middle = dict(zip(lo[one_row], ci[(lo + (hi - lo) // 2)[one_row]]))
    buckets = np.array([int(middle[e]) * 1024 // n for e in order[:first]])
    assert (np.diff(buckets) >= 0).all() and buckets[-1] > buckets[0]


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("F", [16, 32, 64, 128])
@pytest.mark.parametrize("m", [3000, 80000, 330000])
def test_segments_of_a_small_graph_fill_whole_waves(B, op, F, m):
    g = gi.rmat(m // 8, m, 44, directed_candidates=True)
    X = gi.normal_matrix(g.n, F, 45)
    plan = B.gnnpre_build_plan(*dev(g), op, F, gin_eps=EPS)
    info = plan.info()
    groups = torch.cuda.get_device_properties(0).multi_processor_count * 28 * 32 // max(4, F // 4)
    waves = -(-info["num_segments"] // groups)
    # the next shorter segments (of whole windows of 8 edges) would need another wave, or are below the least
    assert info["segment_edges"] == 16 or info["nnz_tilde"] > groups * waves * (info["segment_edges"] - 8)
    outs, _ = B.gnnpre_propagate(plan, X.cuda(), 2)
    check_all_hops(op, EPS, g.rowptr.numpy(), g.colidx.numpy(), X.numpy(), outs, single_hop=single_hop_of(B, plan))
    plan.close()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("b", [1, 3, 32])
@pytest.mark.parametrize("F,m", [(16, 480000), (32, 240000), (64, 120000), (64, 180000), (128, 60000)])
def test_rows_longer_than_short_segments_are_not_cut(B, op, F, m, b):
    """Uniform graphs whose segments of 16 or 24 edges fill one wave: rows of fewer than 72 edges are not cut, whichever block they
    lie in, but for those that a block's end cuts."""
    g = gi.erdos_renyi(m // 30, m // 2, 46)
    assert 3 * 16 <= int((g.rowptr[1:] - g.rowptr[:-1]).max()) < 71
    X = gi.normal_matrix(g.n, F, 45)
    plan = B.gnnpre_build_plan(*dev(g), op, F, gin_eps=EPS, force_blocks=b)
    info = plan.info()
    assert info["segment_edges"] in (16, 24) and info["num_row_fixups"] <= b - 1
    outs, _ = B.gnnpre_propagate(plan, X.cuda(), 2)
    check_all_hops(op, EPS, g.rowptr.numpy(), g.colidx.numpy(), X.numpy(), outs, single_hop=single_hop_of(B, plan))
    plan.close()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("F", [4, 16, 20, 32, 36, 64, 68, 132, 260])
@pytest.mark.parametrize("seg", [1, 7, 8, 9, 31, 33])
def test_register_kernel_tile_and_segment_edges(B, op, F, seg):
    """Widths around the lane-group and column-tile sizes, segments around the window and chunk sizes; rows of every
    length from none to several segments, with the segment's last edge ending its row or not."""
    n = 90
    edges = [(i, j) for i in range(0, n, 7) for j in range(i + 1, min(n, i + 1 + 2 * i))]
    g = gi.from_edge_list(n, edges)
    run_case(B, g, op, F, 2, b=3, seg=seg)


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("tail", [1, 15, 16, 17, 31, 40])
def test_last_row_of_a_block_is_not_cut(B, op, flags, tail):
    """Segments of 16 on a graph whose longest row has fewer than 48 entries: a segment that would start inside the last row
    moves to the block's end and is empty; one block (nothing is cut) and several (only rows that a block's end cuts)."""
    n = 60
    g = gi.from_edge_list(n, [(i, i + 1) for i in range(n - 1)] + [(n - 1, j) for j in range(tail)])
    for b in (1, 2, 3, 5):
        run_case(B, g, op, 64, 2, b=b, seg=16, flags=flags)
    drp, dci = dev(g)
    plan = B.gnnpre_build_plan(drp, dci, op, 64, gin_eps=EPS, force_blocks=1, segment_edges=16, flags=flags)
    fixups = plan.info()["num_row_fixups"]
    plan.close()
    assert fixups == 0


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("F", [16, 100, 132])
def test_rows_four_gigabytes_apart(B, op, F):
    """A narrow view of few, very long rows: at a leading dimension of 2^30 floats a row is 2^32 bytes from the next.  Same
    bits as on rows side by side, plain, with a teleport term and with the sum of hops; and the fetch-only yardstick."""
    n, ld = 4, (1 << 30) + 4
    g = gi.from_edge_list(n, [(0, 1), (1, 2), (0, 2)])
    X = gi.normal_matrix(n, F, 3, device="cuda")
    buf = torch.empty((n - 1) * ld + F, device="cuda")
    far = torch.as_strided(buf, (n, F), (ld, 1))
    far.copy_(X)
    drp, dci = dev(g)
    for alpha in (0.0, 0.2):
        plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, segment_edges=2, teleport_alpha=alpha)
        want, got = B.gnnpre_propagate(plan, X, 2)[0], B.gnnpre_propagate(plan, far, 2)[0]
        zw, zg = (B.gnnpre_propagate_weighted(plan, x, [0.5, 0.25, 2.0])[1] for x in (X, far))
        sinks = [torch.empty(plan.info()["num_segments"], device="cuda") for _ in range(2)]
        for x, sink in zip((X, far), sinks):
            B.gnnpre_gather_ceiling(plan, x, sink)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, got)) and torch.equal(zw, zg)
        if F == 100:  # one column tile and whole warps in both (what lane groups add for empty segments means nothing)
            assert torch.equal(*sinks)
        plan.close()


@pytest.mark.parametrize("op", OPS)
def test_rows_of_more_than_two_segments_are_cut_where_segments_run_in_waves(B, op):
    """Rows of 40 entries and segments of 16, 75,000 of them: far more than run at once, so a segment takes its own 16 edges
    and not a whole row's."""
    n = 30000
    g = gi.from_edge_list(n, [(i, (i + j * j) % n) for i in range(n) for j in range(1, 21)])
    run_case(B, g, op, 64, 1, seg=16)
    plan = B.gnnpre_build_plan(*dev(g), op, 64, gin_eps=EPS, segment_edges=16)
    fixups = plan.info()["num_row_fixups"]
    plan.close()
    assert fixups > n // 2


@pytest.mark.parametrize("F", [68, 72, 100, 124, 200])
@pytest.mark.parametrize("seg", [1, 7, 16, 17, 300])
@pytest.mark.parametrize("isolated", [False, True])
def test_bulk_copy_kernel_at_segment_edges(B, F, seg, isolated):
    """The bulk-copy kernel on short, cut and empty segments: segments around its chunks of 16 edges, rows of every length
    from none to several segments, rows that end with their segment or not; plain, with a teleport term, one launch per block,
    and hops with a sum.  The register kernel's bits throughout, and the oracle's hops."""
    n = 300 if isolated else 90
    edges = [(i, j) for i in range(0, 90, 7) for j in range(i + 1, min(90, i + 1 + 2 * i))] + [(i, i + 1) for i in range(89)]
    g = gi.from_edge_list(n, edges)
    drp, dci = dev(g)
    X = gi.normal_matrix(n, F, 9, device="cuda")
    for alpha in (0.0, 0.15):
        for extra in (0, B.GNNPRE_FLAG_LAUNCH_PER_BLOCK):
            res = []
            for flags in (B.GNNPRE_FLAG_BULK_COPY, B.GNNPRE_FLAG_NO_BULK_COPY):
                plan = B.gnnpre_build_plan(drp, dci, 1, F, force_blocks=3, segment_edges=seg, flags=flags | extra, teleport_alpha=alpha)
                hops = B.gnnpre_propagate(plan, X, 2)[0]
                whops, Z = B.gnnpre_propagate_weighted(plan, X, [0.5, 0.25, -2.0])
                torch.cuda.synchronize()
                res.append([*hops, *whops, Z])
                plan.close()
            assert all(torch.equal(a, b) for a, b in zip(*res)), (alpha, extra)
            assert torch.equal(res[0][0], res[0][2]) and torch.equal(res[0][1], res[0][3])
        if alpha == 0.0:
            check_all_hops(1, EPS, g.rowptr.numpy(), g.colidx.numpy(), to_np(X), res[0][:2])


def test_two_tile_rows_on_a_graph_larger_than_the_cache(B):
    """Rows of 132..256 columns are cut into two equal tiles, each a launch of its own, once a 128-column tile of X no
    longer fits the L2 (here 400,000 nodes: 205 MB per tile; F = 200 gives two tiles of 100 columns, F = 252 two of
    128 and 124).  Checked against the oracle, and against one launch over both tiles."""
    g = gi.rmat(400000, 3000000, 23, directed_candidates=True)
    drp, dci = dev(g)
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    for op, F in ((1, 200), (0, 252)):
        X = gi.normal_matrix(g.n, F, 12, device="cuda")
        res = []
        for flags in (0, B.GNNPRE_FLAG_NO_BULK_COPY):
            plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, flags=flags)
            outs, st = B.gnnpre_propagate(plan, X, 2, want_stats=True)
            torch.cuda.synchronize()
            res.append((outs, st.kernel_launches, plan.info()["segment_edges"]))
            plan.close()
        assert res[0][2] >= 256 and res[0][1] > res[1][1]  # long segments, two segment launches per hop
        check_all_hops(op, EPS, rp, ci, to_np(X), res[0][0])
        for k in range(2):
            assert hop_error(to_np(res[0][0][k]), to_np(res[1][0][k]).astype(np.float64)) <= TOL


# ------------------------------------------------------------------ the normalised adjacency itself

@pytest.mark.parametrize("op", OPS)
def test_normalized_adjacency_values_bit_exact(B, op):
    """gnnpre_normalize against the oracle: fp64 evaluation from integer degrees, one rounding to fp32, so
    the comparison is bitwise; resident and block-streamed (host CSR, host output) runs give the same array."""
    for name, g in list(small_graphs()) + [("c1", gi.make_graph(gi.WORKLOADS["c1"]))]:
        rp, ci = g.rowptr.numpy(), g.colidx.numpy()
        want = orc.normalized_values(op, EPS, rp, ci).astype(np.float32)
        if want.size == 0:
            continue
        for b in (1, 3):
            if b > want.size:
                continue
            plan = B.gnnpre_build_plan(*dev(g), op, 16, gin_eps=EPS, force_blocks=b)
            got = B.gnnpre_normalize(plan)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(to_np(got).view(np.uint32), want.view(np.uint32), err_msg=f"{name} b={b}")
            plan.close()
            hplan = B.gnnpre_build_plan(g.rowptr.pin_memory(), g.colidx.pin_memory(), op, 16, gin_eps=EPS,
                                        force_blocks=b)
            assert hplan.info()["structure_mem"] == 1
            for host_out in (True, False):
                got = B.gnnpre_normalize(hplan, host=host_out)
                torch.cuda.synchronize()
                np.testing.assert_array_equal(to_np(got).view(np.uint32), want.view(np.uint32))
            hplan.close()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("seg", [1, 31, 33, 127, 128, 129, 300])
def test_normalized_values_at_segment_edges(B, op, seg):
    """The values kernel walks segments 128 edges at a time: segment lengths around its chunks, rows without edges,
    a hub of degree 5,000, bit for bit."""
    g = gi.from_edge_list(5200, [(0, j) for j in range(100, 5100)] + [(j, j + 3) for j in range(200, 900)])
    want = orc.normalized_values(op, EPS, g.rowptr.numpy(), g.colidx.numpy()).astype(np.float32)
    for b in (1, 4):
        plan = B.gnnpre_build_plan(*dev(g), op, 16, gin_eps=EPS, force_blocks=b, segment_edges=seg)
        got = B.gnnpre_normalize(plan)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(to_np(got).view(np.uint32), want.view(np.uint32))
        plan.close()


@pytest.mark.parametrize("op", (0, 1))
@pytest.mark.parametrize("isolated", [False, True])
def test_normalized_values_of_any_degree_the_caller_gives(B, op, isolated):
    """Bit for bit, the IEEE square root and division of every degree: 0..5000, squares and powers of two and their
    neighbours, random ones up to the largest, whose conversion to single precision rounds - and what no degree is: a row
    with edges given as 0, -1 or less keeps the infinity, NaN or negative value the formula gives."""
    rng = np.random.default_rng(5)
    k = np.arange(2, 46340, 7, dtype=np.int64)
    p = 2 ** np.arange(1, 32, dtype=np.int64)
    d = np.concatenate([np.arange(5000), k * k - 2, k * k - 1, k * k, p - 2, p - 1, p, rng.integers(1 << 24, (1 << 31) - 1, 30000),
                        rng.integers(1, 1 << 24, 20000), [(1 << 31) - 1, (1 << 31) - 2, -1, -2, -7]])
    d = d[d < (1 << 31)].astype(np.int32)
    n = len(d)
    i = torch.arange(n - 1, dtype=torch.int64)
    if isolated:
        i = i[i % 5 != 0]  # 0 and a few more rows stay alone or have one neighbour
    g = gi.from_edge_list(n, torch.stack([i, (i * 7 + 3) % (n - 1) + 1], 1)[(i * 7 + 3) % (n - 1) + 1 != i].tolist())
    plan = B.gnnpre_build_plan(*dev(g), op, 16, degrees=torch.from_numpy(d).cuda())
    got = to_np(B.gnnpre_normalize(plan))
    torch.cuda.synchronize()
    plan.close()
    rp_t, ci_t = orc.support(op, g.rowptr.numpy(), g.colidx.numpy())
    row = np.repeat(np.arange(n), np.diff(rp_t))
    x = d.astype(np.float64)
    with np.errstate(all="ignore"):
        want = 1.0 / np.sqrt(x + 1.0)
        want = (want[row] * want[ci_t] if op == 0 else 1.0 / x[row]).astype(np.float32)
    np.testing.assert_array_equal(got, want)  # (equal NaN are equal)


def test_a_device_wait_that_runs_out_is_reported_and_leaves_the_plan_usable(B):
    """Failure detection without a fault: a warp polls a barrier that nothing completes, gives up after its
    limit and sets the plan's error word; the host reads GNNPRE_ERR_TIMEOUT once, and the same plan then
    propagates correctly."""
    g = gi.erdos_renyi(3000, 20000, 23)
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    plan = B.gnnpre_build_plan(*dev(g), 0, 128)
    assert B.gnnpre_selftest_wait_timeout(plan, 200) == -8
    assert B.gnnpre_status_string(-8) == "timed out"
    X = gi.normal_matrix(g.n, 128, 2, device="cuda")
    outs, st = B.gnnpre_propagate(plan, X, 2, want_stats=True)  # the error word was cleared: no stale timeout
    check_all_hops(0, 0.0, rp, ci, to_np(X), outs)
    plan.close()


# ------------------------------------------------------------------ teleport (personalised PageRank) filter

@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("alpha", [0.15, 1.0])
def test_teleport_filter_matches_oracle(B, op, alpha):
    """X_k = (1 - alpha) A^ X_{k-1} + alpha X_0 for every kernel shape, with blocks and slabs, resident and
    streamed (bitwise equal to each other), against the fp64 oracle."""
    g = gi.rmat(6000, 60000, 27, directed_candidates=True)
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    drp, dci = dev(g)
    K = 3
    for F, b, c in ((16, 1, 1), (100, 3, 1), (128, 2, 2), (256, 1, 1), (72, 4, 3)):
        X = gi.normal_matrix(g.n, F, 7, device="cuda")
        want = orc.propagate_teleport(op, EPS, alpha, rp, ci, to_np(X), K)
        plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, force_blocks=b, force_col_slabs=c, segment_edges=64,
                                   teleport_alpha=alpha)
        outs, _ = B.gnnpre_propagate(plan, X, K)
        torch.cuda.synchronize()
        for k in range(K):
            assert hop_error(to_np(outs[k]), want[k]) <= TOL, (F, b, c, k)
        hplan = B.gnnpre_build_plan(g.rowptr.pin_memory(), g.colidx.pin_memory(), op, F, gin_eps=EPS, force_blocks=b,
                                    force_col_slabs=c, segment_edges=64, teleport_alpha=alpha,
                                    operands_mem=B.GNNPRE_MEM_HOST)
        houts = [torch.empty(g.n, F).pin_memory() for _ in range(K)]
        B.gnnpre_propagate(hplan, X.cpu().pin_memory(), K, houts)
        for k in range(K):
            assert torch.equal(houts[k], outs[k].cpu()), (F, b, c, k)
        plan.close()
        hplan.close()
    with pytest.raises(B.GnnpreError):
        B.gnnpre_build_plan(drp, dci, op, 16, teleport_alpha=1.5)


@pytest.mark.parametrize("F", [72, 100, 200])
def test_weighted_hop_sum_on_a_graph_of_the_copy_engine(B, F):
    """Where the plain hops of the mean operator go through the bulk-copy kernel: the hops, with and without a sum, have the
    register kernel's bits, and Z is their sum (the bound of test_weighted_hop_sum_adds_every_hop_once)."""
    g = gi.rmat(2000000, 33000000, 29, directed_candidates=False, device="cuda")
    X = gi.normal_matrix(g.n, F, 9, device="cuda")
    gamma = [0.3, -0.7, 1.1, 0.4]
    for alpha in (0.0, 0.15):
        res = []
        for flags in (0, B.GNNPRE_FLAG_NO_BULK_COPY):
            plan = B.gnnpre_build_plan(g.rowptr, g.colidx, 1, F, teleport_alpha=alpha, segment_edges=700, flags=flags)
            res.append((B.gnnpre_propagate_weighted(plan, X, gamma), B.gnnpre_propagate(plan, X, 3)[0]))
            torch.cuda.synchronize()
            plan.close()
        (hops, Z), plain = res[0]
        for a, b, c, d in zip(hops, plain, res[1][0][0], res[1][1]):
            assert torch.equal(a, b) and torch.equal(a, c) and torch.equal(a, d)
        assert torch.equal(Z, res[1][0][1])
        terms = [(gk, m) for gk, m in zip(np.float32(gamma).astype(np.float64).tolist(), [X, *hops])]
        for r0 in range(0, g.n, 250000):
            want = sum(gk * m[r0:r0 + 250000].double() for gk, m in terms)
            size = sum(abs(gk) * m[r0:r0 + 250000].abs().double() for gk, m in terms)
            assert bool(((Z[r0:r0 + 250000].double() - want).abs() <= len(gamma) * 2.0**-24 * size).all())


@pytest.mark.parametrize("alpha", [0.0, 0.15])
@pytest.mark.parametrize("F", [4, 16, 20, 32, 36, 64, 68, 132])
def test_weighted_hop_sum_adds_every_hop_once(B, F, alpha):
    """Z takes its hops two at a time, so odd and even K, K = 1 and 2, on segments that cut rows, rows that span chunks
    and rows without edges.  Against the fp64 sum of the hops the same call returned: each of the K + 1 fused
    multiply-adds rounds once, by at most 2^-24 of a partial sum, itself at most sum_k |gamma_k X_k|."""
    n = 90
    g = gi.from_edge_list(n, [(i, j) for i in range(0, n, 7) for j in range(i + 1, min(n, i + 1 + 2 * i))])
    drp, dci = dev(g)
    X = gi.normal_matrix(n, F, 31, device="cuda")
    for op in OPS:
        for seg in (7, 33, 300):
            for K in (1, 2, 3, 4, 5):
                gamma = [0.3, -0.7, 1.1, 0.4, -0.2, 0.9][: K + 1]
                plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, segment_edges=seg, teleport_alpha=alpha)
                hops, Z = B.gnnpre_propagate_weighted(plan, X, gamma)
                torch.cuda.synchronize()
                plan.close()
                terms = [gk * m.double() for gk, m in zip(np.float32(gamma).astype(np.float64).tolist(), [X, *hops])]
                bound = (K + 1) * 2.0**-24 * sum(t.abs() for t in terms)
                assert bool(((Z.double() - sum(terms)).abs() <= bound).all()), (op, seg, K)


@pytest.mark.parametrize("alpha", [0.0, 0.15])
@pytest.mark.parametrize("F", [16, 32, 64, 128])
def test_weighted_hop_sum_behind_cut_rows_takes_its_own_operands(B, F, alpha):
    """What the sum of hops adds to a row is fetched ahead, into one place per lane; a segment that begins inside a row has a
    sum without such operands first.  Row 0, the row such a sum would name, is huge and has no neighbours: a trace of it in
    any other row is far outside the bound (as in test_weighted_hop_sum_adds_every_hop_once)."""
    n = 4000
    g = gi.from_edge_list(n, [(i, 1 + (i * 7 + j * j) % (n - 1)) for i in range(1, n, 5) for j in range(i % 40)
                              if i != 1 + (i * 7 + j * j) % (n - 1)] + [(2, 1000 + j) for j in range(900)])
    X = gi.normal_matrix(n, F, 32, device="cuda")
    X[0] = 1e30
    drp, dci = dev(g)
    for op in OPS:
        for seg in (5, 16, 40):
            gamma = [0.3, -0.7, 1.1, 0.4]
            plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, segment_edges=seg, teleport_alpha=alpha)
            assert plan.info()["num_row_fixups"] > 0
            hops, Z = B.gnnpre_propagate_weighted(plan, X, gamma)
            torch.cuda.synchronize()
            plan.close()
            terms = [gk * m.double() for gk, m in zip(np.float32(gamma).astype(np.float64).tolist(), [X, *hops])]
            bound = len(gamma) * 2.0**-24 * sum(t.abs() for t in terms)
            assert bool(((Z.double() - sum(terms)).abs() <= bound).all()), (op, seg)
            assert bool((hops[-1][1:].abs() < 1e20).all())


@pytest.mark.parametrize("op,n,F", [(0, 140000, 64), (2, 140000, 64), (1, 70000, 128), (1, 90000, 100), (0, 90000, 100), (2, 70000, 128), (0, 50000, 200)])
@pytest.mark.parametrize("rows", ["uneven", "even"])
def test_epilogues_whose_rows_are_fetched_ahead_give_the_bits_of_narrow_ones(B, op, n, F, rows):
    """Matrices that together exceed the L2: wide tiles ask for X_0, Z and X_{k-1} ahead, tiles of 32 columns do not; the mean
    operator's on a graph that has rows without edges, where a row is not its rank.  Where rows are long and even only some do."""
    L2 = torch.cuda.get_device_properties(0).L2_cache_size
    assert n * F * 16 > L2 > n * 32 * 16 and n * min(F, 128) * 4 <= L2 * 4 // 5  # asked for ahead; not at 32 columns; X itself fits
    g = (gi.rmat(n, 1300000, 51, directed_candidates=True, device="cuda") if rows == "uneven" else  # (so many segments that their cuts do not
         gi.erdos_renyi(n, 10 * n, 52, device="cuda"))                                              # depend on the width; here: no cut rows)
    deg = g.rowptr[1:] - g.rowptr[:-1]
    assert (int(deg.min()) == 0 and int(deg.max()) * n > 4 * g.nnz) if rows == "uneven" else (g.nnz > 9 * n and int(deg.max()) * n < 3 * g.nnz)
    X = gi.normal_matrix(n, F, 52, device="cuda")
    gamma, kw = [0.3, -0.5, 0.25, 0.125], dict(gin_eps=EPS, segment_edges=64, force_blocks=1, force_col_slabs=1, teleport_alpha=0.2)
    wide = B.gnnpre_build_plan(g.rowptr, g.colidx, op, F, **kw)
    hops, Z = B.gnnpre_propagate_weighted(wide, X, gamma)
    plain = B.gnnpre_propagate(wide, X, 2)[0]
    assert torch.equal(plain[1], hops[1])
    for lo in range(0, F, 32):
        cols = slice(lo, min(lo + 32, F))
        narrow = B.gnnpre_build_plan(g.rowptr, g.colidx, op, cols.stop - lo, **kw)
        want, want_Z = B.gnnpre_propagate_weighted(narrow, X[:, cols], gamma)
        assert torch.equal(Z[:, cols], want_Z)
        for x, y in zip(hops, want):
            assert torch.equal(x[:, cols], y)
        narrow.close()
    wide.close()


@pytest.mark.parametrize("op", OPS)
def test_weighted_hop_sum_matches_oracle(B, op):
    """Z = gamma_0 X_0 + sum_k gamma_k X_k accumulated in the kernels' epilogues: every kernel shape, blocks and
    slabs, a strided Z with untouched padding, hops kept or rotated through two buffers; then on top of the
    teleport recurrence.  The hops themselves must equal those of gnnpre_propagate bit for bit."""
    g = gi.rmat(6000, 60000, 33, directed_candidates=True)  # has isolated nodes: SAGE's empty rows are covered
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    drp, dci = dev(g)
    gamma = [0.4, -1.5, 0.75, 2.0, -0.6]
    K = len(gamma) - 1
    for F, b, c in ((16, 1, 1), (100, 3, 1), (128, 2, 2), (256, 1, 1), (72, 4, 3), (600, 2, 1)):
        X = gi.normal_matrix(g.n, F, 9, device="cuda")
        want = orc.weighted_hop_sum(op, EPS, rp, ci, to_np(X), gamma)
        plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, force_blocks=b, force_col_slabs=c, segment_edges=64)
        ref, _ = B.gnnpre_propagate(plan, X, K)
        zbuf = torch.full((g.n, F + 4), -3.0, device="cuda")
        hops, Z = B.gnnpre_propagate_weighted(plan, X, gamma, Z=zbuf[:, :F])
        torch.cuda.synchronize()
        assert hop_error(to_np(Z), want) <= TOL, (F, b, c)
        assert bool((zbuf[:, F:] == -3.0).all())
        for k in range(K):
            assert torch.equal(hops[k], ref[k]), (F, b, c, k)
        last2, Z2 = B.gnnpre_propagate_weighted(plan, X, gamma, keep_hops=False)
        torch.cuda.synchronize()
        assert torch.equal(Z2, Z) and torch.equal(last2[K - 1], ref[K - 1])
        plan.close()
    # with a teleport term the summed hops are those of the recurrence
    F, alpha = 100, 0.2
    X = gi.normal_matrix(g.n, F, 10, device="cuda")
    tele = orc.propagate_teleport(op, EPS, alpha, rp, ci, to_np(X), K)
    want = gamma[0] * to_np(X).astype(np.float64) + sum(gamma[k + 1] * tele[k] for k in range(K))
    plan = B.gnnpre_build_plan(drp, dci, op, F, gin_eps=EPS, force_blocks=2, teleport_alpha=alpha)
    _, Z = B.gnnpre_propagate_weighted(plan, X, gamma)
    torch.cuda.synchronize()
    assert hop_error(to_np(Z), want) <= TOL
    # refusals: Z aliasing an input or a hop, a hop written over the one it reads, a plan with host structure
    with pytest.raises(B.GnnpreError):
        B.gnnpre_propagate_weighted(plan, X, gamma, Z=X)
    o = [torch.empty_like(X) for _ in range(2)]
    with pytest.raises(B.GnnpreError):
        B.gnnpre_propagate_weighted(plan, X, gamma, out=[o[0], o[0], o[1], o[0]])
    plan.close()
    hplan = B.gnnpre_build_plan(g.rowptr.pin_memory(), g.colidx.pin_memory(), op, F, operands_mem=B.GNNPRE_MEM_HOST,
                                force_blocks=2)
    if hplan.info()["structure_mem"] == B.GNNPRE_MEM_HOST:
        with pytest.raises(B.GnnpreError):
            B.gnnpre_propagate_weighted(hplan, X, gamma)
    hplan.close()


@pytest.mark.parametrize("world", [2, 3, 8])
def test_column_shards_assemble_to_the_full_result(B, world):
    """Column sharding over `world` ranks, run here one rank after another on the one GPU (the ranks are
    independent: nothing waits on anything): every rank's slab against the oracle's columns, slabs side by side
    cover every column once."""
    from paper_2207_12000_b200.shard import propagate_column_shard
    g = gi.rmat(8000, 90000, 35, directed_candidates=True)
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    drp, dci = dev(g)
    F, K, op = 100, 3, 0
    X = gi.normal_matrix(g.n, F, 3, device="cuda")
    want = orc.propagate(op, 0.0, rp, ci, to_np(X), K)
    covered = np.zeros(F, dtype=np.int32)
    for rank in range(world):
        lo, outs = propagate_column_shard(B, drp, dci, op, X, K, world, rank)
        torch.cuda.synchronize()
        if not outs:
            continue
        width = outs[0].shape[1]
        covered[lo:lo + width] += 1
        for k in range(K):
            assert hop_error(to_np(outs[k]), want[k][:, lo:lo + width]) <= TOL, (rank, k)
    assert (covered == 1).all()


def test_propagate_and_first_layer_inside_a_cuda_graph(B):
    """The device-resident calls only enqueue work, so a CUDA graph can capture them: K hops of configuration 1 and
    the first dense stage over them, replayed twice on fresh outputs, equal the direct calls bit for bit."""
    w = gi.WORKLOADS["c1"]
    g = gi.make_graph(w, device="cuda")
    X = gi.make_features(w, device="cuda")
    plan = B.gnnpre_build_plan(g.rowptr, g.colidx, w.op, w.feat_dim)
    ref, _ = B.gnnpre_propagate(plan, X, w.hops)
    Wt = gi.normal_matrix(64, w.feat_dim, 3, device="cuda")
    batch = torch.arange(0, g.n, 3, dtype=torch.int32, device="cuda")
    ref_y = B.gnnpre_lc_first_layer(ref, batch, Wt, relu_mask=1)
    outs = [torch.zeros_like(X) for _ in range(w.hops)]
    y = torch.zeros_like(ref_y)
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):  # one call outside the capture: one-time set-up of the kernels
        B.gnnpre_propagate(plan, X, w.hops, outs)
        B.gnnpre_lc_first_layer(outs, batch, Wt, relu_mask=1, out=y, check=False)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        B.gnnpre_propagate(plan, X, w.hops, outs)
        B.gnnpre_lc_first_layer(outs, batch, Wt, relu_mask=1, out=y, check=False)
    for _ in range(2):
        for o in outs:
            o.zero_()
        y.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(o, r) for o, r in zip(outs, ref)) and torch.equal(y, ref_y)
    assert int(flag.item()) == 0
    plan.close()


def test_resuming_from_a_finished_hop_gives_the_same_bits(B):
    """Checkpoint/resume: hops 1..2, then hop 3 started from hop 2's output, equal the uninterrupted run."""
    g = gi.rmat(20000, 200000, 29, directed_candidates=True)
    plan = B.gnnpre_build_plan(*dev(g), 1, 100, force_blocks=3)
    X = gi.normal_matrix(g.n, 100, 4, device="cuda")
    full, _ = B.gnnpre_propagate(plan, X, 3)
    first, _ = B.gnnpre_propagate(plan, X, 2)
    rest, _ = B.gnnpre_propagate(plan, first[1], 1)
    torch.cuda.synchronize()
    assert torch.equal(first[0], full[0]) and torch.equal(first[1], full[1]) and torch.equal(rest[0], full[2])
    plan.close()


@pytest.mark.parametrize("op", OPS)
def test_streamed_slabs_through_the_bulk_copy_kernel(B, op):
    """Column slabs of 100 columns (F = 200, c = 2) and tiles of 80 and 128 columns (F = 160, 640): the tensor map of the
    bulk-copy kernel (asked for; the mean operator has it) starts at a column offset, in dense slab buffers and in the
    caller's strided matrix."""
    g = gi.rmat(12000, 150000, 31, directed_candidates=True)
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    for F, c in ((200, 2), (160, 1), (640, 1)):
        X = gi.normal_matrix(g.n, F, 8, device="cuda")
        plan = B.gnnpre_build_plan(*dev(g), op, F, gin_eps=EPS, force_blocks=3, force_col_slabs=c,
                                   operands_mem=B.GNNPRE_MEM_HOST, flags=B.GNNPRE_FLAG_BULK_COPY)
        houts = [torch.empty(g.n, F).pin_memory() for _ in range(2)]
        B.gnnpre_propagate(plan, X.cpu().pin_memory(), 2, houts)
        check_all_hops(op, EPS, rp, ci, to_np(X), houts)
        plan.close()


def test_feature_width_that_is_not_a_multiple_of_four(B):
    """F = 602 (Reddit's width in the paper's dataset table): the matrices carry a leading dimension of 604; the
    two pad columns may hold anything (NaN here) without touching the 602 real ones."""
    g = gi.erdos_renyi(3000, 30000, 33)
    rp, ci = g.rowptr.numpy(), g.colidx.numpy()
    F, ld = 602, 604
    Xbuf = torch.full((g.n, ld), float("nan"), device="cuda")
    Xbuf[:, :F] = gi.normal_matrix(g.n, F, 3, device="cuda")
    obuf = [torch.zeros((g.n, ld), device="cuda") for _ in range(2)]
    plan = B.gnnpre_build_plan(*dev(g), 0, F, force_blocks=2)
    assert plan.info()["feat_dim"] == 604
    B.gnnpre_propagate(plan, Xbuf[:, :F], 2, [o[:, :F] for o in obuf])
    torch.cuda.synchronize()
    check_all_hops(0, 0.0, rp, ci, to_np(Xbuf[:, :F]).copy(), [o[:, :F] for o in obuf])
    with pytest.raises(B.GnnpreError):  # no room for the pad columns
        B.gnnpre_propagate(plan, torch.zeros((g.n, F), device="cuda")[:, :F], 1)
    plan.close()
