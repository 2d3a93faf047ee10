// gnnpre_normalize: the normalised adjacency itself, edge block by edge block (Eq. 1 written block-wise
// as Eq. 10: S = sum_l D~^{-1/2} A~^(l) D~^{-1/2}).  The propagation path never needs these values (it
// applies the per-node scales on the fly); this export serves callers that want S as a matrix.
// Every value is evaluated in fp64 from the integer degrees and rounded once to fp32.
#include <algorithm>
#include <vector>

#include "gnnpre_internal.cuh"

namespace gnnpre {

namespace {

struct ValArgs {
    const Segment* segs;
    int64_t seg_lo, seg_hi;    // segments of this edge range
    const uint32_t* colx;      // entry of edge e at colx[e - colx_base]
    int64_t colx_base;
    const int32_t* deg;
    const float* rank_scale;   // scales of the rows that own an edge, in rank order
    const int32_t* nzrows;     // those rows (nullptr: every row owns one)
    float* out;                // value of edge e goes to out[e - out_base]
    int64_t out_base;
    float diag_weight;         // GIN: 1 + eps, rounded once
};

// 1.0 / sqrt(d + 1.0), both operations rounded to nearest as IEEE 754 does: a single-precision estimate of the
// reciprocal root, one third-order step in fp64, then the square root and its reciprocal corrected by their exact
// residuals (P. Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", IBM J. Res.
// Dev. 34, 1990).  Eleven fp64 operations instead of a general square root and a general division, the same bits (compared
// once for every d in [0, 2^31 - 2]; the tests hold squares, powers of two and random degrees up to 2^31 - 1); NaN below 0.
__device__ __forceinline__ double inverse_sqrt_degree(int32_t d) {
    const double x = (double)d + 1.0;
    const double y0 = (double)rsqrtf((float)x);
    const double e = fma(-(x * y0), y0, 1.0);
    const double y = fma(y0 * e, fma(0.375, e, 0.5), y0);
    const double s0 = x * y;
    const double s = fma(fma(-s0, s0, x), 0.5 * y, s0);
    return fma(fma(-s, y, 1.0), y, y);
}

// What the formula gives for degrees that a caller got wrong: 1 / sqrt(0) is infinite (-1), the root of less NaN.
__device__ float value_of_no_degree(int32_t di, int32_t dj) {
    return (float)((1.0 / sqrt((double)di + 1.0)) * (1.0 / sqrt((double)dj + 1.0)));
}

// One warp per segment of the edge list, 32 edges at a time, kValChunks chunks of loads in flight: entries are read and
// values written in whole lines whatever the rows' lengths, and the row of an edge follows from the row-end marks.
// Bound by the gather of one degree per edge (a 32-byte sector each) from the L2.  54 M edges, GCN: 2307 us with one
// warp per row (mean degree 15) and a general square root and division per edge, 235 us now.
// GIVEN: the degrees are the caller's, so any integer; looking for what no degree is costs 2 %.
constexpr int kValChunks = 4;

template <int OP, bool GIVEN>
__global__ void __launch_bounds__(256) k_edge_values(const ValArgs a) {
    const int64_t sg = a.seg_lo + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (sg >= a.seg_hi) return;
    const int lane = threadIdx.x & 31;
    const int64_t start = a.segs[sg].start;
    const int len = a.segs[sg].len;
    const uint32_t* entries = a.colx + (start - a.colx_base);
    float* out = a.out + (start - a.out_base);
    int rank = a.segs[sg].rank;
    for (int e0 = 0; e0 < len; e0 += 32 * kValChunks) {
        uint32_t c[kValChunks];
        int row[kValChunks];
#pragma unroll
        for (int k = 0; k < kValChunks; ++k) {
            const int e = e0 + 32 * k + lane;
            c[k] = e < len ? __ldg(entries + e) : 0u;
        }
#pragma unroll
        for (int k = 0; k < kValChunks; ++k) {
            const unsigned ends = __ballot_sync(0xffffffffu, (c[k] & kRowEndBit) != 0);
            row[k] = rank + __popc(ends & ((1u << lane) - 1u));
            rank += __popc(ends);
        }
#pragma unroll
        for (int k = 0; k < kValChunks; ++k) {
            const int e = e0 + 32 * k + lane;
            if (e >= len) continue;
            const int32_t col = (int32_t)(c[k] & ~kRowEndBit);
            float v;
            if (OP == GNNPRE_OP_GCN_SYM) {
                const int32_t di = __ldg(a.deg + row[k]), dj = __ldg(a.deg + col);
                v = (float)(inverse_sqrt_degree(di) * inverse_sqrt_degree(dj));
                if (GIVEN && v != v) v = value_of_no_degree(di, dj);
            } else if (OP == GNNPRE_OP_SAGE_MEAN) {
                v = __ldg(a.rank_scale + row[k]);  // 1 / D_i in fp64, rounded once; 0 stands for a caller's degree below 1
                if (GIVEN && v == 0.f) v = (float)(1.0 / (double)a.deg[a.nzrows ? a.nzrows[row[k]] : row[k]]);
            } else {
                v = col == row[k] ? a.diag_weight : 1.f;  // every row owns its self-loop: rank == row
            }
            out[e] = v;
        }
    }
}

int launch_values(const gnnpre_plan* P, const ValArgs& a, cudaStream_t st) {
    if (a.seg_hi <= a.seg_lo) return GNNPRE_OK;
    const unsigned grid = (unsigned)(((a.seg_hi - a.seg_lo) * 32 + 255) / 256);
    const bool given = P->degrees_given;
    if (P->op == GNNPRE_OP_GIN_SUM) k_edge_values<GNNPRE_OP_GIN_SUM, false><<<grid, 256, 0, st>>>(a);
    else if (P->op == GNNPRE_OP_GCN_SYM && !given) k_edge_values<GNNPRE_OP_GCN_SYM, false><<<grid, 256, 0, st>>>(a);
    else if (P->op == GNNPRE_OP_GCN_SYM) k_edge_values<GNNPRE_OP_GCN_SYM, true><<<grid, 256, 0, st>>>(a);
    else if (!given) k_edge_values<GNNPRE_OP_SAGE_MEAN, false><<<grid, 256, 0, st>>>(a);
    else k_edge_values<GNNPRE_OP_SAGE_MEAN, true><<<grid, 256, 0, st>>>(a);
    GNNPRE_CUDA(cudaGetLastError());
    return GNNPRE_OK;
}

}  // namespace

}  // namespace gnnpre

using namespace gnnpre;

extern "C" int gnnpre_normalize(gnnpre_plan_t* P, float* vals_out, int32_t vals_mem, void* stream) {
    if (!P || !vals_out) return GNNPRE_ERR_INVALID_ARG;
    if (vals_mem != GNNPRE_MEM_DEVICE && vals_mem != GNNPRE_MEM_HOST) return GNNPRE_ERR_INVALID_ARG;
    if (P->nnz_tilde == 0) return GNNPRE_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ValArgs a;
    a.segs = P->segments.p;
    a.deg = P->deg.p;
    a.rank_scale = P->rows_all_nonempty ? P->rscale.p : P->nzscale.p;
    a.nzrows = P->rows_all_nonempty ? nullptr : P->nzrows.p;
    a.diag_weight = (float)(1.0 + (double)P->gin_eps);
    const bool e_host = P->structure_mem == GNNPRE_MEM_HOST;
    if (!e_host && vals_mem == GNNPRE_MEM_DEVICE) {  // everything resident: all blocks in one launch
        a.seg_lo = 0;
        a.seg_hi = P->num_segments;
        a.colx = P->colx.p;
        a.colx_base = 0;
        a.out = vals_out;
        a.out_base = 0;
        return launch_values(P, a, st);
    }
    // Block by block (the paper's a passes): E^(l) goes up on the plan's upload stream if it lives on the
    // host, the kernel runs on its compute stream, the values of block l go down on its download stream if
    // the caller wants them on the host.  Two buffers of each kind take turns and events order the three
    // streams, so block l+1 uploads and block l-1 downloads while block l computes.
    if (__sync_lock_test_and_set(&P->busy, 1)) return GNNPRE_ERR_BUSY;
    int64_t longest = 0;
    for (const Block& B : P->blocks) longest = std::max(longest, B.e_hi - B.e_lo);
    DevBuf<float> stage[2];
    std::vector<cudaEvent_t> events;
    auto record = [&](cudaStream_t s, cudaEvent_t* out) -> int {
        cudaEvent_t e = nullptr;
        GNNPRE_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        events.push_back(e);
        GNNPRE_CUDA(cudaEventRecord(e, s));
        *out = e;
        return GNNPRE_OK;
    };
    auto wait = [&](cudaStream_t s, cudaEvent_t e) -> int {
        if (e) GNNPRE_CUDA(cudaStreamWaitEvent(s, e, 0));
        return GNNPRE_OK;
    };
    auto body = [&]() -> int {
        GNNPRE_TRY(ensure_streams(P));
        if (vals_mem == GNNPRE_MEM_HOST) {
            GNNPRE_TRY(stage[0].alloc((size_t)longest));
            if (P->blocks.size() > 1) GNNPRE_TRY(stage[1].alloc((size_t)longest));
        }
        cudaEvent_t start = nullptr;
        GNNPRE_TRY(record(st, &start));
        GNNPRE_TRY(wait(P->s_h2d, start));
        GNNPRE_TRY(wait(P->s_compute, start));
        GNNPRE_TRY(wait(P->s_d2h, start));
        cudaEvent_t kernel_done[2] = {nullptr, nullptr};  // last kernel that read edge buffer sb / wrote value buffer sb
        cudaEvent_t drained[2] = {nullptr, nullptr};      // last download out of value buffer sb
        for (size_t j = 0; j < P->blocks.size(); ++j) {
            const Block& B = P->blocks[j];
            const int sb = (int)(j & 1);
            a.seg_lo = B.seg_lo;
            a.seg_hi = B.seg_hi;
            if (e_host) {
                if (P->stage_holds[sb] != (int64_t)j) {
                    GNNPRE_TRY(wait(P->s_h2d, kernel_done[sb]));
                    GNNPRE_CUDA(cudaMemcpyAsync(P->colx_stage[sb].p, P->colx_host.p + B.e_lo,
                                                sizeof(uint32_t) * (size_t)(B.e_hi - B.e_lo), cudaMemcpyHostToDevice,
                                                P->s_h2d));
                    P->stage_holds[sb] = (int64_t)j;
                    cudaEvent_t up = nullptr;
                    GNNPRE_TRY(record(P->s_h2d, &up));
                    GNNPRE_TRY(wait(P->s_compute, up));
                }
                a.colx = P->colx_stage[sb].p;
                a.colx_base = B.e_lo;
            } else {
                a.colx = P->colx.p;
                a.colx_base = 0;
            }
            if (vals_mem == GNNPRE_MEM_HOST) {
                GNNPRE_TRY(wait(P->s_compute, drained[sb]));
                a.out = stage[sb].p;
                a.out_base = B.e_lo;
            } else {
                a.out = vals_out;
                a.out_base = 0;
            }
            GNNPRE_TRY(launch_values(P, a, P->s_compute));
            GNNPRE_TRY(record(P->s_compute, &kernel_done[sb]));
            if (vals_mem == GNNPRE_MEM_HOST) {
                GNNPRE_TRY(wait(P->s_d2h, kernel_done[sb]));
                GNNPRE_CUDA(cudaMemcpyAsync(vals_out + B.e_lo, stage[sb].p, sizeof(float) * (size_t)(B.e_hi - B.e_lo),
                                            cudaMemcpyDeviceToHost, P->s_d2h));
                GNNPRE_TRY(record(P->s_d2h, &drained[sb]));
            }
        }
        return GNNPRE_OK;
    };
    int rc = body();
    // the staging buffers die with this call, and host results are promised on return
    for (cudaStream_t s : {P->s_h2d, P->s_compute, P->s_d2h})
        if (s && cudaStreamSynchronize(s) != cudaSuccess && rc == GNNPRE_OK) rc = GNNPRE_ERR_CUDA;
    for (cudaEvent_t e : events) cudaEventDestroy(e);
    if (rc != GNNPRE_OK) {
        (void)cudaGetLastError();
        P->stage_holds[0] = P->stage_holds[1] = -1;
    }
    __sync_lock_release(&P->busy);
    return rc;
}

// Eq. 11: least a with ceil((alpha_A B_A + alpha_S B_S) / a) + alpha_D B_D <= B_GPU (closed form).
extern "C" int gnnpre_solve_normalisation_blocks(int64_t B_A, int64_t B_S, int64_t B_D, int64_t alpha_A, int64_t alpha_S,
                                                 int64_t alpha_D, int64_t B_GPU, int64_t max_a, int64_t* a_out) {
    if (!a_out || B_A < 0 || B_S < 0 || B_D < 0 || alpha_A < 0 || alpha_S < 0 || alpha_D < 0 || max_a < 1)
        return GNNPRE_ERR_INVALID_ARG;
    const int64_t need = alpha_A * B_A + alpha_S * B_S;
    const int64_t room = B_GPU - alpha_D * B_D;
    if (room < 0 || (room == 0 && need > 0)) return GNNPRE_ERR_BUDGET_TOO_SMALL;
    const int64_t a = need == 0 ? 1 : (need + room - 1) / room;
    if (a > max_a) return GNNPRE_ERR_BUDGET_TOO_SMALL;
    *a_out = std::max<int64_t>(a, 1);
    return GNNPRE_OK;
}
