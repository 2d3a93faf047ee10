// Propagation kernels: one hop  X_out = A^ X_prev  over a range of warp-level edge segments
// (Algorithm 1's block product Z = S^(j) X^(i) and its accumulation X_tmp += Z, fused; the
// operator's normalisation of Eq. 1 / Eq. 10 is applied on the fly from per-node scales, so S is
// never materialised).
//
// Work decomposition.  The edge list E of the support is cut, inside every edge block, into short
// contiguous segments.  A group of G lanes (G = 4..32, a lane holds one float4 of a column tile) walks
// one segment edge by edge: the group reads its column indices with coalesced loads, then gathers the
// neighbours' feature rows with 128-bit loads, eight rows in flight per lane, and accumulates in fp32
// registers.  Bit 31 of a column entry marks the last edge
// of a row: there the group scales the sum by r_i and stores the output row.  Rows cut by a segment
// boundary leave their partial sums in scratch rows, which k_finish_rows adds up in a fixed order.
#include <algorithm>
#include <atomic>
#include <type_traits>
#include <utility>

#include "gnnpre_internal.cuh"

namespace gnnpre {

namespace {

#include "segments_common.cuh"
#include "segments.cuh"
#include "segments_tma.cuh"

// A wait on a barrier that nothing ever completes: the polls run out, the error word is set, the warp
// leaves.  This is the give-up path of k_segments_tma, exercised on its own.
__global__ void k_wait_that_runs_out(int* error, uint32_t polls) {
    __shared__ __align__(8) unsigned long long bar;
    const uint32_t b = smem_u32(&bar);
    if (threadIdx.x == 0) mbar_init(b, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    bool done = false;
    for (uint32_t i = 0; i < polls && !done; ++i) done = mbar_try_wait(b, 0);
    if (!done && threadIdx.x == 0) atomicExch(error, 1);
}

#include "fixups.cuh"
#include "ceiling.cuh"

template <int G, int OP, bool HAS_EMPTY, int EP, bool FAR>
int launch_segments_epilogue(const SegArgs& a, dim3 grid, cudaStream_t st) {
    if constexpr (!FAR && kFetchesAhead<G, OP, EP>) {
        // the two that gain on long rows of equal length too
        constexpr int kFrom = EP == kEpTeleport && ((G == 16 && OP == GNNPRE_OP_GCN_SYM) || (G == 32 && OP == GNNPRE_OP_GIN_SUM)) ? 1 : 2;
        if (a.tp.ahead >= kFrom) return launch_dependent(k_segments<G, OP, HAS_EMPTY, EP, FAR, true>, grid, kSegThreads, 0, a.back_to_back, st, a);
    }
    return launch_dependent(k_segments<G, OP, HAS_EMPTY, EP, FAR, false>, grid, kSegThreads, 0, a.back_to_back, st, a);
}

template <int G, bool FAR = false>
int launch_segments_shape(const gnnpre_plan* P, const SegArgs& a, cudaStream_t st) {
    const int64_t groups = a.seg_hi - a.seg_lo;
    const dim3 grid((unsigned)((groups * G + kSegThreads - 1) / kSegThreads), (unsigned)((a.f4 + a.tile_f4 - 1) / a.tile_f4));
    const int ep = epilogue_of(a.tp);
#define GNNPRE_LAUNCH_SEGMENTS(OP_, EMPTY_)                                                             \
    do {                                                                                                \
        if (ep == kEpSum) return launch_segments_epilogue<G, OP_, EMPTY_, kEpSum, FAR>(a, grid, st);       \
        if (ep == kEpTeleport) return launch_segments_epilogue<G, OP_, EMPTY_, kEpTeleport, FAR>(a, grid, st); \
        return launch_segments_epilogue<G, OP_, EMPTY_, kEpPlain, FAR>(a, grid, st);                      \
    } while (0)
    switch (P->op) {
    case GNNPRE_OP_GCN_SYM: GNNPRE_LAUNCH_SEGMENTS(GNNPRE_OP_GCN_SYM, false);
    case GNNPRE_OP_GIN_SUM: GNNPRE_LAUNCH_SEGMENTS(GNNPRE_OP_GIN_SUM, false);
    default:
        if (P->rows_all_nonempty) GNNPRE_LAUNCH_SEGMENTS(GNNPRE_OP_SAGE_MEAN, false);
        GNNPRE_LAUNCH_SEGMENTS(GNNPRE_OP_SAGE_MEAN, true);
    }
#undef GNNPRE_LAUNCH_SEGMENTS
}

// Float4 per column tile of the register kernels: equal tiles of at most 128 columns.
int32_t equal_tile_f4(int32_t f4) {
    const int32_t tiles = (f4 + 31) / 32;
    return (f4 + tiles - 1) / tiles;
}

// The register kernel on all columns of `a`, one launch.
int launch_segments_gather(const gnnpre_plan* P, SegArgs a, cudaStream_t st) {
    a.tile_f4 = equal_tile_f4(a.f4);
    if (far_rows(a.ldx)) return launch_segments_shape<32, true>(P, a, st);
    if (a.tile_f4 <= 4) return launch_segments_shape<4>(P, a, st);
    if (a.tile_f4 <= 8) return launch_segments_shape<8>(P, a, st);
    if (a.tile_f4 <= 16) return launch_segments_shape<16>(P, a, st);
    return launch_segments_shape<32>(P, a, st);
}

// Bulk-copy variant: one persistent CTA per SM, as many warps (at most kTmaMaxWarps) as fit into the
// SM's shared memory with kTmaStages stages of kTmaRows rows each.
constexpr size_t kTmaSmemBudget = 227 * 1024 - 1024;

uint32_t tma_stage_bytes(int32_t f4) { return (kTmaRows / 4) * ((4u * 16u * (uint32_t)f4 + 127u) & ~127u); }

int tma_warps(int32_t f4) {
    const size_t per_warp = (size_t)kTmaStages * tma_stage_bytes(f4);
    return (int)std::min<size_t>(kTmaMaxWarps, kTmaSmemBudget / per_warp);
}

// Tensor map of the [n, width] fp32 matrix at `x` with row stride ldx: box = one row of `width` columns,
// no swizzle, no interleave.  The driver entry point is looked up once (no link-time dependency on libcuda).
int make_row_tensor_map(const float* x, int64_t n, int32_t width, int64_t ldx, CUtensorMap* out) {
    typedef CUresult (*encode_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static std::atomic<encode_fn> cached{nullptr};  // threads may race to fill it; they all store the same pointer
    encode_fn encode = cached.load(std::memory_order_acquire);
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        GNNPRE_CUDA(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q));
        if (q != cudaDriverEntryPointSuccess || !fn) return GNNPRE_ERR_CUDA;
        encode = reinterpret_cast<encode_fn>(fn);
        cached.store(encode, std::memory_order_release);
    }
    const cuuint64_t dims[2] = {(cuuint64_t)width, (cuuint64_t)n};
    const cuuint64_t strides[1] = {(cuuint64_t)ldx * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)width, 1u};
    const cuuint32_t elem[2] = {1u, 1u};
    const CUresult r = encode(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(x), dims, strides, box, elem,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_last_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled", __FILE__, __LINE__);
        return GNNPRE_ERR_CUDA;
    }
    return GNNPRE_OK;
}

template <bool HAS_EMPTY, int F4C, int EP>
int launch_segments_tma_width(const gnnpre_plan* P, const SegArgs& a, cudaStream_t st) {
    const int nwarps = tma_warps(a.f4);
    const size_t smem = (size_t)nwarps * kTmaStages * tma_stage_bytes(a.f4);
    CUtensorMap tmap;
    GNNPRE_TRY(make_row_tensor_map(a.x, P->n, 4 * a.f4, a.ldx, &tmap));
    auto kernel = k_segments_tma<HAS_EMPTY, F4C, EP>;
    // the opt-in to large dynamic shared memory is per kernel and device: once, and again only if a launch needs more
    static std::atomic<int> smem_set[kMaxDevices];
    const int dev = P->device < kMaxDevices ? P->device : 0;
    if (P->device >= kMaxDevices || smem_set[dev].load(std::memory_order_relaxed) < (int)smem) {
        GNNPRE_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        smem_set[dev].store((int)smem, std::memory_order_relaxed);
    }
    const int64_t nseg = a.seg_hi - a.seg_lo;
    const unsigned grid = (unsigned)std::min<int64_t>(P->num_sms, (nseg + nwarps - 1) / nwarps);
    return launch_dependent(kernel, dim3(grid), (unsigned)(nwarps * 32), smem, a.back_to_back, st, a, tmap, P->dev_error.p);
}

// Rows (or column tiles) of 100 columns get kernels with the row size compiled in.
template <bool HAS_EMPTY>
int launch_segments_tma_rows(const gnnpre_plan* P, const SegArgs& a, cudaStream_t st) {
    const int ep = epilogue_of(a.tp);
    if (ep == kEpTeleport) return launch_segments_tma_width<HAS_EMPTY, 0, kEpTeleport>(P, a, st);
    if (a.f4 == 25) return launch_segments_tma_width<HAS_EMPTY, 25, kEpPlain>(P, a, st);
    return launch_segments_tma_width<HAS_EMPTY, 0, kEpPlain>(P, a, st);
}

int launch_segments_tma(const gnnpre_plan* P, const SegArgs& a, cudaStream_t st) {
    return P->rows_all_nonempty ? launch_segments_tma_rows<false>(P, a, st) : launch_segments_tma_rows<true>(P, a, st);
}

template <int G>
int launch_finish_shape(const FixArgs& a, cudaStream_t st) {
    const int64_t rows_per_cta = kThreads / 32, empty_per_cta = kThreads / G * kEmptyPerGroup;
    const int64_t ctas = (a.hub_hi - a.hub_lo) + (a.fix_hi - a.fix_lo + rows_per_cta - 1) / rows_per_cta +
                         (a.num_empty + empty_per_cta - 1) / empty_per_cta;
    const dim3 grid((unsigned)ctas, (unsigned)((a.f4 + a.tile_f4 - 1) / a.tile_f4));
    const int ep = epilogue_of(a.tp);
    if (ep == kEpSum) return launch_dependent(k_finish_rows<G, kEpSum>, grid, kThreads, 0, a.back_to_back, st, a);
    if (ep == kEpTeleport) return launch_dependent(k_finish_rows<G, kEpTeleport>, grid, kThreads, 0, a.back_to_back, st, a);
    return launch_dependent(k_finish_rows<G, kEpPlain>, grid, kThreads, 0, a.back_to_back, st, a);
}

int64_t l2_cache_bytes() {
    static std::atomic<int64_t> cached{0};
    int64_t bytes = cached.load(std::memory_order_relaxed);
    if (bytes == 0) {
        int dev = 0, got = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&got, cudaDevAttrL2CacheSize, dev) != cudaSuccess || got <= 0)
            got = 126 << 20;
        cached.store(bytes = got, std::memory_order_relaxed);
    }
    return bytes;
}

Teleport teleport_of(const gnnpre_plan* P, const HopArgs& h, int32_t f0) {
    Teleport tp;
    tp.x0 = h.x0 ? h.x0 + f0 : nullptr;
    tp.ldx0 = h.ldx0;
    tp.alpha = h.x0 ? P->teleport_alpha : 0.f;
    tp.keep = (float)(1.0 - (double)tp.alpha);
    tp.zsum = h.zsum ? h.zsum + f0 : nullptr;
    tp.ldz = h.ldz;
    tp.xprev = h.zsum_prev ? h.xprev + f0 : nullptr;
    tp.ldp = h.ldx;
    tp.gamma = h.gamma;
    tp.gamma_prev = h.gamma_prev;
    tp.gamma0 = h.gamma0;
    tp.zsum_first = h.zsum_first ? 1 : 0;
    // with X_0 and Z a hop has three to five matrices; tiles of more than 64 columns that exceed the L2 alone gain nothing
    // (600 K nodes, 128 columns: 10.3 ms without, 10.5 with; 1 M nodes, 64 columns 6.1 / 5.8)
    const bool from_memory = P->n * h.width * 16 > l2_cache_bytes() && (h.width <= 64 || !beyond_cache(P, h.width));
    tp.ahead = !from_memory ? 0 : P->short_rows ? 2 : 1;  // 1: long rows of equal length (see kFetchesAhead)
    return tp;
}

}  // namespace

namespace {

// The mean operator's column tiles of 68..124 columns go through the bulk-copy kernel when X's tile is at least four times
// the L2 and rows are long (mean degree >= 32).  Its rows in flight (213 KB per SM) then hide the DRAM latency that the
// register kernel's 90 KB do not; everywhere else its copy engine, about 33 ps per row whatever the row's width, is the
// slower path.  us per hop, bulk copy / register: 2.4 M nodes of mean degree 51, mean operator, 72 columns 3634 / 3845,
// 100 columns 4085 / 4509, 124 columns 4670 / 5150, but 128 columns, rows of whole cache lines, 4641 / 4461; degree 34,
// 100 columns 3187 / 3368.  (In the order of the edge list; in that of the sources 100 columns 3637 / 3870, in long runs three hops
// 12.7 / 13.0 ms.)  With a weight per edge the rows wait for their weights instead: GCN, degree 51, 72 / 100 / 128
// columns 4583 / 4243, 4971 / 4927, 5519 / 4792; GIN, whose few weighted edges are marked, in turn on one device 4239 / 4039,
// 4874 / 4887, 5226 / 4739.  800 K nodes of degree 63, mean, 100 columns (2.4 x L2): register; 1.7 M nodes of degree 15 as well.  What the rule gives away: rows of equal length
// and sources without hubs, X about as large as the L2 - 200,000 nodes of degree 160, 100 columns 898 / 1006, degree 96 523 / 571 -
// where an R-MAT graph of the same size and degree takes 771 / 623; the two differ in nothing that n and |E| tell.
bool tile_uses_bulk_copy(const gnnpre_plan* P, int32_t width) {
    const int32_t f4 = width / 4;
    if (P->op != GNNPRE_OP_SAGE_MEAN || (P->flags & GNNPRE_FLAG_NO_BULK_COPY) || f4 <= 16 || f4 >= 32) return false;
    return (P->flags & GNNPRE_FLAG_BULK_COPY) || (P->n * (int64_t)width * 4 > 4 * l2_cache_bytes() && P->nnz_tilde >= 32 * P->n);
}

// Columns one segment launch covers: all of them, as tiles of one launch, while a 128-column tile of X fits the L2.
// Beyond that each tile is a launch of its own, so that only one tile's rows compete for the cache at a time.
int32_t segment_tile_width(const gnnpre_plan* P, int32_t width) {
    const bool one_launch = (P->flags & GNNPRE_FLAG_NO_BULK_COPY) || P->n * 512 <= l2_cache_bytes();
    if (one_launch && !(P->flags & GNNPRE_FLAG_BULK_COPY)) return width;
    return 4 * equal_tile_f4(width / 4);
}

}  // namespace

// Whether the rows that one segment launch over a slab of this width gathers from are more than the L2 holds (from some four
// fifths of its size on it misses: see k_segment_order).
bool beyond_cache(const gnnpre_plan* P, int32_t width) {
    if (P->n * 512 <= l2_cache_bytes() * 4 / 5) return false;
    return P->n * 4 * (int64_t)std::min(width, segment_tile_width(P, width)) > l2_cache_bytes() * 4 / 5;
}

// Whether a slab of this width is (mostly) summed by the bulk-copy kernel; the plan sizes its segments for it.
bool uses_bulk_copy(const gnnpre_plan* P, int32_t width) {
    return tile_uses_bulk_copy(P, std::min(width, segment_tile_width(P, width)));
}

int launch_segments(const gnnpre_plan* P, const HopArgs& h, int64_t seg_lo, int64_t seg_hi, cudaStream_t st) {
    if (seg_hi <= seg_lo) return GNNPRE_OK;
    const int32_t tile = segment_tile_width(P, h.width);
    for (int32_t f0 = 0; f0 < h.width; f0 += tile) {
        const int32_t w = std::min<int32_t>(tile, h.width - f0);
        SegArgs a;
        a.segs = P->by_source.p && seg_hi - seg_lo == P->num_segments ? P->by_source.p : P->segments.p;
        a.seg_lo = seg_lo;
        a.seg_hi = seg_hi;
        a.colx = h.colx;
        a.colx_base = h.colx_edge_base;
        a.x = h.xprev + f0;
        a.ldx = h.ldx;
        a.out = h.xout + f0;
        a.ldo = h.ldo;
        a.scratch = P->scratch.p + f0;
        a.scratch_ld = P->slab_width;
        a.rscale = P->rscale.p;
        a.cscale = P->cscale.p;
        a.nzrows = P->nzrows.p;
        a.rank_scale = P->rows_all_nonempty ? P->rscale.p : P->nzscale.p;
        a.num_ranks = (int32_t)P->num_nonempty;
        a.f4 = a.tile_f4 = w / 4;
        a.diag_weight = 1.0f + P->gin_eps;
        a.tp = teleport_of(P, h, f0);
        a.back_to_back = h.back_to_back;
        // A hop that adds to Z goes through the register kernel on any graph: it has the rows of X_0, Z and X_{k-1} on their way
        // when a row ends, the bulk-copy kernel would wait for them there.  Mean operator, 100 columns, four hops with a
        // teleport term, both hops of a pair by bulk copy / so: 2.4 M nodes of degree 51 23.1 / 22.3 ms, 2 M of 40
        // 16.4 / 14.9, 1.5 M of 34 11.3 / 9.7; without the term 21.8 / 21.2, 15.2 / 13.9, 10.5 / 8.9.
        if (tile_uses_bulk_copy(P, w) && !a.tp.zsum) GNNPRE_TRY(launch_segments_tma(P, a, st));
        else GNNPRE_TRY(launch_segments_gather(P, a, st));
    }
    return GNNPRE_OK;
}

int launch_finish(const gnnpre_plan* P, const HopArgs& h, int64_t fix_lo, int64_t fix_hi, int64_t hub_lo, int64_t hub_hi,
                  bool empty_rows, int64_t* launches, cudaStream_t st) {
    FixArgs a;
    a.num_empty = empty_rows ? P->num_empty : 0;
    if (fix_hi <= fix_lo && a.num_empty == 0) return GNNPRE_OK;
    a.fix = P->fixups.p;
    a.fix_lo = fix_lo;
    a.fix_hi = fix_hi;
    a.hubs = P->hubs.p;
    a.hub_lo = hub_lo;
    a.hub_hi = hub_hi;
    a.hub_parts = P->hub_parts;
    a.emptyrows = P->emptyrows.p;
    a.scratch = P->scratch.p;
    a.scratch_ld = P->slab_width;
    a.rscale = P->rscale.p;
    a.out = h.xout;
    a.ldo = h.ldo;
    a.f4 = h.width / 4;
    a.tile_f4 = equal_tile_f4(a.f4);
    a.back_to_back = h.back_to_back;
    a.tp = teleport_of(P, h, 0);
    ++*launches;
    if (a.tile_f4 <= 4) return launch_finish_shape<4>(a, st);
    if (a.tile_f4 <= 8) return launch_finish_shape<8>(a, st);
    if (a.tile_f4 <= 16) return launch_finish_shape<16>(a, st);
    return launch_finish_shape<32>(a, st);
}

namespace {

template <int F4C>
int launch_ceiling_tma(const gnnpre_plan* P, const SegArgs& a, float* sink, cudaStream_t st) {
    const int nwarps = tma_warps(a.f4);
    const size_t smem = (size_t)nwarps * kTmaStages * tma_stage_bytes(a.f4);
    CUtensorMap tmap;
    GNNPRE_TRY(make_row_tensor_map(a.x, P->n, 4 * a.f4, a.ldx, &tmap));
    auto kernel = k_ceiling_tma<F4C>;
    GNNPRE_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int64_t nseg = a.seg_hi - a.seg_lo;
    const unsigned grid = (unsigned)std::min<int64_t>(P->num_sms, (nseg + nwarps - 1) / nwarps);
    kernel<<<grid, nwarps * 32, smem, st>>>(a, tmap, sink, P->dev_error.p);
    GNNPRE_CUDA(cudaGetLastError());
    return GNNPRE_OK;
}

template <int G, bool FAR = false>
int launch_ceiling_shape(const SegArgs& a, float* sink, cudaStream_t st) {
    const dim3 grid((unsigned)(((a.seg_hi - a.seg_lo) * G + kThreads - 1) / kThreads), (unsigned)((a.f4 + a.tile_f4 - 1) / a.tile_f4));
    k_ceiling<G, FAR><<<grid, kThreads, 0, st>>>(a, sink);
    GNNPRE_CUDA(cudaGetLastError());
    return GNNPRE_OK;
}

// The fetches of one hop over all column tiles of a slab, tiled and dispatched exactly as launch_segments does.
int launch_ceiling(const gnnpre_plan* P, const HopArgs& h, int64_t seg_lo, int64_t seg_hi, float* sink, cudaStream_t st) {
    if (seg_hi <= seg_lo) return GNNPRE_OK;
    const int32_t tile = segment_tile_width(P, h.width);
    for (int32_t f0 = 0; f0 < h.width; f0 += tile) {
        const int32_t w = std::min<int32_t>(tile, h.width - f0);
        SegArgs a{};
        a.segs = P->by_source.p ? P->by_source.p : P->segments.p;
        a.seg_lo = seg_lo;
        a.seg_hi = seg_hi;
        a.colx = h.colx;
        a.colx_base = h.colx_edge_base;
        a.x = h.xprev + f0;
        a.ldx = h.ldx;
        a.f4 = w / 4;
        if (tile_uses_bulk_copy(P, w)) {
            if (a.f4 == 25) GNNPRE_TRY(launch_ceiling_tma<25>(P, a, sink, st));
            else GNNPRE_TRY(launch_ceiling_tma<0>(P, a, sink, st));
        } else {
            a.tile_f4 = equal_tile_f4(a.f4);
            if (far_rows(a.ldx)) GNNPRE_TRY((launch_ceiling_shape<32, true>(a, sink, st)));
            else if (a.tile_f4 <= 4) GNNPRE_TRY(launch_ceiling_shape<4>(a, sink, st));
            else if (a.tile_f4 <= 8) GNNPRE_TRY(launch_ceiling_shape<8>(a, sink, st));
            else if (a.tile_f4 <= 16) GNNPRE_TRY(launch_ceiling_shape<16>(a, sink, st));
            else GNNPRE_TRY(launch_ceiling_shape<32>(a, sink, st));
        }
    }
    return GNNPRE_OK;
}

}  // namespace

// Everything on the device: K hops, each a sweep over the column slabs and the edge blocks.
int propagate_resident(gnnpre_plan* P, const float* X, int64_t ldx, int32_t K, float* const* out, int64_t ldo,
                       cudaStream_t st, gnnpre_stats_t* stats, const WeightedSum* wsum) {
    // With stats, events bracket every hop and every launch of the segment kernel.
    std::vector<cudaEvent_t> hop_ev, seg_ev;
    auto mark = [&](std::vector<cudaEvent_t>& v) -> int {
        if (!stats) return GNNPRE_OK;
        cudaEvent_t e;
        GNNPRE_CUDA(cudaEventCreate(&e));
        v.push_back(e);
        GNNPRE_CUDA(cudaEventRecord(e, st));
        return GNNPRE_OK;
    };
    int64_t launches = 0, seg_launches = 0;
    int rc = mark(hop_ev);
    for (int32_t k = 0; k < K && rc == GNNPRE_OK; ++k) {
        const float* xprev = k == 0 ? X : out[k - 1];
        const int64_t ldp = k == 0 ? ldx : ldo;
        for (int32_t i = 0; i < P->c && rc == GNNPRE_OK; ++i) {
            const int64_t f_lo = (int64_t)i * P->slab_width;
            HopArgs h;
            h.colx = P->colx.p;
            h.colx_edge_base = 0;
            h.xprev = xprev + f_lo;
            h.x0 = X + f_lo;
            h.ldx0 = ldx;
            h.ldx = ldp;
            h.xout = out[k] + f_lo;
            h.ldo = ldo;
            h.width = (int32_t)std::min<int64_t>(P->slab_width, P->feat_dim - f_lo);
            h.back_to_back = true;
            // Z takes two hops at a time: X_{k-1} is at hand, the rows being gathered, while every pass over Z costs a read
            // and a write of a whole matrix.  The same additions in the same order.  169 K nodes, 64 columns, ten hops with
            // a teleport term: 126 us per hop with a pass over Z in each, 122 so.
            if (wsum && (K - 1 - k) % 2 == 0) {
                h.zsum = wsum->Z + f_lo;
                h.ldz = wsum->ldz;
                h.gamma = wsum->gamma[k + 1];
                h.gamma0 = wsum->gamma[0];
                h.zsum_prev = k > 0;
                h.gamma_prev = wsum->gamma[k];
                h.zsum_first = k <= 1;
            }
            const int seg_tile = segment_tile_width(P, h.width);
            const int seg_tiles = (h.width + seg_tile - 1) / seg_tile;
            const bool per_block = (P->flags & GNNPRE_FLAG_LAUNCH_PER_BLOCK) != 0;
            const size_t groups = per_block ? P->blocks.size() : 1;
            for (size_t j = 0; j < groups && rc == GNNPRE_OK; ++j) {
                const int64_t seg_lo = per_block ? P->blocks[j].seg_lo : 0;
                const int64_t seg_hi = per_block ? P->blocks[j].seg_hi : P->num_segments;
                const int64_t fix_lo = per_block ? P->blocks[j].fix_lo : 0;
                const int64_t fix_hi = per_block ? P->blocks[j].fix_hi : P->num_fixups;
                const int64_t hub_lo = per_block ? P->blocks[j].hub_lo : 0;
                const int64_t hub_hi = per_block ? P->blocks[j].hub_hi : P->num_hubs;
                if (seg_hi > seg_lo) {
                    rc = mark(seg_ev);
                    if (rc == GNNPRE_OK) rc = launch_segments(P, h, seg_lo, seg_hi, st);
                    if (rc == GNNPRE_OK) rc = mark(seg_ev);
                    launches += seg_tiles;
                    seg_launches += seg_tiles;
                }
                if (rc == GNNPRE_OK) rc = launch_finish(P, h, fix_lo, fix_hi, hub_lo, hub_hi, j == 0, &launches, st);
            }
        }
        if (rc == GNNPRE_OK) rc = mark(hop_ev);
    }
    if (stats) {
        if (rc == GNNPRE_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = GNNPRE_ERR_CUDA;
        if (rc == GNNPRE_OK) rc = check_device_error(P);
        if (rc == GNNPRE_OK) {
            for (int32_t k = 0; k < K; ++k) cudaEventElapsedTime(&stats->hop_ms[k], hop_ev[(size_t)k], hop_ev[(size_t)k + 1]);
            cudaEventElapsedTime(&stats->total_ms, hop_ev[0], hop_ev[(size_t)K]);
            float seg_ms = 0.f;
            for (size_t j = 0; j + 1 < seg_ev.size(); j += 2) {
                float ms = 0.f;
                cudaEventElapsedTime(&ms, seg_ev[j], seg_ev[j + 1]);
                seg_ms += ms;
            }
            stats->segments_ms = seg_ms;
            stats->kernel_launches = launches;
            stats->segments_launches = seg_launches;
            stats->h2d_bytes = 0;
            stats->d2h_bytes = 0;
        }
        for (auto& e : hop_ev) cudaEventDestroy(e);
        for (auto& e : seg_ev) cudaEventDestroy(e);
    }
    return rc;
}

}  // namespace gnnpre

// Failure-detection self-tests: see include/gnnpre.h.
extern "C" int gnnpre_selftest_wait_timeout_async(gnnpre_plan_t* P, uint32_t polls, void* stream) {
    if (!P || !P->dev_error.p || polls == 0 || polls > 100000u) return GNNPRE_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    gnnpre::k_wait_that_runs_out<<<1, 32, 0, st>>>(P->dev_error.p, polls);
    GNNPRE_CUDA(cudaGetLastError());
    return GNNPRE_OK;
}

extern "C" int gnnpre_selftest_wait_timeout(gnnpre_plan_t* P, uint32_t polls, void* stream) {
    GNNPRE_TRY(gnnpre_selftest_wait_timeout_async(P, polls, stream));
    return gnnpre_plan_status(P, stream);
}


// Measurement aid: see include/gnnpre.h.
extern "C" int gnnpre_gather_ceiling(gnnpre_plan_t* P, const float* X, int64_t ldx, float* sink, void* stream) {
    if (!P || !X || !sink) return GNNPRE_ERR_INVALID_ARG;
    if (P->structure_mem != GNNPRE_MEM_DEVICE) return GNNPRE_ERR_INVALID_ARG;
    if (ldx < P->feat_dim) return GNNPRE_ERR_INVALID_ARG;
    if (ldx % 4 != 0 || (reinterpret_cast<uintptr_t>(X) & 15u)) return GNNPRE_ERR_ALIGN;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    for (int32_t i = 0; i < P->c; ++i) {
        const int64_t f_lo = (int64_t)i * P->slab_width;
        gnnpre::HopArgs h;
        h.colx = P->colx.p;
        h.colx_edge_base = 0;
        h.xprev = X + f_lo;
        h.ldx = ldx;
        h.xout = nullptr;
        h.ldo = 0;
        h.x0 = nullptr;
        h.ldx0 = 0;
        h.width = (int32_t)std::min<int64_t>(P->slab_width, P->feat_dim - f_lo);
        GNNPRE_TRY(gnnpre::launch_ceiling(P, h, 0, P->num_segments, sink, st));
    }
    return GNNPRE_OK;
}
