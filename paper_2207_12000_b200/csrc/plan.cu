// Plan construction: degrees, operator scales, the support's edge list, the balanced edge blocks
// (Section 3.2, "Precomputation on GPU"; Algorithm 1's split of S), Eq. 12's block counts, and the
// warp-level segment tables the propagation kernels walk.  All of it runs on the GPU except the
// O(b) block arithmetic and the Eq. 12 search.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>

#include "gnnpre_internal.cuh"
#include "segment_rules.h"

namespace gnnpre {

namespace {

constexpr int kTB = 256;

inline unsigned grid_for(int64_t items, int per_block) {
    int64_t g = (items + per_block - 1) / per_block;
    return (unsigned)std::max<int64_t>(1, g);
}

// ---------------------------------------------------------------- rows: pointers, degrees, scales

enum : int { kErrRowptr = 1, kErrColRange = 2, kErrDiagonal = 4, kErrOrder = 8, kErrDegree = 16, kErrRows = kErrRowptr | kErrDegree };

// One thread per row.  Checks the row pointers; D_i = number of nonzeros in row i of A (Section 2) unless the caller
// gave the degrees; A^_ij = r_i c_j: GCN r = c = (D_i + 1)^{-1/2} (Eq. 1); SAGE r = 1/D_i (0 for D_i = 0), c = 1;
// GIN r = c = 1, evaluated in fp64 (IEEE sqrt and divide) and rounded once to fp32; the support's row pointers (with
// self-loops row i of the support is row i of A plus one entry, so rowptr_t[i] = rowptr[i] + i); whether the row owns
// an edge (flag may be nullptr); the length of A's longest row.
__global__ void k_rows(int op, int64_t n, int64_t nnz, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ deg_in,
                       int32_t* __restrict__ deg, float* __restrict__ rscale, float* __restrict__ cscale,
                       int64_t* __restrict__ rowptr_t, int32_t* __restrict__ flag, int* err, int* longest) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t lo = i < n ? rowptr[i] : 0, hi = i < n ? rowptr[i + 1] : 0;
    const int most = __reduce_max_sync(0xffffffffu, (int)min(hi - lo, (int64_t)INT32_MAX));
    if ((threadIdx.x & 31) == 0 && most > 0) atomicMax(longest, most);
    if (i >= n) return;
    int bad = 0;
    if (lo < 0 || hi < lo || hi > nnz || (i == 0 && lo != 0) || (i == n - 1 && hi != nnz)) bad |= kErrRowptr;
    else if (hi - lo >= 0x7fffffffLL) bad |= kErrDegree;
    if (bad) atomicOr(err, bad);
    const int32_t d = deg_in ? deg_in[i] : (int32_t)(hi - lo);
    deg[i] = d;
    double r = 1.0, c = 1.0;
    if (op == GNNPRE_OP_GCN_SYM) {
        r = c = 1.0 / sqrt((double)d + 1.0);
    } else if (op == GNNPRE_OP_SAGE_MEAN) {
        r = d > 0 ? 1.0 / (double)d : 0.0;
    }
    rscale[i] = (float)r;
    cscale[i] = (float)c;
    const int64_t diag = op != GNNPRE_OP_SAGE_MEAN;
    rowptr_t[i] = lo + diag * i;
    if (i == n - 1) rowptr_t[n] = hi + diag * n;
    if (flag) flag[i] = hi > lo;
}

__global__ void k_degrees(int64_t n, const int64_t* __restrict__ rowptr, int32_t* __restrict__ deg) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) deg[i] = (int32_t)(rowptr[i + 1] - rowptr[i]);
}

// ---------------------------------------------------------------- the support's edge list E

// Row holding edge e: the last i with rowptr[i] <= e (rows without edges are skipped because their successor shares
// their start).  Stays inside [0, n) whatever rowptr holds.
__device__ __forceinline__ int64_t row_of_edge(const int64_t* __restrict__ rowptr, int64_t n, int64_t e) {
    int64_t lo = 0, hi = n;  // invariant: rowptr[lo] <= e < rowptr[hi]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (rowptr[mid] <= e) lo = mid; else hi = mid;
    }
    return lo;
}

// The same by a whole warp, 32 probes at a time: four or five dependent loads instead of twenty.
__device__ __forceinline__ int64_t row_of_edge_warp(const int64_t* __restrict__ rowptr, int64_t n, int64_t e, int lane) {
    int64_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) >> 5;
        const int64_t probe = lo + (lane + 1) * step;
        const bool le = probe < hi && rowptr[probe] <= e;
        const int k = __popc(__ballot_sync(0xffffffffu, le));  // probes are ascending: the first k hold
        hi = min(hi, lo + (k + 1) * step);
        lo += k * step;
    }
    return lo;
}

// Copies the edge list into the support: entry (row, col) with its row-end mark, self-loops (with `diag`) inserted at
// their column-sorted position, and checks the contract of colidx on the way (`check`).  Row pointers that k_rows found
// bad (*err) are left alone.  A warp takes `per_warp` consecutive edges whatever rows they belong to - a warp per row took 148 us for
// 1.8 M edges because one row holds 20,000 of them, and the check a pass of its own (54 us) - and finds the rows of 32
// edges from the next 32 row pointers.  The last blocks, one thread per row, write the self-loops of rows without edges.
__global__ void k_support(int diag, int check, int64_t n, int64_t nnz, int64_t per_warp, int64_t edge_blocks,
                          const int64_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                          uint32_t* __restrict__ colx, int* err) {
    constexpr unsigned kFull = 0xffffffffu;
    if (*(volatile int*)err & kErrRows) return;
    if ((int64_t)blockIdx.x >= edge_blocks) {
        const int64_t i = ((int64_t)blockIdx.x - edge_blocks) * blockDim.x + threadIdx.x;
        if (i < n) {
            const int64_t lo = rowptr[i];
            if (rowptr[i + 1] == lo) colx[lo + i] = (uint32_t)i | kRowEndBit;
        }
        return;
    }
    const int lane = threadIdx.x & 31;
    const int64_t e_beg = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per_warp;
    const int64_t e_end = min(nnz, e_beg + per_warp);
    if (e_beg >= e_end) return;
    int64_t r = row_of_edge_warp(rowptr, n, e_beg, lane);  // row of the first edge of the 32
    int bad = 0;
    for (int64_t e0 = e_beg; e0 < e_end; e0 += 32) {
        const int64_t e = min(e0 + lane, e_end - 1);  // lanes past the end repeat the last edge
        const int32_t c = colidx[e];
        int64_t row = -1;
        for (int tries = 0; tries < 4; ++tries) {  // row = base + number of row ends at or before e among the next 32
            const int64_t base = r + 32 * tries;
            const int64_t end_of = rowptr[min(base + 1 + lane, n)];
            int k = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(kFull, end_of, k + step - 1) <= e) k += step;
            const int64_t last_end = __shfl_sync(kFull, end_of, 31);
            if (row < 0 && !(k == 31 && last_end <= e)) row = base + k;
            if (__all_sync(kFull, row >= 0)) break;
        }
        if (row < 0) row = row_of_edge(rowptr, n, e);  // a long run of rows without edges
        row = min(row, n - 1);
        const int64_t lo = rowptr[row], hi = rowptr[row + 1];
        int32_t prev = __shfl_up_sync(kFull, c, 1), next = __shfl_down_sync(kFull, c, 1);
        if (lane == 0) prev = e > 0 ? colidx[e - 1] : 0;
        if (lane == 31 || e0 + lane + 1 >= e_end) next = e + 1 < nnz ? colidx[e + 1] : 0;
        if (check) {
            if (c < 0 || c >= n) bad |= kErrColRange;
            if (c == row) bad |= kErrDiagonal;
            if (e + 1 < hi && next <= c) bad |= kErrOrder;
        }
        if (e0 + lane < e_end) {
            const bool last = e == hi - 1;
            if (diag) {
                const int above = c > row;  // the self-loop comes before this entry
                colx[e + row + above] = (uint32_t)c | (last && above ? kRowEndBit : 0u);
                if (above && (e == lo || prev < row)) colx[e + row] = (uint32_t)row;
                if (!above && last) colx[e + row + 1] = (uint32_t)row | kRowEndBit;
            } else {
                colx[e] = (uint32_t)c | (last ? kRowEndBit : 0u);
            }
        }
        r = __shfl_sync(kFull, row, 31);
    }
    if (bad) atomicOr(err, bad);
}

// ---------------------------------------------------------------- exclusive scan

constexpr int kScanItems = 8;
constexpr int kScanTile = kTB * kScanItems;

// Scratch rows, fix-ups and hub rows that a segment (or all segments before it) accounts for.
struct SegCounts {
    int32_t slots, fixups, hubs;
};
__device__ __forceinline__ SegCounts operator+(const SegCounts& a, const SegCounts& b) {
    return {a.slots + b.slots, a.fixups + b.fixups, a.hubs + b.hubs};
}
__device__ __forceinline__ SegCounts shfl_up(const SegCounts& v, int d) {
    return {__shfl_up_sync(0xffffffffu, v.slots, d), __shfl_up_sync(0xffffffffu, v.fixups, d),
            __shfl_up_sync(0xffffffffu, v.hubs, d)};
}
__device__ __forceinline__ int32_t shfl_up(int32_t v, int d) { return __shfl_up_sync(0xffffffffu, v, d); }

// Sum over the threads before this one; *total = sum over the block.
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(const T& v, T* total) {
    __shared__ T warp_sums[kTB / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T t = shfl_up(incl, d);
        if (lane >= d) incl = incl + t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    const T before = shfl_up(incl, 1);
    __syncthreads();
    T run{}, off{};
    for (int w = 0; w < kTB / 32; ++w) {
        if (w == warp) off = run;
        run = run + warp_sums[w];
    }
    *total = run;
    __syncthreads();
    return lane > 0 ? off + before : off;
}

template <typename T>
__global__ void k_tile_sums(const T* __restrict__ in, int64_t n, T* __restrict__ sums) {
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T s{};
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < n) s = s + in[base + k];
    T total;
    block_exclusive_scan(s, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// out[i] = tile_off[tile] + exclusive prefix inside the tile; the last tile also writes out[n] = grand total.
template <typename T>
__global__ void k_tile_scan(const T* __restrict__ in, int64_t n, const T* __restrict__ tile_off, T* __restrict__ out) {
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T v[kScanItems];
    T s{};
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = base + k < n ? in[base + k] : T{};
        s = s + v[k];
    }
    T total;
    T run = block_exclusive_scan(s, &total);
    if (tile_off) run = tile_off[blockIdx.x] + run;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n) out[base + k] = run;
        run = run + v[k];
        if (base + k == n - 1) out[n] = run;
    }
}

int64_t scan_tiles(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

// Items of temporary memory exclusive_scan wants.
size_t scan_temp_items(int64_t n) {
    size_t items = 0;
    for (int64_t t = scan_tiles(n); t > 1; t = scan_tiles(t)) items += 2 * (size_t)t + 1;
    return items;
}

// out has n + 1 entries (n >= 1): exclusive prefix sums and the total.  `in` and `out` may not alias.
template <typename T>
int exclusive_scan(const T* in, int64_t n, T* out, T* temp, cudaStream_t st) {
    const int64_t tiles = scan_tiles(n);
    const T* offs = nullptr;
    if (tiles > 1) {
        T* sums = temp;
        T* tile_offs = temp + tiles;
        k_tile_sums<<<(unsigned)tiles, kTB, 0, st>>>(in, n, sums);
        GNNPRE_CUDA(cudaGetLastError());
        GNNPRE_TRY(exclusive_scan(sums, tiles, tile_offs, tile_offs + tiles + 1, st));
        offs = tile_offs;
    }
    k_tile_scan<<<(unsigned)tiles, kTB, 0, st>>>(in, n, offs, out);
    GNNPRE_CUDA(cudaGetLastError());
    return GNNPRE_OK;
}

// ---------------------------------------------------------------- what the host has to know

struct BlockRows {
    int32_t row_lo, row_hi, first_partial, last_partial;
    int64_t done_row_hi;
};

// Warp l <= b: block l's rows (l < b), and what the segments before the block account for.
__global__ void k_block_report(int b, const int64_t* __restrict__ e_off, const int64_t* __restrict__ seg_base,
                               const SegCounts* __restrict__ before, const int64_t* __restrict__ rowptr_t, int64_t n,
                               BlockRows* __restrict__ rows, SegCounts* __restrict__ at) {
    const int l = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (l > b) return;
    if (lane == 0) at[l] = before[seg_base[l]];
    if (l == b) return;
    const int64_t lo = e_off[l], hi = e_off[l + 1];
    const int64_t r0 = row_of_edge_warp(rowptr_t, n, lo, lane), r1 = row_of_edge_warp(rowptr_t, n, hi - 1, lane);
    BlockRows o;
    o.row_lo = (int32_t)r0;
    o.row_hi = (int32_t)r1;
    o.first_partial = rowptr_t[r0] < lo;
    o.last_partial = rowptr_t[r1 + 1] > hi;
    // rows complete after this block, i.e. whose end offset is <= hi: those before the row of the next block's first edge
    // (all but those behind the last edge are found so; the last block is the host's)
    o.done_row_hi = hi < rowptr_t[n] ? row_of_edge_warp(rowptr_t, n, hi, lane) : n;
    if (lane == 0) rows[l] = o;
}

// ---------------------------------------------------------------- rows with and without edges

__global__ void k_split_rows(int64_t n, const int32_t* __restrict__ flag, const int32_t* __restrict__ rank,
                             const float* __restrict__ rscale, int32_t* __restrict__ nzrows, float* __restrict__ nzscale,
                             int32_t* __restrict__ emptyrows) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (flag[i]) {
        nzrows[rank[i]] = (int32_t)i;
        nzscale[rank[i]] = rscale[i];
    } else {
        emptyrows[i - rank[i]] = (int32_t)i;
    }
}

// ---------------------------------------------------------------- warp-level segments

// Segment t of block l nominally starts at e_lo(l) + t*L.  A start that falls inside a row is moved
// forward to the next row start when that lies within `snap` edges (and inside the block), so that
// short rows are never cut; long rows are cut and their parts summed by a fix-up.  Where no row of the graph is longer
// than `uncut` edges the start always moves (two may then meet, or one the block's end: an empty segment), and nothing is
// left for the finishing launch (see longest_uncut_row).
// Until k_segment_finalize: slot_head holds the "first row began earlier" flag and len the first row's index.
__global__ void k_segment_starts(int64_t nseg, int b, const int64_t* __restrict__ seg_base,
                                 const int64_t* __restrict__ e_off, int32_t L, int32_t snap, int64_t uncut, const int* __restrict__ longest,
                                 const int64_t* __restrict__ rowptr_t, int64_t n, const int32_t* __restrict__ rank,
                                 Segment* __restrict__ segs) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s > nseg) return;
    Segment g;
    if (s == nseg) {  // sentinel
        g.start = e_off[b];
        g.rank = 0;
        g.slot_head = 0;
        g.slot_tail = -1;
        g.len = (int32_t)n;
        segs[s] = g;
        return;
    }
    int lo = 0, hi = b;  // block holding segment s: seg_base[lo] <= s < seg_base[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (seg_base[mid] <= s) lo = mid; else hi = mid;
    }
    const int64_t t = s - seg_base[lo];
    int64_t start = e_off[lo] + t * (int64_t)L;
    int64_t row = row_of_edge(rowptr_t, n, start);
    if (t > 0 && rowptr_t[row] < start) {
        const int64_t next = rowptr_t[row + 1];
        if ((next - start <= snap || *longest < uncut) && next <= e_off[lo + 1]) {
            start = next;
            // at the very end: empty, as the sentinel
            row = start >= e_off[b] ? n : row + 2 <= n && rowptr_t[row + 2] > start ? row + 1 : row_of_edge(rowptr_t, n, start);
        }
    }
    g.start = start;
    g.rank = row == n ? 0 : rank ? rank[row] : (int32_t)row;
    g.slot_head = row < n && rowptr_t[row] < start;
    g.slot_tail = -1;
    g.len = (int32_t)row;
    segs[s] = g;
}

// What segment s accounts for: a scratch row if its first row began earlier (head), one if the row of its last edge
// goes on and began in it (tail), a fix-up if the row that began earlier ends in it.  first[s] = the segment that row
// began in.
__global__ void k_segment_counts(int64_t nseg, const Segment* __restrict__ segs, const int64_t* __restrict__ rowptr_t,
                                 int32_t hub_parts, SegCounts* __restrict__ counts, int32_t* __restrict__ first) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nseg) return;
    const Segment g = segs[s], nx = segs[s + 1];
    const int head = g.slot_head;
    // the row holding this segment's last edge continues iff the next segment's first row began earlier
    const int tail = nx.slot_head && rowptr_t[nx.len] >= g.start;
    const int emit = head && rowptr_t[(int64_t)g.len + 1] <= nx.start;
    int hub = 0;
    if (emit) {
        const int64_t first_edge = rowptr_t[g.len];
        int64_t lo = max(s - 1, (int64_t)0), hi = s;  // segs[lo].start <= first_edge < segs[hi].start, most often the segment before
        for (int64_t back = 2; lo > 0 && segs[lo].start > first_edge; back *= 2) {
            hi = lo;
            lo = max(lo - back, (int64_t)0);
        }
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if (segs[mid].start <= first_edge) lo = mid; else hi = mid;
        }
        first[s] = (int32_t)lo;
        hub = s - lo + 1 > hub_parts;
    }
    counts[s] = {head + tail, emit, hub};
}

__global__ void k_segment_finalize(int64_t nseg, Segment* __restrict__ segs, const SegCounts* __restrict__ counts,
                                   const SegCounts* __restrict__ before, const int32_t* __restrict__ first,
                                   RowFixup* __restrict__ fixups, int32_t* __restrict__ hubs, const int* err) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s > nseg || *err) return;
    if (s < nseg) {
        const SegCounts c = counts[s], b = before[s];
        const int head = segs[s].slot_head;
        if (c.fixups) {
            RowFixup f;
            f.row = segs[s].len;
            f.seg_first = first[s];
            f.seg_last = (int32_t)s;
            // the tail slot (the last slot) of the row's first segment; the other parts follow it
            f.slot0 = before[first[s] + 1].slots - 1;
            fixups[b.fixups] = f;
            if (c.hubs) hubs[b.hubs] = b.fixups;
        }
        segs[s].slot_head = head ? b.slots : -1;
        segs[s].slot_tail = c.slots > head ? b.slots + head : -1;
    }
    segs[s].len = s < nseg ? (int32_t)(segs[s + 1].start - segs[s].start) : 0;
}

// ---------------------------------------------------------------- the order in which a hop takes its segments

// A hop over a matrix beyond the L2 reads most rows from memory, and in the order of the edge list every segment reads from all
// of it.  But a row's columns ascend, so a segment that lies inside one row reads from a part of the matrix, the narrower the
// longer the row - and most edges belong to long rows.  Taken in the order of their middle columns those segments sweep over
// the matrix together, and the rows that they share are in the L2; the segments of several rows come last.  Every segment does
// what it did, so the bits are the same.  us per hop, edge order / this: 2.4 M nodes, 124 M edges, mean operator, 100 columns
// 3871 / 3637 (bulk copy), 4366 / 3870 (registers); GCN, 128 columns 4971 / 4295; sum, 64 columns 2417 / 2247; 16 columns
// 1386 / 1378; 1 M nodes, 30 M edges, GCN, 128 columns 1072 / 1029; 400 K nodes, 40 M edges, sum, 256 columns 2200 / 2090;
// about the L2's size: 300 K nodes, 40 M edges, GCN, 128 columns 1115 / 1068, 96 columns 997 / 990; well inside it: 169 K
// nodes, 2.5 M edges, GCN, 128 columns 99 / 102.  Four or eight coarse ranges of columns instead: 3 to 6 % slower.
//
// Segments of several rows follow in the order of the edge list: where the caller's numbering has locality (communities, meshes)
// neighbours read the same part of the matrix.  Where hardly any segment lies in one row, or most that do lie near the
// diagonal, the table is left out, as they come.  2 M nodes, GCN, 128 columns, us per hop, edge order / several-row segments in
// order of arrival / so: communities of 20,000, degree 24, 1810 / 3370 / 1790; the same with hubs in each, degree 34, 2280 / 3480 /
// 2285 (2514 with the one-row segments first); a 27-point mesh 1720 / 2080 / 1700; no locality: R-MAT 3260 / 3060 / 3070,
// Erdos-Renyi 3770 / 3765 / 3765.
constexpr int64_t kFewSegments = 64;  // one in so many

// What the host decides by: segments inside one row, and those of them whose row lies near their columns.
struct OrderCounts {
    int32_t one_row, near;
};

// SCATTER false: places[0 .. kOrderBuckets) += segments of the buckets, places[kOrderBuckets + block] = the other segments of the
// block's.  true: places holds the exclusive prefix sums of that, that is, where each bucket and each block's other segments
// begin; copies the segments there.
template <bool SCATTER>
__global__ void __launch_bounds__(kTB) k_segment_order(int64_t nseg, const Segment* __restrict__ segs, const uint32_t* __restrict__ colx,
                                                       const int32_t* __restrict__ nzrows, int64_t n, int32_t* __restrict__ places,
                                                       OrderCounts* report, Segment* __restrict__ ordered, const int* err) {
    constexpr unsigned kFull = 0xffffffffu;
    __shared__ int others[kTB / 32];
    if (*err) return;  // then there is neither a table nor an edge list
    const int64_t s = (int64_t)blockIdx.x * kTB + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int bucket = -1;
    bool near = false;
    Segment g;
    if (s < nseg) {
        g = segs[s];
        const Segment nx = segs[s + 1];
        // all edges in one row (never the last segment: the sentinel has no row)
        if (s + 1 < nseg && g.len > 0 && (nx.rank == g.rank || (nx.rank == g.rank + 1 && nx.slot_head < 0))) {
            const uint32_t col = colx[g.start + g.len / 2] & ~kRowEndBit;
            bucket = column_bucket(col, n);
            if (!SCATTER) near = near_diagonal((uint32_t)(nzrows ? nzrows[g.rank] : g.rank), col, n);
        }
    }
    const unsigned same = __match_any_sync(kFull, bucket);  // one addition per bucket and warp
    const int first = __ffs(same) - 1;
    int at = 0;
    if (lane == first && bucket >= 0) at = atomicAdd(&places[bucket], __popc(same));
    at = __shfl_sync(kFull, at, first) + __popc(same & ((1u << lane) - 1u));
    const unsigned other = __ballot_sync(kFull, s < nseg && bucket < 0);
    if (lane == 0) others[warp] = __popc(other);
    if (!SCATTER) {
        const unsigned one_row = __ballot_sync(kFull, bucket >= 0), nears = __ballot_sync(kFull, near);
        if (lane == 0 && one_row) atomicAdd(&report->one_row, __popc(one_row));
        if (lane == 0 && nears) atomicAdd(&report->near, __popc(nears));
    }
    __syncthreads();
    if (SCATTER) {
        if (s < nseg && bucket < 0) {
            at = places[kOrderBuckets + blockIdx.x] + __popc(other & ((1u << lane) - 1u));
            for (int w = 0; w < warp; ++w) at += others[w];
        }
        if (s < nseg) ordered[at] = g;
    } else if (threadIdx.x == 0) {
        int sum = 0;
        for (int w = 0; w < kTB / 32; ++w) sum += others[w];
        places[kOrderBuckets + blockIdx.x] = sum;
    }
}

// Parts beyond which a cut row counts as a hub and gets a whole CTA of the finishing kernel (64 chains) instead of a
// warp (8 chains).  One value for all widths, because the tree's shape decides the bits and those must not depend on
// how a matrix is cut into column tiles.
constexpr int32_t kHubParts = 64;

// The longest row (edges) of a graph in which no row is cut, so that segments end with rows and the finishing launch has
// nothing to do, at the price of uneven and empty segments.  The launch costs the same whatever the graph, the unevenness
// grows with it; groups of fewer than 32 lanes also wait for the longest segment of their warp.  Mean operator, rows of
// equal length, us per hop never cut / cut:
//   all segments at once (4,096 nodes of degree 16, 64 columns, two hops): 10.4 / 13.7, and no worse up to three segments
//   800,000 edges, L = 32:   32 columns, rows of 1.5 L 25 / 29, 1.8 L 27 / 31, 2 L 29 / 26, 2.4 L 32 / 28; 64 columns
//                            31 / 36, 38 / 38, 40 / 34, 40 / 36; 128 columns 36 / 43, 37 / 49, 42 / 45, 36 / 45
//   4 million, L = 64:       16 columns, 1.6 L 51 / 64, 2 L 60 / 51; 32 columns, 1.6 L 69 / 77, 1.8 L 76 / 72; 64 columns,
//                            1.5 L 99 / 104, 1.8 L 128 / 104; 128 columns, 1.8 L 126 / 151, 2 L 155 / 143, 2.4 L 127 / 142
//   whole waves:             16 columns, 2.4 M edges, L = 80, 1.8 L 26 / 30, 2.2 L 30 / 28; 4.8 M, L = 152, 1.5 L 42 / 48,
//                            1.8 L 50 / 51; 32 columns, 1.2 M, L = 80, 1.8 L 19 / 21, 2.2 L 22 / 19; 2.4 M, L = 152,
//                            1.5 L 31 / 35, 1.8 L 37 / 34; 64 columns, 600,000, L = 80, 1.5 L 15 / 17, 1.8 L 19 / 16
//   20 million, L = 256:     16 columns, 1.25 L 177 / 185, 1.5 L 233 / 219, 2 L 290 / 160; 64 columns, 1.25 L 325 / 332,
//                            1.4 L 391 / 365, 2 L 645 / 302; 128 columns, 1.8 L 529 / 566, 2 L 694 / 538, 2.9 L 549 / 536
int64_t longest_uncut_row(int64_t m, int64_t lanes, int64_t L, bool one_wave) {
    const int64_t work = m * lanes;
    if (one_wave) return 3 * L;
    if (lanes == 32) return work <= (1 << 28) ? 3 * L : 2 * L;
    return work <= (lanes == 16 ? 1 << 23 : 1 << 24) ? 2 * L : work <= (1 << 26) ? 3 * L / 2 : 5 * L / 4;
}

}  // namespace

// ---------------------------------------------------------------- Eq. 12

// For a fixed c the least feasible b has a closed form, so one pass over c suffices.
int solve_budget(int64_t B_S, int64_t B_X, int64_t B_fixed, int64_t beta_S, int64_t beta_X, int64_t B_GPU,
                 int64_t max_b, int64_t max_c, int64_t* b_out, int64_t* c_out) {
    if (B_S < 0 || B_X < 0 || B_fixed < 0 || beta_S < 1 || beta_X < 1 || max_b < 1 || max_c < 1)
        return GNNPRE_ERR_INVALID_ARG;
    bool found = false;
    int64_t best_b = 0, best_c = 0;
    const int64_t need_S = beta_S * B_S;
    for (int64_t c = 1; c <= max_c; ++c) {
        const int64_t x_part = (beta_X * B_X + c - 1) / c;
        const int64_t room = B_GPU - B_fixed - x_part;
        if (room <= 0 && need_S > 0) continue;
        if (room < 0) continue;
        const int64_t b = need_S == 0 ? 1 : (need_S + room - 1) / room;
        if (b > max_b) continue;
        const int64_t bb = std::max<int64_t>(b, 1);
        if (!found || bb * c < best_b * best_c) {  // ascending c: the first minimum has the smallest c
            found = true;
            best_b = bb;
            best_c = c;
        }
    }
    if (!found) return GNNPRE_ERR_BUDGET_TOO_SMALL;
    *b_out = best_b;
    *c_out = best_c;
    return GNNPRE_OK;
}

int check_device_error(gnnpre_plan* P) {
    if (!P->dev_error.p) return GNNPRE_OK;
    int h = 0;
    GNNPRE_CUDA(cudaMemcpy(&h, P->dev_error.p, sizeof(int), cudaMemcpyDeviceToHost));
    if (h == 0) return GNNPRE_OK;
    GNNPRE_CUDA(cudaMemset(P->dev_error.p, 0, sizeof(int)));
    return GNNPRE_ERR_TIMEOUT;
}

int check_device() {
    int dev = 0;
    GNNPRE_CUDA(cudaGetDevice(&dev));
    int major = 0;
    GNNPRE_CUDA(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
    return major == 10 ? GNNPRE_OK : GNNPRE_ERR_UNSUPPORTED_ARCH;
}

}  // namespace gnnpre

using namespace gnnpre;

namespace {

constexpr int kCacheDevices = 64;

int64_t device_memory_bytes(int device) {
    static std::atomic<int64_t> known[kCacheDevices];
    int64_t bytes = device < kCacheDevices ? known[device].load(std::memory_order_relaxed) : 0;
    if (bytes == 0) {
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return 0;
        bytes = (int64_t)total_b;
        if (device < kCacheDevices) known[device].store(bytes, std::memory_order_relaxed);
    }
    return bytes;
}

}  // namespace

// Device memory that calls on the plan may count on: what the caller set, else the device's free memory when the plan was
// built or, if nobody asked then, when somebody first does.
int64_t gnnpre::plan_budget(const gnnpre_plan* P) {
    int64_t budget = P->budget_bytes.load(std::memory_order_relaxed);
    if (budget <= 0) {
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        budget = (int64_t)free_b + P->device_bytes();
        P->budget_bytes.store(budget, std::memory_order_relaxed);
    }
    return budget;
}

namespace {

// One block of device memory per device outlives the plan that used it, so that a program that makes plan after plan (one
// per dataset, or per operator) does not pay 0.7 to 8 ms for an allocation and its release each time.  At most
// kMostCached bytes; only plans for resident operands without a memory budget use it; it is given back when an
// allocation of the library fails and by gnnpre_release_cached_memory.  A block enters it when its device's streams are done.
constexpr size_t kMostCached = 128u << 20, kCachedGrain = 2u << 20;

struct CachedBlock {
    char* p = nullptr;
    size_t bytes = 0;
};
std::mutex g_cache_mutex;
CachedBlock g_cache[kCacheDevices];
void* g_small_page[kCacheDevices];  // four bytes that keep the driver's page of small allocations (see streams_done)

CachedBlock take_cached(int device, size_t bytes) {
    std::lock_guard<std::mutex> lock(g_cache_mutex);
    CachedBlock b;
    if (device < kCacheDevices && g_cache[device].bytes >= bytes) std::swap(b, g_cache[device]);
    return b;
}

// Waits for all streams of the current device; false if that failed.  Freeing device memory does so, be it four bytes - and,
// unlike cudaDeviceSynchronize, it does not invalidate the stream captures in the process.  5 us with the allocation while
// the driver has its page of small allocations, 320 if that came and went with these four bytes.
bool streams_done(int device) {
    if (device < kCacheDevices) {
        std::lock_guard<std::mutex> lock(g_cache_mutex);
        if (!g_small_page[device]) (void)cudaMalloc(&g_small_page[device], 4);
    }
    void* p = nullptr;
    return cudaMalloc(&p, 4) == cudaSuccess && cudaFree(p) == cudaSuccess;
}

// keeps the larger of `b` and what the cache holds, frees the other
void give_cached(int device, CachedBlock b) {
    {
        std::lock_guard<std::mutex> lock(g_cache_mutex);
        if (device < kCacheDevices && g_cache[device].bytes < b.bytes) std::swap(b, g_cache[device]);
    }
    if (b.p) cudaFree(b.p);
}

}  // namespace

bool gnnpre::release_cached_block() {
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return false;
    const CachedBlock b = take_cached(device, 1);
    void* page = nullptr;
    if (device < kCacheDevices) {
        std::lock_guard<std::mutex> lock(g_cache_mutex);
        std::swap(page, g_small_page[device]);
    }
    if (b.p) cudaFree(b.p);
    if (page) cudaFree(page);
    return b.p != nullptr;
}

extern "C" int gnnpre_release_cached_memory(void) {
    (void)release_cached_block();
    return GNNPRE_OK;
}

gnnpre_plan::~gnnpre_plan() {
    if (s_h2d) cudaStreamDestroy(s_h2d);
    if (s_d2h) cudaStreamDestroy(s_d2h);
    if (s_compute) cudaStreamDestroy(s_compute);
    if (s_struct) cudaStreamDestroy(s_struct);
    // kernels on the caller's streams (or of a build that failed) may still use the block: the next plan may have it when they
    // have ended, else it is freed
    if (arena_cached && arena[0].p && streams_done(device)) {
        give_cached(device, {arena[0].p, arena[0].count});
        arena[0].owned = false;
    }
}

int64_t gnnpre_plan::device_bytes() const {
    size_t t = arena[0].bytes() + arena[1].bytes() + colx_stage[0].bytes() + colx_stage[1].bytes();
    for (const auto& s : slab) t += s.bytes();
    for (const auto& s : whole) t += s.bytes();
    return (int64_t)t;
}

int64_t gnnpre_plan::host_bytes() const { return (int64_t)colx_host.bytes(); }

namespace {

// Destroys the plan with its device current, whichever the caller's is, and in the capture mode in which releases of memory
// neither fail nor disturb captures on the caller's streams (a plan may be collected at any time).
void destroy_plan(gnnpre_plan* P) {
    int device = 0;
    const bool other = cudaGetDevice(&device) == cudaSuccess && device != P->device && cudaSetDevice(P->device) == cudaSuccess;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    const bool swapped = cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess;
    delete P;
    if (swapped) cudaThreadExchangeStreamCaptureMode(&mode);
    if (other) cudaSetDevice(device);
    (void)cudaGetLastError();
}

// ask: the free memory is asked for whatever the plan's size.
int build_plan_impl(const gnnpre_csr_t* csr, const int32_t* degrees, const gnnpre_plan_opts_t* opts, bool ask,
                    gnnpre_plan* P) {
    const int64_t n = csr->n, nnz = csr->nnz;
    const bool diag = opts->op != GNNPRE_OP_SAGE_MEAN;
    cudaStream_t st = nullptr;  // the plan is built on the legacy default stream and synchronised
    GNNPRE_CUDA(cudaGetDevice(&P->device));
    P->n = n;
    P->nnz = nnz;
    P->nnz_tilde = nnz + (diag ? n : 0);
    P->feat_dim = (opts->feat_dim + 3) / 4 * 4;  // whole float4 columns; the caller's leading dimensions cover the pad
    P->op = opts->op;
    P->gin_eps = opts->gin_eps;
    P->teleport_alpha = opts->teleport_alpha;
    P->flags = opts->flags;
    P->structure_mem = csr->mem;
    P->degrees_given = degrees != nullptr;
    P->hub_parts = kHubParts;
    const int64_t m = P->nnz_tilde;
    if (csr->mem == GNNPRE_MEM_HOST && (csr->rowptr[0] != 0 || csr->rowptr[n] != nnz)) return GNNPRE_ERR_INVALID_CSR;

    // ---- Eq. 12: (b, c)
    const int64_t F = P->feat_dim;
    P->B_S = 4 * m + 8 * (n + 1);
    P->B_X = 4 * n * F;
    P->B_fixed = 16 * n;
    P->beta_S = csr->mem == GNNPRE_MEM_HOST ? 2 : 1;
    P->beta_X = opts->operands_mem == GNNPRE_MEM_HOST ? 4 : 2;
    P->budget_bytes = opts->budget_bytes;
    const bool resident = opts->operands_mem == GNNPRE_MEM_DEVICE && csr->mem == GNNPRE_MEM_DEVICE;
    int64_t budget = P->budget_bytes;
    if (budget <= 0) {
        // The free memory, but for the question: on a busy machine the driver takes 0.06 to 100 ms to answer it (median 0.4),
        // longer than everything else a small plan needs.  A resident plan whose volumes are a sixteenth of the device at
        // most is not asked about (unless it turns out not to fit: gnnpre_build_plan).
        const int64_t device_bytes = device_memory_bytes(P->device);
        if (resident && !ask && P->B_S + P->beta_X * P->B_X + P->B_fixed <= device_bytes / 16) {
            budget = device_bytes;
        } else {
            size_t free_b = 0, total_b = 0;  // nothing of the plan has been allocated yet
            GNNPRE_CUDA(cudaMemGetInfo(&free_b, &total_b));
            budget = (int64_t)free_b;
            P->budget_bytes = budget;
        }
    }
    P->solved_budget = budget;
    const int64_t max_c = (F + 3) / 4;
    const int64_t max_b = std::min<int64_t>(std::max<int64_t>(m, 1), 1 << 20);
    int64_t b = opts->force_blocks, c = opts->force_col_slabs;
    if (b < 0 || c < 0 || c > max_c) return GNNPRE_ERR_INVALID_ARG;
    P->col_slabs_forced = c > 0;
    if (b > 0 && b > m) return GNNPRE_ERR_INVALID_ARG;
    if (b == 0 || c == 0) {
        // a forced value pins that variable; the other is searched
        int64_t sb = 0, sc = 0;
        const int64_t lo_c = c ? c : 1, hi_c = c ? c : max_c;
        bool found = false;
        for (int64_t cc = lo_c; cc <= hi_c; ++cc) {
            int64_t tb = 0, tc = 0;
            // restrict the search to this c by scaling: solve with max_c = 1 on B_X / cc
            const int64_t x_part = (P->beta_X * P->B_X + cc - 1) / cc;
            int rc = solve_budget(P->B_S, 0, P->B_fixed + x_part, P->beta_S, 1, budget, max_b, 1, &tb, &tc);
            if (rc != GNNPRE_OK) continue;
            if (b > 0) {
                if (tb > b) continue;  // the forced b is too small for this c
                tb = b;
            }
            if (!found || tb * cc < sb * sc) {
                found = true;
                sb = tb;
                sc = cc;
            }
        }
        if (!found) return GNNPRE_ERR_BUDGET_TOO_SMALL;
        b = sb;
        c = sc;
        // Host-resident operands: Eq. 12's model charges every block product the same, but with copies
        // overlapped a second slab lets the upload of X and the first hop's kernels run side by side.
        // Two slabs are used when the budget alone asks for one and the row pieces stay >= 256 bytes
        // (narrower strided pieces travel the host link below full speed); below 256 columns only for
        // two equal slabs, so that the pieces also start on 128-byte lines.
        if (opts->force_col_slabs == 0 && opts->operands_mem == GNNPRE_MEM_HOST && c == 1 && F >= 128 &&
            (F % 8 == 0 || F >= 256))
            c = 2;
        // Likewise a single edge block would hold every output row back until the whole hop is done;
        // eight blocks let finished rows leave for the host while the rest of the hop computes.
        if (opts->force_blocks == 0 && b == 1) {
            // E fits the budget whole: it stays on the device even when the caller's CSR lives on the host
            P->structure_mem = GNNPRE_MEM_DEVICE;
            if (opts->operands_mem == GNNPRE_MEM_HOST && m >= (1 << 20)) b = 8;
        }
    }
    if (m == 0) b = 1;
    P->b = (int32_t)b;
    P->c = (int32_t)c;
    P->slab_width = 4 * ((F + 4 * c - 1) / (4 * c));
    if (P->slab_width * (c - 1) >= F) return GNNPRE_ERR_INVALID_ARG;  // a slab would be empty
    GNNPRE_CUDA(cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, P->device));
    // edges one launch covers: a hop when everything is resident, one block when blocks are launched singly
    const bool streamed = opts->operands_mem == GNNPRE_MEM_HOST || P->structure_mem == GNNPRE_MEM_HOST;
    const bool per_block = (opts->flags & GNNPRE_FLAG_LAUNCH_PER_BLOCK) || streamed;
    const int64_t m_launch = per_block ? m / b : m;
    P->segment_edges = opts->segment_edges > 0
                           ? opts->segment_edges
                           : auto_segment_edges(P->slab_width, m_launch, per_block ? 1 : b, uses_bulk_copy(P, (int32_t)P->slab_width),
                                                !streamed && beyond_cache(P, (int32_t)P->slab_width), !per_block, P->num_sms);
    if (P->segment_edges < 1) return GNNPRE_ERR_INVALID_ARG;

    // ---- block table: block l = edges [floor(l m / b), floor((l+1) m / b))
    P->blocks.assign((size_t)b, Block{});
    std::vector<int64_t> e_off((size_t)b + 1), seg_base((size_t)b + 1);
    {
        const int64_t q = m / b, r = m % b;
        for (int64_t l = 0; l <= b; ++l) e_off[(size_t)l] = l * q + (l * r) / b;
    }
    const int32_t L = P->segment_edges;
    seg_base[0] = 0;
    for (int64_t l = 0; l < b; ++l)
        seg_base[(size_t)l + 1] = seg_base[(size_t)l] + (e_off[(size_t)l + 1] - e_off[(size_t)l] + L - 1) / L;
    const int64_t nseg = seg_base[(size_t)b];
    if (nseg >= 0x3fffffffLL) return GNNPRE_ERR_INVALID_ARG;
    P->num_segments = nseg;
    const bool e_host = P->structure_mem == GNNPRE_MEM_HOST;
    const bool by_source = !per_block && beyond_cache(P, (int32_t)P->slab_width);

    // ---- device memory: one allocation for what has a known size, one for what the segments turn out to need - or, if the
    // caller set no budget, nothing is streamed and what they can need at most is small, a single one.  (An allocation of a
    // few MB takes 370 to 1600 us and its release 300, one of 64 MB no more; one of up to 1 MB, a piece of a page the
    // driver mostly has at hand, about 1 us.)  The temporaries of the build live where E goes at the very end,
    // if there is room.
    struct Report {  // followed by BlockRows[b] and SegCounts[b + 1]
        int32_t err, nonempty, longest_row;
        int32_t unused;
        OrderCounts order;
    };
    static_assert(sizeof(Report) % 8 == 0 && sizeof(BlockRows) % 8 == 0, "the report's parts stay aligned");
    // (the report has a place of its own: E overwrites the temporaries before the host reads it)
    DevBuf<char> report;
    const size_t report_bytes = sizeof(Report) + sizeof(BlockRows) * (size_t)b + sizeof(SegCounts) * (size_t)(b + 1);
    DevBuf<uint32_t> e_temp;
    DevBuf<uint32_t>& colx = e_host ? e_temp : P->colx;  // E of a host-resident structure is on the device for the build only
    const bool small_report = b <= 4096;
    const int64_t places = kOrderBuckets + (nseg + kTB - 1) / kTB;  // see k_segment_order
    auto want_fixed = [&](Carve& carve) {
        carve.want(P->deg, (size_t)n);
        carve.want(P->rscale, (size_t)n);
        carve.want(P->cscale, (size_t)n);
        carve.want(P->rowptr_t, (size_t)n + 1);
        carve.want(P->segments, (size_t)nseg + 1);
        carve.want(P->dev_error, 1);
        if (small_report) carve.want(report, report_bytes);
        if (by_source) {
            carve.want(P->by_source, (size_t)nseg);
            carve.want(P->by_source_counts, 2 * (size_t)places + 1 + scan_temp_items(places));
        }
        if (!e_host) carve.want(P->colx, (size_t)m);
    };
    Carve fixed;
    want_fixed(fixed);
    auto want_sized = [&](Carve& carve, int64_t fixups, int64_t hubs, int64_t nonempty, int64_t empty, int64_t slots) {
        carve.want(P->fixups, (size_t)fixups);
        carve.want(P->hubs, (size_t)hubs);
        if (empty > 0) {
            carve.want(P->nzrows, (size_t)nonempty);
            carve.want(P->nzscale, (size_t)nonempty);
            carve.want(P->emptyrows, (size_t)empty);
        }
        carve.want(P->scratch, (size_t)slots * (size_t)P->slab_width);
    };
    // a segment has at most a head and a tail part and ends at most one cut row, a hub has more than kHubParts parts
    const int64_t most_rows = diag ? 0 : n;
    const int64_t most_bytes = 16 * nseg + 12 * most_rows + 2 * nseg * P->slab_width * 4;
    // (a plan over a matrix beyond the L2 has up to twice the segments, and as much room for them: 2 M nodes, 80 M edges, GCN, 128
    // columns, us for a build with two allocations / one 2550 / 1950; one hop with its plan 5310 / 4710)
    bool one_allocation = !ask && opts->budget_bytes <= 0 && opts->operands_mem == GNNPRE_MEM_DEVICE &&
                          most_bytes <= (by_source ? 256 << 20 : 128 << 20) && fixed.bytes() > (1 << 20);
    if (one_allocation) want_sized(fixed, nseg, nseg / kHubParts, most_rows, most_rows, 2 * nseg);
    const int64_t refused = refused_allocations();
    int placed;
    if (one_allocation && fixed.bytes() <= kMostCached - kCachedGrain) {  // in whole grains, so that the next plan's may fit
        const size_t bytes = (fixed.bytes() + kCachedGrain - 1) / kCachedGrain * kCachedGrain;
        const CachedBlock block = take_cached(P->device, bytes);
        P->arena_cached = true;
        P->arena[0].p = block.p;
        P->arena[0].count = block.bytes;
        placed = block.p ? GNNPRE_OK : P->arena[0].alloc(bytes);
        if (placed == GNNPRE_OK) placed = fixed.place(P->arena[0].p);
    } else {
        placed = fixed.place(P->arena[0]);
    }
    if (placed != GNNPRE_OK && one_allocation && refused_allocations() > refused) {  // no room for the most: what is needed, then
        one_allocation = P->arena_cached = false;
        Carve exact;
        want_fixed(exact);
        placed = exact.place(P->arena[0]);
    }
    GNNPRE_TRY(placed);
    if (e_host) GNNPRE_TRY(e_temp.alloc((size_t)m));
    DevBuf<char> temp_arena;
    if (!small_report) GNNPRE_TRY(report.alloc(report_bytes));
    DevBuf<int32_t> flag, rank, rank_temp, first;
    DevBuf<SegCounts> counts, before, counts_temp;
    DevBuf<int64_t> offsets;
    Carve temps;
    temps.want(offsets, 2 * ((size_t)b + 1));
    if (!diag) {
        temps.want(flag, (size_t)n);
        temps.want(rank, (size_t)n + 1);
        temps.want(rank_temp, scan_temp_items(n));
    }
    temps.want(first, (size_t)nseg);
    temps.want(counts, (size_t)nseg);
    temps.want(before, (size_t)nseg + 1);
    temps.want(counts_temp, scan_temp_items(nseg));
    if (temps.bytes() <= colx.bytes()) GNNPRE_TRY(temps.place(reinterpret_cast<char*>(colx.p)));
    else GNNPRE_TRY(temps.place(temp_arena));
    Report* d_report = reinterpret_cast<Report*>(report.p);
    BlockRows* d_rows = reinterpret_cast<BlockRows*>(report.p + sizeof(Report));
    SegCounts* d_at = reinterpret_cast<SegCounts*>(d_rows + b);

    // ---- the CSR on the device (a temporary copy when the caller's lives on the host)
    DevBuf<int64_t> tmp_rowptr;
    DevBuf<int32_t> tmp_colidx, tmp_deg;
    const int64_t* d_rowptr = csr->rowptr;
    const int32_t* d_colidx = csr->colidx;
    const int32_t* d_deg_in = degrees;
    if (csr->mem == GNNPRE_MEM_HOST) {
        GNNPRE_TRY(tmp_rowptr.alloc((size_t)n + 1));
        GNNPRE_TRY(tmp_colidx.alloc((size_t)nnz));
        GNNPRE_CUDA(cudaMemcpy(tmp_rowptr.p, csr->rowptr, sizeof(int64_t) * (size_t)(n + 1), cudaMemcpyHostToDevice));
        if (nnz) GNNPRE_CUDA(cudaMemcpy(tmp_colidx.p, csr->colidx, sizeof(int32_t) * (size_t)nnz, cudaMemcpyHostToDevice));
        d_rowptr = tmp_rowptr.p;
        d_colidx = tmp_colidx.p;
        if (degrees) {
            GNNPRE_TRY(tmp_deg.alloc((size_t)n));
            GNNPRE_CUDA(cudaMemcpy(tmp_deg.p, degrees, sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice));
            d_deg_in = tmp_deg.p;
        }
    }

    // ---- rows
    GNNPRE_CUDA(cudaMemsetAsync(d_report, 0, sizeof(Report), st));
    GNNPRE_CUDA(cudaMemsetAsync(P->dev_error.p, 0, sizeof(int), st));
    k_rows<<<grid_for(n, kTB), kTB, 0, st>>>(P->op, n, nnz, d_rowptr, d_deg_in, P->deg.p, P->rscale.p, P->cscale.p,
                                             P->rowptr_t.p, flag.p, &d_report->err, &d_report->longest_row);
    GNNPRE_CUDA(cudaGetLastError());
    if (!diag) {  // only SAGE can have rows without edges
        GNNPRE_TRY(exclusive_scan(flag.p, n, rank.p, rank_temp.p, st));
        GNNPRE_CUDA(cudaMemcpyAsync(&d_report->nonempty, rank.p + n, sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    }

    // ---- segments, scratch slots and row fix-ups
    // How far a nominal cut inside a row may move forward to the next row start.  Half a segment keeps the segments
    // balanced (moving by up to a whole one cost 3-15 % on every larger workload).  A launch so small that all its
    // segments are resident at once is bound by latency, not balance: there the cut may move by up to L - 1 edges.
    const int64_t f4_slab = std::min<int64_t>(P->slab_width, 512) / 4;
    const int64_t lanes = f4_slab <= 4 ? 4 : f4_slab <= 8 ? 8 : f4_slab <= 16 ? 16 : 32;
    const bool one_wave = nseg * lanes <= (int64_t)P->num_sms * 768;
    const int32_t snap = one_wave ? L - 1 : L / 2;
    // Segments of 16 or 24 edges that fill one wave (of 28 warps an SM) cut nearly every row of a uniform graph whose rows are a
    // little longer: rows of up to 72 edges are not cut there (96 in groups of whole warps, which wait for nobody's longer
    // segment).  us for two hops, segments of 32 edges / cut / so: degree 24, mean operator, 480,000 edges, 16 columns 16.5 / 25.5 / 16.1,
    // 240,000, 32 columns 13.1 / 17.4 / 12.6, 120,000, 64 columns 11.6 / 15.6 / 11.6; degree 36 16.7 / 22.9 / 18.3, 14.1 / 16.3 / 15.0,
    // 13.0 / 13.9 / 14.0; degree 60, 128 columns, 60,000 edges 10.6 / 13.7 / 12.0; not cut in narrower groups, degree 60 is slower
    // (240,000 edges, 32 columns 15.0 / 13.9 / 19.6).
    const int64_t uncut = std::max<int64_t>(longest_uncut_row(m_launch, lanes, L, one_wave),
                                            one_wave || L >= 32 || opts->segment_edges > 0 ? 0 : lanes == 32 ? 96 : 72);
    if (m > 0) {
        std::vector<int64_t> h_off(e_off);
        h_off.insert(h_off.end(), seg_base.begin(), seg_base.end());
        GNNPRE_CUDA(cudaMemcpyAsync(offsets.p, h_off.data(), sizeof(int64_t) * h_off.size(), cudaMemcpyHostToDevice, st));
        const int64_t *d_e_off = offsets.p, *d_seg_base = offsets.p + b + 1;
        // (without rows that own no edge the scan's ranks are the row numbers)
        k_segment_starts<<<grid_for(nseg + 1, kTB), kTB, 0, st>>>(nseg, (int)b, d_seg_base, d_e_off, L, snap, uncut,
                                                                  &d_report->longest_row, P->rowptr_t.p, n, rank.p, P->segments.p);
        GNNPRE_CUDA(cudaGetLastError());
        k_segment_counts<<<grid_for(nseg, kTB), kTB, 0, st>>>(nseg, P->segments.p, P->rowptr_t.p, P->hub_parts, counts.p, first.p);
        GNNPRE_CUDA(cudaGetLastError());
        GNNPRE_TRY(exclusive_scan(counts.p, nseg, before.p, counts_temp.p, st));
        k_block_report<<<grid_for(b + 1, kTB / 32), kTB, 0, st>>>((int)b, d_e_off, d_seg_base, before.p, P->rowptr_t.p, n, d_rows, d_at);
        GNNPRE_CUDA(cudaGetLastError());
    }
    // What follows needs nothing that only the device knows yet if all tables have room for the most: then the host looks once,
    // at the end, instead of waiting here as well (with the searches above by warps and by short steps, us for plan, hops and
    // release, before / now: 89 K nodes, 1.9 M edges, 500 columns, GCN, two hops 680 / 651; 64 columns, mean operator 241 / 213).
    std::vector<int64_t> h_report((report_bytes + 7) / 8);
    const Report* rep = reinterpret_cast<const Report*>(h_report.data());
    const BlockRows* h_rows = reinterpret_cast<const BlockRows*>(rep + 1);
    const SegCounts* at = reinterpret_cast<const SegCounts*>(h_rows + b);
    auto read_report = [&]() -> int {
        GNNPRE_CUDA(cudaMemcpy(h_report.data(), report.p, report_bytes, cudaMemcpyDeviceToHost));
        if (rep->err) return GNNPRE_ERR_INVALID_CSR;
        P->num_nonempty = diag ? n : rep->nonempty;
        P->num_empty = n - P->num_nonempty;
        P->rows_all_nonempty = P->num_empty == 0;
        P->short_rows = m <= 8 * n || rep->longest_row * n > 4 * m;
        if (m > 0) {
            P->num_slots = at[b].slots;
            P->num_fixups = at[b].fixups;
            P->num_hubs = at[b].hubs;
        }
        return GNNPRE_OK;
    };
    const bool look_once = one_allocation && m > 0;
    if (!look_once) {
        GNNPRE_TRY(read_report());
        if (!one_allocation) {
            Carve sized;
            want_sized(sized, P->num_fixups, P->num_hubs, P->num_nonempty, P->num_empty, P->num_slots);
            GNNPRE_TRY(sized.place(P->arena[1]));
        }
    }
    if (look_once ? !diag : !P->rows_all_nonempty) {
        k_split_rows<<<grid_for(n, kTB), kTB, 0, st>>>(n, flag.p, rank.p, P->rscale.p, P->nzrows.p, P->nzscale.p, P->emptyrows.p);
        GNNPRE_CUDA(cudaGetLastError());
    }
    if (m == 0) {  // no edges at all: every row is empty; one empty block
        P->blocks[0] = Block{0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, n};
        Segment sentinel{0, 0, -1, -1, 0};
        GNNPRE_CUDA(cudaMemcpy(P->segments.p, &sentinel, sizeof(Segment), cudaMemcpyHostToDevice));
        GNNPRE_CUDA(cudaStreamSynchronize(st));
        return GNNPRE_OK;
    }
    k_segment_finalize<<<grid_for(nseg + 1, kTB), kTB, 0, st>>>(nseg, P->segments.p, counts.p, before.p, first.p, P->fixups.p,
                                                                P->hubs.p, &d_report->err);
    GNNPRE_CUDA(cudaGetLastError());

    // ---- E, the support's edge list: overwrites the temporaries
    {
        const bool check = !(opts->flags & GNNPRE_FLAG_SKIP_VALIDATION);
        // 256 edges per warp, more (up to 2048) only while every warp the device holds still gets its share
        const int64_t per_warp = 256 * std::min<int64_t>(8, 1 + nnz / ((int64_t)P->num_sms * 64 * 512));
        const int64_t edge_blocks = ((nnz + per_warp - 1) / per_warp + kTB / 32 - 1) / (kTB / 32);
        const int64_t row_blocks = diag ? (n + kTB - 1) / kTB : 0;
        k_support<<<(unsigned)(edge_blocks + row_blocks), kTB, 0, st>>>(diag ? 1 : 0, check ? 1 : 0, n, nnz, per_warp, edge_blocks,
                                                                       d_rowptr, d_colidx, colx.p, &d_report->err);
        GNNPRE_CUDA(cudaGetLastError());
    }
    int32_t *counted = P->by_source_counts.p, *begins = counted + places;
    const int32_t* row_of_rank = diag ? nullptr : P->nzrows.p;  // (nullptr as well where every row has edges)
    if (by_source) {
        GNNPRE_CUDA(cudaMemsetAsync(counted, 0, sizeof(int32_t) * kOrderBuckets, st));
        k_segment_order<false><<<grid_for(nseg, kTB), kTB, 0, st>>>(nseg, P->segments.p, P->colx.p, row_of_rank, n, counted,
                                                                    &d_report->order, nullptr, &d_report->err);
        GNNPRE_CUDA(cudaGetLastError());
    }
    GNNPRE_TRY(read_report());  // everything is in place
    for (int64_t l = 0; l < b; ++l) {
        Block& B = P->blocks[(size_t)l];
        const BlockRows& r = h_rows[(size_t)l];
        B.e_lo = e_off[(size_t)l];
        B.e_hi = e_off[(size_t)l + 1];
        B.row_lo = r.row_lo;
        B.row_hi = r.row_hi;
        B.first_partial = r.first_partial;
        B.last_partial = r.last_partial;
        B.seg_lo = seg_base[(size_t)l];
        B.seg_hi = seg_base[(size_t)l + 1];
        B.fix_lo = at[l].fixups;
        B.fix_hi = at[l + 1].fixups;
        B.hub_lo = at[l].hubs;
        B.hub_hi = at[l + 1].hubs;
        B.done_row_lo = l == 0 ? 0 : h_rows[(size_t)l - 1].done_row_hi;
        B.done_row_hi = l == b - 1 ? n : r.done_row_hi;
    }
    if (by_source) {
        if (rep->order.one_row * kFewSegments >= nseg && 2 * (int64_t)rep->order.near <= rep->order.one_row) {
            GNNPRE_TRY(exclusive_scan<int32_t>(counted, places, begins, begins + places + 1, st));
            k_segment_order<true><<<grid_for(nseg, kTB), kTB, 0, st>>>(nseg, P->segments.p, P->colx.p, row_of_rank, n, begins, nullptr,
                                                                       P->by_source.p, &d_report->err);
            GNNPRE_CUDA(cudaGetLastError());
            GNNPRE_CUDA(cudaStreamSynchronize(st));
        } else {
            P->by_source.reset();  // the segments stay as they are
        }
    }

    // ---- a host-resident structure keeps E in pinned memory and streams it block by block
    if (P->structure_mem == GNNPRE_MEM_HOST) {
        GNNPRE_TRY(P->colx_host.alloc((size_t)m));
        GNNPRE_CUDA(cudaMemcpy(P->colx_host.p, colx.p, sizeof(uint32_t) * (size_t)m, cudaMemcpyDeviceToHost));
        int64_t longest = 0;
        for (const Block& B : P->blocks) longest = std::max(longest, B.e_hi - B.e_lo);
        // (the build's copies make room for the staging buffers: a structure kept on the host may be one that hardly fits)
        tmp_rowptr.reset();
        tmp_colidx.reset();
        tmp_deg.reset();
        temp_arena.reset();
        e_temp.reset();
        GNNPRE_TRY(P->colx_stage[0].alloc((size_t)longest));
        if (b > 1) GNNPRE_TRY(P->colx_stage[1].alloc((size_t)longest));
    }
    return GNNPRE_OK;
}

}  // namespace

extern "C" int gnnpre_degrees(const gnnpre_csr_t* csr, int32_t* deg_out, void* stream) {
    if (!csr || !deg_out || !csr->rowptr || csr->n < 0) return GNNPRE_ERR_INVALID_ARG;
    GNNPRE_TRY(check_device());
    const int64_t n = csr->n;
    if (n == 0) return GNNPRE_OK;
    cudaStream_t st = (cudaStream_t)stream;
    if (csr->mem == GNNPRE_MEM_DEVICE) {
        k_degrees<<<grid_for(n, kTB), kTB, 0, st>>>(n, csr->rowptr, deg_out);
        GNNPRE_CUDA(cudaGetLastError());
        return GNNPRE_OK;
    }
    DevBuf<int64_t> rp;
    DevBuf<int32_t> dg;
    GNNPRE_TRY(rp.alloc((size_t)n + 1));
    GNNPRE_TRY(dg.alloc((size_t)n));
    GNNPRE_CUDA(cudaMemcpyAsync(rp.p, csr->rowptr, sizeof(int64_t) * (size_t)(n + 1), cudaMemcpyHostToDevice, st));
    k_degrees<<<grid_for(n, kTB), kTB, 0, st>>>(n, rp.p, dg.p);
    GNNPRE_CUDA(cudaGetLastError());
    GNNPRE_CUDA(cudaMemcpyAsync(deg_out, dg.p, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToHost, st));
    GNNPRE_CUDA(cudaStreamSynchronize(st));
    return GNNPRE_OK;
}

extern "C" int gnnpre_build_plan(const gnnpre_csr_t* csr, const int32_t* degrees, const gnnpre_plan_opts_t* opts,
                                 gnnpre_plan_t** plan_out) {
    if (!csr || !opts || !plan_out) return GNNPRE_ERR_INVALID_ARG;
    *plan_out = nullptr;
    if (csr->n < 1 || csr->n >= 0x7fffffffLL || csr->nnz < 0 || !csr->rowptr || (csr->nnz > 0 && !csr->colidx))
        return GNNPRE_ERR_INVALID_ARG;
    if (csr->mem != GNNPRE_MEM_DEVICE && csr->mem != GNNPRE_MEM_HOST) return GNNPRE_ERR_INVALID_ARG;
    if (opts->op < GNNPRE_OP_GCN_SYM || opts->op > GNNPRE_OP_GIN_SUM) return GNNPRE_ERR_INVALID_ARG;
    if (opts->operands_mem != GNNPRE_MEM_DEVICE && opts->operands_mem != GNNPRE_MEM_HOST) return GNNPRE_ERR_INVALID_ARG;
    if (!(opts->teleport_alpha >= 0.f && opts->teleport_alpha <= 1.f)) return GNNPRE_ERR_INVALID_ARG;
    if (opts->feat_dim < 1) return GNNPRE_ERR_INVALID_ARG;
    if (opts->segment_edges < 0 || opts->segment_edges > (1 << 20)) return GNNPRE_ERR_INVALID_ARG;
    GNNPRE_TRY(check_device());
    const int64_t refused = refused_allocations();
    gnnpre_plan* P = new (std::nothrow) gnnpre_plan();
    if (!P) return GNNPRE_ERR_OOM_HOST;
    int rc = build_plan_impl(csr, degrees, opts, false, P);
    if (rc == GNNPRE_ERR_OOM_DEVICE && P->budget_bytes <= 0 && refused_allocations() > refused) {
        // (b, c) were solved for a device that holds the plan easily, but there is no room: for what is free, then
        destroy_plan(P);
        P = new (std::nothrow) gnnpre_plan();
        if (!P) return GNNPRE_ERR_OOM_HOST;
        rc = build_plan_impl(csr, degrees, opts, true, P);
    }
    if (rc != GNNPRE_OK) {
        destroy_plan(P);
        return rc;
    }
    *plan_out = P;
    return GNNPRE_OK;
}

extern "C" int gnnpre_plan_info(const gnnpre_plan_t* P, gnnpre_plan_info_t* o) {
    if (!P || !o) return GNNPRE_ERR_INVALID_ARG;
    std::memset(o, 0, sizeof(*o));
    o->n = P->n;
    o->nnz = P->nnz;
    o->nnz_tilde = P->nnz_tilde;
    o->feat_dim = P->feat_dim;
    o->op = P->op;
    o->b = P->b;
    o->c = P->c;
    o->slab_width = P->slab_width;
    o->B_S = P->B_S;
    o->B_X = P->B_X;
    o->B_fixed = P->B_fixed;
    o->beta_S = P->beta_S;
    o->beta_X = P->beta_X;
    o->budget_bytes = P->solved_budget;
    o->device_bytes = P->device_bytes();
    o->host_bytes = P->host_bytes();
    o->num_segments = P->num_segments;
    o->num_row_fixups = P->num_fixups;
    o->num_scratch_rows = P->num_slots;
    o->segment_edges = P->segment_edges;
    o->structure_mem = P->structure_mem;
    return GNNPRE_OK;
}

extern "C" int gnnpre_plan_block(const gnnpre_plan_t* P, int32_t l, gnnpre_block_info_t* o) {
    if (!P || !o || l < 0 || l >= P->b) return GNNPRE_ERR_INVALID_ARG;
    const Block& B = P->blocks[(size_t)l];
    o->e_lo = B.e_lo;
    o->e_hi = B.e_hi;
    o->row_lo = B.row_lo;
    o->row_hi = B.row_hi;
    o->first_row_partial = B.first_partial;
    o->last_row_partial = B.last_partial;
    return GNNPRE_OK;
}

extern "C" int gnnpre_plan_hop_order(const gnnpre_plan_t* P, int64_t* first_edges_out) {
    if (!P || !first_edges_out) return GNNPRE_ERR_INVALID_ARG;
    if (P->num_segments == 0) return GNNPRE_OK;
    const Segment* segments = P->by_source.p ? P->by_source.p : P->segments.p;
    GNNPRE_CUDA(cudaMemcpy2D(first_edges_out, sizeof(int64_t), &segments->start, sizeof(Segment), sizeof(int64_t),
                             (size_t)P->num_segments, cudaMemcpyDeviceToHost));
    return GNNPRE_OK;
}

extern "C" int gnnpre_plan_scales(const gnnpre_plan_t* P, int32_t* deg_out, float* rscale_out, float* cscale_out) {
    if (!P) return GNNPRE_ERR_INVALID_ARG;
    const size_t n = (size_t)P->n;
    if (deg_out) GNNPRE_CUDA(cudaMemcpy(deg_out, P->deg.p, sizeof(int32_t) * n, cudaMemcpyDeviceToHost));
    if (rscale_out) GNNPRE_CUDA(cudaMemcpy(rscale_out, P->rscale.p, sizeof(float) * n, cudaMemcpyDeviceToHost));
    if (cscale_out) GNNPRE_CUDA(cudaMemcpy(cscale_out, P->cscale.p, sizeof(float) * n, cudaMemcpyDeviceToHost));
    return GNNPRE_OK;
}

extern "C" int gnnpre_plan_support(const gnnpre_plan_t* P, int64_t* rowptr_out, int32_t* colidx_out) {
    if (!P) return GNNPRE_ERR_INVALID_ARG;
    if (rowptr_out)
        GNNPRE_CUDA(cudaMemcpy(rowptr_out, P->rowptr_t.p, sizeof(int64_t) * (size_t)(P->n + 1), cudaMemcpyDeviceToHost));
    if (colidx_out && P->nnz_tilde > 0) {
        const size_t m = (size_t)P->nnz_tilde;
        if (P->structure_mem == GNNPRE_MEM_HOST) {
            std::memcpy(colidx_out, P->colx_host.p, sizeof(uint32_t) * m);
        } else {
            GNNPRE_CUDA(cudaMemcpy(colidx_out, P->colx.p, sizeof(uint32_t) * m, cudaMemcpyDeviceToHost));
        }
        for (size_t e = 0; e < m; ++e) colidx_out[e] &= 0x7fffffff;  // drop the row-end marks
    }
    return GNNPRE_OK;
}

extern "C" void gnnpre_plan_destroy(gnnpre_plan_t* P) {
    if (P) destroy_plan(P);
}

extern "C" int gnnpre_solve_budget(int64_t B_S, int64_t B_X, int64_t B_fixed, int64_t beta_S, int64_t beta_X,
                                   int64_t B_GPU, int64_t max_b, int64_t max_c, int64_t* b_out, int64_t* c_out) {
    if (!b_out || !c_out) return GNNPRE_ERR_INVALID_ARG;
    return solve_budget(B_S, B_X, B_fixed, beta_S, beta_X, B_GPU, max_b, max_c, b_out, c_out);
}
