// The kernel that finishes what the segment kernels leave: rows cut by segment boundaries, and rows without edges.
// Included by propagate.cu inside its unnamed namespace (uses segments_common.cuh).
#pragma once

struct FixArgs {
    const RowFixup* fix;
    int64_t fix_lo, fix_hi;
    const int32_t* hubs;     // fix-ups with more than hub_parts parts: entries [hub_lo, hub_hi) lie in [fix_lo, fix_hi)
    int64_t hub_lo, hub_hi;
    int32_t hub_parts;
    const int32_t* emptyrows;  // rows without any edge (SAGE, D_i = 0); num_empty = 0 leaves them alone
    int64_t num_empty;
    const float* scratch;
    int64_t scratch_ld;
    const float* rscale;
    float* out;
    int64_t ldo;
    int32_t f4;       // float4 per row of this launch's columns
    int32_t tile_f4;  // float4 per row of one column tile (tile blockIdx.y)
    bool back_to_back;  // see launch_dependent
    Teleport tp;
};

// (s, e) <- (s, e) + (t, f) for sums carried as value + error term: the values are added with the exact rounding
// error of that addition (branch-free two-sum) joining the error terms.  Symmetric in its operands.
__device__ __forceinline__ void pair_add1(float& s, float& e, float t, float f) {
    const float sum = s + t;
    const float bb = sum - s;
    const float lost = (s - (sum - bb)) + (t - bb);
    e = (e + f) + lost;
    s = sum;
}

__device__ __forceinline__ void pair_add4(float4& s, float4& e, const float4& t, const float4& f) {
    pair_add1(s.x, e.x, t.x, f.x);
    pair_add1(s.y, e.y, t.y, f.y);
    pair_add1(s.z, e.z, t.z, f.z);
    pair_add1(s.w, e.w, t.w, f.w);
}

// Adds up the parts of the cut rows, and writes the rows without edges.
// A row's parts are P consecutive scratch rows; they are summed as a tree of fixed shape, so the result is the same
// from run to run and whatever the tile width, so that a matrix cut into column tiles or slabs of any widths comes out
// bit-identical:
//   - chain c of C adds parts c, c + C, c + 2C, ... in that order with compensated additions, its loads issued
//     a batch ahead of its adds; the chains' sums (compensation folded in) then meet pairwise (c with c^1, then c^2,
//     then c^4), each carried as a value and an error term;
//   - an ordinary row gets one warp and C = 8 chains: a group of G lanes covers the tile's width, so a warp holds
//     32 / G groups and every lane carries G / 4 chains;
//   - a hub row (P > hub_parts, listed by the plan) gets a whole CTA, C = 64 chains (8 per warp): the warps'
//     sums meet in shared memory and warp 0 adds them in warp order.
// The first (hub_hi - hub_lo) CTAs of the grid take the hubs, the next ones eight ordinary rows each, the rest the
// rows without edges (zero, or alpha * X_0[i] with a teleport term), kEmptyPerGroup to a lane group.
// Bound by latency: two dependent loads per row, and most rows have two or three parts.  So a row whose chains have one part
// each skips the compensated sums (of one part they are that part), and the longer ones are summed four chains at a time: what
// a lane holds stays small, three CTAs an SM for 64 columns instead of two (169 K nodes, us a call before / now: GCN, three
// hops 210.3 / 205.6; ten hops with a teleport term and their sum 1146 / 1124; 89 K nodes, 500 columns, with its plan 692 / 687;
// 128 columns alike: a third CTA spills there and gains nothing, 253.8 / 255.0 for 100 columns).  A lane keeps at most eight
// parts in flight (with sixteen the kernel held 98 to 174 registers and ran narrow rows in five waves), and the row's
// place and scale are fetched while the segment kernel completes.  169 K nodes, 16 columns, mean operator, three
// hops: 146 -> 100 us a call (three launches per hop before, each after the end of the one before it).
// With a teleport term rows without edges read X_0, four rows ahead of their stores (2.4 M nodes, 100 columns, mean operator:
// 174 us for all that follows a hop's segments, 291 a row at a time; 1.7 M nodes of degree 15 171 / 286).
constexpr int kEmptyPerGroup = 16, kEmptyAhead = 4;

template <int G, int EP>
constexpr int kFinishBlocks = G == 32 ? 2 : G == 16 || EP == kEpSum ? 3 : 4;

template <int G, int EP>
__global__ void __launch_bounds__(kThreads, kFinishBlocks<G, EP>) k_finish_rows(const FixArgs a) {
    constexpr unsigned kFull = 0xffffffffu;
    constexpr int kWarps = kThreads / 32;
    constexpr int S = 32 / G;                         // lane groups per warp
    constexpr int CH = G / 4;                         // chains per lane
    constexpr int CW = S * CH;                        // chains per warp
    constexpr int kAtOnce = CH < 4 ? CH : 4, kRounds = CH >= 4 ? 2 : 4;  // chains summed at a time, parts in flight of each
    static_assert(CW == 8, "the tree's shape must not depend on the width");
    __shared__ float4 meet[kWarps][2][G];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gl = lane & (G - 1), sub = lane / G;
    const int q0 = blockIdx.y * a.tile_f4;
    const bool on = gl < min(a.tile_f4, a.f4 - q0);
    const int64_t nhub = a.hub_hi - a.hub_lo;
    const int64_t ordinary = (a.fix_hi - a.fix_lo + kWarps - 1) / kWarps;
    if ((int64_t)blockIdx.x >= nhub + ordinary) {
        const int64_t i0 = ((int64_t)blockIdx.x - nhub - ordinary) * (kThreads / G * kEmptyPerGroup) + threadIdx.x / G;
        int row[kEmptyPerGroup];
#pragma unroll
        for (int k = 0; k < kEmptyPerGroup; ++k) {
            const int64_t i = i0 + k * (kThreads / G);
            row[k] = i < a.num_empty ? a.emptyrows[i] : -1;
        }
        wait_previous_kernel();
#pragma unroll
        for (int k0 = 0; k0 < kEmptyPerGroup; k0 += kEmptyAhead) {
            EpiloguePiece<EP> piece[kEmptyAhead];
#pragma unroll
            for (int k = 0; k < kEmptyAhead; ++k) piece[k].load(a.tp, max(row[k0 + k], 0), 0, q0 + gl, on && row[k0 + k] >= 0);
#pragma unroll
            for (int k = 0; k < kEmptyAhead; ++k)
                if (on && row[k0 + k] >= 0)
                    *(reinterpret_cast<float4*>(a.out + (int64_t)row[k0 + k] * a.ldo) + q0 + gl) =
                        piece[k].finish(make_float4(0.f, 0.f, 0.f, 0.f), 0.f, a.tp, row[k0 + k], 0, q0 + gl);
        }
        return;
    }
    const bool hub_cta = (int64_t)blockIdx.x < nhub;
    const int64_t i = hub_cta ? (int64_t)a.hubs[a.hub_lo + blockIdx.x]
                              : a.fix_lo + ((int64_t)blockIdx.x - nhub) * kWarps + warp;
    const int chains = hub_cta ? CW * kWarps : CW;           // chains that share the row
    const int chain0 = (hub_cta ? warp * CW : 0) + sub * CH;  // this lane's first chain
    int parts = 0, row = 0;
    float scale = 0.f;
    const float* base = a.scratch + 4 * (q0 + (on ? gl : 0));
    if (i < a.fix_hi) {
        const RowFixup f = a.fix[i];
        parts = f.seg_last - f.seg_first + 1;
        row = f.row;
        scale = a.rscale[row];
        base += (int64_t)f.slot0 * a.scratch_ld;
    }
    const bool mine = i < a.fix_hi && (hub_cta || parts <= a.hub_parts);  // hubs are left to their CTAs
    if (!mine) parts = 0;
    wait_previous_kernel();

    auto part_at = [&](int p) {
        return p < parts ? *reinterpret_cast<const float4*>(base + (int64_t)p * a.scratch_ld) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // The chains meet pairwise, first inside the lane (chains chain0 .. chain0 + CH - 1), then across the lane
    // groups of the warp.  A hub's partial sums can be far larger than their total (40,000 terms of either sign), so
    // every sum travels as a pair (value, error term) and each pairwise addition keeps its exact rounding error.
    float4 tot, err;
    if (parts <= chains) {  // most rows: no chain has more than one part
        float4 one[CH], none[CH];
#pragma unroll
        for (int j = 0; j < CH; ++j) one[j] = part_at(chain0 + j);
#pragma unroll
        for (int j = 0; j < CH; ++j) none[j] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int step = 1; step < CH; step <<= 1) {
#pragma unroll
            for (int j = 0; j < CH; j += 2 * step) pair_add4(one[j], none[j], one[j + step], none[j + step]);
        }
        tot = one[0];
        err = none[0];
    } else {
#pragma unroll 1
        for (int j0 = 0; j0 < CH; j0 += kAtOnce) {
            float4 acc[kAtOnce], cmp[kAtOnce];
#pragma unroll
            for (int j = 0; j < kAtOnce; ++j) acc[j] = cmp[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int p0 = chain0 + j0; p0 < parts; p0 += chains * kRounds) {
                float4 part[kRounds][kAtOnce];
#pragma unroll
                for (int r = 0; r < kRounds; ++r) {
#pragma unroll
                    for (int j = 0; j < kAtOnce; ++j) part[r][j] = part_at(p0 + r * chains + j);
                }
#pragma unroll
                for (int r = 0; r < kRounds; ++r) {
#pragma unroll
                    for (int j = 0; j < kAtOnce; ++j)
                        if (p0 + r * chains + j < parts) kahan4(acc[j], cmp[j], part[r][j]);
                }
            }
#pragma unroll
            for (int j = 0; j < kAtOnce; ++j)  // a compensated sum stands for acc - cmp
                cmp[j] = make_float4(-cmp[j].x, -cmp[j].y, -cmp[j].z, -cmp[j].w);
#pragma unroll
            for (int step = 1; step < kAtOnce; step <<= 1) {
#pragma unroll
                for (int j = 0; j < kAtOnce; j += 2 * step) pair_add4(acc[j], cmp[j], acc[j + step], cmp[j + step]);
            }
            if (j0 == 0) {
                tot = acc[0];
                err = cmp[0];
            } else {
                pair_add4(tot, err, acc[0], cmp[0]);
            }
        }
    }
#pragma unroll
    for (int off = G; off < 32; off <<= 1) {
        float4 os, oe;
        os.x = __shfl_xor_sync(kFull, tot.x, off); os.y = __shfl_xor_sync(kFull, tot.y, off);
        os.z = __shfl_xor_sync(kFull, tot.z, off); os.w = __shfl_xor_sync(kFull, tot.w, off);
        oe.x = __shfl_xor_sync(kFull, err.x, off); oe.y = __shfl_xor_sync(kFull, err.y, off);
        oe.z = __shfl_xor_sync(kFull, err.z, off); oe.w = __shfl_xor_sync(kFull, err.w, off);
        pair_add4(tot, err, os, oe);
    }
    if (hub_cta) {  // uniform over the CTA
        if (sub == 0) {
            meet[warp][0][gl] = tot;
            meet[warp][1][gl] = err;
        }
        __syncthreads();
        if (warp != 0) return;
        tot = meet[0][0][gl];
        err = meet[0][1][gl];
        for (int w = 1; w < kWarps; ++w) pair_add4(tot, err, meet[w][0][gl], meet[w][1][gl]);
    }
    tot.x += err.x; tot.y += err.y; tot.z += err.z; tot.w += err.w;
    if (mine && sub == 0 && on)
        *(reinterpret_cast<float4*>(a.out + (int64_t)row * a.ldo) + q0 + gl) = finish_row_piece<EP>(tot, scale, a.tp, row, q0 + gl);
}
