// Register-gather segment kernel.  Included by propagate.cu inside its unnamed namespace (uses segments_common.cuh).
#pragma once

// A group of G lanes walks one segment of the edge list; lane q of the group owns float4 q of the column tile, so a
// tile is at most 4 G columns wide (wider rows are cut into equal tiles, blockIdx.y).
//
// Column entries are taken G (at least 8) at a time, fetched one chunk ahead, and the group reads them back from
// shared memory four to a 128-bit broadcast load, weights as ready-made pairs.  Eight neighbour rows are then
// requested back to back (a "window"), summed in a plain fp32 chain, and that sum joins the row's running sum by a
// compensated (Kahan) addition: rounding stays at a few ulps of sum_j |w_j x_j| whatever the row's length.  Windows
// are counted from the segment's start and a row end closes the sum inside its window, so the order of the additions
// depends on the segment alone - not on G, the tile, the launch or the other segments of the warp.
//
// Where every sum of a chunk goes is worked out by the lanes side by side when the chunk is staged (RowOut): a
// finished row goes to its output row, the first sum to a scratch row if its row began in an earlier segment, and the
// segment's last edge always closes a sum - into a scratch row if its row continues in the next segment.  What the
// padding behind that edge adds is therefore never stored.
//
// Bound by what an SM can draw from the L2 (64 bytes per cycle: a loop that only gathers takes 59 us on 169 K nodes,
// 2.3 M edges, 128 columns) and, on short rows, by the instructions around the row ends.  On that graph, us per launch,
// before (rows of 68..128 columns through the copy engine, one shuffle per edge and operand elsewhere) / now: 128
// columns GCN 148 / 97, mean 123 / 77; 64 columns GCN 105 / 66, mean 75 / 51; 16 columns GCN 45 / 39, mean 35 / 29;
// 256 columns, sum operator 223 / 173.  A persistent grid, four rows in flight at 48 registers, and 256-thread CTAs were
// each slower.
constexpr int kSegWindow = 8;

// What a sum needs when its row ends.  Shared memory is set aside in steps of 8, 16, 32, 64 KB an SM and the L1 gets the rest of
// 256: with 8 bytes a row instead of 16 the plain kernels of whole warps stay within 32 KB, and those of four lanes store less
// per chunk; the address is worked out at the row's end instead.  us a call, 16 / 8 bytes: 233 K nodes, 602 columns, GCN
// 7613 / 7447; 89 K nodes, 500 columns, with its plan 692 / 680; 169 K nodes, GCN, 128 columns 311.4 / 308.2, 16 columns
// 113.8 / 108.5, mean operator, 100 columns 253.8 / 249.8, 16 columns 88.3 / 85.9.  Groups of 8 and 16 lanes and the wide
// kernels with an epilogue have no registers left for that (GCN, 64 columns 210 / 225).
struct __align__(16) RowOutLong {
    char* dst;    // first byte of this column tile in the row the sum goes to
    float scale;  // r_i; 1 for a scratch row
    int row;      // output row; -1 for a scratch row (no epilogue)
};
struct __align__(8) RowOutShort {
    float scale;
    int row;  // output row; ~slot for scratch row `slot`
};

// A shared-memory load returns its bytes to every lane, 128 bytes per cycle and SM, as a row's 512 do: entry and weight of
// an edge cost a cycle each beside the row's four.  Groups of 32 lanes therefore keep weights as single floats (169 K nodes,
// GCN, 128 columns: 102.7 us per launch with weights stored twice, 97.3 so); narrower groups, where the instructions
// count, as pairs ready for the packed multiply-add (64 columns: 66.0 us, 72.8 with single floats).
template <int G, bool WEIGHTED, typename RowOut>
struct __align__(16) SegStage {  // read in 16-byte pieces
    static constexpr int kChunk = G < kSegWindow ? kSegWindow : G;  // edges staged at a time
    static constexpr bool kPairs = G < 32;
    using Weight = std::conditional_t<kPairs, float2, float>;
    RowOut out[kChunk];
    uint32_t col[kChunk];
    Weight w[WEIGHTED ? kChunk : 1];

    __device__ __forceinline__ void set_weight(int i, float v) {
        if constexpr (kPairs) w[i] = make_float2(v, v);
        else w[i] = v;
    }
    __device__ __forceinline__ void add_weighted(Quad& acc, int i, const Quad& x) const {
        if constexpr (kPairs) quad_fma_pair(acc, w[i], x);
        else quad_fma(acc, w[i], x);
    }
    __device__ __forceinline__ void add_weighted4(Quad& acc, int i, const Quad* x) const {
        const float4 p = *reinterpret_cast<const float4*>(&w[i]);
        if constexpr (kPairs) {
            quad_fma_pair(acc, make_float2(p.x, p.y), x[0]);
            quad_fma_pair(acc, make_float2(p.z, p.w), x[1]);
            const float4 q = *reinterpret_cast<const float4*>(&w[i + 2]);
            quad_fma_pair(acc, make_float2(q.x, q.y), x[2]);
            quad_fma_pair(acc, make_float2(q.z, q.w), x[3]);
        } else {
            quad_fma(acc, p.x, x[0]);
            quad_fma(acc, p.y, x[1]);
            quad_fma(acc, p.z, x[2]);
            quad_fma(acc, p.w, x[3]);
        }
    }
};

// AHEAD: epilogue operands come from memory where the hop's matrices together exceed the L2, and one row ahead is too late for that:
// each lane asks for the pieces that belong to its row end when the chunk is staged.  169 K nodes, without / with, us a
// call: teleport term, three hops, GCN, 64 columns 302 / 270, 128 394 / 385, sum operator, 100 columns 386 / 359; with
// the sum of ten hops GCN, 64 columns 1125 / 1035, 100 1517 / 1458, sum operator, 64 columns 1042 / 996, mean, 128
// 1315 / 1283.  Not the mean operator's 64 columns (889 / 918) nor narrower rows (16 columns 15 % slower).  A kernel of its own: the
// code alone, not taken, cost 2 to 3 % (ten hops and their sum, GCN, 60,000 nodes of degree 20, 128 columns 638 / 655).  Those are
// R-MAT graphs, whose many short rows end soon after one another.  Long rows of equal length leave the time that one row ahead
// needs, and the requests cost: Erdos-Renyi graphs of 1.3 times the L2, ten hops and their sum, degree 6 / 12 / 16 / 32, with against
// without: GCN, 64 columns 0.98 / 1.00 / 1.03 / 1.02, 128 1.01 / 1.04 / 1.01 / 1.06, sum operator, 64 columns 1.00 / 1.06 / 1.07 / 1.07; with
// a teleport term only 0.92 / 0.95 / 0.94 / 0.92, 0.97 / 1.02 / 1.03 / 1.04, 0.96 / 1.02 / 1.03 / 1.02, sum operator, 128 columns 0.95 / 0.98 /
// 0.98 / 0.99.  Hence where rows are short, or uneven, and in the two kernels that gain anyway.
template <int G, int OP, int EP>
constexpr bool kFetchesAhead = EP != kEpPlain && (G == 32 || (G == 16 && OP != GNNPRE_OP_SAGE_MEAN));

template <int G, int OP, bool HAS_EMPTY, int EP, bool FAR, bool AHEAD>
__global__ void __launch_bounds__(kSegThreads, kSegBlocks) k_segments(const SegArgs a) {
    constexpr unsigned kFull = 0xffffffffu;
    // GIN's weights are 1 but for the self-loops': groups of 16 lanes and more mark those in a bit mask and add the rest
    // (169 K nodes, 256 columns: 195 us per hop with a weight per edge, 181 so; 24 M edges, 64 columns: 460 / 430); narrower
    // groups lose more by the extra votes than the weights cost (169 K nodes, 32 columns: 42 / 45).  Beside the masks the
    // teleport term's X_0 piece is spilled, that is, waited for as soon as it is asked for: with that term every edge has its
    // weight (1 M nodes of degree 50, 100 columns: 3131 us per hop, 3966 with masks; 169 K nodes, 64 columns: 92 / 102; masks
    // and the piece in shared memory: 3144, 100).
    constexpr bool kDiagonal = OP == GNNPRE_OP_GIN_SUM && G >= 16 && EP != kEpTeleport;
    constexpr bool kWeighted = OP != GNNPRE_OP_SAGE_MEAN && !kDiagonal;
    constexpr bool kShort = G == 4 || (G == 32 && EP == kEpPlain);
    using RowOut = std::conditional_t<kShort, RowOutShort, RowOutLong>;
    using Stage = SegStage<G, kWeighted, RowOut>;
    constexpr int C = Stage::kChunk;
    constexpr int M = C / G;  // entries per lane and chunk
    __shared__ __align__(16) Stage stages[kSegThreads / G];
    __shared__ EpiloguePiece<EP> pieces[EP == kEpSum ? kSegThreads : 1];
    const int lane = threadIdx.x & 31;
    const int gl = lane & (G - 1);
    const int gshift = lane & ~(G - 1);
    constexpr unsigned kGroupLow = G == 32 ? kFull : ((1u << G) - 1u);
    Stage& stage = stages[threadIdx.x / G];
    const int64_t s = a.seg_lo + ((int64_t)blockIdx.x * kSegThreads + threadIdx.x) / G;

    const int q0 = blockIdx.y * a.tile_f4;
    const bool on = gl < min(a.tile_f4, a.f4 - q0);
    // lanes beyond the row's width re-read its first float4: every load is unconditional and in bounds
    const char* const xlane = reinterpret_cast<const char*>(a.x) + 16 * (q0 + (on ? gl : 0));
    const RowStride<FAR> row_bytes = (RowStride<FAR>)a.ldx * 4u;
    const int out_off = 16 * gl;

    const uint32_t* entries = a.colx;
    int left = 0, rank = 0, slot_head = -1, slot_tail = -1;
    if (s < a.seg_hi) {
        const Segment g = a.segs[s];
        entries += g.start - a.colx_base;
        left = g.len;
        rank = g.rank;
        slot_head = g.slot_head;
        slot_tail = g.slot_tail;
    }
    uint32_t c_cur[M], c_next[M];
    float w[M], scale[M];
    int row[M];
    auto fetch_rows = [&]() {  // rows and scales of the next C sums
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const int i = min(rank + gl + m * G, a.num_ranks - 1);
            row[m] = HAS_EMPTY ? __ldg(a.nzrows + i) : i;
            scale[m] = OP == GNNPRE_OP_GIN_SUM ? 1.f : __ldg(a.rank_scale + i);
        }
    };
#pragma unroll
    for (int m = 0; m < M; ++m) c_cur[m] = gl + m * G < left ? __ldg(entries + gl + m * G) : 0u;
#pragma unroll
    for (int m = 0; m < M; ++m) c_next[m] = gl + m * G + C < left ? __ldg(entries + gl + m * G + C) : 0u;
    fetch_rows();
    if (OP == GNNPRE_OP_GCN_SYM) {
#pragma unroll
        for (int m = 0; m < M; ++m) w[m] = __ldg(a.cscale + (c_cur[m] & ~kRowEndBit));
    }
    Quad acc = quad_zero(), tot = quad_zero(), cmp = quad_zero();  // this window's plain sum; the row's running sum
    using Piece = std::conditional_t<EP == kEpSum, EpilogueAhead<EP>, EpiloguePiece<EP>>;
    Piece piece;
    if constexpr (EP == kEpSum) piece.at = &pieces[threadIdx.x];
    bool asked = false;  // the operands of the next row's epilogue are on their way
    wait_previous_kernel();

    while (G == 32 ? left > 0 : __any_sync(kFull, left > 0)) {
        // ---- stage this chunk: lanes past the end hold column 0 without a row-end mark
        unsigned ends = 0, loops = 0;  // last edges of rows; self-loops
#pragma unroll
        for (int m = 0; m < M; ++m)
            ends |= ((__ballot_sync(kFull, (int)c_cur[m] < 0) >> gshift) & kGroupLow) << (m * G);
        if (kDiagonal) {
#pragma unroll
            for (int m = 0; m < M; ++m) {  // every row owns its self-loop, so the rank of a row is its index
                const int i = gl + m * G;
                const bool loop = i < left && (int)(c_cur[m] & ~kRowEndBit) == rank + __popc(ends & ((1u << i) - 1u));
                loops |= ((__ballot_sync(kFull, loop) >> gshift) & kGroupLow) << (m * G);
            }
        }
        const int rank_after = rank + __popc(ends);
        int slot_last = -1;  // scratch row of this chunk's last sum, if its row is cut by the segment's end
        if (left > 0 && left <= C && ((ends >> (left - 1)) & 1u) == 0) {
            slot_last = ends == 0 && slot_head >= 0 ? slot_head : slot_tail;
            ends |= 1u << (left - 1);
        }
        const int last = __popc(ends) - 1;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const int i = gl + m * G;
            const uint32_t col = c_cur[m] & ~kRowEndBit;
            stage.col[i] = col;
            int slot = i == 0 ? slot_head : -1;
            if (slot_last >= 0 && i == last) slot = slot_last;
            if (OP == GNNPRE_OP_GIN_SUM && kWeighted)
                w[m] = (int)col == rank + __popc(ends & ((1u << i) - 1u)) ? a.diag_weight : 1.f;
            RowOut o;
            if constexpr (!kShort)
                o.dst = reinterpret_cast<char*>(slot >= 0 ? a.scratch + (int64_t)slot * a.scratch_ld : a.out + (int64_t)row[m] * a.ldo) + 16 * q0;
            o.scale = slot >= 0 ? 1.f : scale[m];
            if constexpr (kShort) o.row = slot >= 0 ? ~slot : row[m];
            else o.row = slot >= 0 ? -1 : row[m];
            stage.out[i] = o;
            if constexpr (AHEAD) {
                if (a.tp.ahead && i <= last && slot < 0) {  // (always ahead here; without the look the compiler spills more: 1 %)
                    constexpr int kLines = G / 8;
                    const int tile_w = min(a.tile_f4, a.f4 - q0);
                    if (EP == kEpTeleport || a.tp.alpha != 0.f || a.tp.zsum_first)
                        prefetch_piece<kLines>(a.tp.x0 + (int64_t)row[m] * a.tp.ldx0 + 4 * q0, tile_w);
                    if (EP == kEpSum && !a.tp.zsum_first) prefetch_piece<kLines>(a.tp.zsum + (int64_t)row[m] * a.tp.ldz + 4 * q0, tile_w);
                    if (EP == kEpSum && a.tp.xprev) prefetch_piece<kLines>(a.tp.xprev + (int64_t)row[m] * a.tp.ldp + 4 * q0, tile_w);
                }
            }
        }
        if (ends != 0) slot_head = -1;
        rank = rank_after;
        entries += C;
        left -= C;
        float w_next[M];
#pragma unroll
        for (int m = 0; m < M; ++m) {
            c_cur[m] = c_next[m];
            c_next[m] = gl + m * G + C < left ? __ldg(entries + gl + m * G + C) : 0u;
            if (OP == GNNPRE_OP_GCN_SYM) w_next[m] = __ldg(a.cscale + (c_cur[m] & ~kRowEndBit));
        }
        fetch_rows();
        const int here = left + C;  // edges of this group from here to the segment's end
        const int cnt = G == 32 ? min(here, C) : C == kSegWindow ? C : __reduce_max_sync(kFull, min(here, C));
        const unsigned busy = G == 32 ? ends | loops : __reduce_or_sync(kFull, ends | loops);
        const RowOut* out = stage.out;
        __syncwarp();
        if (EP != kEpPlain && !asked) piece.load(a.tp, max(out->row, 0), 4 * q0, gl, on);
        asked = true;

        auto flush = [&]() {  // the last edge added closes a sum
            const RowOut o = *out++;
            quad_kahan(tot, cmp, acc);
            float4 v = make_float4(tot.lo.x, tot.lo.y, tot.hi.x, tot.hi.y);
            if (on) {
                if (EP == kEpSum && o.row < 0) wait_copies_ahead();  // no epilogue, but the next row's copies go to the same place
                if (EP == kEpPlain || o.row < 0) v = make_float4(v.x * o.scale, v.y * o.scale, v.z * o.scale, v.w * o.scale);
                else v = piece.finish(v, o.scale, a.tp, o.row, 4 * q0, gl);
                if constexpr (kShort) {
                    char* const dst = o.row >= 0 ? reinterpret_cast<char*>(a.out + (int64_t)o.row * a.ldo) + 16 * q0
                                                 : reinterpret_cast<char*>(a.scratch + (int64_t)~o.row * a.scratch_ld) + 16 * q0;
                    *reinterpret_cast<float4*>(dst + out_off) = v;
                } else {
                    *reinterpret_cast<float4*>(o.dst + out_off) = v;
                }
            }
            acc = tot = cmp = quad_zero();
            asked = out < stage.out + C;
            if (EP != kEpPlain && asked) piece.load(a.tp, max(out->row, 0), 4 * q0, gl, on);
        };

#pragma unroll 1
        for (int t0 = 0; t0 < cnt; t0 += kSegWindow) {
            Quad x[kSegWindow];
#pragma unroll
            for (int u = 0; u < kSegWindow; u += 4) {
                const uint4 c = *reinterpret_cast<const uint4*>(&stage.col[t0 + u]);
                x[u] = quad_gather(xlane, c.x, row_bytes);
                x[u + 1] = quad_gather(xlane, c.y, row_bytes);
                x[u + 2] = quad_gather(xlane, c.z, row_bytes);
                x[u + 3] = quad_gather(xlane, c.w, row_bytes);
            }
            if (kWeighted && t0 == 0) {  // the weights follow behind the chunk's first row requests
#pragma unroll
                for (int m = 0; m < M; ++m) stage.set_weight(gl + m * G, w[m]);
                __syncwarp();
            }
            if (((busy >> t0) & 0xffu) == 0) {
#pragma unroll
                for (int u = 0; u < kSegWindow; u += 4) {
                    if (kWeighted) {
                        stage.add_weighted4(acc, t0 + u, x + u);
                    } else {
#pragma unroll
                        for (int v = 0; v < 4; ++v) quad_add(acc, x[u + v]);
                    }
                }
            } else {
                const unsigned we = ends >> t0, wl = loops >> t0;
#pragma unroll
                for (int u = 0; u < kSegWindow; ++u) {
                    if (kWeighted) stage.add_weighted(acc, t0 + u, x[u]);
                    else if (kDiagonal && ((wl >> u) & 1u)) quad_fma(acc, a.diag_weight, x[u]);
                    else quad_add(acc, x[u]);
                    if ((we >> u) & 1u) flush();
                }
            }
            quad_kahan(tot, cmp, acc);
            acc = quad_zero();
        }
        __syncwarp();
        if (OP == GNNPRE_OP_GCN_SYM) {
#pragma unroll
            for (int m = 0; m < M; ++m) w[m] = w_next[m];
        }
    }
    if (EP == kEpSum) wait_copies_ahead();  // the row after the segment's last was asked for too
}
