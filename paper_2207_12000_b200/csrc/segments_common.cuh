// What every propagation kernel shares: the epilogue of a finished row, the launch arguments, compensated addition.
// Included by propagate.cu inside its unnamed namespace, before the kernels.
#pragma once

// The optional teleport term: a finished row r_i * sum becomes keep * (r_i * sum) + alpha * X_0[i].
struct Teleport {
    const float* x0;
    int64_t ldx0;
    float alpha, keep;  // keep = 1 - alpha
    // fixed-weight sum of hops (zsum == nullptr: this hop leaves Z alone): Z += gamma * (the value stored for this hop),
    // after gamma_prev * (the hop before it, xprev) if that one left Z alone (xprev == nullptr: it did not)
    float* zsum;
    int64_t ldz;
    const float* xprev;
    int64_t ldp;
    float gamma, gamma_prev, gamma0;
    int zsum_first;
    int ahead;  // fetch the rows that the epilogues read into the L2 ahead of time
};

// EP, the epilogue of a finished row: 0 = scale only; 1 = scale and teleport term; 2 = the launch also accumulates the
// fixed-weight sum of hops (teleport decided at run time).  A compile-time switch, because the mere presence of the
// optional code slowed the plain kernels down although its branches were never taken (the L2-resident workload by
// 10 % for the teleport term and by 40 % for the sum).
constexpr int kEpPlain = 0, kEpTeleport = 1, kEpSum = 2;
// What the epilogue of one row reads besides its sum (column tile at f0, float4 q); loaded before the sum is complete
// where the kernel knows the row ahead of time.
template <int EP>
struct EpiloguePiece {
    float4 x0;
    float4 z[EP == kEpSum ? 2 : 1];  // Z, X_{k-1}
    __device__ __forceinline__ void load(const Teleport& tp, int64_t row, int f0, int q, bool on) {
        if (EP == kEpPlain || !on) return;
        if (EP == kEpTeleport || tp.alpha != 0.f || tp.zsum_first)
            x0 = __ldg(reinterpret_cast<const float4*>(tp.x0 + row * tp.ldx0 + f0) + q);
        if (EP == kEpSum && !tp.zsum_first) z[0] = *(reinterpret_cast<const float4*>(tp.zsum + row * tp.ldz + f0) + q);
        if (EP == kEpSum && tp.xprev) z[1] = __ldg(reinterpret_cast<const float4*>(tp.xprev + row * tp.ldp + f0) + q);
    }
    // the value to store for the row; adds it to the sum of hops (every finished row piece passes here once per hop)
    __device__ __forceinline__ float4 finish(const float4& sum, float scale, const Teleport& tp, int64_t row, int f0, int q) const {
        float4 o = make_float4(sum.x * scale, sum.y * scale, sum.z * scale, sum.w * scale);
        if (EP == kEpTeleport || (EP == kEpSum && tp.alpha != 0.f)) {
            o.x = fmaf(tp.keep, o.x, tp.alpha * x0.x);
            o.y = fmaf(tp.keep, o.y, tp.alpha * x0.y);
            o.z = fmaf(tp.keep, o.z, tp.alpha * x0.z);
            o.w = fmaf(tp.keep, o.w, tp.alpha * x0.w);
        }
        if (EP == kEpSum) {
            float4 acc = z[0];
            if (tp.zsum_first) acc = make_float4(tp.gamma0 * x0.x, tp.gamma0 * x0.y, tp.gamma0 * x0.z, tp.gamma0 * x0.w);
            if (tp.xprev) {
                acc.x = fmaf(tp.gamma_prev, z[1].x, acc.x);
                acc.y = fmaf(tp.gamma_prev, z[1].y, acc.y);
                acc.z = fmaf(tp.gamma_prev, z[1].z, acc.z);
                acc.w = fmaf(tp.gamma_prev, z[1].w, acc.w);
            }
            acc.x = fmaf(tp.gamma, o.x, acc.x);
            acc.y = fmaf(tp.gamma, o.y, acc.y);
            acc.z = fmaf(tp.gamma, o.z, acc.z);
            acc.w = fmaf(tp.gamma, o.w, acc.w);
            *(reinterpret_cast<float4*>(tp.zsum + row * tp.ldz + f0) + q) = acc;
        }
        return o;
    }
};

// Asks for the row piece of f4 float4 (at most 8 * LINES) at p to be brought into the L2.
template <int LINES>
__device__ __forceinline__ void prefetch_piece(const float* p, int f4) {
#pragma unroll
    for (int i = 0; i < LINES; ++i)
        if (8 * i < f4) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 32 * i));
}

__device__ __forceinline__ void copy_ahead(float4* dst, const float4* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void wait_copies_ahead() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The same, its operands copied to shared memory meanwhile (copies are not ordered among themselves: those of one sum are
// waited for before the next sum's are issued, whether or not they were wanted): held in registers beside the eight rows in flight, the twelve
// floats of a sum of hops were spilled, which waits for them at once.  Copies through the L1 (.ca), where the halves of a
// line that neighbouring rows share meet.  24 M edges, ten hops with a teleport term, us per hop, registers / shared memory:
// 16 columns 283 / 254, 64 columns 659 / 598, 128 columns 978 / 920.  The teleport term alone stays in registers (64 columns
// 586 / 608).
template <int EP>
struct EpilogueAhead {
    EpiloguePiece<EP>* at;  // this lane's own
    __device__ __forceinline__ void load(const Teleport& tp, int64_t row, int f0, int q, bool on) const {
        if (EP == kEpPlain || !on) return;
        if (EP == kEpTeleport || tp.alpha != 0.f || tp.zsum_first)
            copy_ahead(&at->x0, reinterpret_cast<const float4*>(tp.x0 + row * tp.ldx0 + f0) + q);
        if (EP == kEpSum && !tp.zsum_first) copy_ahead(&at->z[0], reinterpret_cast<const float4*>(tp.zsum + row * tp.ldz + f0) + q);
        if (EP == kEpSum && tp.xprev) copy_ahead(&at->z[1], reinterpret_cast<const float4*>(tp.xprev + row * tp.ldp + f0) + q);
    }
    __device__ __forceinline__ float4 finish(const float4& sum, float scale, const Teleport& tp, int64_t row, int f0, int q) const {
        wait_copies_ahead();
        return at->finish(sum, scale, tp, row, f0, q);
    }
};

// Both at once, for a row whose sum is already there.
template <int EP>
__device__ __forceinline__ float4 finish_row_piece(float4 sum, float scale, const Teleport& tp, int64_t row, int q) {
    EpiloguePiece<EP> piece;
    piece.load(tp, row, 0, q, true);
    return piece.finish(sum, scale, tp, row, 0, q);
}

// Which epilogue a launch needs.
inline int epilogue_of(const Teleport& tp) { return tp.zsum != nullptr ? kEpSum : tp.alpha != 0.f ? kEpTeleport : kEpPlain; }

struct SegArgs {
    const Segment* segs;
    int64_t seg_lo, seg_hi;
    const uint32_t* colx;
    int64_t colx_base;
    const float* x;
    int64_t ldx;
    float* out;
    int64_t ldo;
    float* scratch;
    int64_t scratch_ld;
    const float* rscale;
    const float* cscale;
    const float* rank_scale;  // row scales in rank order: rank_scale[k] = rscale[row of rank k]
    const int32_t* nzrows;
    int32_t num_ranks;  // rows that own an edge
    int32_t f4;         // float4 per row of this launch's columns
    int32_t tile_f4;    // float4 per row of one column tile (register kernel: tile blockIdx.y)
    bool back_to_back;  // see launch_dependent
    float diag_weight;  // GIN: 1 + eps
    Teleport tp;
};

// A float4 handled as two packed pairs: Blackwell adds and multiplies two fp32 per instruction
// (add/fma .f32x2).  Each lane of each pair is an ordinary IEEE operation, so results equal the scalar
// code's bit for bit.
struct Quad {
    float2 lo, hi;
};

__device__ __forceinline__ Quad quad_zero() { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }

__device__ __forceinline__ Quad quad_load(const unsigned char* p) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

__device__ __forceinline__ void quad_add(Quad& a, const Quad& x) {
    a.lo = __fadd2_rn(a.lo, x.lo);
    a.hi = __fadd2_rn(a.hi, x.hi);
}

// w holds the weight twice
__device__ __forceinline__ void quad_fma_pair(Quad& a, float2 w, const Quad& x) {
    a.lo = __ffma2_rn(w, x.lo, a.lo);
    a.hi = __ffma2_rn(w, x.hi, a.hi);
}

__device__ __forceinline__ void quad_fma(Quad& a, float w, const Quad& x) { quad_fma_pair(a, make_float2(w, w), x); }

// Bytes from one row to the next.  FAR: from 4 GB on (a narrow view of few, very long rows), where a gather needs more than
// one 32-bit multiply-add; those take kernels of their own, compiled for whole warps only.
template <bool FAR>
using RowStride = std::conditional_t<FAR, uint64_t, uint32_t>;
inline bool far_rows(int64_t ldx) { return ldx >= (int64_t)1 << 30; }

// float4 of row `col` through the read-only path; `base` points at this lane's piece of row 0
template <typename Stride>
__device__ __forceinline__ Quad quad_gather(const char* base, uint32_t col, Stride row_bytes) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(base + (uint64_t)col * row_bytes));
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

// Compensated addition of x into (sum, comp), as kahan1 does per component: a - b is evaluated as
// fma(-1, b, a), which rounds the same.
__device__ __forceinline__ void kahan_pair(float2& sum, float2& comp, const float2& x) {
    const float2 neg = make_float2(-1.f, -1.f);
    const float2 y = __ffma2_rn(neg, comp, x);
    const float2 t = __fadd2_rn(sum, y);
    comp = __ffma2_rn(neg, y, __ffma2_rn(neg, sum, t));
    sum = t;
}

__device__ __forceinline__ void quad_kahan(Quad& sum, Quad& comp, const Quad& x) {
    kahan_pair(sum.lo, comp.lo, x.lo);
    kahan_pair(sum.hi, comp.hi, x.hi);
}

// Programmatic dependent launch: the kernels of resident calls follow one another in a stream, and each is launched when
// the last CTA of the one before it has left, without waiting for that kernel's completion and the flush of its stores: what
// is hidden is the latency of launch and completion.  What a kernel reads of the plan's own tables it may read at once;
// wait_previous_kernel() comes before its first access to a matrix or to scratch rows and returns when the previous
// kernel has completed and its stores are visible; every thread of every kernel passes it, so the guarantee carries
// over to the kernels before that one.  It is a no-op in a kernel launched without the attribute, as the streamed
// schedules launch theirs: there copies on other streams bring the tables and matrices in.  No kernel asks for the
// next one early (griddepcontrol.launch_dependents): waiting CTAs beside working ones cost more than they save (4,096
// nodes, two hops: 16 columns 17.5 us with, 10.5 without; 64 columns 12.1 and 9.8; no difference on large graphs).
__device__ __forceinline__ void wait_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... Params, typename... Args>
int launch_dependent(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, bool overlap, cudaStream_t st,
                     Args&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap ? 1 : 0;
    GNNPRE_CUDA(cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...));
    return GNNPRE_OK;
}

// Compensated (Kahan) addition of x into the pair (sum, comp): the low-order bits that the addition
// drops are carried in comp.
__device__ __forceinline__ void kahan1(float& sum, float& comp, float x) {
    const float y = x - comp;
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

__device__ __forceinline__ void kahan4(float4& sum, float4& comp, const float4& x) {
    kahan1(sum.x, comp.x, x.x);
    kahan1(sum.y, comp.y, x.y);
    kahan1(sum.z, comp.z, x.z);
    kahan1(sum.w, comp.w, x.w);
}

constexpr int kThreads = 256;
// Register segment kernel: 14 CTAs of two warps per SM, i.e. 72 registers per thread.  Small CTAs, because segments
// differ in length and a finished warp's place should not wait for seven others.
constexpr int kSegThreads = 64;
#ifndef GNNPRE_SEG_BLOCKS
#define GNNPRE_SEG_BLOCKS 14
#endif
constexpr int kSegBlocks = GNNPRE_SEG_BLOCKS;
constexpr int kMaxDevices = 64;

