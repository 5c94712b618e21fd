// pair_common.cuh -- parameters, tile constants and device helpers shared by the pair
// kernel (pair.cuh) and the passes that prepare it (gbs.cu).
#pragma once

#include <math.h>

#include "gbt_internal.h"

namespace gbt {

constexpr int kWarpsFwd = 16;               // warps per CTA of the pair kernel (one CTA per SM)
constexpr size_t kSmemBudget = 227 * 1024;  // dynamic shared memory of one pair-kernel CTA (the maximum)
constexpr int kR = 2;                       // receivers per lane
constexpr int kWarpRecv = 32 * kR;          // receivers per warp tile
constexpr int kTileWarps = 15;              // warp tiles per CTA tile (dispatch order, lists)
constexpr int kChunkWords = 16;             // warp-tile words per 32-entry chunk of a tile list
constexpr int kCtaRecv = kTileWarps * kWarpRecv;
constexpr int kBatch = 32;                  // segments per staged batch
constexpr float kWinMargin = 0.01f;         // window slack of the ball tests and the prefilter (m)
constexpr int kGroupFreq = 8;               // most frequency slots of one pair launch

// Per-frequency constants.  The forward pass works in units of the beam parameter,
// s' = s / b, so that 1/E = (s' + i) / (b (1 + s'^2)): with r = n^2 / (1 + s'^2) the
// Gaussian exponent, the second phase term and the cutoff are r times a constant.  The
// adjoint and the counting pass work in metres (r = n^2 / (s^2 + b^2)).
struct alignas(16) FreqConst {
    float kb2;            // k b / 2  (kept iff kb2 n^2 <= C D, D = s^2 + b^2)
    float b2;             // b^2
    float K_hi, K_lo;     // f / c in turns per metre, float-float
    float hK;             // second phase term, hK r s turns: K / (2 b), adjoint K / 2
    float ne;             // Gaussian exponent ne r: -k / (2 b) log2(e), adjoint -k b / 2 log2(e)
    float rc;             // kept iff r <= rc: C b / (k / 2), adjoint C / (k b / 2)
    float invb;           // 1 / b
    float sA;             // adjoint amplitude k b / (8 pi^2) (forward: k / (8 pi^2), by the merge)
    float nal;            // exponent of the air absorption nal s: -a b log2(e), adjoint -a log2(e)
    float nkh;            // -k / 2 (adjoint)
    float b;              // b (adjoint)
};
static_assert(sizeof(FreqConst) == 48, "three 16-byte words");

struct alignas(16) FwdParams {
    const float *recv;
    const int32_t *order;
    int64_t n_recv;
    const int32_t *n_seg_ptr;
    const float *rec;          // AoS records, kRecFloats per segment
    const float4 *crec;        // cull records: (o_hi, s0_hi), (t_hi, L_hi) per segment
    int nf;
    int uniform_b;             // all b of the launch equal: frequencies sorted by k, loop stops at first cull
    int tile_cull;             // counting pass: skip segments that reach none of a warp's receivers
    float cutoff;
    float pre_alpha, pre_beta; // union cull: keep iff alpha n^2 <= s^2 + beta
    float kmax_turns;          // largest f / c of the launch's frequencies, turns per metre
    float s_scale;             // staged s is s times this: 1 / b when uniform and forward, else 1
    int splits;
    int64_t n_items;           // CTA tiles x splits x warp tiles (weighted: at most)
    // weighted splits: by dispatch rank (n_tiles + 1), the first tile-split of each CTA tile,
    // or null; partial is then [tile-split][nf][part_recv]
    const int32_t *item_off;
    int n_tiles, part_recv;
    int *work_counter;         // zero at launch (prepass); warps take items from it
    const int32_t *tile_perm;  // dispatch rank -> CTA tile (heaviest first), or null
    // tile pre-cull: per CTA tile, the segments whose beams can reach its receivers
    const int32_t *list;       // segment indices, each tile's in segment order, or null
    const int64_t *list_off;   // per tile: first entry in list
    const int32_t *list_n;     // per tile: entries, or -1 (no list: test every segment)
    // per 32-entry chunk of a tile's list (every list starts on a chunk boundary), one
    // word per warp tile w: bit b set if entry b of the chunk can reach warp tile w
    const uint32_t *list_words;
    float4 *partial;           // [splits][nf][n_recv], processing order: re_hi, im_hi, re_lo, im_lo
    unsigned long long *stats; // counting pass when non-null: [1] prefiltered, [2] kept
    unsigned int *status;      // device status word (timeouts)
    // adjoint mode
    const float2 *grad_out;    // g = dL/dRe p + i dL/dIm p, [user frequency][n_recv]
    float *seg_G;              // per segment: sum over (r, f) of Re(conj(g) c~)
    float *seg_H;              // per (sorted frequency, segment): sum over r of Re(conj(g) dc~/db)
    int64_t seg_stride;        // stride of seg_H rows
    int fperm[GBT_MAX_FREQ];   // sorted frequency slot -> user frequency index
    // losses of porous surfaces (lossy instantiation): per user frequency f and segment j,
    // seg_rf[f * rf_stride + j] = (log2 |R|, arg R / 2 pi) of the path's reflection factor
    const float2 *seg_rf;
    int64_t rf_stride;
    // batched launch: per-instance parameters and the first global item of each
    const struct FwdParams *inst;
    const int64_t *inst_off;   // n_inst + 1 entries
    int n_inst;
    FreqConst fc[kGroupFreq];
};

static_assert(sizeof(FwdParams) % 16 == 0, "instance parameters are copied as 16-byte words");

// Launchers of the pair kernel (pair_fwd.cu, pair_bwd.cu, pair_batched.cu).
void pair_fwd_launch(const FwdParams &p, int window, cudaStream_t s, bool timed);
void pair_unordered_launch(const FwdParams &p, int window, cudaStream_t s, bool timed);   // no lists, no order or few
void pair_bwd_launch(const FwdParams &p, int window, cudaStream_t s, bool timed);
void pair_field_launch(const FwdParams &p, int window, cudaStream_t s, bool timed);   // its forward
int pair_batched_prepare(int nf_max, int window);                  // resident CTAs per SM
void pair_batched_launch(const FwdParams &p, int nf_max, int window, int grid, cudaStream_t s);

namespace {

// Error-free transformations depend on every operation being rounded as written:
// nvcc contracts a product feeding an add into one FMA by default, which would
// round differently in each inlined copy.  The __f*_rn intrinsics are never
// contracted, so these sites use them wherever a rounding is relied upon.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bv = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bv)), __fsub_rn(b, bv));
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Kahan's difference of products a*b - c*d, accurate to about one ulp.
__device__ __forceinline__ float dop(float a, float b, float c, float d)
{
    const float w = __fmul_rn(c, d);
    const float e = fmaf(-c, d, w);
    const float f = fmaf(a, b, -w);
    return f + e;
}

typedef unsigned long long f2x;   // two packed floats (lo = receiver 0, hi = receiver 1)
__device__ __forceinline__ f2x pk(float a, float b)
{
    f2x r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f2x v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2x fma2(f2x a, f2x b, f2x c)
{
    f2x r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2x add2(f2x a, f2x b)
{
    f2x r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x sub2(f2x a, f2x b)
{
    f2x r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x mul2(f2x a, f2x b)
{
    f2x r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x neg2(f2x a) { return mul2(a, 0xbf800000bf800000ull); }
__device__ __forceinline__ f2x splat(float a) { return pk(a, a); }

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, int src_bytes)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem),
                 "r"(src_bytes));
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n"
                 ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bulk copy (TMA) of `bytes` contiguous bytes into shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

__device__ __forceinline__ unsigned int ordered_bits(float f)
{
    unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_ordered(unsigned int u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Whether a receiver takes part: its coordinates are finite and small enough for their squares
// to be FP32 numbers.  One that does not gets a zero field and leaves its neighbours alone: it
// stays out of the frames, balls and boxes of its warp and tile.
__device__ __forceinline__ bool takes_part(float x, float y, float z)
{
    return fabsf(x) < 1e18f && fabsf(y) < 1e18f && fabsf(z) < 1e18f;      // false for a NaN
}
// The warp's first receiver that takes part (part: per receiver of the lane; 0 when there is
// none), which is the frame of the float-float kernels.
__device__ __forceinline__ float3 first_receiver(const bool (&part)[kR], const float (&x)[kR],
                                                 const float (&y)[kR], const float (&z)[kR])
{
    static_assert(kR == 2, "two receivers per lane");
    const uint32_t m0 = __ballot_sync(0xffffffffu, part[0]), m1 = __ballot_sync(0xffffffffu, part[1]);
    const int k = m0 ? 0 : 1, src = (m0 | m1) ? __ffs(m0 ? m0 : m1) - 1 : 0;
    const bool any = (m0 | m1) != 0u;
    const float cx = __shfl_sync(0xffffffffu, k ? x[1] : x[0], src);
    const float cy = __shfl_sync(0xffffffffu, k ? y[1] : y[0], src);
    const float cz = __shfl_sync(0xffffffffu, k ? z[1] : z[0], src);
    return any ? make_float3(cx, cy, cz) : make_float3(0.f, 0.f, 0.f);
}

// Two values, each duplicated into both halves of a float pair.
__device__ __forceinline__ float4 dup2(float a, float b) { return make_float4(a, a, b, b); }

// ---- can a segment keep any receiver inside a ball?
// The distance from the segment's line to a point is 1-Lipschitz, so shrinking the ball
// centre's distance by the radius bounds n from below and |s| from above over the whole
// ball.  The radius carries slack for FP32 rounding at these magnitudes, split between the
// ball (a "reach ball": centre, W = r 1.0001 + 0.05 + 1e-5 (|cx| + |cy| + |cz|)) and the
// segment (1e-5 (|ox| + |oy| + |oz|)), so each (segment, ball) pair pays one add for it.
__device__ __forceinline__ float4 reach_ball(const float4 &b)
{
    return make_float4(b.x, b.y, b.z,
                       fmaf(b.w, 1.0001f, 0.05f) + 1e-5f * (fabsf(b.x) + fabsf(b.y) + fabsf(b.z)));
}
__device__ __forceinline__ float segment_slack(const float4 &r0)
{
    return 1e-5f * (fabsf(r0.x) + fabsf(r0.y) + fabsf(r0.z));
}

// A segment's terms of the test, formed once for all the balls it meets: with d = c - o,
// d.t = c.t - o.t and d x t = c x t - o x t, whose extra rounding (a few ulp of |c| and
// |o|) the slack's 1e-5 (|o| + |c|) far exceeds.
struct SegCull {
    float tx, ty, tz, len, s0;   // direction, length, start
    float ot, ox, oy, oz;        // o.t and o x t
    float slack;                 // the segment's share of the slack
};
__device__ __forceinline__ SegCull seg_cull(const float4 &r0, const float4 &r1)
{
    SegCull g;
    g.tx = r1.x; g.ty = r1.y; g.tz = r1.z; g.len = r1.w; g.s0 = r0.w;
    g.ot = fmaf(r0.x, r1.x, fmaf(r0.y, r1.y, r0.z * r1.z));
    g.ox = fmaf(r0.y, r1.z, -r0.z * r1.y);
    g.oy = fmaf(r0.z, r1.x, -r0.x * r1.z);
    g.oz = fmaf(r0.x, r1.y, -r0.y * r1.x);
    g.slack = segment_slack(r0);
    return g;
}
template <int WINDOW>
__device__ __forceinline__ bool seg_reaches_ball(const SegCull &g, const float4 &rb, float alpha,
                                                 float beta)
{
    const float sc = fmaf(rb.x, g.tx, fmaf(rb.y, g.ty, fmaf(rb.z, g.tz, -g.ot)));
    const float cxr = fmaf(rb.y, g.tz, fmaf(-rb.z, g.ty, -g.ox));
    const float cyr = fmaf(rb.z, g.tx, fmaf(-rb.x, g.tz, -g.oy));
    const float czr = fmaf(rb.x, g.ty, fmaf(-rb.y, g.tx, -g.oz));
    // |d x t| from below: the approximate square root is within a few ulp, and the factor
    // takes it under the exact root
    float nc;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(nc) : "f"(fmaf(cxr, cxr, fmaf(cyr, cyr, czr * czr))));
    nc *= 0.999999f;
    const float R = rb.w + g.slack;
    bool win;
    if (WINDOW == GBT_WINDOW_LINE) win = g.s0 + sc + R >= -kWinMargin;
    else win = (sc + R >= -kWinMargin) && (sc - R <= g.len + kWinMargin);
    const float sabs = fabsf(g.s0 + sc) + R;
    const float nn = nc - R;
    return win && (nn <= 0.f || alpha * nn * nn <= fmaf(sabs, sabs, beta));
}

}  // namespace
}  // namespace gbt
