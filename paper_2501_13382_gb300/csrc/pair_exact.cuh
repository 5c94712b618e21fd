// pair_exact.cuh -- the float-float geometry of one (receiver, segment) pair in its warp
// tile's frame, as the adjoint pair kernel (pair_bwd.cu) and the counting pass (gbs.cu)
// evaluate it, and the staging of segment batches both use.
#pragma once

#include "pair_common.cuh"

namespace gbt {
namespace {

constexpr int kWRaw = 2;                    // raw record buffers per warp (double buffering)
constexpr long long kSpinLimit = 1LL << 22; // bounded mbarrier waits

// Bounded wait: true when the phase of `parity` completed; false on abort or
// when the iteration limit ran out (then the device status word is flagged).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                          unsigned int *status)
{
    for (long long it = 0; it < kSpinLimit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
    }
    atomicOr(status, STATUS_TIMEOUT);
    *abort_flag = 1;
    return false;
}

// One staged batch of a warp: the prefilter (hot) view relative to the warp
// tile's first receiver c and the exact-path view in the same frame.  With
// d = c - o (float-float) the exact view holds, per segment, A = d.t and
// S = s0 + A as float-float pairs, AL = A - L (the segment window), the
// compensated N = d x t and the direction as (hi, lo), so that for a receiver
// at x = c + x' the pair needs only x'.t and x' x t:
//   s_loc = A + x'.t,  s = S + x'.t,  n = N + x' x t.
struct StageSmem {
    float4 O[kBatch];               // o' = o - c, s0_hi (per-warp ball test)
    // prefilter constants, each duplicated into both halves of a float pair:
    // P[0] = t_z, -o'.t;  P[1..2] = 2a o'_x, 2a o'_y, 2a o'_z, beta - a |o'|^2;
    // P[3] = s0 + margin, L + margin;  P[4] = t_x, t_y
    float4 P[kBatch][5];
    // exact view, two values per word, each in both halves of a float pair; component-major,
    // so lanes loading different segments hit different banks:
    // D[0] t_hi.x, t_hi.y | D[1] t_hi.z, S_hi | D[2] t_lo.x, t_lo.y | D[3] t_lo.z, S_lo
    // D[4] N.x, N.y | D[5] N.z, W Gamma_path | D[6] A_hi, A_lo | D[7] AL_hi, AL_lo
    float4 D[8][kBatch];
    int32_t seg[kBatch];            // global segment index of each staged record
};

// Exact geometry of one (receiver, segment) pair in the warp tile's frame, in
// float-float: x' = (xh + xl) exactly; returns false when the pair falls outside
// the window.  `fast`: the warp item's choice of the FP32 local projection, within eps
// of x'.t; a pair within eps of an end of its window is decided and evaluated with the
// float-float projection instead, so the window test is as exact as on that path.
template <int WINDOW>
__device__ __forceinline__ bool frame_geometry(float xh, float yh, float zh, float xl, float yl,
                                               float zl, const StageSmem &w, int j, bool fast,
                                               float eps, float &sh, float &sl, float &n2)
{
    const float4 d0 = w.D[0][j], d1 = w.D[1][j], d2 = w.D[2][j], d3 = w.D[3][j];
    const float4 d4 = w.D[4][j], d5 = w.D[5][j];
    const float4 T = make_float4(d0.x, d0.z, d1.x, d1.z), TL = make_float4(d2.x, d2.z, d3.x, d3.z);
    const float4 NN = make_float4(d4.x, d4.z, d5.x, d5.z);
    // u = x'.t as (U + ul)
    float U, ul;
    auto exact_u = [&]() {
        const float p0 = __fmul_rn(xh, T.x), p1 = __fmul_rn(yh, T.y), p2 = __fmul_rn(zh, T.z);
        const float r0 = fmaf(xh, TL.x, fmaf(xl, T.x, fmaf(xh, T.x, -p0)));
        const float r1 = fmaf(yh, TL.y, fmaf(yl, T.y, fmaf(yh, T.y, -p1)));
        const float r2 = fmaf(zh, TL.z, fmaf(zl, T.z, fmaf(zh, T.z, -p2)));
        float S1, E1, E2;
        two_sum(p0, p1, S1, E1);
        two_sum(S1, p2, U, E2);
        ul = __fadd_rn(__fadd_rn(E1, E2), __fadd_rn(__fadd_rn(r0, r1), r2));
    };
    if (fast) {
        U = fmaf(xh, T.x, fmaf(yh, T.y, __fmul_rn(zh, T.z)));
        ul = fmaf(xl, T.x, fmaf(yl, T.y, fmaf(zl, T.z, fmaf(xh, TL.x, fmaf(yh, TL.y, __fmul_rn(zh, TL.z))))));
    } else {
        exact_u();
    }
    if (WINDOW == GBT_WINDOW_SEGMENT) {
        const float4 d6 = w.D[6][j], d7 = w.D[7][j];
        float wa = __fadd_rn(__fadd_rn(d6.x, U), __fadd_rn(d6.z, ul));
        float wb = __fadd_rn(__fadd_rn(d7.x, U), __fadd_rn(d7.z, ul));
        if (fast && fminf(fabsf(wa), fabsf(wb)) <= eps) {
            fast = false;
            exact_u();
            wa = __fadd_rn(__fadd_rn(d6.x, U), __fadd_rn(d6.z, ul));
            wb = __fadd_rn(__fadd_rn(d7.x, U), __fadd_rn(d7.z, ul));
        }
        if (!(wa >= 0.0f)) return false;
        if (!(wb < 0.0f)) return false;
    }
    float e3;
    two_sum(T.w, U, sh, e3);
    sl = __fadd_rn(e3, __fadd_rn(ul, TL.w));
    if (WINDOW == GBT_WINDOW_LINE) {
        float ss = __fadd_rn(sh, sl);
        if (fast && fabsf(ss) <= eps) {
            fast = false;
            exact_u();
            two_sum(T.w, U, sh, e3);
            sl = __fadd_rn(e3, __fadd_rn(ul, TL.w));
            ss = __fadd_rn(sh, sl);
        }
        if (!(ss >= 0.0f)) return false;
    }
    // n = N + x' x t: the small terms first (float-float projection only), then the
    // main products
    float n0x = NN.x, n0y = NN.y, n0z = NN.z;
    if (!fast) {
        n0x = __fadd_rn(n0x, fmaf(yl, T.z, fmaf(-zl, T.y, fmaf(yh, TL.z, __fmul_rn(-zh, TL.y)))));
        n0y = __fadd_rn(n0y, fmaf(zl, T.x, fmaf(-xl, T.z, fmaf(zh, TL.x, __fmul_rn(-xh, TL.z)))));
        n0z = __fadd_rn(n0z, fmaf(xl, T.y, fmaf(-yl, T.x, fmaf(xh, TL.y, __fmul_rn(-yh, TL.x)))));
    }
    const float nx = fmaf(yh, T.z, fmaf(-zh, T.y, n0x));
    const float ny = fmaf(zh, T.x, fmaf(-xh, T.z, n0y));
    const float nz = fmaf(xh, T.y, fmaf(-yh, T.x, n0z));
    n2 = fmaf(nx, nx, fmaf(ny, ny, __fmul_rn(nz, nz)));
    return true;
}

// Conservative test: can the segment (origin (ox, oy, oz) relative to the frame
// of `sphere`, record words r0 / r1) keep any receiver inside the ball `sphere`
// (centre xyz, radius w)?  The distance from the segment line to a point is
// 1-Lipschitz, so shrinking the ball's centre distance by the radius bounds n
// from below and |s| from above over the whole ball; the radius carries slack
// for FP32 rounding at these magnitudes.
template <int WINDOW>
__device__ __forceinline__ bool ball_may_keep(const float4 &r0, const float4 &r1, float ox, float oy,
                                              float oz, const float4 &sphere, float alpha, float beta)
{
    const float dx = sphere.x - ox, dy = sphere.y - oy, dz = sphere.z - oz;
    const float sc = fmaf(dx, r1.x, fmaf(dy, r1.y, dz * r1.z));
    const float cxr = dy * r1.z - dz * r1.y, cyr = dz * r1.x - dx * r1.z, czr = dx * r1.y - dy * r1.x;
    // |d x t| from below: the approximate square root is within a few ulp, and the
    // factor takes it under the exact root
    float nc;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(nc) : "f"(fmaf(cxr, cxr, fmaf(cyr, cyr, czr * czr))));
    nc *= 0.999999f;
    const float R = sphere.w * 1.0001f + 0.05f + 1e-5f * (fabsf(ox) + fabsf(oy) + fabsf(oz));
    bool win;
    if (WINDOW == GBT_WINDOW_LINE) win = r0.w + sc + R >= -kWinMargin;
    else win = (sc + R >= -kWinMargin) && (sc - R <= r1.w + kWinMargin);
    const float sabs = fabsf(r0.w + sc) + R;
    const float nn = nc - R;
    return win && (nn <= 0.f || alpha * nn * nn <= fmaf(sabs, sabs, beta));
}

// Stage lane's raw record for the warp: the prefilter view relative to the frame
// c = (cx, cy, cz) (the warp tile's first receiver), the origin in that frame for the
// per-warp ball test and the direction.  A record past the segment count becomes one no
// receiver can keep.  Returns L_hi.
__device__ __forceinline__ float stage_batch(StageSmem &w, const float4 (&raw)[kRecFloats / 4],
                                             int lane, bool valid, int32_t seg, float cx,
                                             float cy, float cz, float alpha, float beta)
{
    const float4 r0 = raw[0], r1 = raw[1], r2 = raw[2];
    float4 *P = w.P[lane];
    w.seg[lane] = valid ? seg : -1;
    if (valid) {
        const float ox = (r0.x - cx) + r2.x, oy = (r0.y - cy) + r2.y, oz = (r0.z - cz) + r2.z;
        w.O[lane] = make_float4(ox, oy, oz, r0.w);
        const float ot = fmaf(ox, r1.x, fmaf(oy, r1.y, oz * r1.z));
        const float oo = fmaf(ox, ox, fmaf(oy, oy, oz * oz));
        const float a2 = 2.f * alpha;
        w.D[0][lane] = dup2(r1.x, r1.y);
        P[4] = dup2(r1.x, r1.y);
        P[0] = dup2(r1.z, -ot);
        P[1] = dup2(a2 * ox, a2 * oy);
        P[2] = dup2(a2 * oz, fmaf(-alpha, oo, beta));
        P[3] = dup2(r0.w + kWinMargin, r1.w + kWinMargin);
    } else {
        // far behind its own start
        w.O[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        w.D[0][lane] = dup2(0.f, 0.f);
        P[4] = dup2(0.f, 0.f);
        P[0] = dup2(0.f, -1e15f);
        P[1] = dup2(0.f, 0.f);
        P[2] = dup2(0.f, 0.f);
        P[3] = dup2(0.f, 0.f);
    }
    return valid ? r1.w : 0.f;
}

// Stage lane's raw record's exact-path view in the warp's frame: float-float
// d = c - o, A = d.t, S = s0 + A, AL = A - L and the compensated N = d x t, with the
// direction as (hi, lo) and the amplitude; finite values past the segment count.
__device__ __forceinline__ void stage_exact(StageSmem &w, const float4 (&raw)[kRecFloats / 4],
                                            int lane, bool valid, float cx, float cy, float cz)
{
    const float4 r0 = raw[0], r1 = raw[1], r2 = raw[2], r3 = raw[3], r4 = raw[4];
    if (valid) {
        // d = c - o as (dh + dl)
        float dxh, dxe, dyh, dye, dzh, dze;
        two_sum(cx, -r0.x, dxh, dxe);
        two_sum(cy, -r0.y, dyh, dye);
        two_sum(cz, -r0.z, dzh, dze);
        const float dxl = __fsub_rn(dxe, r2.x), dyl = __fsub_rn(dye, r2.y), dzl = __fsub_rn(dze, r2.z);
        // A = d.t, float-float
        const float q0 = __fmul_rn(dxh, r1.x), q1 = __fmul_rn(dyh, r1.y), q2 = __fmul_rn(dzh, r1.z);
        const float e0 = fmaf(dxh, r3.x, fmaf(dxl, r1.x, fmaf(dxh, r1.x, -q0)));
        const float e1 = fmaf(dyh, r3.y, fmaf(dyl, r1.y, fmaf(dyh, r1.y, -q1)));
        const float e2 = fmaf(dzh, r3.z, fmaf(dzl, r1.z, fmaf(dzh, r1.z, -q2)));
        float S1, E1, Ah, E2;
        two_sum(q0, q1, S1, E1);
        two_sum(S1, q2, Ah, E2);
        const float Al = __fadd_rn(__fadd_rn(E1, E2), __fadd_rn(__fadd_rn(e0, e1), e2));
        // S = s0 + A, AL = A - L
        float Sh, es, ALh, ea;
        two_sum(r0.w, Ah, Sh, es);
        const float Sl = __fadd_rn(es, __fadd_rn(Al, r2.w));
        two_sum(Ah, -r1.w, ALh, ea);
        const float ALl = __fadd_rn(ea, __fsub_rn(Al, r3.w));
        // N = d x t, compensated
        const float nx = dop(dyh, r1.z, dzh, r1.y) +
                         fmaf(dyh, r3.z, fmaf(-dzh, r3.y, fmaf(dyl, r1.z, -dzl * r1.y)));
        const float ny = dop(dzh, r1.x, dxh, r1.z) +
                         fmaf(dzh, r3.x, fmaf(-dxh, r3.z, fmaf(dzl, r1.x, -dxl * r1.z)));
        const float nz = dop(dxh, r1.y, dyh, r1.x) +
                         fmaf(dxh, r3.y, fmaf(-dyh, r3.x, fmaf(dxl, r1.y, -dyl * r1.x)));
        w.D[1][lane] = dup2(r1.z, Sh);
        w.D[2][lane] = dup2(r3.x, r3.y);
        w.D[3][lane] = dup2(r3.z, Sl);
        w.D[4][lane] = dup2(nx, ny);
        w.D[5][lane] = dup2(nz, r4.x);
        w.D[6][lane] = dup2(Ah, Al);
        w.D[7][lane] = dup2(ALh, ALl);
    } else {
        w.D[1][lane] = dup2(0.f, -1e15f);
        w.D[2][lane] = dup2(0.f, 0.f);
        w.D[3][lane] = dup2(0.f, 0.f);
        w.D[4][lane] = dup2(0.f, 0.f);
        w.D[5][lane] = dup2(0.f, 0.f);
        w.D[6][lane] = dup2(-1e15f, 0.f);
        w.D[7][lane] = dup2(-1e15f, 0.f);
    }
}

}  // namespace
}  // namespace gbt
