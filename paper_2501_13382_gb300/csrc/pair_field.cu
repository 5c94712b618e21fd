// pair_field.cu -- the forward sum that the adjoint differentiates (gbt_sum_differentiable).
//
// A least-squares gradient depends on the field's rounding, so this kernel evaluates each
// beam as the adjoint kernel (pair_bwd.cu) does, operation for operation.  Without lists its
// FP32 sums fold every 16 chunks of all segments, whichever of them reach the warp; with lists
// every 16 batches of the tile's own entries, and splits stride chunks of the list.  So a call
// repeats to the bit, and the two forms differ by the rounding of regrouped sums.
//
// Same items and gathering as the forward kernel of pair.cuh: a warp goes through the
// segments whose beams reach its ball.  Each is evaluated for the lane's two receivers in
// paired FP32, in the frame of the warp tile's first receiver c: with d = c - o the staging
// holds A = d.t, S = s0 + A and A - L as float-float pairs and the compensated N = d x t, so
// a receiver at x = c + x' needs u = x'.t and x' x t.  Where the warp is compact for its
// highest band (K max|x'| <= 90 turns) u is FP32, except for a receiver within that
// projection's error bound of an end of its window, which takes the float-float one.
#include "pair_stream.cuh"

namespace gbt {
namespace {

constexpr float kFastTurnsField = 90.0f;   // K max|x'| up to which u is plain FP32
// A segment whose union cutoff radius at the tile is under this many times the ball's radius
// may reach few of its receivers: the paired prefilter (15 instructions per segment) runs
// first and a segment it clears for every lane costs nothing more.  A training step of 131,072
// rays x 4,000 scattered receivers x 4 bands with the line at 0.7, 1, 2, 100: 9.18, 8.54, 8.43,
// 8.42 ms; x 64^2 receivers on a grid 3.92, 3.89, 3.89, 3.89.
constexpr float kSmallBeam = 2.0f;
// Receivers without an order and without lists: where most of a batch's segments are small, every
// receiver evaluates its own candidates, a segment of its own to each lane and half (30,000-ray
// city x 4,000 scattered x 4 bands 1.50 ms with one segment for the warp, 1.10 so; the same bits).
// A kernel of its own, since its registers cost the others.

template <int NF>
struct FieldBuf {
    RawBuf in;
    // every value in both halves of a float pair:
    // D[0] t_hi.x, t_hi.y | D[1] t_hi.z, S_hi | D[2] t_lo.x, t_lo.y | D[3] t_lo.z, S_lo
    // D[4] N.x, N.y | D[5] N.z, W Gamma_path | D[6] A_hi, A_lo | D[7] AL_hi, AL_lo (AL = A - L)
    float4 D[8][kBatch];
    // prefilter: P[0] = t_z, -o'.t;  P[1..2] = 2a o'_x, 2a o'_y, 2a o'_z, beta - a |o'|^2;
    // P[3] = s0 + margin, L + margin  (o' = o - c; t_x, t_y from D[0])
    float4 P[4][kBatch];
    float2 rf[NF][kBatch];     // losses: log2 |R|, arg R / 2 pi
    int32_t seg[kBatch];       // segment index of each staged record
};

struct FieldRecv {               // x' = (X + XL) exactly, and -X
    f2x X, Y, Z, XL, YL, ZL, NX, NY, NZ;
};

// two_sum on both halves; the paired operations round each half exactly like the scalar ones
__device__ __forceinline__ void two_sum2(f2x a, f2x b, f2x &s, f2x &e)
{
    s = add2(a, b);
    const f2x bv = sub2(s, a);
    e = add2(sub2(a, sub2(s, bv)), sub2(b, bv));
}
__device__ __forceinline__ f2x rint2(f2x a)
{
    float x, y;
    upk(a, x, y);
    return pk(rintf(x), rintf(y));
}
__device__ __forceinline__ f2x sel2(bool b0, bool b1, f2x a, f2x b)   // per half a or b
{
    float a0, a1, c0, c1;
    upk(a, a0, a1);
    upk(b, c0, c1);
    return pk(b0 ? a0 : c0, b1 ? a1 : c1);
}

// Stages lane's raw record in the frame c.  Returns whether the segment's union cutoff
// radius is small against the ball of radius rad (kSmallBeam).
template <int NF, bool LOSSY>
__device__ __forceinline__ bool stage_field(const FwdParams &p, FieldBuf<NF> &w, int lane,
                                              const float4 &r0, const float4 &r1, const float4 &r2,
                                              const float4 &r3, float amp, int32_t seg, float cx,
                                              float cy, float cz, float rad)
{
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
    w.D[0][lane] = dup2(r1.x, r1.y);
    w.D[1][lane] = dup2(r1.z, Sh);
    w.D[2][lane] = dup2(r3.x, r3.y);
    w.D[3][lane] = dup2(r3.z, Sl);
    w.D[4][lane] = dup2(nx, ny);
    w.D[5][lane] = dup2(nz, amp);
    w.D[6][lane] = dup2(Ah, Al);
    w.D[7][lane] = dup2(ALh, ALl);
    w.seg[lane] = seg;
    if (LOSSY) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            if (f >= p.nf) break;
            w.rf[f][lane] = p.seg_rf[(int64_t)p.fperm[f] * p.rf_stride + seg];
        }
    }
    const float smax = fabsf(Sh) + 2.0f * rad;
    const bool small = fmaf(smax, smax, p.pre_beta) < kSmallBeam * kSmallBeam * p.pre_alpha * rad * rad;
    if (small) {
        const float ox = (r0.x - cx) + r2.x, oy = (r0.y - cy) + r2.y, oz = (r0.z - cz) + r2.z;
        const float ot = fmaf(ox, r1.x, fmaf(oy, r1.y, oz * r1.z));
        const float oo = fmaf(ox, ox, fmaf(oy, oy, oz * oz));
        const float a2 = 2.f * p.pre_alpha;
        w.P[0][lane] = dup2(r1.z, -ot);
        w.P[1][lane] = dup2(a2 * ox, a2 * oy);
        w.P[2][lane] = dup2(a2 * oz, fmaf(-p.pre_alpha, oo, p.pre_beta));
        w.P[3][lane] = dup2(r0.w + kWinMargin, r1.w + kWinMargin);
    }
    return small;
}

// Whether the staged segment j may keep a beam at one of the lane's receivers (conservative,
// frequency independent):
//   s_loc = x'.t - o'.t,  sm = s_loc + s0 + margin,
//   g = sm^2 + beta - alpha |x' - o'|^2 + alpha s_loc^2  (= q - alpha n^2) >= 0, window.
template <int NF, int WINDOW>
__device__ __forceinline__ void may_keep(const FieldBuf<NF> &w, int j, const FieldRecv &x, f2x NAXX,
                                         f2x AL2, bool &k0, bool &k1)
{
    f2x TX, TY, TZ, OT, OX, OY, OZ, C7, S0, LM;
    staged<false>(w.D[0], j, j, TX, TY);
    staged<false>(w.P[0], j, j, TZ, OT);
    staged<false>(w.P[1], j, j, OX, OY);
    staged<false>(w.P[2], j, j, OZ, C7);
    staged<false>(w.P[3], j, j, S0, LM);
    const f2x sl = fma2(x.X, TX, fma2(x.Y, TY, fma2(x.Z, TZ, OT)));
    const f2x sm = add2(sl, S0);
    const f2x nd = fma2(x.X, OX, fma2(x.Y, OY, fma2(x.Z, OZ, add2(NAXX, C7))));
    const f2x g = fma2(mul2(sl, AL2), sl, fma2(sm, sm, nd));
    float g0, g1, a0, a1;
    upk(g, g0, g1);
    k0 = g0 >= 0.f;
    k1 = g1 >= 0.f;
    if (WINDOW == GBT_WINDOW_LINE) {
        upk(sm, a0, a1);
        k0 = k0 && a0 >= 0.f;
        k1 = k1 && a1 >= 0.f;
        return;
    }
    float b0, b1;
    upk(add2(sl, splat(kWinMargin)), a0, a1);
    upk(sub2(sl, LM), b0, b1);
    k0 = k0 && a0 >= 0.f && b0 < 0.f;
    k1 = k1 && a1 >= 0.f && b1 < 0.f;
}

// Exact geometry of the staged segment j (EACH: and j1 for the second) and the lane's two
// receivers: s = (s + sl), n^2, and which receivers (of v0, v1) lie in the window.
template <int NF, int WINDOW, bool EACH>
__device__ __forceinline__ void field_geometry(const FieldBuf<NF> &w, int j, int j1, const FieldRecv &x,
                                             bool v0, bool v1, bool fast, float eps, f2x &s, f2x &sl, f2x &n2,
                                             f2x &amp, bool &k0, bool &k1)
{
    auto word = [&](int d, f2x &a, f2x &b) { staged<EACH>(w.D[d], j, j1, a, b); };
    f2x TX, TY, TZ, S, TLX, TLY, TLZ, SL, NX, NY, NZ, AH, AL, BH, BL;
    word(0, TX, TY);
    word(1, TZ, S);
    word(2, TLX, TLY);
    word(3, TLZ, SL);
    word(6, AH, AL);
    word(7, BH, BL);
    // u = x'.t as (U + ul)
    f2x U, ul;
    auto exact_u = [&](f2x &u, f2x &l) {
        const f2x p0 = mul2(x.X, TX), p1 = mul2(x.Y, TY), p2 = mul2(x.Z, TZ);
        const f2x r0 = fma2(x.X, TLX, fma2(x.XL, TX, fma2(x.X, TX, neg2(p0))));
        const f2x r1 = fma2(x.Y, TLY, fma2(x.YL, TY, fma2(x.Y, TY, neg2(p1))));
        const f2x r2 = fma2(x.Z, TLZ, fma2(x.ZL, TZ, fma2(x.Z, TZ, neg2(p2))));
        f2x S1, E1, E2;
        two_sum2(p0, p1, S1, E1);
        two_sum2(S1, p2, u, E2);
        l = add2(add2(E1, E2), add2(add2(r0, r1), r2));
    };
    bool x0 = !fast, x1 = !fast;    // receivers on the float-float projection
    float a0, a1, b0, b1;
    auto ends = [&](f2x hi, f2x lo, float &q0, float &q1) { upk(add2(add2(hi, U), add2(lo, ul)), q0, q1); };
    if (fast) {
        U = fma2(x.X, TX, fma2(x.Y, TY, mul2(x.Z, TZ)));
        ul = fma2(x.XL, TX, fma2(x.YL, TY, fma2(x.ZL, TZ,
             fma2(x.X, TLX, fma2(x.Y, TLY, mul2(x.Z, TLZ))))));
        if (WINDOW == GBT_WINDOW_SEGMENT) {
            ends(AH, AL, a0, a1);
            ends(BH, BL, b0, b1);
            x0 = fminf(fabsf(a0), fabsf(b0)) <= eps;
            x1 = fminf(fabsf(a1), fabsf(b1)) <= eps;
        } else {
            f2x q, e;
            two_sum2(S, U, q, e);
            upk(add2(q, add2(e, add2(ul, SL))), a0, a1);
            x0 = fabsf(a0) <= eps;
            x1 = fabsf(a1) <= eps;
        }
        if (x0 || x1) {
            f2x ue, le;
            exact_u(ue, le);
            U = sel2(x0, x1, ue, U);
            ul = sel2(x0, x1, le, ul);
        }
    } else {
        exact_u(U, ul);
    }
    k0 = v0;
    k1 = v1;
    if (WINDOW == GBT_WINDOW_SEGMENT) {
        ends(AH, AL, a0, a1);
        ends(BH, BL, b0, b1);
        k0 = k0 && a0 >= 0.0f && b0 < 0.0f;
        k1 = k1 && a1 >= 0.0f && b1 < 0.0f;
    }
    f2x e3;
    two_sum2(S, U, s, e3);
    sl = add2(e3, add2(ul, SL));
    if (WINDOW == GBT_WINDOW_LINE) {
        upk(add2(s, sl), a0, a1);
        k0 = k0 && a0 >= 0.0f;
        k1 = k1 && a1 >= 0.0f;
    }
    word(4, NX, NY);
    word(5, NZ, amp);
    // n = N + x' x t; the lo parts' products only with the float-float projection
    if (x0 || x1) {
        const f2x mx = add2(NX, fma2(x.YL, TZ, fma2(neg2(x.ZL), TY, fma2(x.Y, TLZ, mul2(x.NZ, TLY)))));
        const f2x my = add2(NY, fma2(x.ZL, TX, fma2(neg2(x.XL), TZ, fma2(x.Z, TLX, mul2(x.NX, TLZ)))));
        const f2x mz = add2(NZ, fma2(x.XL, TY, fma2(neg2(x.YL), TX, fma2(x.X, TLY, mul2(x.NY, TLX)))));
        NX = sel2(x0, x1, mx, NX);
        NY = sel2(x0, x1, my, NY);
        NZ = sel2(x0, x1, mz, NZ);
    }
    const f2x nx = fma2(x.Y, TZ, fma2(x.NZ, TY, NX));
    const f2x ny = fma2(x.Z, TX, fma2(x.NX, TZ, NY));
    const f2x nz = fma2(x.X, TY, fma2(x.NY, TX, NZ));
    n2 = fma2(nx, nx, fma2(ny, ny, mul2(nz, nz)));
}

// Phase of one band's beam in turns, reduced to [-1/2, 1/2]: K s mod 1 from float-float
// products plus the second term K n^2 s / (2 D) and the reflections' phase rph.
template <bool LOSSY>
__device__ __forceinline__ f2x beam_turns(const FreqConst &c, f2x s, f2x sl, f2x n2invD, f2x rph)
{
    const f2x KH = splat(c.K_hi);
    const f2x nph = mul2(splat(-c.K_hi), s);           // -K_hi s, rounded; pe its exact error
    const f2x pe = fma2(KH, s, nph);
    const f2x corr = fma2(KH, sl, fma2(splat(c.K_lo), s, pe));
    f2x tau = add2(sub2(rint2(nph), nph), corr);       // = ph - rint(ph) + corr
    tau = fma2(mul2(splat(c.hK), n2invD), s, tau);
    if (LOSSY) tau = add2(tau, rph);
    // |tau| < 2^22 turns (beyond it FP32 holds no phase): round by 1.5 x 2^23
    return sub2(tau, sub2(add2(tau, splat(12582912.0f)), splat(12582912.0f)));
}
__device__ __forceinline__ void sincos_turns(f2x tau, f2x &sn, f2x &cs)
{
    float t0, t1, sn0, cs0, sn1, cs1;
    upk(mul2(splat(6.283185307179586f), tau), t0, t1);
    __sincosf(t0, &sn0, &cs0);
    __sincosf(t1, &sn1, &cs1);
    sn = pk(sn0, sn1);
    cs = pk(cs0, cs1);
}

// Adds the beams of the staged segment j (EACH: and j1 for the second) to the lane's receivers'
// sums per band.
template <int NF, int WINDOW, bool LOSSY, bool EACH>
__device__ __forceinline__ void eval_field(const FwdParams &p, const FieldBuf<NF> &w, int j, int j1,
                                           const FieldRecv &x, bool v0, bool v1, bool fast, float eps,
                                           f2x (&ax)[NF], f2x (&ay)[NF])
{
    f2x s, sl, n2, amp;
    bool k0, k1;
    field_geometry<NF, WINDOW, EACH>(w, j, j1, x, v0, v1, fast, eps, s, sl, n2, amp, k0, k1);
    f2x invD, n2invD;
    float d0 = 1.f, d1 = 1.f, n20, n21, r0 = 0.f, r1 = 0.f;
    upk(n2, n20, n21);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (NF > 1 && f >= p.nf) break;
        const FreqConst &c = p.fc[f];
        if (f == 0 || !p.uniform_b) {
            upk(fma2(s, s, splat(c.b2)), d0, d1);
            invD = pk(rcp_approx(d0), rcp_approx(d1));
            n2invD = mul2(n2, invD);
            upk(n2invD, r0, r1);
        }
        const bool m0 = k0 && (p.uniform_b ? !(c.kb2 * r0 > p.cutoff) : !(c.kb2 * n20 > p.cutoff * d0));
        const bool m1 = k1 && (p.uniform_b ? !(c.kb2 * r1 > p.cutoff) : !(c.kb2 * n21 > p.cutoff * d1));
        if (!__any_sync(0xffffffffu, m0 || m1)) {
            if (NF == 1 || p.uniform_b) break;
            continue;
        }
        f2x ex = mul2(splat(c.ne), n2invD), RPH = 0ull;
        if (LOSSY) {
            const float2 ra = w.rf[f][j], rb = EACH ? w.rf[f][j1] : ra;
            ex = fma2(splat(c.nal), s, add2(ex, pk(ra.x, rb.x)));
            RPH = pk(ra.y, rb.y);
        }
        float e0, e1;
        upk(ex, e0, e1);
        const f2x ga = pk(m0 ? ex2_approx(e0) : 0.0f, m1 ? ex2_approx(e1) : 0.0f);
        f2x SN, CS;
        sincos_turns(beam_turns<LOSSY>(c, s, sl, n2invD, RPH), SN, CS);
        const f2x g = mul2(mul2(mul2(splat(c.sA), amp), ga), invD);
        ax[f] = fma2(g, fma2(s, CS, mul2(splat(-c.b), SN)), ax[f]);
        ay[f] = fma2(g, fma2(s, SN, mul2(splat(c.b), CS)), ay[f]);
    }
}

// The FP32 sums fold into the item's float-float partials every kFoldEvery batches of list
// entries, or without a list every kFoldEvery chunks of all segments.
template <int NF, int WINDOW, bool LOSSY, bool UNORDERED>
__global__ void __maxnreg__(128) gbs_field_kernel(const __grid_constant__ FwdParams p)
{
    using Cfg = PairCfg<FieldBuf<NF>, false>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    FieldBuf<NF> &B = *reinterpret_cast<FieldBuf<NF> *>(smem_raw + (size_t)warp * Cfg::kPerWarp);

    for (;;) {
        int64_t it = 0;
        if (lane == 0) it = atomicAdd(p.work_counter, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= p.n_items) break;
        Item item;
        if (!decode_item(p, it, item)) continue;

        // receiver k of the lane (lane and lane + 32 of the warp tile) at x = c + x',
        // x' = (xp + xl) exactly
        float xr[kR], yr[kR], zr[kR], xp[kR], yp[kR], zp[kR], xl[kR], yl[kR], zl[kR], xx[kR];
        bool part[kR];
        unsigned bb[6] = {~0u, ~0u, ~0u, 0u, 0u, 0u};
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            const int64_t r = item.wbase + (int64_t)k * 32 + lane;
            part[k] = false;
            xr[k] = yr[k] = zr[k] = xp[k] = yp[k] = zp[k] = xl[k] = yl[k] = zl[k] = xx[k] = 0.0f;
            if (r < p.n_recv) {
                const int64_t o = p.order ? p.order[r] : r;
                xr[k] = p.recv[3 * o]; yr[k] = p.recv[3 * o + 1]; zr[k] = p.recv[3 * o + 2];
                part[k] = takes_part(xr[k], yr[k], zr[k]);
                if (!part[k]) no_partials(p, item, 32 * k + lane);
            }
        }
        // frame of the staged batches: the warp tile's first receiver
        const float3 c0 = first_receiver(part, xr, yr, zr);
        const float cx = c0.x, cy = c0.y, cz = c0.z;
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            if (part[k]) {
                two_sum(xr[k], -cx, xp[k], xl[k]);
                two_sum(yr[k], -cy, yp[k], yl[k]);
                two_sum(zr[k], -cz, zp[k], zl[k]);
                xx[k] = fmaf(xp[k], xp[k], fmaf(yp[k], yp[k], zp[k] * zp[k]));
                const unsigned ux = ordered_bits(xr[k]), uy = ordered_bits(yr[k]), uz = ordered_bits(zr[k]);
                bb[0] = min(bb[0], ux); bb[1] = min(bb[1], uy); bb[2] = min(bb[2], uz);
                bb[3] = max(bb[3], ux); bb[4] = max(bb[4], uy); bb[5] = max(bb[5], uz);
            }
        }
        // ball of the warp tile: about the centre of its bounding box
        float ctr[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            ctr[a] = 0.5f * from_ordered(__reduce_min_sync(0xffffffffu, bb[a])) +
                     0.5f * from_ordered(__reduce_max_sync(0xffffffffu, bb[3 + a]));
        float q2 = 0.0f;
#pragma unroll
        for (int k = 0; k < kR; ++k)
            if (part[k]) {
                const float ex = xr[k] - ctr[0], ey = yr[k] - ctr[1], ez = zr[k] - ctr[2];
                q2 = fmaxf(q2, fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
            }
        const float rad = 1.000001f * sqrtf(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(q2))));
        const float4 rball = reach_ball(make_float4(ctr[0], ctr[1], ctr[2], rad));
        // the FP32 local projection when the warp is compact for its bands; its error bound:
        // the three-term FP32 dot product with |t| = 1 is within about 3 x 2^-24 max|x'| of
        // x'.t, and eps is over five times that
        const float xmax = sqrtf(__uint_as_float(
            __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(xx[0], xx[1])))));
        const bool fast = xmax * p.kmax_turns <= kFastTurnsField;
        const float eps = 1e-6f * xmax;
        FieldRecv x;
        x.X = pk(xp[0], xp[1]); x.Y = pk(yp[0], yp[1]); x.Z = pk(zp[0], zp[1]);
        x.XL = pk(xl[0], xl[1]); x.YL = pk(yl[0], yl[1]); x.ZL = pk(zl[0], zl[1]);
        x.NX = neg2(x.X); x.NY = neg2(x.Y); x.NZ = neg2(x.Z);
        const f2x NAXX = pk(-p.pre_alpha * xx[0], -p.pre_alpha * xx[1]), AL2 = splat(p.pre_alpha);
        f2x ax[NF], ay[NF];     // FP32 sums of the two receivers, per band
#pragma unroll
        for (int f = 0; f < NF; ++f) ax[f] = ay[f] = 0ull;

        bool first = true;
        auto fold_all = [&]() { fold_bands<NF>(p, item, lane, part, ax, ay, first); };
        Gather<WINDOW, true> g(item);
        int group = 0;
        g.issue(p, item, B.in, lane, rball, 0);
        g.issue(p, item, B.in, lane, rball, 1);
        for (uint32_t kb = 0;; ++kb) {
            const int buf = (int)(kb & 1u);
            const int nrec = buf ? g.n1 : g.n0;
            if (nrec <= 0) break;
            if ((buf ? g.group1 : g.group0) != group) {
                group = buf ? g.group1 : g.group0;
                fold_all();
            }
            cp_async_wait1();   // this lane's copies of batch kb
            bool small = false;
            if (lane < nrec)
                small = stage_field<NF, LOSSY>(p, B, lane, B.in.raw[buf][0][lane], B.in.raw[buf][1][lane],
                                                 B.in.raw[buf][2][lane], B.in.raw[buf][3][lane],
                                                 B.in.amp[buf][lane], buf ? g.seg1 : g.seg0, cx, cy, cz, rad);
            const uint32_t smask = __ballot_sync(0xffffffffu, small);
            __syncwarp();       // the batch is staged
            g.issue(p, item, B.in, lane, rball, buf);   // batch kb + 2 into the buffer just read

            const uint32_t all = nrec < 32 ? (1u << nrec) - 1u : 0xffffffffu;
            if (UNORDERED && 2 * __popc(smask) > nrec) {
                // each receiver's own, in segment order
                uint32_t m0 = part[0] ? all & ~smask : 0u, m1 = part[1] ? all & ~smask : 0u;
                for (uint32_t T = smask; T; T &= T - 1u) {
                    const int j = __ffs(T) - 1;
                    bool k0, k1;
                    may_keep<NF, WINDOW>(B, j, x, NAXX, AL2, k0, k1);
                    m0 |= (uint32_t)(part[0] && k0) << j;
                    m1 |= (uint32_t)(part[1] && k1) << j;
                }
                while (__any_sync(0xffffffffu, (m0 | m1) != 0u)) {
                    const bool h0 = m0 != 0u, h1 = m1 != 0u;
                    const int a = h0 ? __ffs(m0) - 1 : h1 ? __ffs(m1) - 1 : 0, c = h1 ? __ffs(m1) - 1 : a;
                    eval_field<NF, WINDOW, LOSSY, true>(p, B, a, c, x, h0, h1, fast, eps, ax, ay);
                    m0 &= m0 - 1u;
                    m1 &= m1 - 1u;
                }
            } else {
                uint32_t mine = 0u;
                for (uint32_t T = smask; T; T &= T - 1u) {
                    const int j = __ffs(T) - 1;
                    bool k0, k1;
                    may_keep<NF, WINDOW>(B, j, x, NAXX, AL2, k0, k1);
                    if ((part[0] && k0) || (part[1] && k1)) mine |= 1u << j;
                }
                uint32_t T = (all & ~smask) | __reduce_or_sync(0xffffffffu, mine);
                while (T) {
                    const int j = __ffs(T) - 1;
                    T &= T - 1u;
                    eval_field<NF, WINDOW, LOSSY, false>(p, B, j, j, x, part[0], part[1], fast, eps, ax, ay);
                }
            }
            __syncwarp();        // before the next batch is staged over this one
        }
        cp_async_wait0();        // every gather of this item has landed
        fold_all();
    }
}

template <int NF, int WINDOW, bool LOSSY>
void launch(const FwdParams &p, cudaStream_t s, bool timed)
{
    static std::atomic<int> known[2][64] = {};
    if (!p.order && !p.list)
        launch_items<PairCfg<FieldBuf<NF>, false>>(gbs_field_kernel<NF, WINDOW, LOSSY, true>, known[1], p, s, timed);
    else
        launch_items<PairCfg<FieldBuf<NF>, false>>(gbs_field_kernel<NF, WINDOW, LOSSY, false>, known[0], p, s, timed);
}

// Frequency slots: 1, 2, 4, 6 (lossless) and 8.
template <int WINDOW>
void launch_nf(const FwdParams &p, cudaStream_t s, bool timed)
{
    if (p.nf > 8) fail(GBT_ERR_UNSUPPORTED, "pair kernel launched with more than 8 frequencies");
    if (p.seg_rf) {
        if (p.nf <= 1) launch<1, WINDOW, true>(p, s, timed);
        else if (p.nf <= 2) launch<2, WINDOW, true>(p, s, timed);
        else if (p.nf <= 4) launch<4, WINDOW, true>(p, s, timed);
        else launch<8, WINDOW, true>(p, s, timed);
        return;
    }
    if (p.nf <= 1) launch<1, WINDOW, false>(p, s, timed);
    else if (p.nf <= 2) launch<2, WINDOW, false>(p, s, timed);
    else if (p.nf <= 4) launch<4, WINDOW, false>(p, s, timed);
    else if (p.nf <= 6) launch<6, WINDOW, false>(p, s, timed);
    else launch<8, WINDOW, false>(p, s, timed);
}
}  // namespace

void pair_field_launch(const FwdParams &p, int window, cudaStream_t s, bool timed)
{
    if (window == GBT_WINDOW_LINE) launch_nf<GBT_WINDOW_LINE>(p, s, timed);
    else launch_nf<GBT_WINDOW_SEGMENT>(p, s, timed);
}
}  // namespace gbt
