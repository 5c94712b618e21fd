// pair.cuh -- the FP32 pair kernel: beams of Eq. 1 / Eq. 2 summed over (receiver, segment,
// frequency), forward only (the adjoint is in pair_bwd.cu).
//
// Every warp works on its own.  It takes (warp tile of 64 receivers, segment split) items
// from a global queue (CTA tiles of 960 receivers heaviest first), collects the segments
// whose beams can reach the warp tile's ball, and evaluates each of them for its 64
// receivers, two per lane in paired FP32 (f32x2).  Where the segments come from:
//  * a tile list (the pre-cull): the warp reads its own 32-bit word of 32 list chunks at
//    once and gathers the entries whose bit is set;
//  * no list: the warp tests the 32-byte cull records of four chunks of 32 segments at a
//    time against its ball.  About 35 instructions per 32 segments, where a test of every
//    (receiver, segment) pair took 15 per segment.  That test comes back for receivers that
//    have no order either (small_beam).
// Gathered records arrive by per-lane cp.async, double buffered, and each lane stages one.
//
// What bounds it: operand reads.  On this chip an FFMA2 with three operand pairs of its own
// issues every 3.1 cycles (2.1 when it shares one with its neighbour, as in a mul2 or add2),
// and ALU, MUFU and shared loads add to that instead of hiding behind it (an FFMA2 and a
// LOP3: 4.9 cycles); more warps or longer chains change little.  So the number of operands
// per pair is what counts.
//  * The frame is the centre of the warp tile's bounding box, x = c + x'.  The staging forms
//    per segment A = (c - o).t and S = s0 + A in float-float, N = (c - o) x t rounded once,
//    and per band the phase of S reduced to one turn, so a pair needs
//      u = x'.t,  s = S + u,  n = N + x' x t
//    and the phase K u + phi_f, reduced by adding and subtracting 1.5 x 2^23: no
//    float-float arithmetic per pair (38 paired operations with one band, where float-float
//    geometry and phase took 63).
//  * u = Um + Uc: x' and t are split on grids of 11 and 12 bits of their magnitude, so the three
//    products of Um and their sum are exact in FP32, and Uc holds the rest to about 2^-36 |x'|.
//    Nine products, where float-float sums took 31 operations; window decisions are those of
//    the exact arithmetic to 1e-10 m.
//  * One band, a compact warp (K max|x'| <= kFastTurns) and a segment without an end of its
//    window inside the warp tile's ball: u is one FP32 dot product plus that of t's low words,
//    six products.  Its rounding, 3 x 2^-24 |x'| at most, moves the phase by up to 1.8e-5 rad
//    (small open plane: relative L2 error 2.3e-7, with the split form 1.7e-7), which spares
//    the 1M-ray city 8 % of its time.  Several bands spend their time on the beams: there the
//    split form is free.  Which of the two a segment takes is uniform over the warp.
//  * Precision.  Relative L2 error against 64 bits over 37 inputs (listed, drawn and bench
//    sizes, 8 seeds each): 0.60 of that of float-float pairs in the geometric mean, 0.24 to
//    1.005 by input; 1M-ray city 1.3e-7 (1.8e-7), with losses 1.4e-7 (1.8e-7), open plane with 6
//    bands 1.3e-7 (1.7e-7), 8 bands with losses 1.85e-7 (1.88e-7), scattered receivers 2.8e-7
//    (4.6e-7).  Dropping t's low word, reducing the phase once and a compensated N with two
//    roundings gave 0.77 and up to 1.26.  What is left is mostly MUFU's sine and cosine (0.39
//    with sincospif); their mean loss of amplitude goes into the merge's factor.  n as exact
//    head products and a rest (15 operations more) would give 0.50, for 8 to 16 % of the time.
//  * The amplitude's common factor k / (8 pi^2) is left to the merge, the pairs' cutoff test
//    is one comparison (r <= rc), and receivers past the last are computed and not stored.
// Summation: FP32 per lane and batch group, folded into the item's float-float partials every
// kFoldEvery batches of list entries and, without a list, twice as often (open plane, 6 bands:
// every 16, 8, 4 batches 1.42e-7, 1.36e-7, 1.32e-7 and 2.08, 2.08, 2.14 ms), merged in split
// order by reduce_kernel, so results do not depend on scheduling.
// Measured (kernel alone, with float-float pairs -> now): city, 1,048,576 rays x 512^2
// receivers, lists: 31.0 -> 15.6 ms; open plane, 65,536 rays x 256^2 x 6 bands, no lists:
// 6.06 -> 1.93 ms; city, 65,536 rays x 200^2 x 2 bands, no lists: 6.79 -> 1.49 ms.
#pragma once

#include "pair_stream.cuh"

namespace gbt {
namespace {

// K max|x'| up to which one band's u is a plain dot product (see above).  Everywhere split, the
// 1M-ray city takes 21.8 ms instead of 20.2, at an error of 1.24e-7 instead of 1.26e-7.
constexpr float kFastTurns = 16.0f;

// Receivers without an order and without lists: a warp tile's 64 may lie anywhere, nearly every
// segment reaches its ball and keeps a few of them.  A segment is small if its union cutoff radius
// at the tile is under small_beam() times the ball's radius; where most of a batch are, may_keep
// marks candidates and every receiver evaluates its own, a slot of its own to each lane and half.
// 65,536-ray city x 10,000 scattered x 2 bands: every segment for all 64 5.36 ms, so 3.85; 8 bands
// 10.0, 6.87; rows of a 200^2 grid 9.26, 6.13; rows of the 256^2 open plane, 6 bands 4.91, 4.58.  Line
// at 0.5, 1, 2, 4: 8 bands 8.62, 6.86, 6.87, 6.87, with a cutoff of 100 (23,296 rays x 17,737 x 5) -,
// 10.43, 7.81, 7.84.  A few hundred ordered receivers (a CTA tile or less) take it too, as they may
// be as far apart, with the line at 1: 56 over 1 km, one split 7.66, 3.01; 900 on 40 m, 6 bands .19,
// .20 (.22 at 2).  The candidates' loop unrolled 1, 2, 4, 8 times: 8 bands 7.03, 6.92, 6.87, 7.92.
// Other ordered receivers have kernels of their own without this (registers).
__device__ __forceinline__ float small_beam(const FwdParams &p) { return p.order ? 1.0f : 2.0f; }

// Shape by the number of band slots: segments evaluated together (plain, which only one band has,
// and split), bands per vote, and warps.  One band needs several segments for independent
// chains and shared operands (1M-ray city step: one segment, 16 warps 27.4 ms; two 26.0;
// four, 12 warps 25.1); two or more bands have the chains themselves.  Bands in pairs spare
// votes where most bands are kept (open plane, 6 bands: 2.06 -> 1.94 ms), and cost where
// few are or the losses take the registers (9,973 scattered receivers, 3 bands: 0.72 ->
// 0.76 ms; 8 bands with losses: 10.25 -> 10.43 ms).
template <int NF, bool LOSSY>
struct PairShape {
    static constexpr int NS = NF == 1 ? 4 : 1, NP = NF == 1 ? 2 : 1;
    static constexpr int FG = NF >= 6 && !LOSSY ? 2 : 1;
    static constexpr int kWarps = NF == 1 ? 12 : 16;
    // the fused batch: 8 bands read 14 warps' constants from shared memory (16 sources x 256^2 x
    // 8 bands, lists: 16 warps 99.6, 14 95.1, 12 97.0 ms)
    static constexpr int kWarpsBatched = NF >= 6 ? 14 : kWarps;
};

// Per-warp shared memory: the raw records and the staged batch, every value in both halves of
// a float pair (a segment is shared by the warp, so the operands of the paired arithmetic are
// broadcast loads).  Segments sit in slots: those whose u is a plain dot product first, then the
// split ones, padded to whole groups with a slot of zero amplitude.
template <int NF, bool LOSSY>
struct WarpBuf {
    static constexpr int kSlots = kBatch + 1;   // padding
    RawBuf in;
    // D[0] t.x, t.y | D[1] t.z, S (times s_scale) | D[2] N.x, N.y | D[3] N.z, amplitude |
    // D[4..6] t on its grid (3) and the rest (3); a plain slot's D[4..5]: t's low words (3)
    float4 D[7][kSlots];
    float4 W[kSlots];               // SEGMENT: A, A - L as (hi, lo); LINE: S as (hi, lo)
    float4 F[(NF + 1) / 2][kSlots]; // bands 2 i, 2 i + 1: phase of S in turns
    float4 R[LOSSY ? (NF + 1) / 2 : 1][LOSSY ? kSlots : 1];   // and amplitude with the losses
};

// A lane's two receivers relative to the frame, as float pairs: x', -x', x' on its grid, the
// rest.
struct LaneRecv {
    f2x X, Y, Z, NX, NY, NZ, XH, YH, ZH, XL, YL, ZL;
};

// Adds the beams of the staged slots j .. j + NS - 1 to the lane's two receivers' sums per
// band.  `cross`: slots with an end of their window inside the warp tile's ball.  EACH: of a slot
// of its own to each receiver (j and j1; h0, h1: whether it has one).
template <int NF, int WINDOW, bool LOSSY, bool PREC, int NS, int FG, bool BATCHED, bool EACH = false>
__device__ __forceinline__ void eval_segments(const FwdParams &p, const WarpBuf<NF, LOSSY> &w,
                                              int j, uint64_t cross, const LaneRecv &x,
                                              f2x (&ax)[NF], f2x (&ay)[NF], int j1 = 0,
                                              bool h0 = true, bool h1 = true)
{
    static_assert(!EACH || (PREC && NS == 1), "slots apart are split ones, one at a time");
    const f2x MAGIC = splat(12582912.0f), ONE = splat(1.0f);
    f2x U[NS], UC[NS], s[NS], nn[NS], amp[NS];
    bool k0[NS], k1[NS];
    auto word = [&](int d, int q, f2x &a, f2x &b) { staged<EACH>(w.D[d], j + q, j1, a, b); };
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        k0[q] = h0;
        k1[q] = h1;
        f2x TX, TY, TZ, S, NX, NY, NZ;
        word(0, q, TX, TY);
        word(1, q, TZ, S);
        word(2, q, NX, NY);
        word(3, q, NZ, amp[q]);
        f2x u;
        if (PREC) {
            f2x HX, HY, HZ, LX, LY, LZ;
            word(4, q, HX, HY);
            word(5, q, HZ, LX);
            word(6, q, LY, LZ);
            U[q] = fma2(x.XH, HX, fma2(x.YH, HY, mul2(x.ZH, HZ)));            // exact
            UC[q] = fma2(x.XL, TX, fma2(x.YL, TY, fma2(x.ZL, TZ,
                    fma2(x.XH, LX, fma2(x.YH, LY, mul2(x.ZH, LZ))))));
            u = add2(U[q], UC[q]);
            if (EACH || ((cross >> (j + q)) & 1u)) {
                const float4 e = w.W[j + q], o = EACH ? w.W[j1] : e;
                float a0, a1;
                upk(add2(add2(pk(e.x, o.x), U[q]), add2(pk(e.y, o.y), UC[q])), a0, a1);
                k0[q] = k0[q] && a0 >= 0.0f;
                k1[q] = k1[q] && a1 >= 0.0f;
                if (WINDOW == GBT_WINDOW_SEGMENT) {
                    upk(add2(add2(pk(e.z, o.z), U[q]), add2(pk(e.w, o.w), UC[q])), a0, a1);
                    k0[q] = k0[q] && a0 < 0.0f;
                    k1[q] = k1[q] && a1 < 0.0f;
                }
            }
        } else {
            f2x LX, LY, LZ, none;
            word(4, q, LX, LY);
            word(5, q, LZ, none);
            U[q] = u = fma2(x.X, TX, fma2(x.Y, TY, mul2(x.Z, TZ)));
            UC[q] = fma2(x.X, LX, fma2(x.Y, LY, mul2(x.Z, LZ)));
        }
        s[q] = fma2(u, splat(p.s_scale), S);
        // n = N + x' x t
        const f2x nx = fma2(x.Y, TZ, fma2(x.NZ, TY, NX));
        const f2x ny = fma2(x.Z, TX, fma2(x.NX, TZ, NY));
        const f2x nz = fma2(x.X, TY, fma2(x.NY, TX, NZ));
        nn[q] = fma2(nx, nx, fma2(ny, ny, mul2(nz, nz)));
    }
    // FG bands at a time, one vote for each group: their chains interleave
    f2x sc[NS][FG], nsc[NS][FG], AD[NS][FG], r[NS][FG], rs[NS][FG];
#pragma unroll
    for (int f0 = 0; f0 < NF; f0 += FG) {
        if (NF > 1 && f0 >= p.nf) break;
        bool m0[NS][FG], m1[NS][FG], any = false;
#pragma unroll
        for (int i = 0; i < FG; ++i) {
            const int f = f0 + i;
            FreqConst cs;
            if (BATCHED) {      // instance constants in shared memory, by whole words (that batch:
                                // 103.4 ms by floats, 99.6 by words)
                const float4 v = reinterpret_cast<const float4 *>(&p.fc[f])[1];
                cs.rc = v.z;
                cs.invb = v.w;
            }
            const FreqConst &c = BATCHED ? cs : p.fc[f];
            const bool live = NF == 1 || FG == 1 || f < p.nf;
#pragma unroll
            for (int q = 0; q < NS; ++q) {
                if (f == 0 || !p.uniform_b) {
                    sc[q][i] = (NF == 1 || p.uniform_b) ? s[q] : mul2(splat(c.invb), s[q]);
                    nsc[q][i] = neg2(sc[q][i]);
                    float d0, d1;
                    upk(fma2(sc[q][i], sc[q][i], ONE), d0, d1);
                    const f2x invD = pk(rcp_approx(d0), rcp_approx(d1));
                    r[q][i] = mul2(nn[q], invD);
                    rs[q][i] = mul2(r[q][i], sc[q][i]);
                    AD[q][i] = LOSSY ? invD : mul2(amp[q], invD);
                } else if (i > 0) {
                    sc[q][i] = sc[q][0]; nsc[q][i] = nsc[q][0]; AD[q][i] = AD[q][0];
                    r[q][i] = r[q][0]; rs[q][i] = rs[q][0];
                }
                float r0, r1;
                upk(r[q][i], r0, r1);
                m0[q][i] = live && (PREC ? k0[q] && r0 <= c.rc : r0 <= c.rc);
                m1[q][i] = live && (PREC ? k1[q] && r1 <= c.rc : r1 <= c.rc);
                any = any || m0[q][i] || m1[q][i];
            }
        }
        // narrower bands keep no more (one b: the kept bands are a prefix); a compact warp's
        // only band seldom misses all its receivers
        if ((NF > 1 || PREC) && !__any_sync(0xffffffffu, any)) {
            if (NF == 1 || p.uniform_b) break;
            continue;
        }
#pragma unroll
        for (int i = 0; i < FG; ++i) {
            const int f = f0 + i;
            FreqConst cs;
            if (BATCHED) {
                const float4 u = reinterpret_cast<const float4 *>(&p.fc[f])[0];
                const float4 v = reinterpret_cast<const float4 *>(&p.fc[f])[1];
                cs.K_hi = u.z;
                cs.K_lo = u.w;
                cs.hK = v.x;
                cs.ne = v.y;
            }
            const FreqConst &c = BATCHED ? cs : p.fc[f];
#pragma unroll
            for (int q = 0; q < NS; ++q) {
                f2x ph, pq;
                staged<EACH>(w.F[f / 2], j + q, j1, ph, pq);
                if (f & 1) ph = pq;
                f2x g = AD[q][i];
                if (LOSSY) {
                    f2x ra, rb;
                    staged<EACH>(w.R[f / 2], j + q, j1, ra, rb);
                    g = mul2(f & 1 ? rb : ra, g);
                }
                f2x ex = mul2(splat(c.ne), r[q][i]);
                if (LOSSY) ex = fma2(splat(c.nal), sc[q][i], ex);
                float e0, e1;
                upk(ex, e0, e1);
                g = mul2(g, pk(m0[q][i] ? ex2_approx(e0) : 0.0f, m1[q][i] ? ex2_approx(e1) : 0.0f));
                const f2x KH = splat(c.K_hi);
                if (PREC) ph = fma2(splat(c.K_lo), U[q], ph);
                ph = fma2(KH, UC[q], ph);
                // less whole turns before and after the second term: every sum is rounded near
                // its smallest size
                const f2x nr = sub2(MAGIC, fma2(KH, U[q], MAGIC));
                f2x tau = fma2(splat(c.hK), rs[q][i], add2(fma2(KH, U[q], nr), ph));
                tau = add2(tau, sub2(MAGIC, add2(tau, MAGIC)));
                float t0, t1, sn0, cs0, sn1, cs1;
                upk(mul2(splat(-6.283185307179586f), tau), t0, t1);
                __sincosf(t0, &sn0, &cs0);
                __sincosf(t1, &sn1, &cs1);
                const f2x NSN = pk(sn0, sn1), CS = pk(cs0, cs1);                // -sin, cos
                ax[f] = fma2(g, fma2(sc[q][i], CS, NSN), ax[f]);
                ay[f] = fma2(g, fma2(nsc[q][i], NSN, CS), ay[f]);
            }
        }
    }
}

// Whether the staged (split) slot j may keep a beam at the lane's receivers: the union of the
// bands' cutoffs and the window, in plain FP32 with margins: u, s and n are within 1e-6 of rad and
// of their own sizes, so n^2 is within 1e-3 of itself and 1e-9 rad^2 (al, be: see the caller).
// The signs' outcome is shifted into m0, m1.
template <int NF, int WINDOW, bool LOSSY>
__device__ __forceinline__ void may_keep(const WarpBuf<NF, LOSSY> &w, int j, const LaneRecv &x, float scale,
                                         float al, float be, float rad, uint32_t &m0, uint32_t &m1)
{
    f2x TX, TY, TZ, S, NX, NY, NZ, amp;
    staged<false>(w.D[0], j, j, TX, TY);
    staged<false>(w.D[1], j, j, TZ, S);
    staged<false>(w.D[2], j, j, NX, NY);
    staged<false>(w.D[3], j, j, NZ, amp);
    const f2x u = fma2(x.X, TX, fma2(x.Y, TY, mul2(x.Z, TZ)));
    const f2x s = fma2(u, splat(scale), S);
    const f2x nx = fma2(x.Y, TZ, fma2(x.NZ, TY, NX));
    const f2x ny = fma2(x.Z, TX, fma2(x.NX, TZ, NY));
    const f2x nz = fma2(x.X, TY, fma2(x.NY, TX, NZ));
    const f2x nn = fma2(nx, nx, fma2(ny, ny, mul2(nz, nz)));
    float g0, g1, a0, a1;
    upk(fma2(s, s, fma2(splat(-al), nn, splat(be))), g0, g1);
    const float4 e = w.W[j];
    upk(add2(u, splat(e.x + kWinMargin + 1e-6f * (fabsf(e.x) + rad))), a0, a1);
    uint32_t b0 = ~(__float_as_uint(g0) | __float_as_uint(a0)), b1 = ~(__float_as_uint(g1) | __float_as_uint(a1));
    if (WINDOW == GBT_WINDOW_SEGMENT) {
        upk(add2(u, splat(e.z - kWinMargin - 1e-6f * (fabsf(e.z) + rad))), a0, a1);
        b0 &= __float_as_uint(a0);
        b1 &= __float_as_uint(a1);
    }
    m0 = __funnelshift_l(b0, m0, 1);
    m1 = __funnelshift_l(b1, m1, 1);
}

// Slots of a staged batch: [0, n_plain) with a plain u, [n_plain, end) with the split one, and
// which slots may have an end of their window inside the ball.
struct StagedBatch {
    int n_plain, end;
    uint64_t cross;
    uint32_t small;            // segments whose beam is small against the ball (small_beam)
};

// Stages the batch's raw records (a lane each) in the frame c, for the 64 receivers within rad
// of it: see WarpBuf.  A segment is split where the warp is not `fast` (one band, compact, every
// x' one float) or an end of its window may lie inside the ball (a margin of 1 mm covers the
// rounding of the float-float heads).
template <int NF, int WINDOW, bool LOSSY, int NS, int NP, bool UNORDERED>
__device__ __forceinline__ StagedBatch stage(const FwdParams &p, WarpBuf<NF, LOSSY> &w, int lane,
                                             int nrec, int buf, int32_t seg, float cx, float cy,
                                             float cz, float rad, bool fast)
{
    const bool have = lane < nrec;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 r0 = have ? w.in.raw[buf][0][lane] : zero, r1 = have ? w.in.raw[buf][1][lane] : zero;
    const float4 r2 = have ? w.in.raw[buf][2][lane] : zero, r3 = have ? w.in.raw[buf][3][lane] : zero;
    const float amp = have ? w.in.amp[buf][lane] : 0.0f;
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
    // S = s0 + A
    float Sh, es;
    two_sum(r0.w, Ah, Sh, es);
    const float Sl = __fadd_rn(es, __fadd_rn(Al, r2.w));
    bool cross;
    float4 W;
    if (WINDOW == GBT_WINDOW_SEGMENT) {
        float ALh, ea;
        two_sum(Ah, -r1.w, ALh, ea);
        const float ALl = __fadd_rn(ea, __fsub_rn(Al, r3.w));
        W = make_float4(Ah, Al, ALh, ALl);
        cross = !(Ah - rad >= 1e-3f && ALh + rad <= -1e-3f);
    } else {
        W = make_float4(Sh, Sl, 0.f, 0.f);
        cross = !(Sh - rad >= 1e-3f);
    }
    // slots: whole groups of NS plain segments first, then the others (the last few plain ones
    // among them), padded to whole groups of NP with slots of zero amplitude
    const uint32_t xm = __ballot_sync(0xffffffffu, have && cross);
    const uint32_t all = nrec < 32 ? (1u << nrec) - 1u : 0xffffffffu;
    const uint32_t below = (1u << lane) - 1u;
    uint32_t plain = fast ? all & ~xm : 0u;
    StagedBatch b;
    b.small = 0u;
    if (UNORDERED) {
        const float smax = fabsf(Sh) + rad;
        const float line = small_beam(p) * rad;
        b.small = __ballot_sync(0xffffffffu, have && fmaf(smax, smax, p.pre_beta) < p.pre_alpha * line * line);
    }
    b.n_plain = __popc(plain) / NS * NS;
#pragma unroll
    for (int q = 1; q < NS; ++q)
        if (__popc(plain) > b.n_plain) plain &= plain - 1u;
    b.end = nrec;
    b.cross = fast ? ~0ull : (uint64_t)xm;     // fast warps: every split segment
    const bool mine_plain = (plain >> lane) & 1u;
    const int slot = mine_plain ? __popc(plain & below) : b.n_plain + __popc(all & ~plain & below);
    // N = d x t, each component (ah + al) (th + tl) - (bh + bl) (uh + ul) rounded once
    auto cross_term = [](float ah, float al, float th, float tl, float bh, float bl, float uh, float ul) {
        const float p = __fmul_rn(ah, th), q = __fmul_rn(bh, uh);
        float d, e;
        two_sum(p, -q, d, e);
        e = __fadd_rn(e, __fsub_rn(fmaf(ah, th, -p), fmaf(bh, uh, -q)));
        return __fadd_rn(d, __fadd_rn(e, fmaf(ah, tl, fmaf(-bh, ul, fmaf(al, th, -bl * uh)))));
    };
    const float nx = cross_term(dyh, dyl, r1.z, r3.z, dzh, dzl, r1.y, r3.y);
    const float ny = cross_term(dzh, dzl, r1.x, r3.x, dxh, dxl, r1.z, r3.z);
    const float nz = cross_term(dxh, dxl, r1.y, r3.y, dyh, dyl, r1.x, r3.x);
    if (have) {
        w.D[0][slot] = dup2(r1.x, r1.y);
        w.D[1][slot] = dup2(r1.z, Sh * p.s_scale);
        w.D[2][slot] = dup2(nx, ny);
        w.D[3][slot] = dup2(nz, amp);
        if (mine_plain) {
            // one band: with K_lo / K_hi of t in its low words, K_hi (U + u_lo) is K u
            const float ks = p.fc[0].K_lo * rcp_approx(p.fc[0].K_hi);
            w.D[4][slot] = dup2(fmaf(r1.x, ks, r3.x), fmaf(r1.y, ks, r3.y));
            w.D[5][slot] = dup2(fmaf(r1.z, ks, r3.z), 0.f);
        } else {
            // t rounded to multiples of 2^-12 (by 1.5 x 2^11, whose ulp that is), and the rest
            const float hx = __fsub_rn(__fadd_rn(r1.x, 3072.f), 3072.f);
            const float hy = __fsub_rn(__fadd_rn(r1.y, 3072.f), 3072.f);
            const float hz = __fsub_rn(__fadd_rn(r1.z, 3072.f), 3072.f);
            w.D[4][slot] = dup2(hx, hy);
            w.D[5][slot] = dup2(hz, __fadd_rn(__fsub_rn(r1.x, hx), r3.x));
            w.D[6][slot] = dup2(__fadd_rn(__fsub_rn(r1.y, hy), r3.y), __fadd_rn(__fsub_rn(r1.z, hz), r3.z));
            w.W[slot] = W;
        }
    }
#pragma unroll
    for (int f0 = 0; f0 < NF; f0 += 2) {
        float phi[2] = {0.f, 0.f}, a[2] = {0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int f = f0 + i;
            if (f >= NF || (NF > 1 && f >= p.nf)) continue;
            const FreqConst &c = p.fc[f];
            const float ph = __fmul_rn(c.K_hi, Sh);
            const float pe = fmaf(c.K_hi, Sh, -ph);                    // exact
            phi[i] = __fsub_rn(ph, rintf(ph)) + fmaf(c.K_hi, Sl, fmaf(c.K_lo, Sh, pe));
            if (LOSSY && have) {
                const float2 rf = p.seg_rf[(int64_t)p.fperm[f] * p.rf_stride + seg];
                phi[i] += rf.y;
                a[i] = amp * exp2f(rf.x);
            }
        }
        if (have) {
            w.F[f0 / 2][slot] = dup2(phi[0], phi[1]);
            if (LOSSY) w.R[f0 / 2][slot] = dup2(a[0], a[1]);
        }
    }
    if (NP > 1 && lane < (NP - (b.end - b.n_plain) % NP) % NP) {
        const int q = b.end + lane;
#pragma unroll
        for (int d = 0; d < 7; ++d) w.D[d][q] = zero;
        w.W[q] = zero;
#pragma unroll
        for (int f0 = 0; f0 < NF; f0 += 2) {
            w.F[f0 / 2][q] = zero;
            if (LOSSY) w.R[f0 / 2][q] = zero;
        }
    }
    return b;
}

// The frame of a warp tile with stray receivers (points far off the map), so that their |x'| does
// not coarsen the others': the tile's first, middle or last receiver (part: those that count),
// if most of them lie within sqrt(close2) of it; else c as it is.  Out of line and without a
// search for the median: inside the kernel its registers cost the main loop (open plane, 6 bands:
// median 2.11 ms, inline 2.10, so 2.04).
__device__ __noinline__ void stray_frame(const bool (&part)[kR], const float (&x)[kR], const float (&y)[kR],
                                         const float (&z)[kR], float close2, float (&c)[3])
{
    const uint32_t m0 = __ballot_sync(0xffffffffu, part[0]), m1 = __ballot_sync(0xffffffffu, part[1]);
#pragma unroll 1
    for (int q = 0; q < 3; ++q) {
        const int k = q == 0 ? m0 == 0u : m1 != 0u;
        const uint32_t m = k ? m1 : m0;
        const int src = q < 2 ? __ffs(m) - 1 : 31 - __clz(m);
        const float cx = __shfl_sync(0xffffffffu, k ? x[1] : x[0], src);
        const float cy = __shfl_sync(0xffffffffu, k ? y[1] : y[0], src);
        const float cz = __shfl_sync(0xffffffffu, k ? z[1] : z[0], src);
        int close = 0;
#pragma unroll
        for (int r = 0; r < kR; ++r) {
            const float ex = x[r] - cx, ey = y[r] - cy, ez = z[r] - cz;
            close += __popc(__ballot_sync(0xffffffffu, part[r] && fmaf(ex, ex, fmaf(ey, ey, ez * ez)) < close2));
        }
        if (2 * close > __popc(m0) + __popc(m1)) {
            c[0] = cx; c[1] = cy; c[2] = cz;
            break;
        }
    }
}

template <int NF, int WINDOW, bool BATCHED, bool LOSSY, bool UNORDERED = false>
__global__ void __launch_bounds__(32 * PairCfg<WarpBuf<NF, LOSSY>, BATCHED, BATCHED ? PairShape<NF, LOSSY>::kWarpsBatched : PairShape<NF, LOSSY>::kWarps>::kWarps, 1) gbs_pair_kernel(const __grid_constant__ FwdParams prm)
{
    using Cfg = PairCfg<WarpBuf<NF, LOSSY>, BATCHED, BATCHED ? PairShape<NF, LOSSY>::kWarpsBatched : PairShape<NF, LOSSY>::kWarps>;
    static_assert(!(LOSSY && BATCHED), "batches with losses run the single-sum kernel");
    using Shape = PairShape<NF, LOSSY>;
    constexpr int NS = Shape::NS, NP = Shape::NP, FG = Shape::FG;
    static_assert(NF % FG == 0 && NS <= 4, "whole band groups");
    static_assert(NP <= 2, "one padding slot");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char *const mine = smem_raw + (size_t)warp * Cfg::kPerWarp;
    WarpBuf<NF, LOSSY> &B = *reinterpret_cast<WarpBuf<NF, LOSSY> *>(mine);
    FwdParams &inst = *reinterpret_cast<FwdParams *>(mine + sizeof(WarpBuf<NF, LOSSY>));

    for (;;) {
        int64_t it = 0;
        if (lane == 0) it = atomicAdd(prm.work_counter, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= (BATCHED ? prm.n_items : item_count(prm))) break;
        if (BATCHED) {
            int lo = 0, hi = prm.n_inst - 1;      // last instance with inst_off <= it
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (prm.inst_off[mid] <= it) lo = mid;
                else hi = mid - 1;
            }
            it -= prm.inst_off[lo];
            __syncwarp();
            const int4 *src = reinterpret_cast<const int4 *>(prm.inst + lo);
            int4 *dst = reinterpret_cast<int4 *>(&inst);
            for (int q = lane; q < (int)(sizeof(FwdParams) / 16); q += 32) dst[q] = src[q];
            __syncwarp();
        }
        const FwdParams &p = BATCHED ? inst : prm;
        Item item;
        if (!decode_item(p, it, item)) continue;

        // the lane's receivers: lane and lane + 32 of the warp tile, the two halves of its
        // Morton patch, so a beam edge splits work evenly over lanes
        float xr[kR], yr[kR], zr[kR];
        bool part[kR];
        unsigned bb[6] = {~0u, ~0u, ~0u, 0u, 0u, 0u};
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            const int64_t r = item.wbase + (int64_t)k * 32 + lane;
            part[k] = false;
            xr[k] = yr[k] = zr[k] = 0.0f;
            if (r < p.n_recv) {
                const int64_t o = p.order ? p.order[r] : r;
                xr[k] = p.recv[3 * o]; yr[k] = p.recv[3 * o + 1]; zr[k] = p.recv[3 * o + 2];
                part[k] = takes_part(xr[k], yr[k], zr[k]);
                if (!part[k]) no_partials(p, item, 32 * k + lane);
            }
            if (part[k]) {
                const unsigned ux = ordered_bits(xr[k]), uy = ordered_bits(yr[k]), uz = ordered_bits(zr[k]);
                bb[0] = min(bb[0], ux); bb[1] = min(bb[1], uy); bb[2] = min(bb[2], uz);
                bb[3] = max(bb[3], ux); bb[4] = max(bb[4], uy); bb[5] = max(bb[5], uz);
            }
        }
        f2x ax[NF], ay[NF];     // FP32 sums of the two receivers, per band
#pragma unroll
        for (int f = 0; f < NF; ++f) ax[f] = ay[f] = 0ull;
        // frame: the centre c of the bounding box; rad bounds |x'|
        float ctr[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float lo = from_ordered(__reduce_min_sync(0xffffffffu, bb[a]));
            const float hi = from_ordered(__reduce_max_sync(0xffffffffu, bb[3 + a]));
            ctr[a] = 0.5f * lo + 0.5f * hi;
        }
        float4 rball;
        {
            unsigned far2 = 0u, near2 = ~0u;      // bits of the largest and the smallest |x - c|^2
#pragma unroll
            for (int k = 0; k < kR; ++k)
                if (part[k]) {
                    const float ex = xr[k] - ctr[0], ey = yr[k] - ctr[1], ez = zr[k] - ctr[2];
                    const unsigned e2 = __float_as_uint(fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
                    far2 = max(far2, e2);
                    near2 = min(near2, e2);
                }
            const float f2 = __uint_as_float(__reduce_max_sync(0xffffffffu, far2));
            const float n2 = __uint_as_float(__reduce_min_sync(0xffffffffu, near2));
            rball = reach_ball(make_float4(ctr[0], ctr[1], ctr[2], 1.000001f * sqrtf(f2)));
            // a centre without a receiver within half the radius may lie between the others and a
            // stray one
            if (n2 > 0.25f * f2) stray_frame(part, xr, yr, zr, 0.0625f * f2, ctr);
        }
        float xp[kR], yp[kR], zp[kR], xl[kR], yl[kR], zl[kR], xx[kR];
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            xp[k] = yp[k] = zp[k] = xl[k] = yl[k] = zl[k] = xx[k] = 0.0f;
            if (part[k]) {
                two_sum(xr[k], -ctr[0], xp[k], xl[k]);
                two_sum(yr[k], -ctr[1], yp[k], yl[k]);
                two_sum(zr[k], -ctr[2], zp[k], zl[k]);
                xx[k] = fmaf(xp[k], xp[k], fmaf(yp[k], yp[k], zp[k] * zp[k]));
            }
        }
        const float cx = ctr[0], cy = ctr[1], cz = ctr[2];
        const float rad = 1.000001f * sqrtf(__uint_as_float(
            __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(xx[0], xx[1])))));
        bool fast = false;
        if (NF == 1) {
            bool rest = false;          // x' is not one float
#pragma unroll
            for (int k = 0; k < kR; ++k) rest = rest || xl[k] != 0.0f || yl[k] != 0.0f || zl[k] != 0.0f;
            fast = rad * p.kmax_turns <= kFastTurns && !__any_sync(0xffffffffu, rest);
        }
        // grid of a receiver's x': a power of two q with |x'| <= 2^11 q, by adding 1.5 x 2^23 q
        float grid[kR];
#pragma unroll
        for (int k = 0; k < kR; ++k)
            grid[k] = xx[k] > 1e-36f ? scalbnf(12582912.0f, (int)ceilf(0.5f * log2f(xx[k]) + 1e-5f) - 11) : 0.0f;
        LaneRecv x;
        {
            float h[3][kR];
#pragma unroll
            for (int k = 0; k < kR; ++k) {
                h[0][k] = __fsub_rn(__fadd_rn(xp[k], grid[k]), grid[k]);
                h[1][k] = __fsub_rn(__fadd_rn(yp[k], grid[k]), grid[k]);
                h[2][k] = __fsub_rn(__fadd_rn(zp[k], grid[k]), grid[k]);
                xl[k] = __fadd_rn(__fsub_rn(xp[k], h[0][k]), xl[k]);
                yl[k] = __fadd_rn(__fsub_rn(yp[k], h[1][k]), yl[k]);
                zl[k] = __fadd_rn(__fsub_rn(zp[k], h[2][k]), zl[k]);
            }
            x.X = pk(xp[0], xp[1]); x.Y = pk(yp[0], yp[1]); x.Z = pk(zp[0], zp[1]);
            x.NX = neg2(x.X); x.NY = neg2(x.Y); x.NZ = neg2(x.Z);
            x.XH = pk(h[0][0], h[0][1]); x.YH = pk(h[1][0], h[1][1]); x.ZH = pk(h[2][0], h[2][1]);
            x.XL = pk(xl[0], xl[1]); x.YL = pk(yl[0], yl[1]); x.ZL = pk(zl[0], zl[1]);
        }
        // the candidates' test in the units of the staged s, with its margins
        const float al = 0.999f * p.pre_alpha * p.s_scale * p.s_scale;
        const float be = fmaf(1.001e-9f * al, rad * rad, 1.001f * p.pre_beta * p.s_scale * p.s_scale);
        bool first = true;
        auto fold_all = [&]() { fold_bands<NF>(p, item, lane, part, ax, ay, first); };

        Gather<WINDOW, false> g(item);
        g.issue(p, item, B.in, lane, rball, 0);
        g.issue(p, item, B.in, lane, rball, 1);
        for (uint32_t kb = 0;; ++kb) {
            const int buf = (int)(kb & 1u);
            const int nrec = buf ? g.n1 : g.n0;
            if (nrec <= 0) break;
            cp_async_wait1();   // this lane's copies of batch kb
            const StagedBatch b = stage<NF, WINDOW, LOSSY, NS, NP, UNORDERED>(
                p, B, lane, nrec, buf, buf ? g.seg1 : g.seg0, cx, cy, cz, rad, fast);
            __syncwarp();       // the batch is staged
            g.issue(p, item, B.in, lane, rball, buf);   // batch kb + 2 into the buffer just read
            if (NF == 1)
                for (int j = 0; j < b.n_plain; j += NS)
                    eval_segments<NF, WINDOW, LOSSY, false, NS, FG, BATCHED>(p, B, j, 0ull, x, ax, ay);
            if (UNORDERED && !fast && 2 * __popc(b.small) > nrec) {
                // small beams: each receiver's own candidates, in segment order
                uint32_t m0 = 0u, m1 = 0u;      // slot j at bit 31 - j
#pragma unroll 4
                for (int j = 0; j < nrec; ++j)
                    may_keep<NF, WINDOW, LOSSY>(B, j, x, p.s_scale, al, be, rad, m0, m1);
                m0 = part[0] ? m0 << (32 - nrec) : 0u;
                m1 = part[1] ? m1 << (32 - nrec) : 0u;
                while (__any_sync(0xffffffffu, (m0 | m1) != 0u)) {
                    const bool h0 = m0 != 0u, h1 = m1 != 0u;
                    const int a = __clz(h0 ? m0 : h1 ? m1 : 0x80000000u), c = h1 ? __clz(m1) : a;
                    eval_segments<NF, WINDOW, LOSSY, true, 1, 1, BATCHED, true>(p, B, a, 0ull, x, ax, ay, c, h0, h1);
                    m0 &= ~(0x80000000u >> a);
                    m1 &= ~(0x80000000u >> c);
                }
            } else {
                for (int j = b.n_plain; j < b.end; j += NP)
                    eval_segments<NF, WINDOW, LOSSY, true, NP, FG, BATCHED>(p, B, j, b.cross, x, ax, ay);
            }
            // without a list every entry of a batch reaches the warp: twice as often
            const uint32_t every = item.lst ? kFoldEvery : kFoldEvery / 2;
            if (kb % every == every - 1) fold_all();
            __syncwarp();        // before the next batch is staged over this one
        }
        cp_async_wait0();        // every gather of this item has landed
        fold_all();
    }
}

}  // namespace
}  // namespace gbt
