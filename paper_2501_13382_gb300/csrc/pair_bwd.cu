// pair_bwd.cu -- the adjoint pair kernel: per segment the sums over receivers and bands of
// Re(conj(g) c~) and, per band, of Re(conj(g) dc~/db), with c~ the contribution without
// W Gamma_path, by recomputation.
//
// Persistent CTAs of warps that work on their own: a warp takes (warp tile of 64 receivers,
// segment split) items from a global queue and double-buffers its 32-record batches (a bulk
// asynchronous copy completed on a per-warp mbarrier, or per-lane cp.async gathers from the
// tile's segment list with the pre-cull; every wait is bounded and raises a status flag).  A
// paired FP32 prefilter (the union of the bands' cutoffs and the window, with a margin)
// gives one keep bit per pair; survivors are evaluated in the warp's frame (pair_exact.cuh),
// segment by segment, and the warp's sums go to the segment's global G and H.
#include "pair_exact.cuh"
#include "pair_stream.cuh"

namespace gbt {
namespace {

// The FP32 local projection x'.t (instead of float-float) when K_max max|x'| <= kFastTurns:
// its rounding, at most about 3 ulp of |x'|, moves a term's phase by at most
// 3 x 2^-24 x 90 turns = 1.0e-4 rad.
constexpr float kFastTurnsAdj = 90.0f;

// Losses of the staged batch: per frequency slot and staged segment, log2 |R| and
// arg R / 2 pi of its porous reflections' factor.
template <int NF>
struct LossSmem {
    float2 rf[NF][kBatch];
};

// Adjoint terms of one beam: with c~ the contribution without W Gamma_path,
// G += Re(conj(g) c~) and H += Re(conj(g) dc~/db), where
// d log c / db = 1/b + i/E - k n^2 / (2 E^2), E = s - i b.  With losses c~ carries
// the porous reflections' factor (rf: log2 |R|, arg R in turns) and exp(-a s); neither
// depends on b, so the logarithmic derivative is the same.
template <bool LOSSY>
__device__ __forceinline__ void beam_adjoint(const FreqConst &q, float sh, float sl, float n2,
                                             float invD, float2 g, float &G, float &H,
                                             float2 rf = make_float2(0.f, 0.f))
{
    const float n2invD = n2 * invD;
    float ex = q.ne * n2invD;
    if (LOSSY) ex = fmaf(q.nal, sh, ex + rf.x);
    const float ga = ex2_approx(ex);
    const float ph = __fmul_rn(q.K_hi, sh);       // rounded: pe below is its exact error
    const float pe = fmaf(q.K_hi, sh, -ph);
    const float corr = fmaf(q.K_hi, sl, fmaf(q.K_lo, sh, pe));
    float tau = __fsub_rn(ph, rintf(ph)) + corr;
    tau = fmaf(q.hK * n2invD, sh, tau);
    if (LOSSY) tau += rf.y;
    tau = tau - rintf(tau);
    float sn, cs;
    __sincosf(6.283185307179586f * tau, &sn, &cs);
    const float gs = q.sA * ga * invD;
    const float cr = gs * fmaf(sh, cs, -q.b * sn);
    const float ci = gs * fmaf(sh, sn, q.b * cs);
    G = fmaf(g.x, cr, fmaf(g.y, ci, G));
    const float t = -q.nkh * n2 * invD * invD;                        // k n^2 / (2 D^2)
    const float dr = q.invb - q.b * invD - t * (sh * sh - q.b2);      // Re d log c / db
    const float di = sh * invD - t * (2.0f * sh * q.b);               // Im d log c / db
    H = fmaf(g.x, cr * dr - ci * di, fmaf(g.y, cr * di + ci * dr, H));
}

// Adjoint terms of one surviving pair added into G and H[f] (gk: this receiver's
// g per sorted frequency, stride kR * 32 float2).
template <int NF, int WINDOW, bool LOSSY>
__device__ __forceinline__ void survivor_adjoint(const FwdParams &p, float xh, float yh, float zh,
                                                 float xl, float yl, float zl, const StageSmem &w,
                                                 const LossSmem<NF> *loss, int j, bool fast,
                                                 float eps, const float2 *gk, float &G,
                                                 float (&H)[NF])
{
    float sh, sl, n2;
    if (!frame_geometry<WINDOW>(xh, yh, zh, xl, yl, zl, w, j, fast, eps, sh, sl, n2)) return;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (f >= p.nf) break;
        const FreqConst &q = p.fc[f];
        const float D = fmaf(sh, sh, q.b2);
        if (q.kb2 * n2 > p.cutoff * D) {
            if (p.uniform_b) break;
            continue;
        }
        beam_adjoint<LOSSY>(q, sh, sl, n2, rcp_approx(D), gk[f * (kR * 32)], G, H[f],
                            LOSSY ? loss->rf[f][j] : make_float2(0.f, 0.f));
    }
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int NF>
struct AdjSmem {
    float2 g[NF][kR][32];      // the warp's receivers' g, per sorted frequency
};
// Per-warp shared memory of the pair kernel: two raw record buffers (bulk-copy
// or cp.async targets), the staged batch, and the completion barriers of the
// bulk copies.
struct AdjWarpBuf {
    float4 raw[kWRaw][kBatch][kRecFloats / 4];
    StageSmem stg;
    unsigned long long bar[kWRaw];
    int32_t queue[kBatch];           // list positions of the next batch for this warp tile
    int abort_flag, pad[3];
};

template <int NF, bool LOSSY>
struct AdjCfg {
    static constexpr size_t kAdj = sizeof(AdjSmem<NF>);
    static constexpr size_t kLoss = LOSSY ? sizeof(LossSmem<NF>) : 0;
    static constexpr size_t kPerWarp = (sizeof(AdjWarpBuf) + kAdj + kLoss + 127) / 128 * 128;
    // as many warps as fit in the shared memory budget, at most kWarpsFwd
    static constexpr int kFit = (int)(kSmemBudget / kPerWarp);
    static constexpr int kWarps = kFit < kWarpsFwd ? kFit : kWarpsFwd;
    static constexpr size_t kSmem = kWarps * kPerWarp;
};

template <int NF, int WINDOW, bool LOSSY>
__global__ void __maxnreg__(128) gbs_adjoint_kernel(const __grid_constant__ FwdParams prm)
{
    using Cfg = AdjCfg<NF, LOSSY>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char *const mine = smem_raw + (size_t)warp * Cfg::kPerWarp;
    AdjWarpBuf &B = *reinterpret_cast<AdjWarpBuf *>(mine);
    AdjSmem<NF> &adj = *reinterpret_cast<AdjSmem<NF> *>(mine + sizeof(AdjWarpBuf));
    LossSmem<NF> *const loss =
        reinterpret_cast<LossSmem<NF> *>(mine + sizeof(AdjWarpBuf) + Cfg::kAdj);

    if (lane == 0) {
        for (int i = 0; i < kWRaw; ++i) mbar_init(smem_addr(&B.bar[i]), 1);
        B.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncwarp();
    volatile int *abort_flag = &B.abort_flag;
    uint32_t ph = 0;   // bit i: parity of the next completion of bar[i]

    for (;;) {
        int64_t it = 0;
        if (lane == 0) it = atomicAdd(prm.work_counter, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        const FwdParams &p = prm;
        if (it >= p.n_items || *abort_flag) break;

        // item -> (CTA tile by dispatch rank, split, warp tile within the CTA tile)
        const int64_t per_tile = (int64_t)kTileWarps * p.splits;
        const int64_t tile_rank = it / per_tile;
        const int64_t rem = it - tile_rank * per_tile;
        const int split = (int)(rem / kTileWarps);
        const int wl = (int)(rem - (int64_t)split * kTileWarps);
        const int64_t tile = p.tile_perm ? (int64_t)p.tile_perm[tile_rank] : tile_rank;
        const int64_t wbase = tile * kCtaRecv + (int64_t)wl * kWarpRecv;
        if (wbase >= p.n_recv) continue;
        // the segments this item streams: the CTA tile's list, or every segment
        const int32_t *lst = nullptr;
        int64_t n_seg = *p.n_seg_ptr;
        if (p.list) {
            const int32_t ln = p.list_n[tile];
            if (ln >= 0) {
                lst = p.list + p.list_off[tile];
                n_seg = ln;
            }
        }
        const int64_t n_batches = (n_seg + kBatch - 1) / kBatch;
        const uint32_t nb = split < n_batches ? (uint32_t)((n_batches - 1 - split) / p.splits + 1) : 0u;
        const float alpha = p.pre_alpha, beta = p.pre_beta;
        // receiver k of the lane at x = c + x', x' = (xp + xl) exactly
        float xa[kR], ya[kR], za[kR], xp[kR], yp[kR], zp[kR], xl[kR], yl[kR], zl[kR], xx[kR];
        int32_t ridx[kR];
        bool part[kR];
        uint32_t valid = 0;
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            // lane holds receivers lane and lane + 32 of the warp tile: the two halves
            // of its Morton patch, so a beam edge splits work evenly over lanes
            const int64_t r = wbase + (int64_t)k * 32 + lane;
            xa[k] = ya[k] = za[k] = xp[k] = yp[k] = zp[k] = xl[k] = yl[k] = zl[k] = xx[k] = 0.0f;
            ridx[k] = -1;
            part[k] = false;
            if (r < p.n_recv) {
                const int64_t o = p.order ? p.order[r] : r;
                xa[k] = p.recv[3 * o]; ya[k] = p.recv[3 * o + 1]; za[k] = p.recv[3 * o + 2];
                part[k] = takes_part(xa[k], ya[k], za[k]);
                if (part[k]) ridx[k] = (int32_t)o;
            }
        }
        // frame of the staged batches: the warp tile's first receiver
        const float3 c0 = first_receiver(part, xa, ya, za);
        const float cx = c0.x, cy = c0.y, cz = c0.z;
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            if (part[k]) {
                two_sum(xa[k], -cx, xp[k], xl[k]);
                two_sum(ya[k], -cy, yp[k], yl[k]);
                two_sum(za[k], -cz, zp[k], zl[k]);
                xx[k] = fmaf(xp[k], xp[k], fmaf(yp[k], yp[k], zp[k] * zp[k]));
                valid |= 1u << k;
            }
#pragma unroll
            for (int f = 0; f < NF; ++f)
                adj.g[f][k][lane] = (f < p.nf && ridx[k] >= 0)
                                        ? p.grad_out[(int64_t)p.fperm[f] * p.n_recv + ridx[k]]
                                        : make_float2(0.f, 0.f);
        }
        // bounding ball of the warp tile's receivers (relative to its first receiver)
        float4 sphere = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p.tile_cull) {
            float sx = 0.f, sy = 0.f, sz = 0.f, nv = 0.f;
#pragma unroll
            for (int k = 0; k < kR; ++k)
                if ((valid >> k) & 1u) { sx += xp[k]; sy += yp[k]; sz += zp[k]; nv += 1.f; }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sx += __shfl_xor_sync(0xffffffffu, sx, o);
                sy += __shfl_xor_sync(0xffffffffu, sy, o);
                sz += __shfl_xor_sync(0xffffffffu, sz, o);
                nv += __shfl_xor_sync(0xffffffffu, nv, o);
            }
            if (nv > 0.f) { sx /= nv; sy /= nv; sz /= nv; }
            float r2 = 0.f;
#pragma unroll
            for (int k = 0; k < kR; ++k)
                if ((valid >> k) & 1u) {
                    const float ex = xp[k] - sx, ey = yp[k] - sy, ez = zp[k] - sz;
                    r2 = fmaxf(r2, fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
            sphere = make_float4(sx, sy, sz, sqrtf(r2));
        }
        // the FP32 local projection when the warp is compact enough for its frequencies
        float xmax2 = fmaxf((valid & 1u) ? xx[0] : 0.f, (valid & 2u) ? xx[1] : 0.f);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) xmax2 = fmaxf(xmax2, __shfl_xor_sync(0xffffffffu, xmax2, o));
        const bool fast_u = sqrtf(xmax2) * p.kmax_turns <= kFastTurnsAdj;
        // its error bound: the three-term FP32 dot product with |t| = 1 is within about
        // 3 x 2^-24 max|x'| of x'.t; eps is over five times that
        const float eps_u = 1e-6f * sqrtf(xmax2);
        static_assert(kR == 2, "the paired prefilter handles two receivers per lane");
        const f2x X2 = pk(xp[0], xp[1]), Y2 = pk(yp[0], yp[1]), Z2 = pk(zp[0], zp[1]);
        const f2x NAXX = pk(-alpha * xx[0], -alpha * xx[1]);
        const f2x AL2 = pk(alpha, alpha);
        const f2x MG2 = pk(kWinMargin, kWinMargin);
        // Batches of the item, double-buffered: raw buffer k % 2 receives batch k.  Consecutive
        // segments: batch k is split + k * splits, one bulk copy (lane 0) on the buffer's
        // mbarrier.  A tile list: the item takes the list's 32-entry chunks split, split +
        // splits, ..., reads this warp tile's word of 32 such chunks at once (one per lane),
        // queues the set bits' list positions in order, gathers the entries of each full
        // batch, and every lane copies its own record with 16-byte async copies (one commit
        // group per batch, empty past the end).
        // Per buffer: records in the batch, and this lane's segment index (or -1).
        int nrec0 = 0, nrec1 = 0;
        int32_t seg0 = -1, seg1 = -1;
        const int64_t n_chunks = (n_seg + kBatch - 1) / kBatch;
        const uint32_t *lw =
            lst ? p.list_words + (p.list_off[tile] / kBatch) * kChunkWords + wl : nullptr;
        int64_t wnext = split;   // list: lane 0's chunk of the next window
        int64_t wchunk = 0;      // list: this lane's chunk in the current window
        uint32_t word = 0u;      // list: its entries for this warp tile not yet queued
        auto next_list_batch = [&](int32_t &pos) -> int {
            int n = 0;
            for (;;) {
                if (!__any_sync(0xffffffffu, word != 0u)) {
                    if (wnext >= n_chunks) break;
                    wchunk = wnext + (int64_t)lane * p.splits;
                    word = wchunk < n_chunks ? lw[wchunk * kChunkWords] : 0u;
                    wnext += (int64_t)kBatch * p.splits;
                    continue;
                }
                // lanes in chunk order, bits in entry order
                const int cnt = __popc(word);
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const int total = __shfl_sync(0xffffffffu, incl, 31);
                int slot = n + incl - cnt;
                while (word != 0u && slot < kBatch) {
                    B.queue[slot++] = (int32_t)(wchunk * kBatch + __ffs(word) - 1);
                    word &= word - 1u;
                }
                n = min(n + total, kBatch);
                if (n == kBatch) break;
            }
            __syncwarp();
            pos = lane < n ? B.queue[lane] : -1;
            __syncwarp();
            return n;
        };
        auto issue = [&](uint32_t k) {   // all lanes, k in increasing order
            const int buf = (int)(k & 1u);
            int n = 0;
            int32_t idx = -1;
            if (lst) {
                int32_t pos;
                n = next_list_batch(pos);
                idx = pos >= 0 ? lst[pos] : -1;
                if (idx >= 0) {
                    const float4 *src =
                        reinterpret_cast<const float4 *>(p.rec + (int64_t)idx * kRecFloats);
#pragma unroll
                    for (int c = 0; c < kRecFloats / 4; ++c) cp_async16(&B.raw[buf][lane][c], src + c, 16);
                }
                cp_async_commit();
            } else if (k < nb) {
                const int64_t b = split + (int64_t)k * p.splits;
                n = (int)min((int64_t)kBatch, n_seg - b * kBatch);
                idx = lane < n ? (int32_t)(b * kBatch + lane) : -1;
                if (lane == 0) {
                    const uint32_t bytes = (uint32_t)n * kRecFloats * 4;
                    mbar_arrive_expect_tx(smem_addr(&B.bar[buf]), bytes);
                    bulk_g2s(smem_addr(&B.raw[buf][0][0]), p.rec + b * kBatch * kRecFloats, bytes,
                             smem_addr(&B.bar[buf]));
                }
            }
            if (buf) { nrec1 = n; seg1 = idx; } else { nrec0 = n; seg0 = idx; }
        };
        issue(0);
        issue(1);
        uint32_t waited = 0;   // bulk batches whose copy has landed
        for (uint32_t kb_ = 0;; ++kb_) {
            const int buf = (int)(kb_ & 1u);
            const int nrec = buf ? nrec1 : nrec0;
            if (nrec <= 0) break;
            const int32_t my_seg = buf ? seg1 : seg0;
            if (lst) {
                cp_async_wait1();   // this lane's copies of batch kb_
            } else {
                bool ok = mbar_wait(smem_addr(&B.bar[buf]), (ph >> buf) & 1u, abort_flag, p.status);
                if (!__all_sync(0xffffffffu, ok)) break;
                ph ^= 1u << buf;
                waited = kb_ + 1;
            }
            const bool seg_ok = lane < nrec;
            StageSmem &w = B.stg;
            const float my_len = stage_batch(w, B.raw[buf][lane], lane, seg_ok, my_seg, cx, cy, cz,
                                             alpha, beta);
            // The exact view: with the pre-cull at once (nearly every batch has survivors);
            // testing every pair only after the prefilter, and only for a batch in which the
            // warp has a survivor (most such batches have none), before raw[buf] is reused.
            if (lst) stage_exact(w, B.raw[buf][lane], lane, seg_ok, cx, cy, cz);
            if (LOSSY) {
#pragma unroll
                for (int f = 0; f < NF; ++f)
                    loss->rf[f][lane] = (seg_ok && f < p.nf)
                                            ? p.seg_rf[(int64_t)p.fperm[f] * p.rf_stride + my_seg]
                                            : make_float2(0.f, 0.f);
            }
            uint32_t tmask = 0u;
            if (p.tile_cull) {
                // this lane's segment against the warp tile's ball (own lane's staging only)
                const float4 O = w.O[lane];
                const float4 *R1 = &B.raw[buf][lane][1];   // t_hi, L_hi of the raw record
                // a list entry carrying this warp tile's bit already passed the same test
                // against the warp tile's ball when the lists were built
                const bool pass = seg_ok && (lst != nullptr ||
                                  ball_may_keep<WINDOW>(O, make_float4(R1->x, R1->y, R1->z, my_len),
                                                        O.x, O.y, O.z, sphere, alpha, beta));
                tmask = __ballot_sync(0xffffffffu, pass);
            }
            if (lst) {
                __syncwarp();    // the batch is staged and raw[buf] is free again
                issue(kb_ + 2);
            }

            // ---- prefilter: one keep bit per (receiver, segment); segment jj at bit 31 - jj.
            // Both receivers of the lane go through paired FP32 instructions:
            //   s_loc = x'.t - o'.t,  sm = s_loc + s0 + margin,
            //   g = sm^2 + beta - alpha |x' - o'|^2 + alpha s_loc^2  (= q - alpha n^2),
            // keep iff g >= 0 and the window test holds.
            uint32_t m[kR];
#pragma unroll
            for (int k = 0; k < kR; ++k) m[k] = 0u;
            auto pair_bits = [&](int jj, uint32_t &kb0, uint32_t &kb1) {
                const float4 *P = w.P[jj];
                const float4 p0 = P[4], p1 = P[0], p2 = P[1], p3 = P[2], p4 = P[3];
                const f2x TX = pk(p0.x, p0.y), TY = pk(p0.z, p0.w), TZ = pk(p1.x, p1.y);
                const f2x OT = pk(p1.z, p1.w);
                const f2x OX = pk(p2.x, p2.y), OY = pk(p2.z, p2.w), OZ = pk(p3.x, p3.y);
                const f2x C7 = pk(p3.z, p3.w), S0 = pk(p4.x, p4.y);
                const f2x sl = fma2(X2, TX, fma2(Y2, TY, fma2(Z2, TZ, OT)));
                const f2x sm2 = add2(sl, S0);
                const f2x nd = fma2(X2, OX, fma2(Y2, OY, fma2(Z2, OZ, add2(NAXX, C7))));
                const f2x gg = fma2(mul2(sl, AL2), sl, fma2(sm2, sm2, nd));
                float g0, g1, s0_, s1_;
                upk(gg, g0, g1);
                if (WINDOW == GBT_WINDOW_LINE) {
                    upk(sm2, s0_, s1_);
                    kb0 = ~(__float_as_uint(g0) | __float_as_uint(s0_));
                    kb1 = ~(__float_as_uint(g1) | __float_as_uint(s1_));
                } else {
                    const f2x a = add2(sl, MG2);
                    const f2x bb = sub2(sl, pk(p4.z, p4.w));
                    float a0, a1, b0_, b1_;
                    upk(a, a0, a1);
                    upk(bb, b0_, b1_);
                    kb0 = ~(__float_as_uint(g0) | __float_as_uint(a0)) & __float_as_uint(b0_);
                    kb1 = ~(__float_as_uint(g1) | __float_as_uint(a1)) & __float_as_uint(b1_);
                }
            };
if (p.tile_cull) {
                // only the segments that can reach this warp tile's receivers
                uint32_t T = tmask;
                while (T) {
                    const int jj = __ffs(T) - 1;
                    T &= T - 1;
                    uint32_t kb0, kb1;
                    pair_bits(jj, kb0, kb1);
                    m[0] |= (kb0 >> 31) << (31 - jj);
                    m[1] |= (kb1 >> 31) << (31 - jj);
                }
            } else {
#pragma unroll 4
                for (int jj = 0; jj < kBatch; ++jj) {
                    uint32_t kb0, kb1;
                    pair_bits(jj, kb0, kb1);
                    m[0] = __funnelshift_l(kb0, m[0], 1);
                    m[1] = __funnelshift_l(kb1, m[1], 1);
                }
            }
            if (!lst) {
                if (__any_sync(0xffffffffu, (((valid & 1u) ? m[0] : 0u) | ((valid & 2u) ? m[1] : 0u)) != 0u))
                    stage_exact(w, B.raw[buf][lane], lane, seg_ok, cx, cy, cz);
                __syncwarp();    // the batch is staged and raw[buf] is free again
                issue(kb_ + 2);
            }
            // ---- survivors
            {
                // segment by segment: the lanes holding a survivor of segment jj add their
                // receivers' terms, the warp sums them, and one lane adds the sums to the
                // segment's global G and H (no shared-memory atomics between lanes)
                const uint32_t mm0 = (valid & 1u) ? m[0] : 0u, mm1 = (valid & 2u) ? m[1] : 0u;
                uint32_t any = __reduce_or_sync(0xffffffffu, mm0 | mm1);
                while (any) {
                    const int jj = __clz(any);
                    any ^= 0x80000000u >> jj;
                    float G = 0.f, H[NF];
#pragma unroll
                    for (int f = 0; f < NF; ++f) H[f] = 0.f;
                    if ((mm0 << jj) >> 31)
                        survivor_adjoint<NF, WINDOW, LOSSY>(p, xp[0], yp[0], zp[0], xl[0], yl[0],
                                                            zl[0], w, loss, jj, fast_u, eps_u,
                                                            &adj.g[0][0][lane],
                                                            G, H);
                    if ((mm1 << jj) >> 31)
                        survivor_adjoint<NF, WINDOW, LOSSY>(p, xp[1], yp[1], zp[1], xl[1], yl[1],
                                                            zl[1], w, loss, jj, fast_u, eps_u,
                                                            &adj.g[0][1][lane],
                                                            G, H);
                    G = warp_sum(G);
#pragma unroll
                    for (int f = 0; f < NF; ++f)
                        if (f < p.nf) H[f] = warp_sum(H[f]);
                    const int32_t jg = w.seg[jj];
                    if (lane == 0 && jg >= 0) {
                        if (G != 0.f) atomicAdd(&p.seg_G[jg], G);
#pragma unroll
                        for (int f = 0; f < NF; ++f)
                            if (f < p.nf && H[f] != 0.f) atomicAdd(&p.seg_H[(int64_t)f * p.seg_stride + jg], H[f]);
                    }
                }
            }
            __syncwarp();        // before the next batch is staged over this one
        }
        if (lst) {
            cp_async_wait0();    // every gather of this item has landed
        } else if (*abort_flag && lane == 0) {
            // a wait gave up: let the bulk copies still in flight land before leaving
            const uint32_t issued = min(nb, waited + 2u);
            for (uint32_t k = waited; k < issued; ++k) {
                const int bf = (int)(k & 1u);
                for (long long i2 = 0; i2 < kSpinLimit; ++i2)
                    if (mbar_try_wait(smem_addr(&B.bar[bf]), (ph >> bf) & 1u)) break;
                ph ^= 1u << bf;
            }
        }
    }
}

template <int NF, int WINDOW, bool LOSSY>
void launch(const FwdParams &p, cudaStream_t s, bool timed)
{
    static std::atomic<int> known[64] = {};
    launch_items<AdjCfg<NF, LOSSY>>(gbs_adjoint_kernel<NF, WINDOW, LOSSY>, known, p, s, timed);
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

void pair_bwd_launch(const FwdParams &p, int window, cudaStream_t s, bool timed)
{
    if (window == GBT_WINDOW_LINE) launch_nf<GBT_WINDOW_LINE>(p, s, timed);
    else launch_nf<GBT_WINDOW_SEGMENT>(p, s, timed);
}
}  // namespace gbt
