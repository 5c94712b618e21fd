// gbs.cu -- everything around the pair kernel (pair.cuh): the prepass of traced segments
// into kernel records, the tile order and the pre-cull's segment lists, the counting pass,
// the all-FP64 path, the merge of partial sums, the adjoint's per-ray map, batches, time
// synthesis and the receiver order.
//
//  * A prepass turns every traced segment into an 80-byte record (origin, start distance,
//    direction and length as float-float, amplitude) and a 32-byte cull record.
//  * Receivers are visited in Morton order, in warp tiles of 64; CTA tiles of 15 warp tiles
//    are dispatched heaviest first, with segment splits sized so that the queue drains on
//    short items.
//  * The per-split partials are merged in float-float (error-free FP32 sums) in a fixed
//    order, so results do not depend on scheduling.
//  * The pair kernel holds the sums of up to 8 frequencies in registers; more (up to 16)
//    run as one launch per group of 8, each with its own partials and output rows.

#include <math.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>
#include <cmath>
#include <string>

#include "pair_exact.cuh"
#include "pair_stream.cuh"

namespace gbt {
namespace {

// ------------------------------------------------------ counting pass --
// Every pair (or, with the pre-cull, every pair of the segments that reach a warp tile)
// goes through a paired FP32 prefilter, the union of the bands' cutoffs and the window with
// a margin, and the survivors through the exact test in float-float (pair_exact.cuh); only
// counts come out (gbt_sum_stats_get).

// The kept (pair, frequency) triples of one surviving pair.
template <int NF, int WINDOW>
__device__ __forceinline__ void survivor_count(const FwdParams &p, float xh, float yh, float zh,
                                               float xl, float yl, float zl, const StageSmem &w,
                                               int j, uint32_t &kept)
{
    float sh, sl, n2;
    if (!frame_geometry<WINDOW>(xh, yh, zh, xl, yl, zl, w, j, false, 0.f, sh, sl, n2)) return;
    if (p.uniform_b) {
        const float D = fmaf(sh, sh, p.fc[0].b2);
        const float r = n2 * rcp_approx(D);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            if (f >= p.nf) break;
            if (p.fc[f].kb2 * r > p.cutoff) break;
            ++kept;
        }
    } else {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            if (f >= p.nf) break;
            const float D = fmaf(sh, sh, p.fc[f].b2);
            if (p.fc[f].kb2 * n2 > p.cutoff * D) continue;
            ++kept;
        }
    }
}

// Per-warp shared memory of the counting pass: two raw record buffers (bulk-copy or
// cp.async targets), the staged batch, and the completion barriers of the bulk copies.
struct CountBuf {
    float4 raw[kWRaw][kBatch][kRecFloats / 4];
    StageSmem stg;
    unsigned long long bar[kWRaw];
    int32_t queue[kBatch];           // list positions of the next batch for this warp tile
    int abort_flag, pad[3];
};
constexpr size_t kCountPerWarp = (sizeof(CountBuf) + 127) / 128 * 128;
constexpr int kCountWarps = (int)(kSmemBudget / kCountPerWarp) < kWarpsFwd
                                ? (int)(kSmemBudget / kCountPerWarp) : kWarpsFwd;
constexpr size_t kCountSmem = kCountWarps * kCountPerWarp;

// Persistent and warp-autonomous like the pair kernel: consecutive segments arrive by one
// bulk copy per batch, a tile list's by one 16-byte cp.async per lane and word.
template <int NF, int WINDOW>
__global__ void __maxnreg__(128) gbs_count_kernel(const __grid_constant__ FwdParams prm)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char *const mine = smem_raw + (size_t)warp * kCountPerWarp;
    CountBuf &B = *reinterpret_cast<CountBuf *>(mine);

    if (lane == 0) {
        for (int i = 0; i < kWRaw; ++i) mbar_init(smem_addr(&B.bar[i]), 1);
        B.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncwarp();
    volatile int *abort_flag = &B.abort_flag;
    uint32_t n_pre = 0, n_kept = 0;
    unsigned long long n_test = 0;
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
        bool part[kR];
        uint32_t valid = 0;
#pragma unroll
        for (int k = 0; k < kR; ++k) {
            // lane holds receivers lane and lane + 32 of the warp tile: the two halves
            // of its Morton patch, so a beam edge splits work evenly over lanes
            const int64_t r = wbase + (int64_t)k * 32 + lane;
            xa[k] = ya[k] = za[k] = xp[k] = yp[k] = zp[k] = xl[k] = yl[k] = zl[k] = xx[k] = 0.0f;
            part[k] = false;
            if (r < p.n_recv) {
                const int64_t o = p.order ? p.order[r] : r;
                xa[k] = p.recv[3 * o]; ya[k] = p.recv[3 * o + 1]; za[k] = p.recv[3 * o + 2];
                part[k] = takes_part(xa[k], ya[k], za[k]);
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
        int nrec0 = 0, nrec1 = 0;   // per buffer: records in the batch
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
            if (lst) {
                int32_t pos;
                n = next_list_batch(pos);
                const int32_t idx = pos >= 0 ? lst[pos] : -1;
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
                if (lane == 0) {
                    const uint32_t bytes = (uint32_t)n * kRecFloats * 4;
                    mbar_arrive_expect_tx(smem_addr(&B.bar[buf]), bytes);
                    bulk_g2s(smem_addr(&B.raw[buf][0][0]), p.rec + b * kBatch * kRecFloats, bytes,
                             smem_addr(&B.bar[buf]));
                }
            }
            if (buf) nrec1 = n; else nrec0 = n;
        };
        issue(0);
        issue(1);
        uint32_t waited = 0;   // bulk batches whose copy has landed
        for (uint32_t kb_ = 0;; ++kb_) {
            const int buf = (int)(kb_ & 1u);
            const int nrec = buf ? nrec1 : nrec0;
            if (nrec <= 0) break;
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
            const float my_len = stage_batch(w, B.raw[buf][lane], lane, seg_ok, -1, cx, cy, cz, alpha,
                                             beta);
            // the exact view: with the pre-cull at once, testing every pair only for a batch in
            // which the warp has a survivor, before raw[buf] is reused
            if (lst) stage_exact(w, B.raw[buf][lane], lane, seg_ok, cx, cy, cz);
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
                n_test += __popc(T) * __popc(valid);
                while (T) {
                    const int jj = __ffs(T) - 1;
                    T &= T - 1;
                    uint32_t kb0, kb1;
                    pair_bits(jj, kb0, kb1);
                    m[0] |= (kb0 >> 31) << (31 - jj);
                    m[1] |= (kb1 >> 31) << (31 - jj);
                }
            } else {
                n_test += (uint32_t)nrec * __popc(valid);
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
#pragma unroll
            for (int k = 0; k < kR; ++k) {
                uint32_t mm = ((valid >> k) & 1u) ? m[k] : 0u;
                n_pre += __popc(mm);
                while (mm) {
                    const int jj = __clz(mm);
                    mm ^= 0x80000000u >> jj;
                    survivor_count<NF, WINDOW>(p, xp[k], yp[k], zp[k], xl[k], yl[k], zl[k], w, jj, n_kept);
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
    atomicAdd(&prm.stats[1], (unsigned long long)n_pre);
    atomicAdd(&prm.stats[2], (unsigned long long)n_kept);
    atomicAdd(&prm.stats[3], n_test);
}

// ------------------------------------------------------------- prepass --

struct PrepParams {
    const int32_t *n_seg_ptr;
    const double *o, *t, *L, *s0;
    const int32_t *ray, *depth, *bmat;
    const float *gamma;
    const float *weight;       // per global ray, or nullptr -> the fan's own weight
    FanDev fan;
    int64_t n_fan;
    int n_materials;
    float *rec;
    float4 *crec;              // cull records (origin, s0, direction, length), 32 B each
    // F64 path records (nullptr when not needed)
    double *amp64;
    unsigned int *status;
    double w0;                 // weight of every ray of a Fibonacci or explicit fan
    int *counters;             // kCounters work counters to zero, or nullptr
};
constexpr int kCounters = GBT_MAX_FREQ / kGroupFreq;   // one per pair launch of a sum

// v = hi + lo, each rounded to nearest: hi = (float)v, lo = (float)(v - hi).  By integer
// operations on v's bits in the range where neither part can leave FP32 (2^-60 .. 2^120, and
// zero): the four FP64 and conversion instructions per value issue at a 64th of the integer
// rate and were most of the prepass (3.06e6 segments: 405 us with them).
__device__ __forceinline__ void split_ff(double v, float &hi, float &lo)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const uint32_t h = (uint32_t)(bits >> 32), l = (uint32_t)bits;
    const uint32_t e = (h >> 20) & 0x7ffu;
    if (e - 963u <= 180u) {
        const uint32_t m = ((h & 0xfffffu) << 3) | (l >> 29);      // hi's 23 fraction bits
        int32_t r = (int32_t)(l & 0x1fffffffu);                    // the 29 below, in 2^(e - 1075)
        const bool up = r > 0x10000000 || (r == 0x10000000 && (m & 1u));
        hi = __uint_as_float((h & 0x80000000u) | ((((e - 896u) << 23) | m) + (up ? 1u : 0u)));
        if (up) r -= 0x20000000;
        if (h & 0x80000000u) r = -r;
        lo = __int2float_rn(r) * __uint_as_float((e - 948u) << 23);
    } else if ((bits << 1) == 0ull) {
        hi = (float)v;
        lo = 0.0f;
    } else {
        hi = (float)v;
        lo = (float)(v - (double)hi);
    }
}

// Writes segment j's 80-byte record and 32-byte cull record.
__device__ __forceinline__ void write_record(float *rec, float4 *crec, int64_t j, const double *o,
                                             const double *t, double s0, double L, double amp)
{
    float4 *R = reinterpret_cast<float4 *>(rec + j * kRecFloats);
    float oh[3], ol[3], th[3], tl[3], s0h, s0l, Lh, Ll;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        split_ff(o[a], oh[a], ol[a]);
        split_ff(t[a], th[a], tl[a]);
    }
    split_ff(s0, s0h, s0l);
    split_ff(L, Lh, Ll);
    R[0] = make_float4(oh[0], oh[1], oh[2], s0h);     // R_OXH .. R_S0H
    R[1] = make_float4(th[0], th[1], th[2], Lh);      // R_TXH .. R_LH
    R[2] = make_float4(ol[0], ol[1], ol[2], s0l);     // R_OXL .. R_S0L
    R[3] = make_float4(tl[0], tl[1], tl[2], Ll);      // R_TXL .. R_LL
    R[4] = make_float4((float)amp, 0.f, 0.f, 0.f);    // R_AMP
    crec[2 * j] = R[0];
    crec[2 * j + 1] = R[1];
}

// Product of gamma over the reflections before a segment: materials bmat[1 .. dep].
__device__ __forceinline__ double path_gamma(const PrepParams &p, const int32_t *bmat, int dep)
{
    double g = 1.0;
    for (int q = 1; q <= dep; ++q) {
        const int m = bmat[q];
        if (m < 0 || m >= p.n_materials) {
            atomicOr(p.status, STATUS_BOUNDS);
            continue;
        }
        g *= (double)p.gamma[m];
    }
    return g;
}
__device__ __forceinline__ double ray_amplitude(const PrepParams &p, int64_t ray)
{
    if (p.weight) return (double)p.weight[ray];
    return p.fan.kind == GBT_FAN_LATLONG ? fan_weight(p.fan, p.n_fan, ray) : p.w0;
}

__global__ void prepass_kernel(PrepParams p)
{
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j < kCounters && p.counters) p.counters[j] = 0;
    if (j >= *p.n_seg_ptr) return;
    const int dep = p.depth[j];
    const double amp = ray_amplitude(p, p.ray[j]) * path_gamma(p, p.bmat + j - dep, dep);
    write_record(p.rec, p.crec, j, p.o + 3 * j, p.t + 3 * j, p.s0[j], p.L[j], amp);
    if (p.amp64) p.amp64[j] = amp;
}

// Records straight from the tracer's padded rows (gbt_solve: nobody sees the segment list):
// a block takes kPackRays rays, finds its first segment from the blocks' counts, and its
// threads run over its segments, not its slots (most rows are short).  Replaces the scan, the
// compaction and the prepass: 101 bytes less written and read per segment (1M-ray city: 610
// us for the five kernels, 258 us).
__global__ void __launch_bounds__(kPackRays) pack_kernel(PrepParams p, PaddedRays r)
{
    __shared__ int32_t first[kPackRays + 1];     // segments of the block before each ray
    __shared__ int32_t ws[kPackRays / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (blockIdx.x == 0 && threadIdx.x < kCounters) p.counters[threadIdx.x] = 0;
    auto block_sum = [&](int32_t v) {            // of every thread's v
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) ws[wid] = v;
        __syncthreads();
        int32_t s = 0;
        for (int w = 0; w < kPackRays / 32; ++w) s += ws[w];
        __syncthreads();
        return s;
    };
    int32_t before = 0;
    if (r.scanned) {
        before = r.bsum[blockIdx.x];
    } else {
        for (int64_t q = threadIdx.x; q < blockIdx.x; q += kPackRays) before += r.bsum[q];
        before = block_sum(before);
    }
    const int64_t i = (int64_t)blockIdx.x * kPackRays + threadIdx.x;
    const int32_t cnt = i < r.n_rays ? r.cnt[i] : 0;
    int32_t x = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    for (int w = 0; w < wid; ++w) x += ws[w];
    first[threadIdx.x + 1] = x;
    if (threadIdx.x == 0) first[0] = 0;
    __syncthreads();
    const int32_t total = first[kPackRays];
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *r.n_seg = before + total;
    for (int32_t k = threadIdx.x; k < total; k += kPackRays) {
        int lo = 0;                              // last ray with first[lo] <= k
#pragma unroll
        for (int st = kPackRays / 2; st > 0; st >>= 1)
            if (first[lo + st] <= k) lo += st;
        const int dep = k - first[lo];
        const int64_t ray = (int64_t)blockIdx.x * kPackRays + lo;
        const int64_t slot = ray * r.stride + dep;
        const double amp = ray_amplitude(p, r.ray_begin + ray) * path_gamma(p, r.bmat + slot - dep, dep);
        write_record(p.rec, p.crec, before + k, r.o + 3 * slot, r.t + 3 * slot, r.s0[slot], r.L[slot], amp);
    }
}

// ---- losses of porous surfaces
struct LossParams {
    const int32_t *ray_off;
    int64_t n_rays;
    const double *t;
    const int32_t *bmat, *hit;
    const float *sigma;        // per material, kPa s m^-2 (<= 0 hard), or nullptr: all hard
    const double *tri;         // the scene's triangles (unit normal at 9..11)
    int64_t n_tri;
    int n_materials, nf;
    double freq[GBT_MAX_FREQ];
    double2 *z;                // [f][material] impedance
    float2 *seg_rf;            // [f][rf_stride] (log2 |R|, arg R / 2 pi), or nullptr
    double2 *seg_r64;          // [f][rf_stride] R for the F64 path, or nullptr
    int64_t rf_stride;
    unsigned int *status;
};

// Normalised impedance of a porous, locally reacting surface of flow resistivity sigma
// (kPa s m^-2) at frequency f, Delany-Bazley for exp(-i omega t):
// Z = 1 + 9.08 (f/sigma)^-0.75 + i 11.9 (f/sigma)^-0.73.  Once per (band, material): the two
// pow() of a bounce were most of the prepass (8 bands, 448,870 segments: 4.45 ms).
__global__ void porous_impedance_kernel(LossParams p)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.nf * p.n_materials) return;
    const double sg = (double)p.sigma[i % p.n_materials];
    if (!(sg > 0.0)) return;
    const double x = p.freq[i / p.n_materials] / sg;
    p.z[i] = make_double2(1.0 + 9.08 * pow(x, -0.75), 11.9 * pow(x, -0.73));
}

// Cosine of the angle of incidence at the reflection that starts segment j (depth >= 1):
// |t_j . n| with n the unit normal of the primitive that ended segment j - 1 (ground:
// +z); a mirror reflection keeps |d . n|.  An unknown primitive is flagged.
__device__ __forceinline__ double incidence_cos(const LossParams &p, int64_t j)
{
    const int prim = p.hit[j - 1];
    double nx = 0.0, ny = 0.0, nz = 1.0;
    if (prim >= 1 && prim <= p.n_tri) {
        const double *n = p.tri + 12 * (int64_t)(prim - 1) + 9;
        nx = n[0]; ny = n[1]; nz = n[2];
    } else if (prim != 0) {
        atomicOr(p.status, STATUS_BAD_INPUT);
    }
    return fabs(p.t[3 * j] * nx + p.t[3 * j + 1] * ny + p.t[3 * j + 2] * nz);
}

// One thread per (ray, band) walks the ray's segments with the product of the plane-wave
// reflection factors R = (Z c - 1) / (Z c + 1) of its porous reflections so far; the F32
// path keeps their logarithms and arguments as running sums, one logarithm and arctangent
// per porous bounce instead of one per segment.  Bound by FP64 issue.
__global__ void __launch_bounds__(128) porous_path_kernel(LossParams p)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= p.n_rays) return;
    const int f = blockIdx.y;
    const int32_t a = p.ray_off[i], e = p.ray_off[i + 1];
    double rr = 1.0, ri = 0.0, lg = 0.0, turns = 0.0;
    for (int32_t j = a; j < e; ++j) {
        const int m = j > a ? p.bmat[j] : -1;
        if (p.sigma && m >= 0 && m < p.n_materials && p.sigma[m] > 0.0f) {
            const double2 z = p.z[f * p.n_materials + m];
            const double c = incidence_cos(p, j);
            const double ar = z.x * c - 1.0, ai = z.y * c, br = z.x * c + 1.0;
            const double inv = 1.0 / (br * br + ai * ai);
            const double x = (ar * br + ai * ai) * inv, y = (ai * br - ar * ai) * inv;
            if (p.seg_rf) {
                lg += 0.5 * log2(x * x + y * y);
                turns += atan2(y, x) * (0.5 / kPi);
                turns -= rint(turns);
            } else {
                const double nr = rr * x - ri * y;
                ri = rr * y + ri * x;
                rr = nr;
            }
        }
        const int64_t k = (int64_t)f * p.rf_stride + j;
        if (p.seg_rf) p.seg_rf[k] = make_float2((float)lg, (float)turns);
        else p.seg_r64[k] = make_double2(rr, ri);
    }
}

// ------------------------------------------------------ FP64 variant --

constexpr int kWarps64 = 2;        // warps per block, each on its own 32 receivers

struct F64Params {
    FwdParams g;               // what the gathering of segments reads (records, splits, cull)
    const float *recv;
    const int32_t *order;
    int64_t n_recv;
    const double *o, *t, *L, *s0, *amp;
    int nf;
    double cutoff;
    double k[GBT_MAX_FREQ], b[GBT_MAX_FREQ], kb[GBT_MAX_FREQ], b2[GBT_MAX_FREQ];
    double2 *partial;          // [splits][nf][n_recv]
    double absorb[GBT_MAX_FREQ];   // amplitude decay rate of air per frequency (Np/m)
    const double2 *r64;        // [f][r64_stride] porous reflections' factor, or nullptr
    int64_t r64_stride;
};

template <int NF>
struct Warp64 {
    RawBuf in;
    // prefilter constants of a staged segment (o' = o - c): (t, -o'.t), (2a o', beta - a |o'|^2),
    // (s0 + margin, L + margin, margin)
    float4 P[3][kBatch];
    int32_t seg[kBatch];
    // a window of candidate pairs: s and n^2, segment, kept frequencies, terms
    double2 geo[32];
    int32_t pair_seg[32];
    uint32_t kept[32];
    double2 term[NF][32];
};

// Position of the n-th set bit of m (n < popc(m)).
__device__ __forceinline__ int nth_bit(uint32_t m, int n)
{
    int pos = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int c = __popc(m & ((1u << w) - 1u));
        if (n >= c) {
            n -= c;
            pos += w;
            m >>= w;
        }
    }
    return pos;
}

__device__ __forceinline__ int warp_scan(int v, int lane)     // inclusive
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// The lane in whose range [its predecessor's incl, incl) slot lies (31 past the last).
__device__ __forceinline__ int list_owner(int incl, int slot)
{
    int own = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1) {
        const int e = __shfl_sync(0xffffffffu, incl, own + st - 1);
        if (e <= slot) own += st;
    }
    return own;
}

// Every step of a kept beam in FP64: geometry, cull, beam, Neumaier accumulation.  FP64
// issues at 1/64 of the FP32 rate, so what bounds it is the number of FP64 instructions in
// which lanes idle or reject: a warp gathers the segments that reach the ball of its 32
// receivers (as the FP32 kernels do) and an FP32 prefilter with a margin marks the candidates
// among 32 of them.  The marked pairs go through the FP64 geometry and cull 32 at a time, a
// lane per pair, and what they keep through the beam 32 at a time, a lane per (pair, band),
// whoever owns the receiver; each receiver's lane then adds its terms in segment order.
// Candidates are listed segment by segment, so that a window's terms belong to many lanes
// (listed lane by lane, 10 of 32 lanes were active).  16,384 rays x 128^2 receivers x 2
// bands: 35.4 ms testing every pair in FP64, 2.2 ms so,
// bit for bit the same field.
template <int WINDOW, int NF>
__global__ void __launch_bounds__(32 * kWarps64) gbs_fwd_f64_kernel(const __grid_constant__ F64Params p)
{
    __shared__ Warp64<NF> all[kWarps64];
    const int lane = threadIdx.x & 31;
    Warp64<NF> &w = all[threadIdx.x >> 5];
    Item m;
    m.wbase = ((int64_t)blockIdx.x * kWarps64 + (threadIdx.x >> 5)) * 32;
    if (m.wbase >= p.n_recv) return;            // warps never wait for one another
    m.split = blockIdx.y;
    m.splits = p.g.splits;
    m.lst = nullptr;
    m.lw = nullptr;
    m.n_seg = *p.g.n_seg_ptr;
    const int64_t r = m.wbase + lane;
    const bool valid = r < p.n_recv;
    const int64_t ri = valid ? (p.order ? p.order[r] : r) : 0;
    const float xf = valid ? p.recv[3 * ri] : 0.f, yf = valid ? p.recv[3 * ri + 1] : 0.f,
                zf = valid ? p.recv[3 * ri + 2] : 0.f;
    // ball about the centre c of the receivers' bounding box
    const bool part = valid && takes_part(xf, yf, zf);
    const float v[3] = {xf, yf, zf};
    float ctr[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const unsigned u = ordered_bits(v[a]);
        ctr[a] = 0.5f * from_ordered(__reduce_min_sync(0xffffffffu, part ? u : ~0u)) +
                 0.5f * from_ordered(__reduce_max_sync(0xffffffffu, part ? u : 0u));
    }
    const float xp = xf - ctr[0], yp = yf - ctr[1], zp = zf - ctr[2];
    const float xx = fmaf(xp, xp, fmaf(yp, yp, zp * zp));
    const float rad = 1.000001f * sqrtf(__uint_as_float(
        __reduce_max_sync(0xffffffffu, part ? __float_as_uint(xx) : 0u)));
    const float4 rball = reach_ball(make_float4(ctr[0], ctr[1], ctr[2], rad));
    const float alpha = p.g.pre_alpha, beta = p.g.pre_beta, naxx = -alpha * xx;
    const double c2 = 2.0 * p.cutoff;

    double sr[NF], cr[NF], si[NF], ci[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) sr[f] = cr[f] = si[f] = ci[f] = 0.0;
    Gather<WINDOW, false> g(m);
    g.issue(p.g, m, w.in, lane, rball, 0);
    g.issue(p.g, m, w.in, lane, rball, 1);
    for (uint32_t kb = 0;; ++kb) {
        const int buf = (int)(kb & 1u);
        const int nrec = buf ? g.n1 : g.n0;
        if (nrec <= 0) break;
        cp_async_wait1();   // this lane's copies of batch kb
        if (lane < nrec) {
            const float4 r0 = w.in.raw[buf][0][lane], r1 = w.in.raw[buf][1][lane], r2 = w.in.raw[buf][2][lane];
            const float ox = (r0.x - ctr[0]) + r2.x, oy = (r0.y - ctr[1]) + r2.y, oz = (r0.z - ctr[2]) + r2.z;
            const float ot = fmaf(ox, r1.x, fmaf(oy, r1.y, oz * r1.z));
            const float oo = fmaf(ox, ox, fmaf(oy, oy, oz * oz));
            const float a2 = 2.f * alpha;
            w.P[0][lane] = make_float4(r1.x, r1.y, r1.z, -ot);
            // What the prefilter's terms may lose: with M = |o'| + |x'| the rounding of o', x' and t
            // moves n^2 by at most 10 x 2^-24 M^2, that of the sums alpha s_loc^2 and alpha |x' - o'|^2,
            // which cancel, by about 30 x 2^-24 alpha M^2 more, whatever s is; and s by 6 x 2^-24 M.
            const float M = sqrtf(oo) + rad;
            w.P[1][lane] = make_float4(a2 * ox, a2 * oy, a2 * oz,
                                       fmaf(-alpha, oo, beta) + 3e-6f * alpha * M * M);
            const float mg = kWinMargin + 1e-6f * (fabsf(ox) + fabsf(oy) + fabsf(oz) + rad);
            w.P[2][lane] = make_float4(r0.w + mg, r1.w + mg, mg, 0.f);
            w.seg[lane] = buf ? g.seg1 : g.seg0;
        }
        __syncwarp();
        g.issue(p.g, m, w.in, lane, rball, buf);
        // candidates, frequency independent: s_loc = x'.t - o'.t, sm = s_loc + s0 + margin,
        // sm^2 + beta - alpha |x' - o'|^2 + alpha s_loc^2 (= q - alpha n^2) >= 0, window
        uint32_t mine = 0u;                   // lane j: the lanes that are candidates of segment j
        for (int j = 0; j < nrec; ++j) {
            const float4 a = w.P[0][j], b = w.P[1][j], q = w.P[2][j];
            const float sl = fmaf(xp, a.x, fmaf(yp, a.y, fmaf(zp, a.z, a.w)));
            const float sm = sl + q.x;
            const float nd = fmaf(xp, b.x, fmaf(yp, b.y, fmaf(zp, b.z, naxx + b.w)));
            // (an overflow leaves the pair a candidate)
            bool keep = part && !(fmaf(alpha * sl, sl, fmaf(sm, sm, nd)) < 0.f);
            if (WINDOW == GBT_WINDOW_LINE) keep = keep && !(sm < 0.f);
            else keep = keep && !(sl + q.z < 0.f) && !(sl >= q.y);
            const uint32_t b32 = __ballot_sync(0xffffffffu, keep);
            if (lane == j) mine = b32;
        }
        // the segments' candidates as one list: segment j's at [incl - cnt, incl) of lane j
        const int cnt = __popc(mine);
        const int incl = warp_scan(cnt, lane);
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        for (int w0 = 0; w0 < total; w0 += 32) {
            const int slot = w0 + lane;
            const int sj = list_owner(incl, slot);
            const int rank = slot - __shfl_sync(0xffffffffu, incl - cnt, sj);
            const uint32_t lanes = __shfl_sync(0xffffffffu, mine, sj);
            const int rl = slot < total ? nth_bit(lanes, rank) : 0;
            const double x = (double)__shfl_sync(0xffffffffu, xf, rl);
            const double y = (double)__shfl_sync(0xffffffffu, yf, rl);
            const double z = (double)__shfl_sync(0xffffffffu, zf, rl);
            uint32_t kf = 0u;                 // frequencies this pair keeps
            if (slot < total) {
                const int64_t j = w.seg[sj];
                const double dx = x - p.o[3 * j], dy = y - p.o[3 * j + 1], dz = z - p.o[3 * j + 2];
                const double tx = p.t[3 * j], ty = p.t[3 * j + 1], tz = p.t[3 * j + 2];
                const double sl = dx * tx + dy * ty + dz * tz;
                const double s = p.s0[j] + sl;
                const bool in = WINDOW == GBT_WINDOW_SEGMENT ? sl >= 0.0 && sl < p.L[j] : s >= 0.0;
                const double cx = dy * tz - dz * ty, cy = dz * tx - dx * tz, cz = dx * ty - dy * tx;
                const double n2 = cx * cx + cy * cy + cz * cz;
                const double ss = s * s;
                if (in) {
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        if (f >= p.nf) break;
                        kf |= (uint32_t)!(p.kb[f] * n2 > c2 * (ss + p.b2[f])) << f;
                    }
                }
                w.geo[lane] = make_double2(s, n2);
                w.pair_seg[lane] = (int32_t)j;
            }
            w.kept[lane] = kf;
            const int kc = __popc(kf), kincl = warp_scan(kc, lane);
            const int ktotal = __shfl_sync(0xffffffffu, kincl, 31);
            __syncwarp();
            for (int v0 = 0; v0 < ktotal; v0 += 32) {
                const int ks = v0 + lane;
                const int ps = list_owner(kincl, ks);
                const int krank = ks - __shfl_sync(0xffffffffu, kincl - kc, ps);
                if (ks < ktotal) {
                    const int f = nth_bit(w.kept[ps], krank);
                    const int64_t j = w.pair_seg[ps];
                    const double s = w.geo[ps].x, n2 = w.geo[ps].y;
                    const double k = p.k[f], b = p.b[f], kb = p.kb[f];
                    // c = amp * (k b / 8 pi^2) / E * exp(i k s + i k n^2 / (2E)), E = s - i b
                    const double invD = 1.0 / (s * s + p.b2[f]);
                    const double re_exp = -0.5 * kb * n2 * invD - p.absorb[f] * s;
                    const double ph = k * s + 0.5 * k * n2 * s * invD;
                    const double a = p.amp[j] * (kb / (8.0 * kPi * kPi)) * exp(re_exp) * invD;
                    double sn, cs;
                    sincos(ph, &sn, &cs);
                    double2 v = make_double2(a * (s * cs - b * sn), a * (s * sn + b * cs));
                    if (p.r64) {
                        const double2 R = p.r64[(int64_t)f * p.r64_stride + j];
                        v = make_double2(v.x * R.x - v.y * R.y, v.x * R.y + v.y * R.x);
                    }
                    w.term[f][ps] = v;
                }
            }
            __syncwarp();
            const int last = __shfl_sync(0xffffffffu, sj, min(total - w0, 32) - 1);
            for (int q = __shfl_sync(0xffffffffu, sj, 0); q <= last; ++q) {
                const uint32_t own = __shfl_sync(0xffffffffu, mine, q);
                const int at = __shfl_sync(0xffffffffu, incl - cnt, q) + __popc(own & ((1u << lane) - 1u)) - w0;
                const uint32_t bits = ((own >> lane) & 1u) && at >= 0 && at < 32 ? w.kept[at] : 0u;
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    if ((bits >> f) & 1u) {
                        const double2 v = w.term[f][at];
                        // Neumaier accumulation
                        const double t1 = sr[f] + v.x;
                        cr[f] += fabs(sr[f]) >= fabs(v.x) ? (sr[f] - t1) + v.x : (v.x - t1) + sr[f];
                        sr[f] = t1;
                        const double t2 = si[f] + v.y;
                        ci[f] += fabs(si[f]) >= fabs(v.y) ? (si[f] - t2) + v.y : (v.y - t2) + si[f];
                        si[f] = t2;
                    }
                }
            }
            __syncwarp();       // before the next window
        }
        __syncwarp();           // before the next batch is staged over this one
    }
    cp_async_wait0();
    if (!valid) return;
#pragma unroll
    for (int f = 0; f < NF; ++f)
        if (f < p.nf)
            p.partial[((int64_t)m.split * p.nf + f) * p.n_recv + ri] =
                make_double2(sr[f] + cr[f], si[f] + ci[f]);
}

template <int WINDOW>
void launch_f64(const F64Params &q, dim3 grid, cudaStream_t s)
{
    if (q.nf <= 1) gbs_fwd_f64_kernel<WINDOW, 1><<<grid, 32 * kWarps64, 0, s>>>(q);
    else if (q.nf <= 2) gbs_fwd_f64_kernel<WINDOW, 2><<<grid, 32 * kWarps64, 0, s>>>(q);
    else if (q.nf <= 4) gbs_fwd_f64_kernel<WINDOW, 4><<<grid, 32 * kWarps64, 0, s>>>(q);
    else if (q.nf <= 8) gbs_fwd_f64_kernel<WINDOW, 8><<<grid, 32 * kWarps64, 0, s>>>(q);
    else gbs_fwd_f64_kernel<WINDOW, GBT_MAX_FREQ><<<grid, 32 * kWarps64, 0, s>>>(q);
}

// ------------------------------------------------------------ adjoint --

// Per ray: the weight gradient sum_j Gamma_path_j G_j, the material gradient
// sum over bounces of W (product of the other bounces' gamma) G_j, and the beam
// parameter gradient sum_j W Gamma_path_j H_jf.  The products of the other bounces are the
// ones before a bounce times a backward recurrence over the ones after it, so gamma = 0 needs
// no special case and a ray costs its length (formed directly they cost its square, with an
// atomic per segment and bounce and per segment and band: 345 us for 262,144 rays, 838,595
// segments, 4 bands; 102 us so).
struct RayGradParams {
    int64_t n_rays, ray_begin;
    const int32_t *ray_off, *bmat;
    const float *gamma, *weight;
    FanDev fan;
    int64_t n_fan;
    const float *seg_G, *seg_H;
    int64_t seg_stride;
    int nf, n_materials;
    float *grad_w;             // n_fan entries (this range written), or nullptr
    double *acc;               // [n_materials] gamma, then [nf] b (sorted slots)
    unsigned int *status;
};

constexpr int kMaxDepth = 65;

template <int NF>
__global__ void __launch_bounds__(128) ray_grad_kernel(RayGradParams p)
{
    extern __shared__ double sacc[];
    const int nacc = p.n_materials + p.nf;
    for (int k = threadIdx.x; k < nacc; k += blockDim.x) sacc[k] = 0.0;
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double hb[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) hb[f] = 0.0;
    if (i < p.n_rays) {
        const int64_t a = p.ray_off[i];
        const int cnt = min((int)(p.ray_off[i + 1] - a), kMaxDepth);
        const double W = p.weight ? (double)p.weight[p.ray_begin + i]
                                  : fan_weight(p.fan, p.n_fan, p.ray_begin + i);
        double pre[kMaxDepth];     // pre[d]: product of gamma over the bounces 1 .. d
        double gp = 1.0, gw = 0.0;
        for (int d = 0; d < cnt; ++d) {
            const int64_t j = a + d;
            if (d >= 1) {
                int m = p.bmat[j];
                if (m < 0 || m >= p.n_materials) {
                    atomicOr(p.status, STATUS_BOUNDS);
                    m = 0;
                }
                gp *= (double)p.gamma[m];
            }
            pre[d] = gp;
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                // a zero adds nothing, whatever the weight and the coefficients are
                const double H = f < p.nf ? (double)p.seg_H[f * p.seg_stride + j] : 0.0;
                if (H != 0.0) hb[f] += W * gp * H;
            }
            gw += gp * (double)p.seg_G[j];
        }
        // S_d = sum over d' >= d of (product of gamma over the bounces d + 1 .. d') G_d'
        double S = 0.0;
        for (int d = cnt - 1; d >= 0; --d) {
            const int64_t j = a + d;
            S += (double)p.seg_G[j];
            if (d >= 1) {
                int m = p.bmat[j];
                if (m < 0 || m >= p.n_materials) m = 0;
                if (S != 0.0) {
                    atomicAdd(&sacc[m], W * pre[d - 1] * S);
                    S *= (double)p.gamma[m];
                }
            }
        }
        if (p.grad_w) p.grad_w[p.ray_begin + i] = (float)gw;
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (f >= p.nf) break;
        double v = hb[f];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(&sacc[p.n_materials + f], v);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nacc; k += blockDim.x)
        if (sacc[k] != 0.0) atomicAdd(&p.acc[k], sacc[k]);
}

struct GradOutParams {
    const double *acc;
    int n_materials, nf;
    int fperm[GBT_MAX_FREQ];
    float *grad_gamma;
    double *grad_b;
};

__global__ void grad_out_kernel(GradOutParams p)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < p.n_materials) p.grad_gamma[k] = (float)p.acc[k];
    else if (k < p.n_materials + p.nf && p.grad_b)
        p.grad_b[p.fperm[k - p.n_materials]] = p.acc[k];
}

// ------------------------------------------------------------- reduce --

// ---- dispatch order of the CTA tiles: heaviest first
// Items of one tile cost about the same (their batches interleave over the whole
// segment list), but tiles differ by the number of beams that reach them.  A
// sampled count of segments whose Gaussian can reach each tile's bounding ball
// ranks the tiles so the persistent CTAs take the heavy ones first and the queue
// drains with light items (longest processing time first).  The order only
// changes which CTA computes an item, never the arithmetic of any sum.
constexpr int kWeightSamples = 1 << 15;        // sampled segments per estimate
constexpr int64_t kMaxOrderedTiles = 1 << 14;  // beyond this the rank pass is skipped
constexpr int64_t kOrderPairs = int64_t(1) << 31;   // (receiver, segment slot) pairs, see tile_ws_layout
constexpr int64_t kOrderTiles = 24;


// Also each tile's reach ball (the list passes' form, with the ball's share of the slack).
__global__ void tile_ball_kernel(const float *recv, const int32_t *order, int64_t n_recv,
                                 float4 *ball, unsigned int *weight, float4 *rball)
{
    __shared__ float red[5][8];
    const int64_t base = (int64_t)blockIdx.x * kCtaRecv;
    const int n = (int)(n_recv - base < (int64_t)kCtaRecv ? n_recv - base : (int64_t)kCtaRecv);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float sx = 0.f, sy = 0.f, sz = 0.f, nv = 0.f;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int64_t o = order ? order[base + j] : base + j;
        const float x = recv[3 * o], y = recv[3 * o + 1], z = recv[3 * o + 2];
        if (takes_part(x, y, z)) { sx += x; sy += y; sz += z; nv += 1.f; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
        sz += __shfl_xor_sync(0xffffffffu, sz, o);
        nv += __shfl_xor_sync(0xffffffffu, nv, o);
    }
    if (lane == 0) { red[0][wid] = sx; red[1][wid] = sy; red[2][wid] = sz; red[4][wid] = nv; }
    __syncthreads();
    sx = sy = sz = nv = 0.f;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
        sx += red[0][k]; sy += red[1][k]; sz += red[2][k]; nv += red[4][k];
    }
    nv = fmaxf(nv, 1.f);
    const float cx = sx / nv, cy = sy / nv, cz = sz / nv;
    float r2 = 0.f;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int64_t o = order ? order[base + j] : base + j;
        const float x = recv[3 * o], y = recv[3 * o + 1], z = recv[3 * o + 2];
        const float dx = x - cx, dy = y - cy, dz = z - cz;
        if (takes_part(x, y, z)) r2 = fmaxf(r2, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    }
    for (int o = 16; o > 0; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
    __syncthreads();
    if (lane == 0) red[3][wid] = r2;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) r2 = fmaxf(r2, red[3][k]);
        ball[blockIdx.x] = make_float4(cx, cy, cz, sqrtf(r2));
        rball[blockIdx.x] = reach_ball(ball[blockIdx.x]);
        weight[blockIdx.x] = 0u;
    }
}

// Bounding ball of each warp tile (64 receivers), one warp per warp tile.
__global__ void warp_ball_kernel(const float *recv, const int32_t *order, int64_t n_recv,
                                 int64_t n_wtiles, float4 *wball)
{
    const int64_t wt = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (wt >= n_wtiles) return;
    float x[2] = {0.f, 0.f}, y[2] = {0.f, 0.f}, z[2] = {0.f, 0.f};
    float sx = 0.f, sy = 0.f, sz = 0.f, nv = 0.f;
    bool ok[2];
    for (int k = 0; k < 2; ++k) {
        const int64_t r = wt * kWarpRecv + k * 32 + lane;
        ok[k] = r < n_recv;
        if (ok[k]) {
            const int64_t o = order ? order[r] : r;
            x[k] = recv[3 * o]; y[k] = recv[3 * o + 1]; z[k] = recv[3 * o + 2];
            ok[k] = takes_part(x[k], y[k], z[k]);
        }
        if (ok[k]) { sx += x[k]; sy += y[k]; sz += z[k]; nv += 1.f; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
        sz += __shfl_xor_sync(0xffffffffu, sz, o);
        nv += __shfl_xor_sync(0xffffffffu, nv, o);
    }
    if (nv > 0.f) { sx /= nv; sy /= nv; sz /= nv; }
    float r2 = 0.f;
    for (int k = 0; k < 2; ++k)
        if (ok[k]) {
            const float dx = x[k] - sx, dy = y[k] - sy, dz = z[k] - sz;
            r2 = fmaxf(r2, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        }
    for (int o = 16; o > 0; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
    if (lane == 0) wball[wt] = make_float4(sx, sy, sz, sqrtf(r2));
}

template <int WINDOW>
__global__ void tile_weight_kernel(const float4 *crec, const int32_t *n_seg_ptr, const float4 *ball,
                                   int64_t n_tiles, float alpha, float beta, unsigned int *weight)
{
    const int64_t ns = *n_seg_ptr;
    const int64_t stride = ns > kWeightSamples ? (ns + kWeightSamples - 1) / kWeightSamples : 1;
    const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * stride;
    const bool ok = j < ns;
    float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
    if (ok) {
        r0 = crec[2 * j];
        r1 = crec[2 * j + 1];
    }
    for (int64_t t = blockIdx.y; t < n_tiles; t += gridDim.y) {
        const float4 b = ball[t];
        bool pass = false;
        if (ok)
            pass = ball_may_keep<WINDOW>(r0, r1, r0.x - b.x, r0.y - b.y, r0.z - b.z,
                                         make_float4(0.f, 0.f, 0.f, b.w), alpha, beta);
        // one atomic per block: a warp each, on a few dozen tiles, took 23 us in contention
        const int c = __syncthreads_count(pass);
        if (threadIdx.x == 0 && c) atomicAdd(&weight[t], (unsigned int)c);
    }
}

// perm[rank] = tile, ranks by weight descending, ties by tile index (a permutation)
__global__ void tile_rank_kernel(const unsigned int *weight, int64_t n_tiles, int32_t *perm)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tiles) return;
    const unsigned int wt = weight[t];
    int64_t rank = 0;
    for (int64_t u = 0; u < n_tiles; ++u) {
        const unsigned int wu = weight[u];
        rank += (wu > wt) || (wu == wt && u < t);
    }
    perm[rank] = (int32_t)t;
}

// ---- tile pre-cull: per CTA tile, the list of segments that can reach it
// Two passes over (chunk of 1024 segments) x (tile) with the ball test of the
// pre-cull: counts, then the indices, each tile's list in segment order (so the
// sums keep their order and stay deterministic).  Tiles take consecutive ranges
// of the list buffer lightest first; a tile that does not fit streams every
// segment, which gives the same field.
constexpr int kListChunk = 1024;

template <int WINDOW>
__global__ void __launch_bounds__(kListChunk) list_count_kernel(
    const float4 *crec, const int32_t *n_seg_ptr, const float4 *rball, int64_t n_tiles,
    int64_t n_chunks, float alpha, float beta, int32_t *counts, uint32_t *bits)
{
    // block (c, g): chunk c against the 32-tile groups g, g + G, ... (G = gridDim.y); lane
    // k of each warp keeps tile k's ballot of the group, so the group ends with one count
    // and one ballot store per lane
    extern __shared__ int32_t cnt_s[];
    const int64_t G = gridDim.y, g = blockIdx.y;
    for (int64_t t = threadIdx.x; t < n_tiles; t += blockDim.x) cnt_s[t] = 0;
    __syncthreads();
    const int64_t ns = *n_seg_ptr;
    const int64_t c = blockIdx.x;
    if (c * kListChunk < ns) {
        const int64_t j = c * kListChunk + threadIdx.x;
        const bool ok = j < ns;
        float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
        if (ok) {
            r0 = crec[2 * j];
            r1 = crec[2 * j + 1];
        }
        const SegCull sg = seg_cull(r0, r1);
        const int lane = threadIdx.x & 31;
        for (int64_t t0 = g * 32; t0 < n_tiles; t0 += G * 32) {
            const int nt = (int)min((int64_t)32, n_tiles - t0);
            uint32_t mine = 0u;
            for (int k = 0; k < nt; ++k) {
                const bool pass = ok && seg_reaches_ball<WINDOW>(sg, rball[t0 + k], alpha, beta);
                const uint32_t m = __ballot_sync(0xffffffffu, pass);
                if (lane == k) mine = m;
            }
            if (lane < nt) {
                if (mine) atomicAdd(&cnt_s[t0 + lane], (int32_t)__popc(mine));
                if (bits) bits[(t0 + lane) * n_chunks * 32 + c * 32 + (threadIdx.x >> 5)] = mine;
            }
        }
    }
    __syncthreads();
    for (int64_t t = threadIdx.x; t < n_tiles; t += blockDim.x)
        if ((t / 32) % G == g) counts[t * n_chunks + c] = cnt_s[t];
}

// Exclusive scan of 1024 values held one per thread; returns the block total.
__device__ __forceinline__ int64_t block_scan_1024(int64_t v, int64_t &excl, int64_t *ws)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int64_t x = ws[lane];
        int64_t xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += y;
        }
        ws[lane] = xi - x;
        if (lane == 31) ws[32] = xi;
    }
    __syncthreads();
    excl = incl - v + ws[wid];
    const int64_t total = ws[32];
    __syncthreads();
    return total;
}

// One block per tile: chunk counts -> exclusive offsets within the tile; the tile's total.
__global__ void __launch_bounds__(1024) list_scan_chunks_kernel(int32_t *counts, int64_t n_chunks,
                                                                unsigned int *total)
{
    __shared__ int64_t ws[33];
    int32_t *row = counts + (int64_t)blockIdx.x * n_chunks;
    int64_t carry = 0;
    for (int64_t base = 0; base < n_chunks; base += 1024) {
        const int64_t c = base + threadIdx.x;
        const int64_t v = c < n_chunks ? row[c] : 0;
        int64_t excl;
        const int64_t tot = block_scan_1024(v, excl, ws);
        if (c < n_chunks) row[c] = (int32_t)(carry + excl);
        carry += tot;
    }
    if (threadIdx.x == 0) total[blockIdx.x] = (unsigned int)carry;
}

// Per 32-entry chunk of a tile list, one word per warp tile of the CTA tile: bit b set
// if entry b can reach the warp tile's ball.  Each warp takes whole chunks (blocks
// (g, t) stride over tile t's chunks) and writes the chunk's 16 words in one store.
template <int WINDOW>
__global__ void list_words_kernel(const float4 *crec, const float4 *wball, int64_t n_wtiles,
                                  float alpha, float beta, const int64_t *list_off,
                                  const int32_t *list_n, const int32_t *list, uint32_t *list_words)
{
    static_assert(kTileWarps <= kChunkWords, "one word per warp tile");
    __shared__ float4 sball[kTileWarps];
    const int64_t t = blockIdx.y;
    const int32_t n = list_n[t];
    if (n <= 0) return;                    // uniform over the block
    const int nw = (int)min((int64_t)kTileWarps, n_wtiles - t * kTileWarps);
    if (threadIdx.x < nw) sball[threadIdx.x] = reach_ball(wball[t * kTileWarps + threadIdx.x]);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t off = list_off[t];       // a multiple of 32
    uint32_t *words = list_words + (off / 32) * kChunkWords;
    const int64_t n_ch = ((int64_t)n + 31) / 32;
    const int64_t wpb = blockDim.x / 32;
    for (int64_t ch = (int64_t)blockIdx.x * wpb + (threadIdx.x >> 5); ch < n_ch;
         ch += (int64_t)gridDim.x * wpb) {
        const int64_t i = ch * 32 + lane;
        const bool in = i < n;
        float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
        if (in) {
            const int64_t jseg = list[off + i];
            r0 = crec[2 * jseg];
            r1 = crec[2 * jseg + 1];
        }
        const SegCull sg = seg_cull(r0, r1);
        uint32_t mine = 0u;
        for (int w = 0; w < nw; ++w) {
            const uint32_t m = __ballot_sync(
                0xffffffffu, in && seg_reaches_ball<WINDOW>(sg, sball[w], alpha, beta));
            if (lane == w) mine = m;
        }
        if (lane < kChunkWords) words[ch * kChunkWords + lane] = mine;
    }
}

// One block: list ranges, tiles lightest first (perm lists them heaviest first), each
// starting on a 32-entry chunk boundary; and, with want > 0, each tile's segment splits,
// want per tile on average (at most (want + 1) x n_tiles in all), numbered heaviest tile
// first.  A tile's share goes with the root of its list length, its cost: equal shares make
// the heavy tiles' items ten times the mean, so that the queue drains well only with three
// times as many of them, whose per-item work and partial sums then cost more than the tail
// they save; shares with the cost itself make the last items as long as the first.  Equal
// (32 items per warp) | root (12) | cost (12), in ms: 1 M rays x 512^2 x 1 band, city,
// 22.4 | 19.4 | 20.4; 192^2 x 8 bands with losses 6.40 | 6.42 | 6.94; batch of 8 sources x
// 128^2 x 8 bands 4.63 | 3.62 | 3.67; 9,973 scattered receivers .724 | .701 | .697.
__global__ void __launch_bounds__(1024) list_layout_kernel(const unsigned int *total,
                                                           const int32_t *perm, int64_t n_tiles,
                                                           int64_t cap, int64_t *list_off,
                                                           int32_t *list_n, const int32_t *n_seg_ptr,
                                                           int64_t want, int32_t *item_off,
                                                           int32_t *tile_first, int32_t *tile_splits)
{
    __shared__ int64_t ws[33];
    const int64_t per = (n_tiles + 1023) / 1024;
    const int64_t i0 = (int64_t)threadIdx.x * per;
    auto tile_at = [&](int64_t i) {   // i-th lightest tile
        const int64_t r = n_tiles - 1 - i;
        return perm ? (int64_t)perm[r] : r;
    };
    auto padded = [](int64_t n) { return (n + 31) / 32 * 32; };   // whole 32-entry chunks
    int64_t sum = 0;
    for (int64_t i = i0; i < i0 + per && i < n_tiles; ++i) sum += padded(total[tile_at(i)]);
    int64_t off;
    block_scan_1024(sum, off, ws);
    for (int64_t i = i0; i < i0 + per && i < n_tiles; ++i) {
        const int64_t t = tile_at(i);
        const int64_t n = total[t];
        list_off[t] = off;
        list_n[t] = off + padded(n) <= cap ? (int32_t)n : -1;
        off += padded(n);
    }
    if (want <= 0) return;
    __syncthreads();       // every list_n is written
    const int64_t scan_cost = *n_seg_ptr / 8;      // a tile without a list tests every segment
    auto rank_tile = [&](int64_t r) { return perm ? (int64_t)perm[r] : r; };
    auto cost = [&](int64_t t) { return (int64_t)total[t] + (list_n[t] < 0 ? scan_cost : 0); };
    auto share = [&](int64_t t) { return (int64_t)(64.0f * sqrtf((float)cost(t))) + 1; };
    sum = 0;
    for (int64_t r = i0; r < i0 + per && r < n_tiles; ++r) sum += share(rank_tile(r));
    int64_t at;
    const int64_t all = block_scan_1024(sum, at, ws);
    const int64_t each = max((all + want - 1) / want, (int64_t)1);
    auto splits = [&](int64_t t) {
        return max(min((share(t) + each - 1) / each, (cost(t) + 63) / 64), (int64_t)1);
    };
    sum = 0;
    for (int64_t r = i0; r < i0 + per && r < n_tiles; ++r) sum += splits(rank_tile(r));
    const int64_t n_items = block_scan_1024(sum, at, ws);
    for (int64_t r = i0; r < i0 + per && r < n_tiles; ++r) {
        const int64_t t = rank_tile(r), s = splits(t);
        item_off[r] = (int32_t)at;
        tile_first[t] = (int32_t)at;
        tile_splits[t] = (int32_t)s;
        at += s;
    }
    if (threadIdx.x == 0) item_off[n_tiles] = (int32_t)n_items;
}

template <int WINDOW>
__global__ void __launch_bounds__(kListChunk) list_write_kernel(
    const float4 *crec, const int32_t *n_seg_ptr, const float4 *rball, int64_t n_tiles,
    int64_t n_chunks, float alpha, float beta, const int32_t *chunk_off, const int64_t *list_off,
    const int32_t *list_n, int32_t *list)
{
    __shared__ int32_t wsum[32];
    const int64_t ns = *n_seg_ptr;
    const int64_t c = blockIdx.x;
    if (c * kListChunk >= ns) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t j = c * kListChunk + threadIdx.x;
    const bool ok = j < ns;
    float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
    if (ok) {
        r0 = crec[2 * j];
        r1 = crec[2 * j + 1];
    }
    const SegCull sg = seg_cull(r0, r1);
    for (int64_t t = 0; t < n_tiles; ++t) {
        if (list_n[t] < 0) continue;
        const bool pass = ok && seg_reaches_ball<WINDOW>(sg, rball[t], alpha, beta);
        const unsigned int m = __ballot_sync(0xffffffffu, pass);
        if (lane == 0) wsum[wid] = __popc(m);
        __syncthreads();
        int before = 0;
        for (int w = 0; w < wid; ++w) before += wsum[w];
        if (pass)
            list[list_off[t] + chunk_off[t * n_chunks + c] + before +
                 __popc(m & ((1u << lane) - 1u))] = (int32_t)j;
        __syncthreads();
    }
}

// The same lists from the ballots the counting pass stored (one 32-bit word per tile and
// 32 segments): no ball test is repeated.  A warp takes a (tile, chunk) row, a word a lane: one
// scan places the words.  A dense row (over a quarter of its bits) then goes out a word at a
// time; in a sparse one each lane writes its entries to shared memory in order, and the row
// leaves in whole lines (dense rows that way too: 11 us for 9,973 scattered receivers instead
// of 4).  (A warp per word, finding its place from the earlier words of its
// row, was bound by those instructions: 1 M rays x 512^2 receivers, 274 tiles: 717 us, 188
// so.)
constexpr int kWriteWarps = 8;
__global__ void __launch_bounds__(32 * kWriteWarps) list_write_bits_kernel(
    const int32_t *n_seg_ptr, int64_t n_tiles, int64_t n_chunks, const uint32_t *bits,
    const int32_t *chunk_off, const int64_t *list_off, const int32_t *list_n, int32_t *list)
{
    __shared__ int32_t rows[kWriteWarps][kListChunk];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *const row = rows[wid];
    const int64_t used = ((int64_t)*n_seg_ptr + kListChunk - 1) / kListChunk;
    for (int64_t t = blockIdx.y; t < n_tiles; t += gridDim.y) {
        if (list_n[t] <= 0) continue;
        for (int64_t c = (int64_t)blockIdx.x * kWriteWarps + wid; c < used;
             c += (int64_t)gridDim.x * kWriteWarps) {
            uint32_t m = bits[(t * n_chunks + c) * 32 + lane];
            const int n = __popc(m);
            int at = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, at, o);
                if (lane >= o) at += y;
            }
            const int total = __shfl_sync(0xffffffffu, at, 31);
            if (total == 0) continue;
            at -= n;
            int32_t *const dst = list + list_off[t] + chunk_off[t * n_chunks + c];
            const int32_t jc = (int32_t)(c * kListChunk);
            if (total > kListChunk / 4) {       // dense: a word at a time, straight to the list
#pragma unroll 4
                for (int w = 0; w < 32; ++w) {
                    const uint32_t mw = __shfl_sync(0xffffffffu, m, w);
                    const int aw = __shfl_sync(0xffffffffu, at, w);
                    if ((mw >> lane) & 1u) dst[aw + __popc(mw & ((1u << lane) - 1u))] = jc + 32 * w + lane;
                }
                continue;
            }
            const int32_t j0 = jc + 32 * lane;
            while (m) {
                row[at++] = j0 + __ffs(m) - 1;
                m &= m - 1u;
            }
            __syncwarp();
            for (int i = lane; i < total; i += 32) dst[i] = row[i];
            __syncwarp();
        }
    }
}

// Time synthesis: out[n, r] (+)= Re sum_f A_f p[f, r] exp(-i omega_f t_n).  Bound by writing
// n_t * n_recv floats, with the FMAs close behind; so samples are taken in pairs about the
// centre t_c of the block's kSynthTile samples: with A_f p exp(-i omega_f t_c) = u - i v,
//   h(t_c +- d) = sum_f u cos(omega_f d) -+ sum_f v sin(omega_f d),
// two FMAs per band and pair of samples instead of four.  The offsets' turns are exact in
// two floats, the centre's reduced in FP64 (one per band and block: FP64 arithmetic in every
// offset held the blocks up as long as the stores), and the sine and cosine of the reduced
// turn take in its low part, so that the error is that of FP32 rounding alone.  2,048 samples
// x 65,536 receivers x 6 bands: 99.6 us before, 77.9 now (6.9 TB/s); relative error
// 1.0e-7 before, 7e-8 now.  Threads run over groups of four adjacent receivers (16-byte
// streaming stores), each holding its receivers' u and v in registers; NF is the exact
// frequency count.
constexpr int kSynthTile = 32;
constexpr int kSynthRecv = 4;                   // receivers per thread

struct SynthParams {
    const float2 *p;           // [nf][n_recv] fields
    int64_t n_recv, n_t;
    double step[GBT_MAX_FREQ], start[GBT_MAX_FREQ];     // f dt modulo 2 and f t0, in turns
    double amp_re[GBT_MAX_FREQ], amp_im[GBT_MAX_FREQ];
    float step_hi[GBT_MAX_FREQ], step_lo[GBT_MAX_FREQ]; // step in two floats
    float *out;                // [n_t][n_recv]
    int accumulate;
};

template <int NF>
__global__ void __launch_bounds__(256) synth_kernel(const SynthParams p)
{
    __shared__ float2 rot[kSynthTile / 2][NF];   // cos, sin of omega_f (k + 1/2) dt
    __shared__ float2 centre[NF];                // A_f exp(-i omega_f t_c)
    const int64_t n0 = (int64_t)blockIdx.y * kSynthTile;
    // cosine and sine of th + tl turns, |th| <= 1/2
    auto phasor = [](float th, float tl) {
        float s, c;
        sincospif(2.0f * th, &s, &c);
        const float e = 6.2831853f * tl;
        return make_float2(fmaf(-s, e, c), fmaf(c, e, s));
    };
    for (int i = threadIdx.x; i < kSynthTile / 2 * NF; i += blockDim.x) {
        const int a = i / NF, f = i - a * NF;
        const float k = (float)a + 0.5f, h = k * p.step_hi[f];
        rot[a][f] = phasor(h - rintf(h), fmaf(k, p.step_hi[f], -h) + k * p.step_lo[f]);
    }
    if (threadIdx.x >= 224 && threadIdx.x < 224 + NF) {
        const int f = threadIdx.x - 224;
        double turns = fma((double)n0 + 0.5 * (kSynthTile - 1), p.step[f], p.start[f]);
        turns -= rint(turns);
        const float th = (float)turns;
        const float2 w = phasor(th, (float)(turns - (double)th));
        centre[f] = make_float2((float)(p.amp_re[f] * w.x + p.amp_im[f] * w.y),    // A (cos - i sin)
                                (float)(p.amp_im[f] * w.x - p.amp_re[f] * w.y));
    }
    __syncthreads();
    const int64_t r = kSynthRecv * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
    if (r >= p.n_recv) return;
    const int nr = (int)min((int64_t)kSynthRecv, p.n_recv - r);
    float u[kSynthRecv][NF], v[kSynthRecv][NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const float2 c = centre[f];
#pragma unroll
        for (int k = 0; k < kSynthRecv; ++k) {
            const float2 q = k < nr ? p.p[(int64_t)f * p.n_recv + r + k] : make_float2(0.f, 0.f);
            u[k][f] = fmaf(q.x, c.x, -q.y * c.y);
            v[k][f] = -fmaf(q.x, c.y, q.y * c.x);
        }
    }
    const int na = (int)min((int64_t)kSynthTile, p.n_t - n0);
    float *o = p.out + n0 * p.n_recv + r;
    // 16-byte stores need a row length divisible by four (every row then starts aligned)
    const bool vec = nr == kSynthRecv && !p.accumulate && (p.n_recv & 3) == 0 &&
                     ((uintptr_t)p.out & 15u) == 0;
    auto store = [&](int row_i, const float (&h)[kSynthRecv]) {
        if (row_i >= na) return;
        float *row = o + row_i * p.n_recv;
        if (vec) {
            __stcs(reinterpret_cast<float4 *>(row), make_float4(h[0], h[1], h[2], h[3]));
        } else {
            for (int k = 0; k < nr; ++k) row[k] = p.accumulate ? row[k] + h[k] : h[k];
        }
    };
    for (int a = 0; a < kSynthTile / 2; ++a) {
        if (kSynthTile / 2 - 1 - a >= na) continue;      // neither sample of the pair exists
        float c[kSynthRecv], s[kSynthRecv];
#pragma unroll
        for (int k = 0; k < kSynthRecv; ++k) c[k] = s[k] = 0.f;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const float2 q = rot[a][f];
#pragma unroll
            for (int k = 0; k < kSynthRecv; ++k) {
                c[k] = fmaf(q.x, u[k][f], c[k]);
                s[k] = fmaf(q.y, v[k][f], s[k]);
            }
        }
        float lo[kSynthRecv], hi[kSynthRecv];
#pragma unroll
        for (int k = 0; k < kSynthRecv; ++k) {
            lo[k] = c[k] + s[k];
            hi[k] = c[k] - s[k];
        }
        store(kSynthTile / 2 - 1 - a, lo);
        store(kSynthTile / 2 + a, hi);
    }
}

struct ReduceParams {
    int64_t n;                 // nf * n_recv
    int64_t n_recv;
    int perm[GBT_MAX_FREQ];    // partial frequency slot -> output frequency
    int splits;
    const float4 *p32;         // in processing order of the receivers
    const int32_t *order;      // processing order -> receiver, or null
    float scale[GBT_MAX_FREQ], scale_lo[GBT_MAX_FREQ];   // per slot: the partials' common factor
    const double2 *p64;        // F64 path: by receiver
    float2 *out;
    int accumulate;
    // weighted splits: per tile its first tile-split and their number, or nullptr
    const int32_t *tile_first, *tile_splits;
    int nf, part_recv;
};

// Float-float partials (hi, running FP32 sum of errors) merged into a float-float total with
// error-free FP32 sums: about 44 bits, far beyond the complex64 output, and no FP64
// arithmetic (GB300 issues FP64 at a small fraction of the FP32 rate).  A block takes 32
// outputs; its kMergeGroups warps each sum a consecutive range of the splits and the first
// warp adds the groups in order, so a few thousand receivers with hundreds of splits still
// fill the chip (9,973 receivers, 3 bands, 471 splits: 160 us with one thread per output).
constexpr int kMergeGroups = 8;
__device__ __forceinline__ void merge_ff(float4 &a, const float4 &v)   // (rh, ih, rl, il)
{
    float t, e;
    two_sum(a.x, v.x, t, e);
    a.x = t;
    a.z = __fadd_rn(a.z, __fadd_rn(e, v.z));
    two_sum(a.y, v.y, t, e);
    a.y = t;
    a.w = __fadd_rn(a.w, __fadd_rn(e, v.w));
}
__global__ void __launch_bounds__(32 * kMergeGroups) reduce_kernel(ReduceParams p)
{
    __shared__ float4 part[kMergeGroups][32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)32 + lane;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < p.n) {
        int64_t n = p.splits, stride = p.n;
        const float4 *src = p.p32 + i;
        if (p.tile_first) {
            const int64_t f = i / p.n_recv, r = i - f * p.n_recv, t = r / kCtaRecv;
            n = p.tile_splits[t];
            stride = (int64_t)p.nf * p.part_recv;
            src = p.p32 + p.tile_first[t] * stride + f * p.part_recv + (r - t * kCtaRecv);
        }
        const int s0 = (int)(n * g / kMergeGroups), s1 = (int)(n * (g + 1) / kMergeGroups);
#pragma unroll 8
        for (int s = s0; s < s1; ++s) merge_ff(a, __ldcs(src + s * stride));
    }
    part[g][lane] = a;
    __syncthreads();
    if (g != 0 || i >= p.n) return;
#pragma unroll
    for (int q = 1; q < kMergeGroups; ++q) merge_ff(a, part[q][lane]);
    const int64_t f = i / p.n_recv, r = i - f * p.n_recv;
    const int64_t oi = (int64_t)p.perm[f] * p.n_recv + (p.order ? p.order[r] : r);
    // times the slot's amplitude factor, in float-float (1 leaves the total as it is)
    const float k = p.scale[f], x = __fmul_rn(a.x, k), y = __fmul_rn(a.y, k);
    const float kl = p.scale_lo[f];
    a = make_float4(x, y, fmaf(a.x, kl, fmaf(a.z, k, fmaf(a.x, k, -x))),
                    fmaf(a.y, kl, fmaf(a.w, k, fmaf(a.y, k, -y))));
    if (p.accumulate) {
        const float2 o = p.out[oi];
        merge_ff(a, make_float4(o.x, o.y, 0.f, 0.f));
    }
    p.out[oi] = make_float2(__fadd_rn(a.x, a.z), __fadd_rn(a.y, a.w));
}

// The same for the FP64 partials, of which few receivers have up to 4,096 splits (one receiver,
// 8,000 rays with up to 20 reflections: .33 ms with one thread per output, .10 so).
constexpr int kMergeGroups64 = 16;
__global__ void __launch_bounds__(32 * kMergeGroups64) reduce64_kernel(ReduceParams p)
{
    __shared__ double2 part[kMergeGroups64][32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)32 + lane;
    double re = 0.0, im = 0.0;
    if (i < p.n) {
        const int s0 = (int)((int64_t)p.splits * g / kMergeGroups64);
        const int s1 = (int)((int64_t)p.splits * (g + 1) / kMergeGroups64);
        const double2 *src = p.p64 + i;
#pragma unroll 8
        for (int s = s0; s < s1; ++s) {
            const double2 v = src[(int64_t)s * p.n];
            re += v.x;
            im += v.y;
        }
    }
    part[g][lane] = make_double2(re, im);
    __syncthreads();
    if (g != 0 || i >= p.n) return;
#pragma unroll
    for (int q = 1; q < kMergeGroups64; ++q) {
        re += part[q][lane].x;
        im += part[q][lane].y;
    }
    const int64_t f = i / p.n_recv, r = i - f * p.n_recv;
    const int64_t oi = (int64_t)p.perm[f] * p.n_recv + r;
    if (p.accumulate) {
        const float2 o = p.out[oi];
        re += (double)o.x;
        im += (double)o.y;
    }
    p.out[oi] = make_float2((float)re, (float)im);
}

// The factor of slot f's partials: 1 for the differentiable sum, else the k / (8 pi^2) that the
// pair kernel leaves out (see FreqConst) and what MUFU's sine and cosine lose, which are cut
// towards zero: their amplitude is 7.3e-8 short on average over a turn (measured at 2^22 phases),
// in every term alike, about a third of the field's error.
constexpr double kMufuShort = 7.3e-8;
static void merge_scale(ReduceParams &rp, int f, double freq_hz, double c, bool differentiable)
{
    const double k = 2.0 * kPi * freq_hz / c;
    const double v = differentiable ? 1.0 : k / (8.0 * kPi * kPi) * (1.0 + kMufuShort);
    rp.scale[f] = (float)v;
    rp.scale_lo[f] = (float)(v - (double)rp.scale[f]);
}

static void reduce_launch(const ReduceParams &rp, cudaStream_t s)
{
    if (rp.p32) reduce_kernel<<<(unsigned)((rp.n + 31) / 32), 32 * kMergeGroups, 0, s>>>(rp);
    else reduce64_kernel<<<(unsigned)((rp.n + 31) / 32), 32 * kMergeGroups64, 0, s>>>(rp);
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
}

// ------------------------------------------------------ receiver order --

__global__ void bbox_kernel(const float *recv, int64_t n, unsigned int *bb)
{
    __shared__ unsigned int lo[3], hi[3];
    if (threadIdx.x < 3) { lo[threadIdx.x] = 0xffffffffu; hi[threadIdx.x] = 0u; }
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        for (int a = 0; a < 3; ++a) {
            unsigned int u = ordered_bits(recv[3 * i + a]);
            atomicMin(&lo[a], u);
            atomicMax(&hi[a], u);
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        atomicMin(&bb[threadIdx.x], lo[threadIdx.x]);
        atomicMax(&bb[3 + threadIdx.x], hi[threadIdx.x]);
    }
}

__device__ __forceinline__ unsigned int spread10(unsigned int v)
{
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// 30-bit code of a position quantised to the bounding box bb (ordered bits, see bbox_kernel).
__device__ __forceinline__ unsigned int morton_code(const float *x, const unsigned int *bb)
{
    unsigned int code = 0;
    for (int a = 0; a < 3; ++a) {
        const float lo = from_ordered(bb[a]), hi = from_ordered(bb[3 + a]);
        const float span = hi - lo;
        float u = span > 0.f ? (x[a] - lo) / span : 0.f;
        unsigned int q = (unsigned int)fminf(fmaxf(u * 1023.0f, 0.0f), 1023.0f);
        code |= spread10(q) << a;
    }
    return code;
}

__global__ void morton_kernel(const float *recv, int64_t n, int64_t npad, const unsigned int *bb,
                              unsigned long long *keys)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= npad) return;
    if (i >= n) { keys[i] = ~0ull; return; }
    keys[i] = ((unsigned long long)morton_code(recv + 3 * i, bb) << 32) | (unsigned long long)i;
}

__global__ void bitonic_step(unsigned long long *keys, int64_t npad, int64_t j, int64_t k)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= npad) return;
    const int64_t l = i ^ j;
    if (l > i) {
        const unsigned long long a = keys[i], b = keys[l];
        const bool up = (i & k) == 0;
        if ((a > b) == up) { keys[i] = b; keys[l] = a; }
    }
}

// ---- stable LSD radix sort of the (Morton code, index) keys on the code's 30 bits,
// 8 bits per pass: the same order as sorting the whole keys, in O(n) per pass
constexpr int kRadixBlock = 1024;   // keys per block, one per thread
constexpr int kRadixBuckets = 256;

__device__ __forceinline__ unsigned int radix_digit(unsigned long long key, int shift)
{
    return (unsigned int)(key >> (32 + shift)) & (kRadixBuckets - 1);
}

// The lanes (of those with ok) that hold the same 8-bit digit: a ballot per bit, a third of
// the time of __match_any_sync.
__device__ __forceinline__ unsigned int same_digit(unsigned int d, bool ok)
{
    unsigned int m = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool set = (d >> b) & 1u;
        const unsigned int v = __ballot_sync(0xffffffffu, set);
        m &= set ? v : ~v;
    }
    return m;
}

// counts[d * nblocks + block]: keys of the block with digit d
__global__ void __launch_bounds__(kRadixBlock) radix_count_kernel(const unsigned long long *keys,
                                                                  int64_t n, int shift,
                                                                  uint32_t *counts, int64_t nblocks)
{
    __shared__ uint32_t c[kRadixBuckets];
    if (threadIdx.x < kRadixBuckets) c[threadIdx.x] = 0u;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * kRadixBlock + threadIdx.x;
    if (i < n) atomicAdd(&c[radix_digit(keys[i], shift)], 1u);
    __syncthreads();
    if (threadIdx.x < kRadixBuckets) counts[(int64_t)threadIdx.x * nblocks + blockIdx.x] = c[threadIdx.x];
}

// One block per digit: exclusive scan of its blocks' counts in place, and its total.  (One
// block for all digits took 47 us a pass at 262,144 keys.)
__global__ void __launch_bounds__(256) radix_scan_kernel(uint32_t *counts, int64_t nblocks, uint32_t *total)
{
    __shared__ uint32_t ws[8];
    uint32_t *row = counts + (int64_t)blockIdx.x * nblocks;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int64_t base = 0; base < nblocks; base += 256) {
        const int64_t c = base + threadIdx.x;
        const uint32_t v = c < nblocks ? row[c] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) ws[wid] = x;
        __syncthreads();
        uint32_t before = carry, all = 0;
        for (int w = 0; w < 8; ++w) {
            if (w < wid) before += ws[w];
            all += ws[w];
        }
        if (c < nblocks) row[c] = before + x - v;
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

// Stable scatter: rank within the warp from the lanes holding the same digit, then the
// counts of earlier warps of the block, then the scanned offset of (digit, block).
__global__ void __launch_bounds__(kRadixBlock) radix_scatter_kernel(const unsigned long long *in,
                                                                    unsigned long long *out,
                                                                    int64_t n, int shift,
                                                                    const uint32_t *offs,
                                                                    const uint32_t *total,
                                                                    int64_t nblocks)
{
    __shared__ uint32_t wc[kRadixBlock / 32][kRadixBuckets];
    __shared__ uint32_t base[kRadixBuckets];     // keys of smaller digits
    for (int q = threadIdx.x; q < (kRadixBlock / 32) * kRadixBuckets; q += kRadixBlock)
        (&wc[0][0])[q] = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * kRadixBlock + threadIdx.x;
    const bool ok = i < n;
    const unsigned long long key = ok ? in[i] : 0ull;
    const unsigned int d = radix_digit(key, shift);
    const unsigned int same = same_digit(d, ok);
    const unsigned int rank = __popc(same & ((1u << lane) - 1u));
    if (ok && rank == 0) wc[wid][d] = __popc(same);
    __syncthreads();
    if (threadIdx.x < kRadixBuckets) {
        uint32_t run = 0u;
        for (int w = 0; w < kRadixBlock / 32; ++w) {
            const uint32_t c = wc[w][threadIdx.x];
            wc[w][threadIdx.x] = run;
            run += c;
        }
    }
    if (wid == 0) {
        uint32_t carry = 0;
#pragma unroll
        for (int q = 0; q < kRadixBuckets / 32; ++q) {
            const uint32_t v = total[q * 32 + lane];
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            base[q * 32 + lane] = carry + x - v;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    __syncthreads();
    if (ok) out[base[d] + offs[(int64_t)d * nblocks + blockIdx.x] + wc[wid][d] + rank] = key;
}

// The whole order in one launch, for up to kOrderSmall receivers, which are bound by launches
// and by the latency of passes over few keys: every block forms the bounding box and all codes
// itself (in shared memory, from L2) and ranks its 128 keys by counting the ones before them,
// four keys a warp and four codes a load.  That is n^2 comparisons, but spread over the chip:
// 4,096 receivers 13 us (the radix passes of the large path in their fifteen launches 65 us,
// in one block 29), 16,384 receivers 45 us (72).
constexpr int kOrderSmall = 16384;
constexpr int kOrderThreads = 1024, kOrderWarps = kOrderThreads / 32;
constexpr int kOrderKeys = 4;      // of a warp
__global__ void __launch_bounds__(kOrderThreads) order_small_kernel(const float *recv, int n, int32_t *order)
{
    extern __shared__ uint4 code4[];               // n codes, padded to whole rows of 128
    uint32_t *const code = reinterpret_cast<uint32_t *>(code4);
    __shared__ unsigned int bb[6];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int rows = (n + 127) / 128;
    if (threadIdx.x < 3) { bb[threadIdx.x] = 0xffffffffu; bb[3 + threadIdx.x] = 0u; }
    __syncthreads();
    unsigned lo[3] = {~0u, ~0u, ~0u}, hi[3] = {0u, 0u, 0u};
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kOrderThreads)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const unsigned u = ordered_bits(recv[3 * i + a]);
            lo[a] = min(lo[a], u);
            hi[a] = max(hi[a], u);
        }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = __reduce_min_sync(0xffffffffu, lo[a]);
        hi[a] = __reduce_max_sync(0xffffffffu, hi[a]);
        if (lane == 0) {
            atomicMin(&bb[a], lo[a]);
            atomicMax(&bb[3 + a], hi[a]);
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < 128 * rows; i += kOrderThreads)
        code[i] = i < n ? morton_code(recv + 3 * i, bb) : 0xffffffffu;     // above any code
    __syncthreads();
    const int i0 = (blockIdx.x * kOrderWarps + wid) * kOrderKeys;          // one uint4 of keys
    if (i0 >= n) return;
    const uint4 own = code4[i0 / 4];
    const uint32_t key[kOrderKeys] = {own.x, own.y, own.z, own.w};
    int before[kOrderKeys] = {0, 0, 0, 0};
    // earlier keys come first on a tie: code <= key before the own four, code < key after
    auto row = [&](int r, bool ties) {
        const uint4 c = code4[32 * r + lane];
#pragma unroll
        for (int m = 0; m < kOrderKeys; ++m) {
            const uint32_t k = key[m] + (ties ? 1u : 0u);
            before[m] += (c.x < k) + (c.y < k) + (c.z < k) + (c.w < k);
        }
    };
    const int r0 = i0 / 128, l0 = (i0 % 128) / 4;
#pragma unroll 4
    for (int r = 0; r < r0; ++r) row(r, true);
    if (lane != l0) {
        row(r0, lane < l0);
    } else {
#pragma unroll
        for (int m = 0; m < kOrderKeys; ++m)
#pragma unroll
            for (int q = 0; q < kOrderKeys; ++q) before[m] += key[q] < key[m] + (q < m ? 1u : 0u);
    }
#pragma unroll 4
    for (int r = r0 + 1; r < rows; ++r) row(r, false);
#pragma unroll
    for (int m = 0; m < kOrderKeys; ++m) {
        const int at = __reduce_add_sync(0xffffffffu, before[m]);
        if (lane == m && i0 + m < n) order[at] = i0 + m;
    }
}

__global__ void extract_order(const unsigned long long *keys, int64_t n, int32_t *order)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) order[i] = (int32_t)(keys[i] & 0xffffffffull);
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// The 32-byte cull records follow the 80-byte records in a sum's record region.
float4 *cull_records(const float *rec, int64_t capacity)
{
    return reinterpret_cast<float4 *>(
        reinterpret_cast<char *>(const_cast<float *>(rec)) +
        align_up((size_t)kRecFloats * (size_t)capacity * sizeof(float), 256));
}

template <int NF, int WINDOW>
void launch_count(const FwdParams &p, cudaStream_t s)
{
    GBT_CUDA(cudaFuncSetAttribute(gbs_count_kernel<NF, WINDOW>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCountSmem));
    const int grid = (int)std::max<int64_t>(
        1, std::min<int64_t>((p.n_items + kCountWarps - 1) / kCountWarps, (int64_t)num_sms()));
    GBT_CUDA(cudaMemsetAsync(p.work_counter, 0, sizeof(int), s));
    gbs_count_kernel<NF, WINDOW><<<grid, 32 * kCountWarps, kCountSmem, s>>>(p);
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
}

template <int WINDOW>
void launch_count_nf(const FwdParams &p, cudaStream_t s)
{
    if (p.nf <= 1) launch_count<1, WINDOW>(p, s);
    else if (p.nf <= 4) launch_count<4, WINDOW>(p, s);
    else launch_count<8, WINDOW>(p, s);
}

// Frequency processing order: when every b is equal, sorted by k so that the kept
// frequencies of a pair form a prefix (wider beams first); otherwise as given.
// perm[slot] = user frequency index.  Returns whether b is uniform.
bool freq_order(const gbt_sum_args &a, int (&perm)[GBT_MAX_FREQ])
{
    for (int f = 0; f < GBT_MAX_FREQ; ++f) perm[f] = f;
    bool uniform = true;
    for (int f = 1; f < a.n_freq; ++f) uniform = uniform && a.beam_b[f] == a.beam_b[0];
    if (uniform)
        std::stable_sort(perm, perm + a.n_freq,
                         [&](int x, int y) { return a.freq_hz[x] < a.freq_hz[y]; });
    return uniform;
}


// Kernel parameters shared by the forward, counting and adjoint launches, for the
// frequency group that starts at processing slot g0 (fperm maps the group's slots to
// user frequency indices).
FwdParams make_pair_params(const TraceDev &td, const SceneDev &sd, const gbt_sum_args &a,
                           const float *rec, int g0 = 0, bool adjoint = false)
{
    FwdParams q{};
    q.recv = a.recv; q.order = a.recv_order; q.n_recv = a.n_recv;
    q.n_seg_ptr = td.ray_off + td.n_rays;
    q.rec = rec;
    q.crec = cull_records(rec, td.capacity);
    q.nf = std::min(kGroupFreq, a.n_freq - g0);
    q.cutoff = (float)a.cutoff;
    q.tile_cull = a.tile_cull ? 1 : 0;
    int perm[GBT_MAX_FREQ];
    q.uniform_b = freq_order(a, perm) || q.nf == 1 ? 1 : 0;     // one band has one b (the ninth alone)
    double amin = 1e300, bmax = 0.0, kmax = 0.0;
    for (int f = 0; f < GBT_MAX_FREQ; ++f) q.fperm[f] = f;
    for (int f = 0; f < q.nf; ++f) {
        const int g = perm[g0 + f];
        q.fperm[f] = g;
        const double K = a.freq_hz[g] / sd.c;       // turns per metre
        const double k = 2.0 * kPi * K;
        const double b = a.beam_b[g];
        FreqConst &c = q.fc[f];
        c.K_hi = (float)K;
        c.K_lo = (float)(K - (double)c.K_hi);
        c.kb2 = (float)(0.5 * k * b);
        c.b2 = (float)(b * b);
        c.invb = (float)(1.0 / b);
        c.b = (float)b;
        c.nkh = (float)(-0.5 * k);
        const double unit = adjoint ? 1.0 : b;      // the pass's unit of length for s
        c.hK = (float)(0.5 * K / unit);
        c.ne = (float)(-0.5 * k * b * 1.4426950408889634 / (unit * unit));
        c.rc = (float)(a.cutoff * unit * unit / (0.5 * k * b));
        c.sA = (float)(k * b / (8.0 * kPi * kPi));
        c.nal = (float)(-a.absorption[g] * 1.4426950408889634 * unit);
        amin = std::min(amin, 0.5 * k * b);
        bmax = std::max(bmax, b * b);
        kmax = std::max(kmax, K);
    }
    q.kmax_turns = (float)kmax;
    q.s_scale = (q.uniform_b && !adjoint) ? (float)(1.0 / a.beam_b[perm[g0]]) : 1.0f;
    q.pre_alpha = (float)(amin / (a.cutoff + 1.0));
    q.pre_beta = (float)bmax;
    q.status = status_word();
    return q;
}

}  // namespace

bool has_losses(const gbt_sum_args &a)
{
    if (a.flow_resistivity) return true;
    for (int f = 0; f < a.n_freq; ++f)
        if (a.absorption[f] != 0.0) return true;
    return false;
}

// Per (frequency, segment) loss factors of a sum: (log2 |R|, arg R / 2 pi) floats for the
// F32 path, complex doubles for the F64 path; then the impedance per (frequency, material);
// none without losses.
static size_t loss_bytes(const TraceDev &td, const gbt_sum_args &a)
{
    if (!has_losses(a)) return 0;
    const size_t per = a.precision == GBT_PRECISION_F64 ? sizeof(double2) : sizeof(float2);
    return align_up((size_t)a.n_freq * (size_t)td.capacity * per, 256) +
           align_up((size_t)a.n_freq * (size_t)td.scene->d.n_materials * sizeof(double2), 256);
}

int choose_splits(const TraceDev &td, const gbt_sum_args &a, bool adjoint)
{
    if (a.seg_split > 0) return a.seg_split;
    const int64_t nseg_est = td.n_seg_host >= 0 ? td.n_seg_host : td.capacity;
    if (a.precision == GBT_PRECISION_F64) {
        // about 512 warps (of 32 receivers) per SM, whose costs differ by ten times and more
        // (16,384 rays x 128^2 x 2 bands: 128 per SM 3.05 ms, 256 2.48, 512 2.24)
        const int64_t tiles = (a.n_recv + 31) / 32;
        int64_t s = (512 * (int64_t)num_sms() + tiles - 1) / (tiles > 0 ? tiles : 1);
        s = std::max<int64_t>(1, std::min<int64_t>(s, (nseg_est + 2 * kBatch - 1) / (2 * kBatch)));
        // partial sums stay under 1 GiB, and under an eighth of a solve's budget (40 MB a band
        // without one, and two chunks may hold them)
        const int64_t room = a.max_device_bytes > 0 ? std::min<int64_t>(1LL << 30, a.max_device_bytes / 8)
                                                    : 1LL << 30;
        const int64_t per_split = (int64_t)a.n_freq * std::max<int64_t>(a.n_recv, 1) * (int64_t)sizeof(double2);
        s = std::min<int64_t>(s, std::max<int64_t>(1, room / per_split));
        return (int)std::min<int64_t>(s, 4096);
    }
    // items are (warp tile, split): about 16 per resident warp, so that the last items to
    // finish are short ones; with the pre-cull 12, shared out by list length (see
    // list_layout_kernel; 16 and 24: 0-5 % slower for a batch, within 1 % elsewhere), and 32
    // equal ones for the differentiable sum, whose tiles are split alike
    const int64_t wtiles = std::max<int64_t>(1, (a.n_recv + kCtaRecv - 1) / kCtaRecv) * kTileWarps;
    const int64_t warps = (int64_t)num_sms() * kWarpsFwd;
    const int64_t per_warp = !a.tile_cull ? 16 : adjoint ? 32 : 12;
    int64_t s = (per_warp * warps + wtiles - 1) / wtiles;
    s = std::max<int64_t>(1, std::min<int64_t>(s, (nseg_est + kBatch - 1) / kBatch));
    // partial sums stay under ~1 GiB
    const int64_t per_split = (int64_t)a.n_freq * std::max<int64_t>(a.n_recv, 1) * 16;
    s = std::min<int64_t>(s, std::max<int64_t>(1, (1LL << 30) / per_split));
    return (int)std::min<int64_t>(s, 4096);
}

static int64_t cta_tiles(int64_t n_recv) { return (n_recv + kCtaRecv - 1) / kCtaRecv; }

// Tile workspace: balls, weights and the dispatch permutation (heaviest tiles
// first), plus, with the tile pre-cull, the per-tile segment lists.
struct TileWs {
    float4 *ball = nullptr;
    float4 *rball = nullptr;       // the balls with their share of the list test's slack
    unsigned int *weight = nullptr;
    int32_t *perm = nullptr;
    int32_t *counts = nullptr;     // [tiles][chunks]: counts, then offsets within the tile
    int64_t *list_off = nullptr;
    int32_t *list_n = nullptr;
    int32_t *list = nullptr;
    uint32_t *words = nullptr;     // per 32-entry list chunk: one word per warp tile
    float4 *wball = nullptr;       // per warp tile: bounding ball
    uint32_t *bits = nullptr;      // [tiles][chunks * 32]: the counting pass's ballots, or null
    int32_t *item_off = nullptr;   // by rank, tiles + 1: first tile-split of each tile (see list_layout_kernel)
    int32_t *tile_first = nullptr, *tile_splits = nullptr;   // the same by tile
    int64_t tiles = 0, chunks = 0, cap = 0, wtiles = 0;
    bool order = false, lists = false;
    size_t bytes = 0;              // workspace the layout needs
};

std::atomic<int64_t> g_list_cap_limit{0};   // set_list_capacity (0: the default)

static TileWs tile_ws_layout(void *ws, int64_t n_recv, int64_t seg_capacity, bool tile_cull,
                             bool adjoint = false)
{
    TileWs t;
    t.tiles = cta_tiles(n_recv);
    // The order's three launches (10 to 14 us) pay where a tile's items are many and long: with
    // few tiles every tile is split finely and the queue drains evenly in any order, until the
    // whole kernel is long.  Measured without / with the order, 5 to 18 tiles: 1.3e7 pairs 36 /
    // 46 us, 6e7 69 / 83, 2.4e8 110 / 120, 7e8 155 / 164, 2.1e9 268 / 257, 9.7e9 703 / 697.
    t.order = t.tiles >= 2 && t.tiles <= kMaxOrderedTiles &&
              (adjoint || tile_cull || t.tiles >= kOrderTiles || n_recv * seg_capacity >= kOrderPairs);
    t.lists = tile_cull && t.tiles >= 1 && t.tiles <= kMaxOrderedTiles && seg_capacity > 0;
    if (!t.order && !t.lists) return t;
    t.chunks = t.lists ? (seg_capacity + kListChunk - 1) / kListChunk : 0;
    // room for an eighth of all (tile, segment) pairs, at least 16M entries
    const int64_t all = t.tiles * seg_capacity;
    // (a multiple of 32: every tile's list starts on a 32-entry chunk boundary)
    t.cap = t.lists ? std::min<int64_t>(all, std::max<int64_t>(int64_t(1) << 24, all / 8)) : 0;
    const int64_t limit = g_list_cap_limit.load();
    if (limit > 0) t.cap = std::min(t.cap, limit);
    t.cap = (t.cap + 31) / 32 * 32;
    t.wtiles = (n_recv + kWarpRecv - 1) / kWarpRecv;
    char *w = static_cast<char *>(ws);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *r = w ? w + off : nullptr;
        off += align_up(bytes, 256);
        return r;
    };
    t.ball = reinterpret_cast<float4 *>(take((size_t)t.tiles * sizeof(float4)));
    t.rball = reinterpret_cast<float4 *>(take((size_t)t.tiles * sizeof(float4)));
    t.weight = reinterpret_cast<unsigned int *>(take((size_t)t.tiles * sizeof(unsigned int)));
    t.perm = reinterpret_cast<int32_t *>(take((size_t)t.tiles * sizeof(int32_t)));
    if (t.lists) {
        t.counts = reinterpret_cast<int32_t *>(take((size_t)(t.tiles * t.chunks) * sizeof(int32_t)));
        t.list_off = reinterpret_cast<int64_t *>(take((size_t)t.tiles * sizeof(int64_t)));
        t.list_n = reinterpret_cast<int32_t *>(take((size_t)t.tiles * sizeof(int32_t)));
        t.item_off = reinterpret_cast<int32_t *>(take((size_t)(t.tiles + 1) * sizeof(int32_t)));
        t.tile_first = reinterpret_cast<int32_t *>(take((size_t)t.tiles * sizeof(int32_t)));
        t.tile_splits = reinterpret_cast<int32_t *>(take((size_t)t.tiles * sizeof(int32_t)));
        t.list = reinterpret_cast<int32_t *>(take((size_t)t.cap * sizeof(int32_t)));
        t.words = reinterpret_cast<uint32_t *>(take((size_t)(t.cap / 32) * kChunkWords * sizeof(uint32_t)));
        t.wball = reinterpret_cast<float4 *>(take((size_t)t.wtiles * sizeof(float4)));
        // the ballots, unless they would take more than 4 GiB (then the write pass repeats
        // the ball tests)
        const size_t bb = (size_t)t.tiles * (size_t)t.chunks * 32 * sizeof(uint32_t);
        if (bb <= (size_t(1) << 32)) t.bits = reinterpret_cast<uint32_t *>(take(bb));
    }
    t.bytes = off;
    return t;
}

static size_t tile_ws_bytes(int64_t n_recv, int64_t seg_capacity, bool tile_cull, bool adjoint = false)
{
    return tile_ws_layout(nullptr, n_recv, seg_capacity, tile_cull, adjoint).bytes;
}

// Whether a sum's tiles are split in proportion to their lists (else every tile alike): the
// automatic split of the pre-culled forward sum.
static bool weighted_splits(const gbt_sum_args &a, const TileWs &t, bool adjoint)
{
    return t.lists && a.seg_split == 0 && !adjoint;
}
// Receivers of a tile-split's partials: a CTA tile's, or all of a single tile.
static int part_receivers(int64_t n_recv) { return (int)std::min<int64_t>(kCtaRecv, n_recv); }
// Points q at a weighted layout: tile-splits instead of splits per tile.
static void set_weighted(FwdParams &q, const TileWs &t)
{
    q.part_recv = part_receivers(q.n_recv);
    q.item_off = t.item_off;
    q.n_tiles = (int32_t)t.tiles;
    q.n_items = ((int64_t)q.splits + 1) * t.tiles * kTileWarps;     // at most (sizes the grid)
}
// Float-float partials of nf bands: [split][band][receiver], or weighted
// [tile-split][band][receiver of the tile].
static size_t partial_count(const gbt_sum_args &a, int nf, int splits, bool weighted)
{
    return weighted ? ((size_t)splits + 1) * (size_t)cta_tiles(a.n_recv) * part_receivers(a.n_recv) * nf
                    : (size_t)splits * nf * (size_t)a.n_recv;
}

// Launches the tile preparation for q's receivers and records (the records must
// be written earlier on s) and points q at its results: the dispatch order and,
// with the pre-cull, the segment lists.  Weights are the exact list sizes when
// the lists are built, else a sampled count.
static void tile_prep_launch(FwdParams &q, int window, const TileWs &t, cudaStream_t s,
                             bool weighted = false)
{
    if (!t.order && !t.lists) return;
    const int64_t T = t.tiles;
    int64_t n = 0;
    tile_ball_kernel<<<(unsigned)T, 256, 0, s>>>(q.recv, q.order, q.n_recv, t.ball, t.weight, t.rball);
    ++n;
    // tile groups of the chunk-major list passes (each block walks 1 / tg of the tiles):
    // one, since more re-read the chunk's records for every group (measured on the city:
    // 8 groups took list_count 1.77 -> 2.19 ms and list_write_bits 1.58 -> 1.75 ms)
    const unsigned tg = 1;
    if (t.lists) {
        const size_t sm = (size_t)T * sizeof(int32_t);
        if (window == GBT_WINDOW_LINE) {
            GBT_CUDA(cudaFuncSetAttribute(list_count_kernel<GBT_WINDOW_LINE>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
            list_count_kernel<GBT_WINDOW_LINE><<<dim3((unsigned)t.chunks, tg), kListChunk, sm, s>>>(
                q.crec, q.n_seg_ptr, t.rball, T, t.chunks, q.pre_alpha, q.pre_beta, t.counts, t.bits);
        } else {
            GBT_CUDA(cudaFuncSetAttribute(list_count_kernel<GBT_WINDOW_SEGMENT>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
            list_count_kernel<GBT_WINDOW_SEGMENT><<<dim3((unsigned)t.chunks, tg), kListChunk, sm, s>>>(
                q.crec, q.n_seg_ptr, t.rball, T, t.chunks, q.pre_alpha, q.pre_beta, t.counts, t.bits);
        }
        list_scan_chunks_kernel<<<(unsigned)T, 1024, 0, s>>>(t.counts, t.chunks, t.weight);
        n += 2;
    } else {
        if (window == GBT_WINDOW_LINE)
            tile_weight_kernel<GBT_WINDOW_LINE><<<dim3(kWeightSamples / 256, 8), 256, 0, s>>>(
                q.crec, q.n_seg_ptr, t.ball, T, q.pre_alpha, q.pre_beta, t.weight);
        else
            tile_weight_kernel<GBT_WINDOW_SEGMENT><<<dim3(kWeightSamples / 256, 8), 256, 0, s>>>(
                q.crec, q.n_seg_ptr, t.ball, T, q.pre_alpha, q.pre_beta, t.weight);
        ++n;
    }
    if (t.order) {
        tile_rank_kernel<<<(unsigned)((T + 255) / 256), 256, 0, s>>>(t.weight, T, t.perm);
        ++n;
        q.tile_perm = t.perm;
    }
    if (t.lists) {
        list_layout_kernel<<<1, 1024, 0, s>>>(t.weight, t.order ? t.perm : nullptr, T, t.cap,
                                              t.list_off, t.list_n, q.n_seg_ptr,
                                              weighted ? (int64_t)q.splits * T : 0, t.item_off,
                                              t.tile_first, t.tile_splits);
        warp_ball_kernel<<<(unsigned)((t.wtiles + 7) / 8), 256, 0, s>>>(q.recv, q.order, q.n_recv,
                                                                         t.wtiles, t.wball);
        const dim3 mgrid(128, (unsigned)T);     // many blocks per tile: the gathers overlap
        // rows: about 1,024 blocks at least, where there are that many
        const dim3 wgrid((unsigned)std::min<int64_t>((t.chunks + kWriteWarps - 1) / kWriteWarps,
                                                     std::max<int64_t>(64, 1024 / T)),
                         (unsigned)std::min<int64_t>(T, 65535));
        if (window == GBT_WINDOW_LINE) {
            if (t.bits)
                list_write_bits_kernel<<<wgrid, 32 * kWriteWarps, 0, s>>>(
                    q.n_seg_ptr, T, t.chunks, t.bits, t.counts, t.list_off, t.list_n, t.list);
            else
                list_write_kernel<GBT_WINDOW_LINE><<<(unsigned)t.chunks, kListChunk, 0, s>>>(
                    q.crec, q.n_seg_ptr, t.rball, T, t.chunks, q.pre_alpha, q.pre_beta, t.counts,
                    t.list_off, t.list_n, t.list);
            list_words_kernel<GBT_WINDOW_LINE><<<mgrid, 256, 0, s>>>(
                q.crec, t.wball, t.wtiles, q.pre_alpha, q.pre_beta, t.list_off, t.list_n, t.list, t.words);
        } else {
            if (t.bits)
                list_write_bits_kernel<<<wgrid, 32 * kWriteWarps, 0, s>>>(
                    q.n_seg_ptr, T, t.chunks, t.bits, t.counts, t.list_off, t.list_n, t.list);
            else
                list_write_kernel<GBT_WINDOW_SEGMENT><<<(unsigned)t.chunks, kListChunk, 0, s>>>(
                    q.crec, q.n_seg_ptr, t.rball, T, t.chunks, q.pre_alpha, q.pre_beta, t.counts,
                    t.list_off, t.list_n, t.list);
            list_words_kernel<GBT_WINDOW_SEGMENT><<<mgrid, 256, 0, s>>>(
                q.crec, t.wball, t.wtiles, q.pre_alpha, q.pre_beta, t.list_off, t.list_n, t.list, t.words);
        }
        n += 4;
        q.list = t.list;
        q.list_off = t.list_off;
        q.list_n = t.list_n;
        q.list_words = t.words;
        if (weighted) set_weighted(q, t);
    }
    GBT_CUDA(cudaGetLastError());
    note_launches(n);
}

// Kernel records: the 80-byte records, then the 32-byte cull records of the list and
// dispatch-order kernels (sector aligned, a fraction of the size, so they stay in L2).
static size_t records_bytes(const TraceDev &td)
{
    return align_up((size_t)kRecFloats * (size_t)td.capacity * sizeof(float), 256) +
           align_up((size_t)td.capacity * 2 * sizeof(float4), 256);
}


// Prepass of a trace's segments into kernel records (and FP64 amplitudes when amp64 is
// set), with the sum's reflection coefficients and ray weights.
static void prepass_launch(const TraceDev &td, const SceneDev &sd, const gbt_sum_args &a,
                           float *rec, double *amp64, int *counters, cudaStream_t s,
                           void *loss = nullptr, const PaddedRays *rays = nullptr)
{
    if (td.capacity == 0) return;
    PrepParams pp{};
    pp.counters = counters;
    pp.w0 = 4.0 * kPi / (double)td.n_fan;
    pp.n_seg_ptr = td.ray_off + td.n_rays;
    pp.o = td.o; pp.t = td.t; pp.L = td.L; pp.s0 = td.s0;
    pp.ray = td.ray; pp.depth = td.depth; pp.bmat = td.bmat;
    pp.gamma = a.gamma;
    pp.weight = a.ray_weight;
    pp.fan = td.fan;
    pp.n_fan = td.n_fan;
    pp.n_materials = sd.n_materials;
    pp.rec = rec;
    pp.crec = cull_records(rec, td.capacity);
    pp.amp64 = amp64;
    pp.status = status_word();
    if (rays) {
        pack_kernel<<<(unsigned)((rays->n_rays + kPackRays - 1) / kPackRays), kPackRays, 0, s>>>(pp, *rays);
        note_launches(1);
        GBT_CUDA(cudaGetLastError());
        return;
    }
    prepass_kernel<<<(unsigned)((td.capacity + 255) / 256), 256, 0, s>>>(pp);
    note_launches(1);
    if (loss) {
        LossParams lp{};
        lp.ray_off = td.ray_off;
        lp.n_rays = td.n_rays;
        lp.t = td.t;
        lp.bmat = td.bmat;
        lp.hit = td.hit;
        lp.sigma = a.flow_resistivity;
        lp.tri = sd.tri;
        lp.n_tri = sd.n_tri;
        lp.n_materials = sd.n_materials;
        lp.nf = a.n_freq;
        for (int f = 0; f < a.n_freq; ++f) lp.freq[f] = a.freq_hz[f];
        lp.rf_stride = td.capacity;
        lp.status = status_word();
        const bool f64 = a.precision == GBT_PRECISION_F64;
        if (f64) lp.seg_r64 = static_cast<double2 *>(loss);
        else lp.seg_rf = static_cast<float2 *>(loss);
        lp.z = reinterpret_cast<double2 *>(
            static_cast<char *>(loss) +
            align_up((size_t)a.n_freq * (size_t)td.capacity * (f64 ? sizeof(double2) : sizeof(float2)), 256));
        const int nz = a.n_freq * sd.n_materials;
        if (lp.sigma) {
            porous_impedance_kernel<<<(unsigned)((nz + 63) / 64), 64, 0, s>>>(lp);
            note_launches(1);
        }
        porous_path_kernel<<<dim3((unsigned)((td.n_rays + 127) / 128), (unsigned)a.n_freq), 128, 0, s>>>(lp);
        note_launches(1);
    }
    GBT_CUDA(cudaGetLastError());
}

// Partials of all of a sum's frequency groups.
static size_t partial_bytes(const TraceDev &td, const gbt_sum_args &a, int splits, bool adjoint)
{
    if (a.precision == GBT_PRECISION_F64)
        return align_up((size_t)splits * a.n_freq * (size_t)a.n_recv * sizeof(double2), 256);
    const bool w = weighted_splits(a, tile_ws_layout(nullptr, a.n_recv, td.capacity, a.tile_cull != 0), adjoint);
    return align_up(partial_count(a, a.n_freq, splits, w) * sizeof(float4), 256);
}

size_t sum_workspace_bytes(const TraceDev &td, const gbt_sum_args &a, int splits, bool adjoint)
{
    size_t b = records_bytes(td);
    b += align_up((size_t)td.capacity * sizeof(double), 256);               // amp64
    b += 256;                                                               // work counter
    b += partial_bytes(td, a, splits, adjoint);
    if (a.precision != GBT_PRECISION_F64) b += tile_ws_bytes(a.n_recv, td.capacity, a.tile_cull != 0);
    b += loss_bytes(td, a);
    return b;
}

void sum_launch(const TraceDev &td, const SceneDev &sd, const gbt_sum_args &a, int splits,
                void *work, cudaStream_t s, unsigned long long *stats, bool differentiable,
                const PaddedRays *rays)
{
    char *w = static_cast<char *>(work);
    float *rec = reinterpret_cast<float *>(w);
    w += records_bytes(td);
    double *amp64 = reinterpret_cast<double *>(w);
    w += align_up((size_t)td.capacity * sizeof(double), 256);
    int *counter = reinterpret_cast<int *>(w);
    w += 256;
    void *partial = w;
    w += partial_bytes(td, a, splits, differentiable);
    void *order_ws = w;
    if (a.precision != GBT_PRECISION_F64) w += tile_ws_bytes(a.n_recv, td.capacity, a.tile_cull != 0);
    void *loss = loss_bytes(td, a) ? static_cast<void *>(w) : nullptr;
    const int32_t *n_seg_ptr = td.ray_off + td.n_rays;

    prepass_launch(td, sd, a, rec, amp64, counter, s, loss, rays);

    if (a.n_recv <= 0) return;
    ReduceParams rp{};
    rp.n_recv = a.n_recv;
    rp.out = reinterpret_cast<float2 *>(a.out);
    rp.accumulate = a.accumulate;
    rp.splits = splits;
    rp.order = a.recv_order;
    if (a.precision == GBT_PRECISION_F64) {
        F64Params q{};
        q.recv = a.recv; q.order = a.recv_order; q.n_recv = a.n_recv;
        q.g.n_seg_ptr = n_seg_ptr;
        q.g.rec = rec;
        q.g.crec = cull_records(rec, td.capacity);
        q.g.splits = splits;
        double kbmin = 1e300, bmax = 0.0;
        q.o = td.o; q.t = td.t; q.L = td.L; q.s0 = td.s0; q.amp = amp64;
        q.nf = a.n_freq;
        q.cutoff = a.cutoff;
        for (int f = 0; f < a.n_freq; ++f) {
            q.k[f] = 2.0 * kPi * a.freq_hz[f] / sd.c;
            q.b[f] = a.beam_b[f];
            q.kb[f] = q.k[f] * q.b[f];
            q.b2[f] = q.b[f] * q.b[f];
            kbmin = std::min(kbmin, q.k[f] * q.b[f]);
            bmax = std::max(bmax, q.b[f]);
        }
        // the union of the bands' cutoffs, with a relative margin of 2e-4 at any cutoff
        q.g.pre_alpha = (float)(0.5 * kbmin / (1.0002 * a.cutoff + 1.0));
        q.g.pre_beta = (float)(bmax * bmax);
        q.partial = reinterpret_cast<double2 *>(partial);
        for (int f = 0; f < a.n_freq; ++f) q.absorb[f] = a.absorption[f];
        q.r64 = static_cast<const double2 *>(loss);
        q.r64_stride = td.capacity;
        dim3 grid((unsigned)((a.n_recv + 32 * kWarps64 - 1) / (32 * kWarps64)), (unsigned)splits);
        if (a.window == GBT_WINDOW_LINE) launch_f64<GBT_WINDOW_LINE>(q, grid, s);
        else launch_f64<GBT_WINDOW_SEGMENT>(q, grid, s);
        note_launches(1);
        GBT_CUDA(cudaGetLastError());
        rp.n = (int64_t)a.n_freq * a.n_recv;
        for (int f = 0; f < GBT_MAX_FREQ; ++f) rp.perm[f] = f;
        rp.p64 = reinterpret_cast<double2 *>(partial);
        reduce_launch(rp, s);
        return;
    }
    // F32: one pair launch and one merge per group of at most 8 frequencies, each
    // group with its own partials (split-major within the group) and output rows
    for (int g0 = 0; g0 < a.n_freq; g0 += kGroupFreq) {
        FwdParams q = make_pair_params(td, sd, a, rec, g0, differentiable);
        q.splits = splits;
        const TileWs tw = tile_ws_layout(order_ws, a.n_recv, td.capacity, a.tile_cull != 0);
        const bool weighted = weighted_splits(a, tw, differentiable) && !stats;
        q.partial = reinterpret_cast<float4 *>(partial) + partial_count(a, g0, splits, weighted);
        q.stats = stats;
        q.seg_rf = static_cast<const float2 *>(loss);
        q.rf_stride = td.capacity;
        q.n_items = cta_tiles(a.n_recv) * kTileWarps * splits;
        q.work_counter = counter + g0 / kGroupFreq;
        tile_prep_launch(q, a.window, tw, s, weighted);
        if (stats) {
            if (a.window == GBT_WINDOW_LINE) launch_count_nf<GBT_WINDOW_LINE>(q, s);
            else launch_count_nf<GBT_WINDOW_SEGMENT>(q, s);
            continue;
        }
        if (differentiable) pair_field_launch(q, a.window, s, true);
        else pair_fwd_launch(q, a.window, s, true);
        rp.n = (int64_t)q.nf * a.n_recv;
        for (int f = 0; f < GBT_MAX_FREQ; ++f) rp.perm[f] = q.fperm[f];
        for (int f = 0; f < q.nf; ++f) merge_scale(rp, f, a.freq_hz[q.fperm[f]], sd.c, differentiable);
        rp.p32 = q.partial;
        rp.tile_first = weighted ? tw.tile_first : nullptr;
        rp.tile_splits = tw.tile_splits;
        rp.nf = q.nf;
        rp.part_recv = q.part_recv;
        reduce_launch(rp, s);
    }
}

void synth_launch(const float *p, int nf, int64_t n_recv, const double *freq_hz,
                  const double *amp, double t0, double dt, int64_t n_t, float *out,
                  int accumulate, cudaStream_t s)
{
    if (n_recv <= 0 || n_t <= 0) return;
    SynthParams sp{};
    sp.p = reinterpret_cast<const float2 *>(p);
    sp.n_recv = n_recv;
    sp.n_t = n_t;
    for (int f = 0; f < nf; ++f) {
        // whole turns of a pair of steps drop out (offsets are odd multiples of half a step)
        sp.step[f] = std::remainder(freq_hz[f] * dt, 2.0);
        sp.start[f] = freq_hz[f] * t0;
        sp.step_hi[f] = (float)sp.step[f];
        sp.step_lo[f] = (float)(sp.step[f] - (double)sp.step_hi[f]);
        sp.amp_re[f] = amp[2 * f];
        sp.amp_im[f] = amp[2 * f + 1];
    }
    sp.out = out;
    sp.accumulate = accumulate;
    const int64_t per_block = 256 * kSynthRecv;
    const dim3 grid((unsigned)((n_recv + per_block - 1) / per_block),
                    (unsigned)((n_t + kSynthTile - 1) / kSynthTile));
    switch (nf) {
#define GBT_SYNTH(NFV) \
    case NFV: synth_kernel<NFV><<<grid, 256, 0, s>>>(sp); break;
        GBT_SYNTH(1) GBT_SYNTH(2) GBT_SYNTH(3) GBT_SYNTH(4) GBT_SYNTH(5) GBT_SYNTH(6)
        GBT_SYNTH(7) GBT_SYNTH(8) GBT_SYNTH(9) GBT_SYNTH(10) GBT_SYNTH(11) GBT_SYNTH(12)
        GBT_SYNTH(13) GBT_SYNTH(14) GBT_SYNTH(15) GBT_SYNTH(16)
#undef GBT_SYNTH
    default: fail(GBT_ERR_INVALID_ARG, "synthesis takes 1 .. 16 frequencies");
    }
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
}

size_t recv_order_scratch_bytes(int64_t n)
{
    const int64_t nblocks = (n + kRadixBlock - 1) / kRadixBlock;
    if (n <= kOrderSmall) return 0;
    return 2 * align_up((size_t)n * sizeof(unsigned long long), 256) +
           align_up((size_t)kRadixBuckets * nblocks * sizeof(uint32_t), 256) +
           align_up(kRadixBuckets * sizeof(uint32_t), 256) + 256;
}

void recv_order_launch(const float *recv, int64_t n, int32_t *order, void *scratch, cudaStream_t s)
{
    if (n <= 0) return;
    if (n <= kOrderSmall) {
        const size_t sm = ((size_t)n + 127) / 128 * 128 * sizeof(uint32_t);
        static std::atomic<bool> set[64] = {};
        int dev = 0;
        GBT_CUDA(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64) fail(GBT_ERR_UNSUPPORTED, "device index >= 64");
        if (!set[dev].load(std::memory_order_acquire)) {
            GBT_CUDA(cudaFuncSetAttribute(order_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(kOrderSmall * sizeof(uint32_t))));
            set[dev].store(true, std::memory_order_release);
        }
        const unsigned blocks = (unsigned)((n + kOrderWarps * kOrderKeys - 1) / (kOrderWarps * kOrderKeys));
        order_small_kernel<<<blocks, kOrderThreads, sm, s>>>(recv, (int)n, order);
        note_launches(1);
        GBT_CUDA(cudaGetLastError());
        return;
    }
    const int64_t nblocks = (n + kRadixBlock - 1) / kRadixBlock;
    char *w = static_cast<char *>(scratch);
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(w);
    w += align_up((size_t)n * sizeof(unsigned long long), 256);
    unsigned long long *tmp = reinterpret_cast<unsigned long long *>(w);
    w += align_up((size_t)n * sizeof(unsigned long long), 256);
    uint32_t *counts = reinterpret_cast<uint32_t *>(w);
    w += align_up((size_t)kRadixBuckets * nblocks * sizeof(uint32_t), 256);
    uint32_t *total = reinterpret_cast<uint32_t *>(w);
    w += align_up(kRadixBuckets * sizeof(uint32_t), 256);
    unsigned int *bb = reinterpret_cast<unsigned int *>(w);
    GBT_CUDA(cudaMemsetAsync(bb, 0xff, 3 * sizeof(unsigned int), s));
    GBT_CUDA(cudaMemsetAsync(bb + 3, 0x00, 3 * sizeof(unsigned int), s));
    bbox_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, s>>>(recv, n, bb);
    note_launches(1);
    morton_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(recv, n, n, bb, keys);
    note_launches(1);
    for (int shift = 0; shift < 30; shift += 8) {   // 30-bit codes: four passes
        radix_count_kernel<<<(unsigned)nblocks, kRadixBlock, 0, s>>>(keys, n, shift, counts, nblocks);
        radix_scan_kernel<<<kRadixBuckets, 256, 0, s>>>(counts, nblocks, total);
        radix_scatter_kernel<<<(unsigned)nblocks, kRadixBlock, 0, s>>>(keys, tmp, n, shift, counts, total,
                                                                         nblocks);
        note_launches(3);
        std::swap(keys, tmp);
    }
    extract_order<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(keys, n, order);
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
}


// ------------------------------------------------------------ adjoint --

static size_t bwd_layout(const TraceDev &td, const gbt_sum_args &a, const SceneDev *sd,
                         size_t *off)
{
    // records | amp64 | counter | seg_G | seg_H | acc | tile order | losses
    size_t b = 0;
    off[0] = b; b += records_bytes(td);
    off[1] = b; b += align_up((size_t)td.capacity * sizeof(double), 256);
    off[2] = b; b += 256;
    off[3] = b; b += align_up((size_t)td.capacity * sizeof(float), 256);
    off[4] = b; b += align_up((size_t)a.n_freq * td.capacity * sizeof(float), 256);
    off[5] = b; b += align_up((size_t)((sd ? sd->n_materials : 1024) + GBT_MAX_FREQ) * sizeof(double), 256);
    off[6] = b; b += tile_ws_bytes(a.n_recv, td.capacity, a.tile_cull != 0, true);
    off[7] = b; b += loss_bytes(td, a);
    return b;
}

size_t bwd_workspace_bytes(const TraceDev &td, const gbt_sum_args &a)
{
    size_t off[8];
    return bwd_layout(td, a, &td.scene->d, off);
}

void bwd_launch(const TraceDev &td, const SceneDev &sd, const gbt_sum_args &a,
                const float *grad_out, float *grad_gamma, float *grad_w, double *grad_b,
                void *work, cudaStream_t s)
{
    size_t off[8];
    bwd_layout(td, a, &sd, off);
    char *w = static_cast<char *>(work);
    float *rec = reinterpret_cast<float *>(w + off[0]);
    double *amp64 = reinterpret_cast<double *>(w + off[1]);
    int *counter = reinterpret_cast<int *>(w + off[2]);
    float *seg_G = reinterpret_cast<float *>(w + off[3]);
    float *seg_H = reinterpret_cast<float *>(w + off[4]);
    double *acc = reinterpret_cast<double *>(w + off[5]);

    GBT_CUDA(cudaMemsetAsync(seg_G, 0, (size_t)td.capacity * sizeof(float), s));
    GBT_CUDA(cudaMemsetAsync(seg_H, 0, (size_t)a.n_freq * td.capacity * sizeof(float), s));
    GBT_CUDA(cudaMemsetAsync(acc, 0, (size_t)(sd.n_materials + GBT_MAX_FREQ) * sizeof(double), s));
    if (grad_w) GBT_CUDA(cudaMemsetAsync(grad_w, 0, (size_t)td.n_fan * sizeof(float), s));

    void *loss = loss_bytes(td, a) ? static_cast<void *>(w + off[7]) : nullptr;
    prepass_launch(td, sd, a, rec, amp64, counter, s, loss);
    // per frequency group: seg_G gathers every frequency's terms, seg_H the group's rows
    // (processing slots g0 .. g0 + nf - 1)
    if (a.n_recv > 0) {
        const int splits = choose_splits(td, a, true);
        for (int g0 = 0; g0 < a.n_freq; g0 += kGroupFreq) {
            FwdParams q = make_pair_params(td, sd, a, rec, g0, true);
            q.splits = splits;
            q.n_items = cta_tiles(a.n_recv) * kTileWarps * splits;
            q.work_counter = counter + g0 / kGroupFreq;
            q.grad_out = reinterpret_cast<const float2 *>(grad_out);
            q.seg_G = seg_G;
            q.seg_H = seg_H + (int64_t)g0 * td.capacity;
            q.seg_stride = td.capacity;
            q.seg_rf = static_cast<const float2 *>(loss);
            q.rf_stride = td.capacity;
            tile_prep_launch(q, a.window, tile_ws_layout(w + off[6], a.n_recv, td.capacity, a.tile_cull != 0, true), s);
            pair_bwd_launch(q, a.window, s, true);
        }
    }
    int fperm[GBT_MAX_FREQ];
    freq_order(a, fperm);
    RayGradParams r{};
    r.n_rays = td.n_rays;
    r.ray_begin = td.ray_begin;
    r.ray_off = td.ray_off;
    r.bmat = td.bmat;
    r.gamma = a.gamma;
    r.weight = a.ray_weight;
    r.fan = td.fan;
    r.n_fan = td.n_fan;
    r.seg_G = seg_G;
    r.seg_H = seg_H;
    r.seg_stride = td.capacity;
    r.nf = a.n_freq;
    r.n_materials = sd.n_materials;
    r.grad_w = grad_w;
    r.acc = acc;
    r.status = status_word();
    const size_t sh = (size_t)(sd.n_materials + a.n_freq) * sizeof(double);
    const unsigned rb = (unsigned)((td.n_rays + 127) / 128);
    if (r.nf <= 1) ray_grad_kernel<1><<<rb, 128, sh, s>>>(r);
    else if (r.nf <= 4) ray_grad_kernel<4><<<rb, 128, sh, s>>>(r);
    else ray_grad_kernel<GBT_MAX_FREQ><<<rb, 128, sh, s>>>(r);
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
    GradOutParams g{};
    g.acc = acc;
    g.n_materials = sd.n_materials;
    g.nf = a.n_freq;
    for (int f = 0; f < GBT_MAX_FREQ; ++f) g.fperm[f] = fperm[f];
    g.grad_gamma = grad_gamma;
    g.grad_b = grad_b;
    const int nk = sd.n_materials + a.n_freq;
    grad_out_kernel<<<(unsigned)((nk + 127) / 128), 128, 0, s>>>(g);
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
}

// ------------------------------------------------------------ batched --

// Many (trace, sum arguments) instances in one persistent launch (pair_batched.cu), or each
// on its own kernels over a few branch streams.
enum { kFused = 0, kConcurrent = 1 };      // how a batch executes
constexpr int kBranches = 4;               // branch streams of a concurrent batch

struct BatchImpl {
    std::vector<const gbt_trace_t *> traces;
    std::vector<gbt_sum_args> args;
    std::vector<int> order;            // instance processing order (cost, descending)
    std::vector<int64_t> n_seg, cost;
    std::vector<int> splits;
    std::vector<size_t> rec_off, part_off, ord_off, loss_off;
    std::vector<FwdParams> table;      // in processing order
    std::vector<int64_t> inst_off;
    void *work = nullptr;
    size_t work_bytes = 0;
    int *counter = nullptr;
    FwdParams *d_table = nullptr;
    int64_t *d_off = nullptr;
    int grid = 1;
    int nf_max = 1, window = 0;
    bool use_graph = false;
    cudaStream_t capture_stream = nullptr;   // private stream the graph is recorded on
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int64_t graph_kernels = 0;               // kernel nodes of the recorded graph
    cudaEvent_t used = nullptr;              // after the latest submit
    // kConcurrent: each instance runs the single-instance pair kernel (parameters
    // in constant space) on one of a few branch streams forked from the submit
    // stream, so one instance's draining tail overlaps the next one's start
    int mode = kFused;
    std::vector<cudaStream_t> branch;
    cudaEvent_t fork = nullptr;
    std::vector<cudaEvent_t> join;
};

static void batch_plan(BatchImpl &B, double items_per_slot)
{
    // splits per instance: items proportional to the instance's cost
    const int64_t slots = (int64_t)B.grid;
    double total = 0.0;
    for (int64_t c : B.cost) total += (double)std::max<int64_t>(c, 1);
    const int n = (int)B.args.size();
    B.splits.assign(n, 1);
    for (int i = 0; i < n; ++i) {
        const gbt_sum_args &a = B.args[i];
        const int64_t tiles = std::max<int64_t>(1, (a.n_recv + kCtaRecv - 1) / kCtaRecv);
        const double want = items_per_slot * slots * (double)std::max<int64_t>(B.cost[i], 1) / total;
        int64_t sp = (int64_t)std::ceil(want / (double)tiles);
        const int64_t nb = std::max<int64_t>(1, (B.n_seg[i] + kBatch - 1) / kBatch);
        sp = std::max<int64_t>(1, std::min<int64_t>(sp, nb));
        const int64_t per_split = (int64_t)a.n_freq * std::max<int64_t>(a.n_recv, 1) * 16;
        sp = std::min<int64_t>(sp, std::max<int64_t>(1, (1LL << 30) / per_split));
        B.splits[i] = (int)std::min<int64_t>(sp, 4096);
    }
}

// Concurrent batches split each instance as a single sum would.
static void batch_plan_concurrent(BatchImpl &B)
{
    const int n = (int)B.args.size();
    B.splits.assign(n, 1);
    for (int i = 0; i < n; ++i) B.splits[i] = choose_splits(B.traces[i]->d, B.args[i]);
}

// The fused form's table holds each instance's items, so its tiles are split alike.
static bool batch_weighted(const BatchImpl &B, int i)
{
    const gbt_sum_args &a = B.args[i];
    return B.mode == kConcurrent &&
           weighted_splits(a, tile_ws_layout(nullptr, a.n_recv, B.traces[i]->d.capacity, a.tile_cull != 0), false);
}

static void batch_layout(BatchImpl &B, cudaStream_t s)
{
    const int n = (int)B.args.size();
    B.rec_off.assign(n, 0);
    B.part_off.assign(n, 0);
    B.ord_off.assign(n, 0);
    B.loss_off.assign(n, 0);
    size_t b = 0;
    for (int i = 0; i < n; ++i) {
        B.rec_off[i] = b;
        b += records_bytes(B.traces[i]->d);
        B.part_off[i] = b;
        b += align_up(partial_count(B.args[i], B.args[i].n_freq, B.splits[i], batch_weighted(B, i)) *
                          sizeof(float4), 256);
        B.ord_off[i] = b;
        b += tile_ws_bytes(B.args[i].n_recv, B.traces[i]->d.capacity, B.args[i].tile_cull != 0);
        B.loss_off[i] = b;
        b += loss_bytes(B.traces[i]->d, B.args[i]);
    }
    // work counters per instance (kCounters, of which an instance of one group uses the first)
    const size_t cnt = align_up((size_t)n * kCounters * sizeof(int), 256);
    const size_t tab = align_up((size_t)n * sizeof(FwdParams), 256);
    const size_t off = align_up((size_t)(n + 1) * sizeof(int64_t), 256);
    const size_t need = b + cnt + tab + off;
    if (need > B.work_bytes) {
        if (B.work) dfree(B.work, s);
        B.work = dalloc(need, s);
        B.work_bytes = need;
    }
    char *w = static_cast<char *>(B.work);
    B.counter = reinterpret_cast<int *>(w + b);
    B.d_table = reinterpret_cast<FwdParams *>(w + b + cnt);
    B.d_off = reinterpret_cast<int64_t *>(w + b + cnt + tab);

    B.table.clear();
    B.inst_off.assign(1, 0);
    for (int k = 0; k < n; ++k) {
        const int i = B.order[k];
        const TraceDev &td = B.traces[i]->d;
        const gbt_sum_args &a = B.args[i];
        float *rec = reinterpret_cast<float *>(w + B.rec_off[i]);
        FwdParams q = make_pair_params(td, td.scene->d, a, rec);
        q.splits = B.splits[i];
        q.n_items = cta_tiles(a.n_recv) * kTileWarps * q.splits;
        q.partial = reinterpret_cast<float4 *>(w + B.part_off[i]);
        q.work_counter = B.mode == kConcurrent ? B.counter + k * kCounters : B.counter;
        if (has_losses(a)) {
            q.seg_rf = reinterpret_cast<const float2 *>(w + B.loss_off[i]);
            q.rf_stride = td.capacity;
        }
        {
            const TileWs t = tile_ws_layout(w + B.ord_off[i], a.n_recv, td.capacity, a.tile_cull != 0);
            q.tile_perm = t.order ? t.perm : nullptr;
            q.list = t.lists ? t.list : nullptr;
            q.list_off = t.lists ? t.list_off : nullptr;
            q.list_n = t.lists ? t.list_n : nullptr;
            q.list_words = t.lists ? t.words : nullptr;
            if (batch_weighted(B, i)) set_weighted(q, t);
        }
        B.table.push_back(q);
        B.inst_off.push_back(B.inst_off.back() + q.n_items);
    }
    GBT_CUDA(cudaMemcpyAsync(B.d_table, B.table.data(), (size_t)n * sizeof(FwdParams),
                             cudaMemcpyHostToDevice, s));
    GBT_CUDA(cudaMemcpyAsync(B.d_off, B.inst_off.data(), (size_t)(n + 1) * sizeof(int64_t),
                             cudaMemcpyHostToDevice, s));
    GBT_CUDA(cudaStreamSynchronize(s));
}

static void batch_prepass(BatchImpl &B, int i, int *counters, cudaStream_t s)
{
    const TraceDev &td = B.traces[i]->d;
    char *w = static_cast<char *>(B.work);
    prepass_launch(td, td.scene->d, B.args[i], reinterpret_cast<float *>(w + B.rec_off[i]), nullptr,
                   counters, s, has_losses(B.args[i]) ? static_cast<void *>(w + B.loss_off[i]) : nullptr);
}

// Merge of instance i (processing index k) into its output.
static void batch_reduce(BatchImpl &B, int k, cudaStream_t s)
{
    const int i = B.order[k];
    const gbt_sum_args &a = B.args[i];
    if (a.n_recv == 0) return;
    ReduceParams rp{};
    rp.n = (int64_t)a.n_freq * a.n_recv;
    rp.n_recv = a.n_recv;
    for (int f = 0; f < GBT_MAX_FREQ; ++f) rp.perm[f] = B.table[k].fperm[f];
    for (int f = 0; f < a.n_freq; ++f)
        merge_scale(rp, f, a.freq_hz[B.table[k].fperm[f]], B.traces[i]->d.scene->d.c, false);
    rp.splits = B.splits[i];
    rp.p32 = reinterpret_cast<float4 *>(static_cast<char *>(B.work) + B.part_off[i]);
    rp.p64 = nullptr;
    rp.order = a.recv_order;
    rp.out = reinterpret_cast<float2 *>(a.out);
    rp.accumulate = a.accumulate;
    if (batch_weighted(B, i)) {
        const TileWs t = tile_ws_layout(static_cast<char *>(B.work) + B.ord_off[i], a.n_recv,
                                        B.traces[i]->d.capacity, a.tile_cull != 0);
        rp.tile_first = t.tile_first;
        rp.tile_splits = t.tile_splits;
        rp.nf = a.n_freq;
        rp.part_recv = part_receivers(a.n_recv);
    }
    reduce_launch(rp, s);
}

// Concurrent form: instances (longest first) dealt round-robin to branch streams
// forked from s and joined back into it; on each branch an instance's prepass,
// tile order, pair kernel and merge follow one another.
static void batch_record_concurrent(BatchImpl &B, cudaStream_t s)
{
    const int n = (int)B.args.size();
    const int nb = std::max(1, std::min(n, kBranches));
    if (B.branch.empty()) {
        B.branch.assign(nb, nullptr);
        B.join.assign(nb, nullptr);
        for (int j = 0; j < nb; ++j) {
            GBT_CUDA(cudaStreamCreateWithFlags(&B.branch[j], cudaStreamNonBlocking));
            GBT_CUDA(cudaEventCreateWithFlags(&B.join[j], cudaEventDisableTiming));
        }
        GBT_CUDA(cudaEventCreateWithFlags(&B.fork, cudaEventDisableTiming));
    }
    GBT_CUDA(cudaEventRecord(B.fork, s));
    for (int j = 0; j < nb; ++j) GBT_CUDA(cudaStreamWaitEvent(B.branch[j], B.fork, 0));
    char *w = static_cast<char *>(B.work);
    for (int k = 0; k < n; ++k) {
        const int i = B.order[k];
        cudaStream_t bs = B.branch[k % nb];
        const FwdParams &q = B.table[k];
        batch_prepass(B, i, q.work_counter, bs);
        if (B.args[i].n_recv == 0) continue;
        {
            FwdParams qq = q;
            tile_prep_launch(qq, B.window,
                             tile_ws_layout(w + B.ord_off[i], B.args[i].n_recv,
                                            B.traces[i]->d.capacity, B.args[i].tile_cull != 0), bs,
                             batch_weighted(B, i));
        }
        pair_fwd_launch(q, B.window, bs, false);
        batch_reduce(B, k, bs);
    }
    for (int j = 0; j < nb; ++j) {
        GBT_CUDA(cudaEventRecord(B.join[j], B.branch[j]));
        GBT_CUDA(cudaStreamWaitEvent(s, B.join[j], 0));
    }
}

static void batch_record(BatchImpl &B, cudaStream_t s)
{
    if (B.mode == kConcurrent) {
        batch_record_concurrent(B, s);
        return;
    }
    const int n = (int)B.args.size();
    char *w = static_cast<char *>(B.work);
    for (int i = 0; i < n; ++i) batch_prepass(B, i, nullptr, s);
    for (int k = 0; k < n; ++k) {
        const int i = B.order[k];
        FwdParams qq = B.table[k];
        tile_prep_launch(qq, B.window,
                         tile_ws_layout(w + B.ord_off[i], B.args[i].n_recv, B.traces[i]->d.capacity,
                                        B.args[i].tile_cull != 0), s);
    }
    FwdParams prm = B.table[0];
    prm.inst = B.d_table;
    prm.inst_off = B.d_off;
    prm.n_inst = n;
    prm.n_items = B.inst_off.back();
    prm.work_counter = B.counter;
    pair_batched_launch(prm, B.nf_max, B.window, B.grid, s);
    for (int k = 0; k < n; ++k) batch_reduce(B, k, s);
}

BatchImpl *batch_create(const gbt_batch_desc &d, cudaStream_t s)
{
    BatchImpl *B = new BatchImpl();
    try {
        // an instance with more than kGroupFreq frequencies becomes one instance per group of
        // consecutive frequencies, each writing its own rows of the caller's output
        for (int i = 0; i < d.n_instances; ++i) {
            const gbt_sum_args &a = d.args[i];
            for (int g0 = 0; g0 < a.n_freq; g0 += kGroupFreq) {
                gbt_sum_args sa = a;
                sa.n_freq = std::min(kGroupFreq, a.n_freq - g0);
                for (int f = 0; f < GBT_MAX_FREQ; ++f) {
                    sa.freq_hz[f] = f < sa.n_freq ? a.freq_hz[g0 + f] : 0.0;
                    sa.beam_b[f] = f < sa.n_freq ? a.beam_b[g0 + f] : 0.0;
                }
                sa.out = a.out + (size_t)g0 * (size_t)a.n_recv * 2;
                B->traces.push_back(d.traces[i]);
                B->args.push_back(sa);
            }
        }
        const int n = (int)B->args.size();
        B->use_graph = d.use_graph != 0;
        B->window = B->args[0].window;
        bool lossy = false;
        for (int i = 0; i < n; ++i) {
            GBT_REQUIRE(B->args[i].window == B->window, "batch instances must share one window");
            GBT_REQUIRE(B->args[i].precision == GBT_PRECISION_F32, "batches are F32 only");
            B->nf_max = std::max(B->nf_max, (int)B->args[i].n_freq);
            lossy = lossy || has_losses(B->args[i]);
        }
        if (lossy && d.form == GBT_BATCH_FUSED)
            fail(GBT_ERR_UNSUPPORTED, "the fused batch form has no losses: use GBT_BATCH_CONCURRENT");
        status_word();   // allocate before any capture
        // segment counts of every trace (each read once its trace is complete)
        B->n_seg.resize(n);
        B->cost.resize(n);
        for (int i = 0; i < n; ++i) {
            const TraceDev &td = B->traces[i]->d;
            const int32_t ns = read_device_i32(td.ray_off + td.n_rays, td.used);
            B->n_seg[i] = ns;
            B->cost[i] = (int64_t)ns * B->args[i].n_recv * B->args[i].n_freq;
        }
        B->order.resize(n);
        for (int i = 0; i < n; ++i) B->order[i] = i;
        std::stable_sort(B->order.begin(), B->order.end(),
                         [&](int x, int y) { return B->cost[x] > B->cost[y]; });
        B->grid = pair_batched_prepare(B->nf_max, B->window) * num_sms();
        // candidates: the concurrent form, then the fused launch at a few work
        // granularities (items per resident CTA); 0 items marks the concurrent form
        auto plan = [&](double ips) {
            B->mode = ips > 0.0 ? kFused : kConcurrent;
            if (ips > 0.0) batch_plan(*B, ips);
            else batch_plan_concurrent(*B);
            batch_layout(*B, s);
        };
        // the fused form's default granularity when it is not tuned
        double best_ips = d.form == GBT_BATCH_FUSED ? 32.0 : 0.0;
        std::vector<double> cands;
        if (d.form != GBT_BATCH_FUSED) cands.push_back(0.0);
        if (d.form != GBT_BATCH_CONCURRENT && !lossy)
            for (double v : {4.0, 8.0, 16.0, 32.0}) cands.push_back(v);
        if (d.autotune && cands.size() > 1) {
            float best = 1e30f;
            cudaEvent_t e0, e1;
            GBT_CUDA(cudaEventCreate(&e0));
            GBT_CUDA(cudaEventCreate(&e1));
            try {
                for (double ips : cands) {
                    plan(ips);
                    batch_record(*B, s);   // warm
                    GBT_CUDA(cudaEventRecord(e0, s));
                    batch_record(*B, s);
                    GBT_CUDA(cudaEventRecord(e1, s));
                    GBT_CUDA(cudaEventSynchronize(e1));
                    float ms = 0.f;
                    GBT_CUDA(cudaEventElapsedTime(&ms, e0, e1));
                    if (ms < best) { best = ms; best_ips = ips; }
                }
            } catch (...) {
                cudaEventDestroy(e0);
                cudaEventDestroy(e1);
                throw;
            }
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
        }
        plan(best_ips);
    } catch (...) {
        batch_destroy(B);
        throw;
    }
    return B;
}

static void batch_mark_used(BatchImpl *B, cudaStream_t s)
{
    mark_used(B->used, s);
    for (const gbt_trace_t *t : B->traces) mark_trace_used(t, s);
}

void batch_submit(BatchImpl *B, cudaStream_t s)
{
    if (!B->use_graph) {
        batch_record(*B, s);
        batch_mark_used(B, s);
        return;
    }
    if (!B->exec) {
        // record on a private stream (the caller's may be the legacy default stream,
        // which cannot be captured); the graph is then launched on the caller's stream
        if (!B->capture_stream)
            GBT_CUDA(cudaStreamCreateWithFlags(&B->capture_stream, cudaStreamNonBlocking));
        cudaStream_t cs = B->capture_stream;
        GBT_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        try {
            batch_record(*B, cs);
        } catch (...) {
            cudaGraph_t g = nullptr;
            cudaStreamEndCapture(cs, &g);
            if (g) cudaGraphDestroy(g);
            throw;
        }
        GBT_CUDA(cudaStreamEndCapture(cs, &B->graph));
        GBT_CUDA(cudaGraphInstantiate(&B->exec, B->graph, 0));
        // the launches were counted while recording; later replays add the graph's kernels
        size_t nn = 0;
        GBT_CUDA(cudaGraphGetNodes(B->graph, nullptr, &nn));
        std::vector<cudaGraphNode_t> nodes(nn);
        if (nn) GBT_CUDA(cudaGraphGetNodes(B->graph, nodes.data(), &nn));
        for (cudaGraphNode_t nd : nodes) {
            cudaGraphNodeType t;
            GBT_CUDA(cudaGraphNodeGetType(nd, &t));
            if (t == cudaGraphNodeTypeKernel) ++B->graph_kernels;
        }
    } else {
        note_launches(B->graph_kernels);
    }
    GBT_CUDA(cudaGraphLaunch(B->exec, s));
    batch_mark_used(B, s);
}

void batch_destroy(BatchImpl *B)
{
    if (!B) return;
    // the batch's workspace is freed behind its latest submit; graphs, streams and
    // events may be destroyed while work they launched is still pending
    cudaStream_t q = nullptr;
    try {
        q = after_last_use(B->used);
    } catch (...) {
        cudaDeviceSynchronize();
    }
    if (B->exec) cudaGraphExecDestroy(B->exec);
    if (B->graph) cudaGraphDestroy(B->graph);
    if (B->capture_stream) cudaStreamDestroy(B->capture_stream);
    for (cudaStream_t b : B->branch) if (b) cudaStreamDestroy(b);
    for (cudaEvent_t e : B->join) if (e) cudaEventDestroy(e);
    if (B->fork) cudaEventDestroy(B->fork);
    if (B->work) dfree(B->work, q);
    if (B->used) cudaEventDestroy(B->used);
    delete B;
}

// ---------------------------------------------------- bounded-wait self test --

// Waits on an mbarrier phase that nothing completes, with the same bounded
// try-wait loop the pair kernel uses; when the limit runs out it flags
// STATUS_TIMEOUT and returns, leaving the context usable.
__global__ void selftest_wait_kernel(long long spins, unsigned int *status)
{
    __shared__ unsigned long long bar;
    if (threadIdx.x != 0) return;
    mbar_init(smem_addr(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    for (long long it = 0; it < spins; ++it)
        if (mbar_try_wait(smem_addr(&bar), 0u)) return;
    atomicOr(status, STATUS_TIMEOUT);
}

void selftest_timeout_launch(long long spins, cudaStream_t s)
{
    selftest_wait_kernel<<<1, 32, 0, s>>>(spins, status_word());
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
}

// ------------------------------------------------- receiver order, no allocation --
//
// Some callers cannot allocate device memory at the point where they need a
// receiver order: a host application that owns every device allocation and
// forbids libraries from calling the CUDA allocator, or a latency-critical
// loop (a real-time auralisation thread, for example) that must not call an
// allocator because an allocation may block or fail under memory pressure.
// For them the sort's scratch lives in a fixed device array below.  The array
// is part of the library image: every GPU that loads the library holds it
// (8 MiB + 256 bytes) until the process exits.  Its contents persist between
// calls, so everything that must start at zero is cleared on each call, and
// calls that overlap on the GPU share (and race on) the array.
constexpr int64_t kNoAllocMaxRecv = 1 << 20;
static __device__ __align__(256) unsigned char
    g_order_scratch[kNoAllocMaxRecv * sizeof(unsigned long long) + 256];

namespace {
std::mutex g_order_scratch_mu;
void *g_order_scratch_dev[64] = {};
}  // namespace

void recv_order_noalloc_launch(const float *recv, int64_t n, int32_t *order, cudaStream_t s)
{
    if (n > kNoAllocMaxRecv)
        fail(GBT_ERR_INVALID_ARG, "gbt_recv_order_noalloc handles at most 1048576 receivers (got " +
                                      std::to_string(n) + ")");
    if (n <= 0) return;
    int dev = 0;
    GBT_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) fail(GBT_ERR_UNSUPPORTED, "device index >= 64");
    void *base = nullptr;
    {
        // set-up, once per device, with that device current: the host-side name of
        // the array is not a device address, so ask the runtime for the address
        std::lock_guard<std::mutex> lk(g_order_scratch_mu);
        if (!g_order_scratch_dev[dev]) {
            void *ptr = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&ptr, g_order_scratch);
            if (e != cudaSuccess) {
                cudaGetLastError();
                fail(GBT_ERR_CUDA, std::string("cudaGetSymbolAddress(order scratch): ") +
                                       cudaGetErrorString(e));
            }
            g_order_scratch_dev[dev] = ptr;
        }
        base = g_order_scratch_dev[dev];
    }
    int64_t npad = 1;
    while (npad < n) npad <<= 1;
    unsigned long long *keys = static_cast<unsigned long long *>(base);
    unsigned int *bb = reinterpret_cast<unsigned int *>(
        static_cast<char *>(base) + align_up((size_t)npad * sizeof(unsigned long long), 256));
    GBT_CUDA(cudaMemsetAsync(bb, 0xff, 3 * sizeof(unsigned int), s));
    GBT_CUDA(cudaMemsetAsync(bb + 3, 0x00, 3 * sizeof(unsigned int), s));
    bbox_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, s>>>(recv, n, bb);
    note_launches(1);
    const unsigned g = (unsigned)((npad + 255) / 256);
    morton_kernel<<<g, 256, 0, s>>>(recv, n, npad, bb, keys);
    note_launches(1);
    for (int64_t k = 2; k <= npad; k <<= 1)
        for (int64_t j = k >> 1; j > 0; j >>= 1) {
            bitonic_step<<<g, 256, 0, s>>>(keys, npad, j, k);
            note_launches(1);
        }
    extract_order<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(keys, n, order);
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
}

void set_list_capacity(int64_t entries) { g_list_cap_limit.store(entries); }

}  // namespace gbt
