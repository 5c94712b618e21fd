// pair_stream.cuh -- what the forward and the adjoint pair kernels share: the items of the
// work queue, the gathering of the segments that reach a warp tile, and the launch.
#pragma once

#include <algorithm>
#include <atomic>

#include "pair_common.cuh"

namespace gbt {
namespace {

constexpr int kScan = 4;                    // chunks tested at a time without a list
constexpr int kFoldEvery = 16;              // batches between float-float folds
static_assert(kFoldEvery % kScan == 0, "fold groups are whole windows");

// One item of the queue: a warp tile and a split of the segments it goes through.
struct Item {
    int64_t wbase;             // first receiver (processing order) of the warp tile
    int split, splits;         // of the tile's
    int64_t part;              // first partial of the warp tile's first receiver, band 0
    int64_t part_band;         // and from band to band
    const int32_t *lst;        // the CTA tile's list, or null: every segment
    const uint32_t *lw;        // this warp tile's words of its chunks
    int64_t n_seg;             // entries of the list, or segments
};
// Item `it` of p: CTA tile by dispatch rank, split, warp tile within the CTA tile; false
// past the last receiver.  (Items of p: see item_count.)
__device__ __forceinline__ int64_t item_count(const FwdParams &p)
{
    return p.item_off ? (int64_t)p.item_off[p.n_tiles] * kTileWarps : p.n_items;
}
__device__ __forceinline__ bool decode_item(const FwdParams &p, int64_t it, Item &m)
{
    const int64_t g = it / kTileWarps;         // tile-split
    const int wl = (int)(it - g * kTileWarps);
    int64_t tile_rank;
    if (p.item_off) {
        int lo = 0, hi = p.n_tiles - 1;        // last rank with item_off <= g
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (p.item_off[mid] <= g) lo = mid;
            else hi = mid - 1;
        }
        tile_rank = lo;
        m.split = (int)(g - p.item_off[lo]);
        m.splits = p.item_off[lo + 1] - p.item_off[lo];
    } else {
        tile_rank = g / p.splits;
        m.split = (int)(g - tile_rank * p.splits);
        m.splits = p.splits;
    }
    const int64_t tile = p.tile_perm ? (int64_t)p.tile_perm[tile_rank] : tile_rank;
    m.wbase = tile * kCtaRecv + (int64_t)wl * kWarpRecv;
    if (m.wbase >= p.n_recv) return false;
    m.part_band = p.item_off ? p.part_recv : p.n_recv;
    m.part = p.item_off ? g * p.nf * p.part_recv + (int64_t)wl * kWarpRecv
                        : (int64_t)m.split * p.nf * p.n_recv + m.wbase;
    m.lst = nullptr;
    m.lw = nullptr;
    m.n_seg = *p.n_seg_ptr;
    if (p.list) {
        const int32_t ln = p.list_n[tile];
        if (ln >= 0) {
            m.lst = p.list + p.list_off[tile];
            m.lw = p.list_words + (p.list_off[tile] / kBatch) * kChunkWords + wl;
            m.n_seg = ln;
        }
    }
    return true;
}

// The raw records of two batches, word-major (each lane copies and reads only its own), and
// the positions of the batch being queued.
struct RawBuf {
    float4 raw[2][4][kBatch];
    float amp[2][kBatch];
    int32_t queue[kBatch];
};

// Batches of an item.  A window is the item's next 32 list chunks (one word per lane) or
// next kScan segment chunks (words of lanes 0 .. kScan - 1, from the ball test); its set
// bits' positions are queued in order and each full batch's records are gathered (one
// commit group per batch, empty past the end).
// GROUPS: each batch also carries its fold group: kFoldEvery batches of list entries, or without
// a list kFoldEvery chunks of segments (a batch ends where its group does).
template <int WINDOW, bool GROUPS>
struct Gather {
    int64_t wnext;             // first chunk of the next window
    int64_t wchunk = 0;        // this lane's chunk of the current window
    uint32_t word = 0u;        // its entries not yet queued
    int n0 = 0, n1 = 0;        // per buffer: records of the batch
    int32_t seg0 = -1, seg1 = -1;   // and this lane's segment
    int count = 0;             // GROUPS: batches issued, or windows scanned
    int group0 = 0, group1 = 0;     // per buffer: fold group

    __device__ __forceinline__ explicit Gather(const Item &m) : wnext(m.split) {}

    __device__ __forceinline__ void issue(const FwdParams &p, const Item &m, RawBuf &B, int lane,
                                          const float4 &rball, int buf)
    {
        const int64_t n_chunks = (m.n_seg + kBatch - 1) / kBatch;
        int n = 0;
        while (n < kBatch) {
            const uint32_t act = __ballot_sync(0xffffffffu, word != 0u);
            if (!act) {
                if (wnext >= n_chunks) break;
                if (GROUPS && !m.lst) {
                    if (n > 0 && count % (kFoldEvery / kScan) == 0) break;
                    ++count;
                }
                wchunk = wnext + (int64_t)lane * m.splits;
                if (m.lst) {
                    word = wchunk < n_chunks ? m.lw[wchunk * kChunkWords] : 0u;
                    wnext += (int64_t)32 * m.splits;
                } else {
                    float4 q0[kScan], q1[kScan];
#pragma unroll
                    for (int i = 0; i < kScan; ++i) {
                        const int64_t sg = (wnext + (int64_t)i * m.splits) * kBatch + lane;
                        q0[i] = q1[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (sg < m.n_seg) {
                            q0[i] = p.crec[2 * sg];
                            q1[i] = p.crec[2 * sg + 1];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < kScan; ++i) {
                        const int64_t sg = (wnext + (int64_t)i * m.splits) * kBatch + lane;
                        const uint32_t b = __ballot_sync(0xffffffffu,
                            sg < m.n_seg && seg_reaches_ball<WINDOW>(seg_cull(q0[i], q1[i]), rball,
                                                                     p.pre_alpha, p.pre_beta));
                        if (lane == i) word = b;
                    }
                    wnext += (int64_t)kScan * m.splits;
                }
                continue;
            }
            if (__any_sync(0xffffffffu, __popc(word) > 6)) {
                // full words: one chunk at a time, a lane per entry
                const int src = __ffs(act) - 1;
                const uint32_t b = __shfl_sync(0xffffffffu, word, src);
                const int32_t base = __shfl_sync(0xffffffffu, (int32_t)wchunk, src) * kBatch;
                const int slot = n + __popc(b & ((1u << lane) - 1u));
                const bool set = (b >> lane) & 1u;
                if (set && slot < kBatch) B.queue[slot] = base + lane;
                const uint32_t rest = __ballot_sync(0xffffffffu, set && slot >= kBatch);
                if (lane == src) word = rest;
                n = min(n + __popc(b), kBatch);
            } else {
                // sparse words: a lane per chunk, its entries one after the other
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
                    B.queue[slot++] = (int32_t)(wchunk * kBatch) + __ffs(word) - 1;
                    word &= word - 1u;
                }
                n = min(n + total, kBatch);
            }
        }
        __syncwarp();
        int32_t idx = -1;
        if (lane < n) {
            idx = B.queue[lane];
            if (m.lst) idx = m.lst[idx];
            const float4 *src = reinterpret_cast<const float4 *>(p.rec + (int64_t)idx * kRecFloats);
#pragma unroll
            for (int c = 0; c < 4; ++c) cp_async16(&B.raw[buf][c][lane], src + c, 16);
            cp_async4(&B.amp[buf][lane], p.rec + (int64_t)idx * kRecFloats + R_AMP);
        }
        cp_async_commit();
        __syncwarp();
        if (GROUPS) {
            const int grp = m.lst ? count++ / kFoldEvery : (count - 1) / (kFoldEvery / kScan);
            if (buf) group1 = grp; else group0 = grp;
        }
        if (buf) { n1 = n; seg1 = idx; } else { n0 = n; seg0 = idx; }
    }
};

// A staged word's two values as float pairs: of slot j, or (EACH) of slot j for the lane's first
// receiver and j1 for its second.
template <bool EACH>
__device__ __forceinline__ void staged(const float4 *w, int j, int j1, f2x &a, f2x &b)
{
    if (EACH) {
        const float4 u = w[j], v = w[j1];
        a = pk(u.x, v.x);
        b = pk(u.z, v.z);
    } else {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(w + j);
        a = v.x;
        b = v.y;
    }
}

// Adds an FP32 partial sum (x, y) into a float-float accumulator (hi, hi, lo, lo); the
// item's first fold only writes it.
__device__ __forceinline__ void fold(float4 *acc, float x, float y, bool first)
{
    if (first) {
        __stcg(acc, make_float4(x, y, 0.0f, 0.0f));
    } else if (x != 0.0f || y != 0.0f) {
        float4 a = __ldcg(acc);
        float s, e;
        two_sum(a.x, x, s, e);
        a.x = s;
        a.z += e;
        two_sum(a.y, y, s, e);
        a.y = s;
        a.w += e;
        __stcg(acc, a);
    }
}

// Zero partials of the item's receiver `at` (of its warp tile), which takes no part.
__device__ __forceinline__ void no_partials(const FwdParams &p, const Item &m, int at)
{
    for (int f = 0; f < p.nf; ++f)
        __stcg(p.partial + m.part + f * m.part_band + at, make_float4(0.f, 0.f, 0.f, 0.f));
}

// Folds a lane's two receivers' sums per band into the item's partials and zeroes them.
template <int NF>
__device__ __forceinline__ void fold_bands(const FwdParams &p, const Item &m, int lane, const bool (&part_of)[kR],
                                           f2x (&ax)[NF], f2x (&ay)[NF], bool &first)
{
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (f < p.nf) {
            float x0, x1, y0, y1;
            upk(ax[f], x0, x1);
            upk(ay[f], y0, y1);
            float4 *const part = p.partial + m.part + f * m.part_band + lane;
            if (part_of[0]) fold(part, x0, y0, first);
            if (part_of[1]) fold(part + 32, x1, y1, first);
        }
        ax[f] = ay[f] = 0ull;
    }
    first = false;
}

// Launch shape of a kernel with per-warp shared memory BUF (and, batched, the instance's
// parameters): as many warps as fit in the shared memory budget, at most MOST.
template <class BUF, bool BATCHED, int MOST = kWarpsFwd>
struct PairCfg {
    static constexpr size_t kInst = BATCHED ? sizeof(FwdParams) : 0;
    static constexpr size_t kPerWarp = (sizeof(BUF) + kInst + 127) / 128 * 128;
    static constexpr int kFit = (int)(kSmemBudget / kPerWarp);
    static constexpr int kWarps = kFit < MOST ? kFit : MOST;
    static constexpr size_t kSmem = kWarps * kPerWarp;
};

// Resident CTAs per SM of a kernel (its shared memory attribute set), asked once per device.
template <class CFG, class FN>
int resident_ctas(FN fn, std::atomic<int> (&known)[64])
{
    int dev = 0;
    GBT_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) fail(GBT_ERR_UNSUPPORTED, "device index >= 64");
    int per_sm = known[dev].load(std::memory_order_acquire);
    if (per_sm) return per_sm;
    GBT_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CFG::kSmem));
    GBT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * CFG::kWarps, CFG::kSmem));
    if (per_sm < 1) fail(GBT_ERR_UNSUPPORTED, "GBS kernel does not fit on one SM");
    known[dev].store(per_sm, std::memory_order_release);
    return per_sm;
}

// Launches one persistent kernel over p's items (p.work_counter zeroed by the prepass).
template <class CFG, class FN>
void launch_items(FN fn, std::atomic<int> (&known)[64], const FwdParams &p, cudaStream_t s, bool timed)
{
    const int per_sm = resident_ctas<CFG>(fn, known);
    const int grid = (int)std::max<int64_t>(
        1, std::min<int64_t>((p.n_items + CFG::kWarps - 1) / CFG::kWarps, (int64_t)per_sm * num_sms()));
    if (timed) timing_begin(s);
    fn<<<grid, 32 * CFG::kWarps, CFG::kSmem, s>>>(p);
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
    if (timed) timing_end(s);
}

}  // namespace
}  // namespace gbt
