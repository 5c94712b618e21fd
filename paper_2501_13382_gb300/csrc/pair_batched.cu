// pair_batched.cu -- the pair kernel over many instances in one persistent launch: one work
// counter over the items of all instances (longest first), each warp loading the item's
// instance parameters into shared memory.
#include "pair.cuh"

namespace gbt {
namespace {
template <int NF, int WINDOW>
int run(const FwdParams *p, int grid, cudaStream_t s)
{
    using Cfg = PairCfg<WarpBuf<NF, false>, true, PairShape<NF, false>::kWarpsBatched>;
    static std::atomic<int> known[64] = {};
    auto *fn = gbs_pair_kernel<NF, WINDOW, true, false>;
    const int per_sm = resident_ctas<Cfg>(fn, known);
    if (!p) return per_sm;
    GBT_CUDA(cudaMemsetAsync(p->work_counter, 0, sizeof(int), s));
    fn<<<grid, 32 * Cfg::kWarps, Cfg::kSmem, s>>>(*p);
    note_launches(1);
    GBT_CUDA(cudaGetLastError());
    return per_sm;
}
template <int WINDOW>
int run_nf(const FwdParams *p, int nf, int grid, cudaStream_t s)
{
    return nf <= 1   ? run<1, WINDOW>(p, grid, s)
           : nf <= 2 ? run<2, WINDOW>(p, grid, s)
           : nf <= 4 ? run<4, WINDOW>(p, grid, s)
                     : run<8, WINDOW>(p, grid, s);
}
}  // namespace

int pair_batched_prepare(int nf_max, int window)
{
    return window == GBT_WINDOW_LINE ? run_nf<GBT_WINDOW_LINE>(nullptr, nf_max, 0, nullptr)
                                     : run_nf<GBT_WINDOW_SEGMENT>(nullptr, nf_max, 0, nullptr);
}

void pair_batched_launch(const FwdParams &p, int nf_max, int window, int grid, cudaStream_t s)
{
    if (window == GBT_WINDOW_LINE) run_nf<GBT_WINDOW_LINE>(&p, nf_max, grid, s);
    else run_nf<GBT_WINDOW_SEGMENT>(&p, nf_max, grid, s);
}
}  // namespace gbt
