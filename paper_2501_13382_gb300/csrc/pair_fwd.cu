// pair_fwd.cu -- forward instantiations of the pair kernel.
#include "pair.cuh"

namespace gbt {
namespace {
template <int NF, int WINDOW, bool LOSSY>
void launch(const FwdParams &p, cudaStream_t s, bool timed)
{
    static std::atomic<int> known[64] = {};
    launch_items<PairCfg<WarpBuf<NF, LOSSY>, false, PairShape<NF, LOSSY>::kWarps>>(gbs_pair_kernel<NF, WINDOW, false, LOSSY>, known, p, s, timed);
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

void pair_fwd_launch(const FwdParams &p, int window, cudaStream_t s, bool timed)
{
    if ((!p.order || p.n_recv <= kCtaRecv) && !p.list) pair_unordered_launch(p, window, s, timed);
    else if (window == GBT_WINDOW_LINE) launch_nf<GBT_WINDOW_LINE>(p, s, timed);
    else launch_nf<GBT_WINDOW_SEGMENT>(p, s, timed);
}
}  // namespace gbt
