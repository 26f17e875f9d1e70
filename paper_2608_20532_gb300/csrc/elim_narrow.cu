// Elimination of the contexts of SMALL_WD + 1 .. NARROW_WD words (96 < d <= 288).
#include "elim.cuh"

namespace f2 {
namespace {

// CTA-owned contexts first (longest first), then warp-owned ones, 16 warps per
// SM at 128 registers.  A CTA-owned context's insertions run one warp at a time,
// so CTAs of four warps waste less (2,388 against 2,434 us on the 77,926-context
// learn), but a long context takes longer in them: calls of fewer than
// DEFAULT_LONG_CALL_ROWS rows, which one such context can hold up, take eight.
// 4,096 contexts with a few of 10,000 and more rows: 398 us with four, 307 with
// eight; where no context stands out 265 and 268, 10,000 contexts of parsed
// values 1,051 and 1,061.
__global__ void __launch_bounds__(LEARN_WARPS * 32, 2) elim_narrow_kernel(StoreDev s, LearnArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) uint32_t smem[];
    elim_queues<CLS_CTA, CLS_WARP, CLS_RESUME>(s, a, smem, a.warp_region_words, [&](int c, auto cta, uint32_t* region, int words) {
        switch (s.desc[c].wd) {
        case 4: elim_one<4, decltype(cta)::value>(s, a, c, region, words); break;
        case 5: elim_one<5, decltype(cta)::value>(s, a, c, region, words); break;
        case 6: elim_one<6, decltype(cta)::value>(s, a, c, region, words); break;
        case 7: elim_one<7, decltype(cta)::value>(s, a, c, region, words); break;
        case 8: elim_one<8, decltype(cta)::value>(s, a, c, region, words); break;
        case 9: elim_one<9, decltype(cta)::value>(s, a, c, region, words); break;
        default: break;
        }
    });
}

}  // namespace

cudaError_t elim_launch_narrow(const StoreDev& sd, LearnArgs la, int max_words, int warps, int num_sms, cudaStream_t cs)
{
    return launch_queues(elim_narrow_kernel, sd, la, max_words, la.warp_region_words, warps, 16 / warps, num_sms, cs);
}

cudaError_t elim_load_narrow()
{
    cudaFuncAttributes fa;
    return cudaFuncGetAttributes(&fa, elim_narrow_kernel);
}

}  // namespace f2
