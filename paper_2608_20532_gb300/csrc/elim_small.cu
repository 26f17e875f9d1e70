// Elimination of the contexts of at most SMALL_WD words (d <= 96).
#include "elim.cuh"

namespace f2 {
namespace {

static_assert(DEFAULT_SMALL_REGION_BYTES / 4 >= 32 * SMALL_WD * row_stride(SMALL_WD) + CTL_WORDS + FL_WORDS,
              "a warp region holds the basis of any small-width context");

// CTA-owned contexts first (longest first), then warp-owned ones, at three
// CTAs per SM (80 registers; four CTAs at 64 registers spill and ran 6%
// slower on the 78k-context, 81M-row learn).
__global__ void __launch_bounds__(LEARN_WARPS * 32, 3) elim_small_kernel(StoreDev s, LearnArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) uint32_t smem[];
    elim_queues<CLS_CTA_S, CLS_WARP_S, CLS_RESUME_S>(s, a, smem, a.small_region_words, [&](int c, auto cta, uint32_t* region, int words) {
        switch (s.desc[c].wd) {
        case 1: elim_one<1, decltype(cta)::value>(s, a, c, region, words); break;
        case 2: elim_one<2, decltype(cta)::value>(s, a, c, region, words); break;
        case 3: elim_one<3, decltype(cta)::value>(s, a, c, region, words); break;
        default: break;
        }
    });
}

}  // namespace

cudaError_t elim_launch_small(const StoreDev& sd, LearnArgs la, int max_words, int num_sms, cudaStream_t cs)
{
    return launch_queues(elim_small_kernel, sd, la, max_words, la.small_region_words, LEARN_WARPS, 3, num_sms, cs);
}

cudaError_t elim_load_small()
{
    cudaFuncAttributes fa;
    return cudaFuncGetAttributes(&fa, elim_small_kernel);
}

}  // namespace f2
