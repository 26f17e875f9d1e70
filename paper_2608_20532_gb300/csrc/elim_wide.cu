// Elimination of the contexts of more than NARROW_WD words, a CTA each.
#include "elim.cuh"

namespace f2 {
namespace {

template <int WDT, int CLS, int RESUME>
__global__ void __launch_bounds__(WIDE_WARPS * 32, WDT <= WIDE_M_WD ? 2 : 1) elim_wide_kernel(StoreDev s, LearnArgs a)
{
    extern __shared__ __align__(16) uint32_t smem[];
    elim_cta_queue<CLS, RESUME>(s, a, [&](int c) { elim_cta<WDT>(s, a, c, smem, a.cta_region_words); });
}

template <typename K>
cudaError_t launch(K kernel, const StoreDev& sd, LearnArgs la, int max_d, int wdt, int per_sm, int num_sms,
                   cudaStream_t cs)
{
    la.cta_region_words = elim_words(max_d, wdt);
    const size_t smem = 4 * (size_t)la.cta_region_words;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<num_sms * resident_ctas(smem, per_sm), WIDE_WARPS * 32, smem, cs>>>(sd, la);
    return cudaGetLastError();
}

}  // namespace

cudaError_t elim_launch_wide(const StoreDev& sd, LearnArgs la, int max_d, bool medium, int num_sms, cudaStream_t cs)
{
    if (medium)
        return launch(elim_wide_kernel<WIDE_M_WD, CLS_WIDE_M, CLS_RESUME_W>, sd, la, max_d, WIDE_M_WD, 2, num_sms, cs);
    return launch(elim_wide_kernel<WIDE_WD, CLS_WIDE, CLS_RESUME_W>, sd, la, max_d, WIDE_WD, 1, num_sms, cs);
}

cudaError_t elim_load_wide()
{
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, elim_wide_kernel<WIDE_M_WD, CLS_WIDE_M, CLS_RESUME_W>);
    return e != cudaSuccess ? e : cudaFuncGetAttributes(&fa, elim_wide_kernel<WIDE_WD, CLS_WIDE, CLS_RESUME_W>);
}

}  // namespace f2
