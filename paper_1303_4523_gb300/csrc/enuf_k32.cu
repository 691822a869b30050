// FP32 instantiation of the ENUF-DPD kernels and launch sequences.
#include "enuf_enqueue.cuh"
namespace enuf {
ENUF_INSTANTIATE(float)

cudaError_t configure_fft2(const FftShape& fs, const FftPlanDev& fp, int max_smem) {
    auto set = [&](auto passes) { return passes.configure(max_smem); };
    return fft2_dispatch(fs, fp, set, set);
}
}  // namespace enuf
