// The batched launch sequence (FP32 systems).
#include "enuf_enqueue.cuh"
namespace enuf {
template size_t batch_bytes<float>(const BatchSys*, int);
template cudaError_t configure_batch<float>(int);
template cudaError_t batch_build<float>(void*, const BatchSys*, int, BatchLaunch*);
template cudaError_t batch_enqueue<float>(const BatchLaunch&, cudaStream_t, cudaStream_t, cudaEvent_t, cudaEvent_t,
                                          LaunchLog*);
}  // namespace enuf
