// Stockham FFT passes (FP32).
#include "enuf_enqueue.cuh"

namespace enuf {
template struct StockhamPasses<float, false>;
template struct StockhamPasses<float, true>;
}  // namespace enuf
