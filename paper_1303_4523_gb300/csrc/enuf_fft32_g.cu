// Two-factor FFT passes of any length (FP32).
#include "enuf_enqueue.cuh"

namespace enuf {
template struct Fft2Lines<0, 0>;
}  // namespace enuf
