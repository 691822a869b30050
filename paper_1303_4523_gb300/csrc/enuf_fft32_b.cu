// Two-factor FFT passes of single lengths (FP32), part b.
#include "enuf_enqueue.cuh"

namespace enuf {
#define ENUF_INST(a, b) template struct Fft2Planes<a, b>;
ENUF_FFT2_PLANES_B(ENUF_INST)
}  // namespace enuf
