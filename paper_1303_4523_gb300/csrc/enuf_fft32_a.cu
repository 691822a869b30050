// Two-factor FFT passes of single lengths (FP32), part a.
#include "enuf_enqueue.cuh"

namespace enuf {
#define ENUF_INST(a, b) template struct Fft2Planes<a, b>;
ENUF_FFT2_PLANES_A(ENUF_INST)
}  // namespace enuf
