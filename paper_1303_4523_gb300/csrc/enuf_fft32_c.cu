// Two-factor FFT passes of single lengths (FP32), part c.
#include "enuf_enqueue.cuh"

namespace enuf {
#define ENUF_INST(a, b) template struct Fft2Lines<a, b>;
ENUF_FFT2_LINES_A(ENUF_INST)
}  // namespace enuf
