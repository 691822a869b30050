// Two-factor FFT passes of single lengths (FP32), part d.
#include "enuf_enqueue.cuh"

namespace enuf {
#define ENUF_INST(a, b) template struct Fft2Lines<a, b>;
ENUF_FFT2_LINES_B(ENUF_INST)
}  // namespace enuf
