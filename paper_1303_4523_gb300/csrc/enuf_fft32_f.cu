// Two-factor FFT passes of single lengths (FP32), part f.
#include "enuf_enqueue.cuh"

namespace enuf {
#define ENUF_INST(a, b) template struct Fft2Lines<a, b>;
ENUF_FFT2_LINES_D(ENUF_INST)
}  // namespace enuf
