// The FFT passes of the sides 384 and 768.
#include "fft_passes.cuh"

namespace hrt {

template struct Passes<12>;
template struct Passes<24>;

}  // namespace hrt
