// The FFT passes of the sides 64, 96, 128 and 192.
#include "fft_passes.cuh"

namespace hrt {

template struct Passes<2>;
template struct Passes<3>;
template struct Passes<4>;
template struct Passes<6>;

}  // namespace hrt
