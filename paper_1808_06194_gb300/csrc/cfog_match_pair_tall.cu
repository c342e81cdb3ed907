// The FFT matcher's kernel, planes up to 96 x 96, with twice the threads and one CTA per
// SM: launches with so few CPs that an SM would not get two.
#include "cfog_match_fft.cuh"

namespace cfog {
MatchKernel match_kernel_pair_tall() { return make_kernel<Geometry<kFftThreadsTall, 1, 256>>(); }
}  // namespace cfog
