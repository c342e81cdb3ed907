// The FFT matcher's kernel, planes up to 128 x 128, with twice the threads and one CTA per
// SM: launches with so few CPs that an SM would not get two.
#include "cfog_match_fft.cuh"

namespace cfog {
MatchKernel match_kernel_wide_tall() { return make_kernel<Geometry<kFftThreadsTall, 1, 512>>(); }
}  // namespace cfog
