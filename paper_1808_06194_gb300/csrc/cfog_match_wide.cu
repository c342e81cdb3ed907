// The FFT matcher's kernel, planes up to 128 x 128 (WIDE; the kernel of cfog_match).
// One translation unit per geometry: the build compiles them in parallel.
#include "cfog_match_fft.cuh"

namespace cfog {
MatchKernel match_kernel_wide() { return make_kernel<Geometry<kFftThreads, 2, 512>>(); }
}  // namespace cfog
