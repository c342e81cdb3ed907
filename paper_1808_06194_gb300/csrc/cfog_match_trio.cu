// The FFT matcher's kernel, three CPs per SM (TRIO).
// One translation unit per geometry: the build compiles them in parallel.
#include "cfog_match_fft.cuh"

namespace cfog {
MatchKernel match_kernel_trio() { return make_kernel<Geometry<kFftThreads, 3, 256>>(); }
}  // namespace cfog
