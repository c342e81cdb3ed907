// The FFT matcher's kernel, planes up to 96 x 96 (PAIR and PAIRT).
// One translation unit per geometry: the build compiles them in parallel.
#include "cfog_match_fft.cuh"

namespace cfog {
MatchKernel match_kernel_pair() { return make_kernel<Geometry<kFftThreads, 2, 256>>(); }
}  // namespace cfog
