// Mixed-radix transforms, one per thread, for launches too small to fill the GPU.
#include "fft_mixed_pair.cuh"

namespace gb300fft {
const void *mixed_one_fn(bool cols, bool fs) { return pair_fn<float2, 16>(cols, fs); }
}  // namespace gb300fft
