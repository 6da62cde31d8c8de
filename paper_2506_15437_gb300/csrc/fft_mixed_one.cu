// Mixed-radix transforms, one per thread: launches too small to fill the GPU, the
// passes of a four-step transform, lengths beyond 7000 and odd row widths.
#include "fft_mixed_pair.cuh"

namespace gb300fft {
const void *mixed_one_fn(bool cols, bool fs) {
    return fs ? (const void *)k_mixed_pair<float2, 16, false, true> : pair_fn<float2, 16>(cols);
}
}  // namespace gb300fft
