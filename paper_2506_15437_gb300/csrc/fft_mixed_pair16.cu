// Mixed-radix transforms, two per thread: radices up to 16.
#include "fft_mixed_pair.cuh"

namespace gb300fft {
const void *mixed_pair16_fn(bool cols) { return pair_fn<C2, 16>(cols); }
}  // namespace gb300fft
