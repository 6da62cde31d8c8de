// Mixed-radix transforms, two per thread: radices up to 13.
#include "fft_mixed_pair.cuh"

namespace gb300fft {
const void *mixed_pair13_fn(bool cols) { return pair_fn<C2, 13>(cols); }
}  // namespace gb300fft
