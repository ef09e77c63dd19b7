// The column-strip smoother in float arithmetic.
#include "fmg_strip_impl.cuh"

namespace fm {
template void strip_launch<float>(fm_ctx*, const StripCall<float>&, cudaStream_t);
template void strip_init<float>(int);
}  // namespace fm
