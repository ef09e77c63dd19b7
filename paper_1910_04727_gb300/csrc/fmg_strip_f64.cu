// The column-strip smoother in double arithmetic.
#include "fmg_strip_impl.cuh"

namespace fm {
template void strip_launch<double>(fm_ctx*, const StripCall<double>&, cudaStream_t);
template void strip_init<double>(int);
}  // namespace fm
