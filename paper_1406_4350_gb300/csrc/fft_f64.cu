// The compile-time-length FFT passes in the FP64 units.
#include "fft_launch_impl.cuh"

namespace chebfi {
template void fft_tables<double>();
template bool fast_dispatch<double>(chebfi_ctx*, const cplx<double>*, int64_t, int64_t, cplx<double>*, LocalEpi<double>, cudaStream_t,
                                const double*);
template bool fast_real_space<double>(chebfi_ctx*, const cplx<double>*, int64_t, int64_t, cplx<double>*, cplx<double>*, bool, cudaStream_t);
}  // namespace chebfi
