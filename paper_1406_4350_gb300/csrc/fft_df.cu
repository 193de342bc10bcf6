// The compile-time-length FFT passes in double-float.
#define CHEBFI_FFT_DF
#include "fft_launch_impl.cuh"

namespace chebfi {
template void fft_tables<dfl>();
template bool fast_dispatch<dfl>(chebfi_ctx*, const cplx<double>*, int64_t, int64_t, cplx<dfl>*, LocalEpi<double>, cudaStream_t,
                                const double*);
}  // namespace chebfi
