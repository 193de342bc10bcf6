// The compile-time-length FFT passes in FP32.
#include "fft_launch_impl.cuh"

namespace chebfi {
template void fft_tables<float>();
template bool fast_dispatch<float>(chebfi_ctx*, const cplx<float>*, int64_t, int64_t, cplx<float>*, LocalEpi<float>, cudaStream_t,
                                const float*);
template bool fast_real_space<float>(chebfi_ctx*, const cplx<float>*, int64_t, int64_t, cplx<float>*, cplx<float>*, bool, cudaStream_t);
}  // namespace chebfi
