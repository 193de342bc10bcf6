// Kernels and launches of the compile-time-length FFT path of the local-potential operator
// (Section 2.1), instantiated once per arithmetic: fft_f32.cu, fft_f64.cu, fft_df.cu.
#pragma once

#include "fft_core.cuh"
#include "fft_fast.cuh"
#include "fft_fast_kernels.cuh"
#include "internal.cuh"
#include "kernels.cuh"

namespace chebfi {

// (K + V_loc) with the compiled kernels of the context's grid; false if its size has none
template <typename R>
bool fast_dispatch(chebfi_ctx* ctx, const cplx<typename SphT<R>::type>* Y, int64_t ldy, int64_t nb, cplx<R>* T,
                   LocalEpi<typename SphT<R>::type> ep, cudaStream_t st, const typename SphT<R>::type* K);

}  // namespace chebfi
