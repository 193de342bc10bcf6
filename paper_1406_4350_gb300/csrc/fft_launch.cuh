// Kernels and launches of the compile-time-length FFT path of the local-potential operator
// (Section 2.1), instantiated once per arithmetic: fft_f32.cu, fft_f64.cu, fft_df.cu.
#pragma once

#include "fft_core.cuh"
#include "fft_fast.cuh"
#include "fft_fast_kernels.cuh"
#include "internal.cuh"
#include "kernels.cuh"

namespace chebfi {

// The constant tables of the compiled passes on the current device: filled once per device and
// complete on return.  A context fills them when it takes a potential on a compiled grid, so
// that its launches, which may be inside a stream capture, have nothing to set up.
template <typename R> void fft_tables();
void fixed_tables();

// (K + V_loc) with the compiled kernels of the context's grid; false if its size has none
template <typename R>
bool fast_dispatch(chebfi_ctx* ctx, const cplx<typename SphT<R>::type>* Y, int64_t ldy, int64_t nb, cplx<R>* T,
                   LocalEpi<typename SphT<R>::type> ep, cudaStream_t st, const typename SphT<R>::type* K);

// Real-space values of nb <= 65535 bands on a compiled grid, out[band][z'][x'][y'] in split
// order (T: column buffer): the z pass, and with `planes` the plane pass; false if the size
// has no compiled kernels.  fixed_planes_real: the plane pass from an FP64 column buffer in
// fixed point (false at sizes without it).
template <typename R>
bool fast_real_space(chebfi_ctx* ctx, const cplx<R>* Y, int64_t ldy, int64_t nb, cplx<R>* T, cplx<R>* out, bool planes,
                     cudaStream_t st);
bool fixed_planes_real(chebfi_ctx* ctx, int64_t nb, const double2* T, double2* out, cudaStream_t st);
// The plane pass (multiply by V_loc included) of nb <= 65535 bands in fixed point; false where
// the context's FP64 path does not take it.
bool fixed_planes(chebfi_ctx* ctx, int64_t nb, cdf* T, cudaStream_t st);
bool fixed_planes(chebfi_ctx* ctx, int64_t nb, double2* T, cudaStream_t st);
inline bool fixed_planes(chebfi_ctx*, int64_t, float2*, cudaStream_t) { return false; }

}  // namespace chebfi
