// Kernels and launches of the compile-time-length FFT path of the local-potential operator
// (Section 2.1): the definition of fast_dispatch<R>, included by one translation unit per
// arithmetic R.
#pragma once

#include <type_traits>

#include "fft_launch.cuh"

namespace chebfi {
namespace {
constexpr int kThreads = 256;

// ---------------------------------------------------------------- compile-time-length path
// The pass bodies live in fft_fast_kernels.cuh; here each block finds its columns or plane
// from its grid position.
using fk::FastArgs;
using fk::kCBF;

// Threads of a z pass's block (kCBF lines): its two transform passes have kCBF NB and kCBF NA
// items, mostly fewer than 256, so smaller blocks leave fewer threads idle at their barriers;
// measured with 64, 128, 192 and 256 (ms for 512 bands; 256 threads and the choice).  Inverse:
// FP32 60^3 0.070 and 0.065, 80^3 0.164 and 0.145, double-float 72^3 0.424 and 0.356, 96^3 0.974
// and 0.907.  Forward, whose epilogue wants more loads in flight: FP32 60^3 0.089 and 0.079,
// double-float 72^3 0.493 and 0.431, but FP32 64^3 0.080 with 256 and 0.088 with 128.
// The FP64 units bind theirs whatever the block (36^3: 0.152 ms with 256, 0.157 with 128).
template <typename R, int N> constexpr int zinv_threads() {
  return std::is_same<R, double>::value ? kThreads : N < 96 ? 128 : 192;
}
template <typename R, int N> constexpr int zfwd_threads() {
  return std::is_same<R, dfl>::value ? (N < 96 ? 128 : 192) : std::is_same<R, float>::value && N < 64 ? 128 : kThreads;
}

// R: the arithmetic of the transforms (float, double, or dfl, the double-float form of the
// FP64 path); blocks, the kinetic diagonal and the epilogue's operands are stored in
// SphT<R> (double for dfl), the column buffer and the planes in cplx<R>.
template <typename R, int N3>
__global__ void __launch_bounds__(zinv_threads<R, N3>()) k_zinv_f(const cplx<typename SphT<R>::type>* __restrict__ Y, int64_t ldy,
                                                     cplx<R>* __restrict__ T, FastArgs fa) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fk::zinv_body<R, N3>(Y, ldy, T, fa, blockIdx.x * kCBF, blockIdx.y, smem_raw);
}

// Threads of an FP32 plane's block, measured over 64 to 768 per length: small planes run in
// small blocks, whose barriers more of their neighbours fill (32^3, 512 bands: 128 threads
// 0.070 ms, 256 0.076; 64^3: 0.425 and 0.438); above 96 only two planes fit an SM, and it
// takes 512 threads each to fill it (100^3, 256 bands: 1.02 and 1.13 ms).  At 48 to 96 other
// counts are slower (48^3: 128 0.205, 256 0.201, 384 0.246 ms; 96^3: 192-384 0.79-0.81, 256
// 0.783, 512 0.89).
template <typename R, int N> constexpr int plane_threads() {
  return sizeof(R) != 4 ? kThreads : N < 48 || N == 64 ? 128 : N > 96 ? 512 : 256;
}
template <typename R, int N>
__global__ void __launch_bounds__(plane_threads<R, N>()) k_plane_f(cplx<R>* __restrict__ T, const R* __restrict__ Vs, FastArgs fa) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fk::plane_body_pruned<R, N, plane_threads<R, N>()>(T, Vs, fa, blockIdx.x, blockIdx.y, smem_raw);
}

#ifndef CHEBFI_FFT_DF
template <typename R, int N>
__global__ void __launch_bounds__(kThreads) k_plane_real_f(const cplx<R>* __restrict__ T, cplx<R>* __restrict__ out,
                                                           FastArgs fa) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fk::plane_real_body<R, N, kThreads>(T, out + ((int64_t)blockIdx.y * N + blockIdx.x) * N * N, fa, blockIdx.x, blockIdx.y,
                                      smem_raw);
}
#endif

template <typename R, int N3>
__global__ void __launch_bounds__(zfwd_threads<R, N3>()) k_zfwd_f(const cplx<R>* __restrict__ T, FastArgs fa,
                                                     const typename SphT<R>::type* __restrict__ K,
                                                     LocalEpi<typename SphT<R>::type> ep) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fk::zfwd_body<R, N3>(T, fa, K, ep, blockIdx.x * kCBF, blockIdx.y, smem_raw);
}

template <typename R> void set_smem(const void* f, size_t bytes) {
  CHEBFI_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

template <typename R> const R* vtable(const chebfi_ctx* c);
template <> const float* vtable<float>(const chebfi_ctx* c) { return c->d_vsf.p; }
template <> const double* vtable<double>(const chebfi_ctx* c) { return c->d_vs.p; }

template <typename R, int N>
void fast_launch(chebfi_ctx* ctx, const cplx<typename SphT<R>::type>* Y, int64_t ldy, int64_t nb, cplx<R>* T,
                 LocalEpi<typename SphT<R>::type> ep, cudaStream_t st, const typename SphT<R>::type* K) {
  using S = typename SphT<R>::type;
  const SphereFFT& s = ctx->sph;
  const FastArgs fa = fk::fast_args(ctx);
  CHEBFI_REQUIRE(s.pitch == fk::plane_pitch(N), CHEBFI_ERR_STATE, "plane pitch of the compile-time path");
  const size_t zbytes = (size_t)(kCBF * s.zpitch) * sizeof(cplx<R>);
  const size_t pbytes = (size_t)(N * s.pitch) * sizeof(cplx<R>);
#ifndef CHEBFI_FFT_DF
  set_smem<R>((const void*)k_plane_f<R, N>, pbytes);
#endif
  set_smem<R>((const void*)k_zinv_f<R, N>, zbytes);
  set_smem<R>((const void*)k_zfwd_f<R, N>, zbytes);
  for (int64_t b0 = 0; b0 < nb; b0 += 65535) {
    const int nbc = (int)std::min<int64_t>(65535, nb - b0);
    dim3 gz((s.ncol + kCBF - 1) / kCBF, nbc);
    const double esz = sizeof(cplx<R>), col = (double)N * s.ncol * nbc * esz, sph = (double)ctx->npw * nbc * esz;
    CHEBFI_LAUNCH_W("k_zinv", st, sph + col, k_zinv_f<R, N><<<gz, zinv_threads<R, N>(), zbytes, st>>>(Y + b0 * ldy, ldy, T, fa));
    if (!fixed_planes(ctx, nbc, T, st)) {
#ifndef CHEBFI_FFT_DF
      CHEBFI_LAUNCH_W("k_plane", st, 2.0 * col, k_plane_f<R, N><<<dim3(N, nbc), plane_threads<R, N>(), pbytes, st>>>(T, vtable<R>(ctx), fa));
#else
      CHEBFI_REQUIRE(false, CHEBFI_ERR_STATE, "double-float columns without fixed-point planes");
#endif
    }
    LocalEpi<S> e = ep;
    e.Y = ep.Y + b0 * ep.ldy;
    if (e.Z) e.Z = ep.Z + b0 * ep.ldz;
    if (e.Zhi) {
      e.Zhi = ep.Zhi + b0 * ep.ldzb;
      e.Zlo = ep.Zlo + b0 * ep.ldzb;
    }
    if (e.T) e.T = ep.T + b0 * ep.ldt;
    if (e.Yprev) e.Yprev = ep.Yprev + b0 * ep.ldt;
    e.inv_n3 = (S)(1.0 / ((double)N * N * N));
    const double epi = sph * (1.0 + (e.Z ? 1.0 : 0.0) + (e.T ? 1.0 : 0.0) + (e.Yprev ? 1.0 : 0.0)) +
                       (e.Zhi ? (double)ctx->npw * nbc * (e.zplane ? 12.0 : 8.0) : 0.0);
    CHEBFI_LAUNCH_W("k_zfwd", st, col + epi, k_zfwd_f<R, N><<<gz, zfwd_threads<R, N>(), zbytes, st>>>(T, fa, K, e));
  }
}

#ifndef CHEBFI_FFT_DF
template <typename R, int N>
void real_launch(chebfi_ctx* ctx, const cplx<R>* Y, int64_t ldy, int64_t nb, cplx<R>* T, cplx<R>* out, bool planes,
                 cudaStream_t st) {
  const SphereFFT& s = ctx->sph;
  const FastArgs fa = fk::fast_args(ctx);
  CHEBFI_REQUIRE(nb <= 65535, CHEBFI_ERR_ARG, "too many bands in a chunk");
  const size_t zbytes = (size_t)(kCBF * s.zpitch) * sizeof(cplx<R>), pbytes = (size_t)(N * s.pitch) * sizeof(cplx<R>);
  set_smem<R>((const void*)k_zinv_f<R, N>, zbytes);
  const dim3 gz((s.ncol + kCBF - 1) / kCBF, (unsigned)nb);
  CHEBFI_LAUNCH("k_zinv", st, k_zinv_f<R, N><<<gz, zinv_threads<R, N>(), zbytes, st>>>(Y, ldy, T, fa));
  if (!planes) return;
  set_smem<R>((const void*)k_plane_real_f<R, N>, pbytes);
  CHEBFI_LAUNCH("k_plane_real", st, k_plane_real_f<R, N><<<dim3(N, (unsigned)nb), kThreads, pbytes, st>>>(T, out, fa));
}
#endif

}  // namespace

template <typename R> void fft_tables() {
  static fk::OncePerDevice once;
  once(fk::fill_twiddles);
}

// Compile-time-length path for cubic grids of the compiled sizes; false = not taken.
template <typename R>
bool fast_dispatch(chebfi_ctx* ctx, const cplx<typename SphT<R>::type>* Y, int64_t ldy, int64_t nb, cplx<R>* T,
                   LocalEpi<typename SphT<R>::type> ep, cudaStream_t st, const typename SphT<R>::type* K) {
  switch (ctx->grid[0]) {
#define CHEBFI_X(n) \
  case n: fast_launch<R, n>(ctx, Y, ldy, nb, T, ep, st, K); return true;
#ifdef CHEBFI_FFT_DF
    CHEBFI_FFT_DF_SIZES(CHEBFI_X)
#else
    CHEBFI_FFT_SIZES(CHEBFI_X)
#endif
#undef CHEBFI_X
    default: return false;
  }
}


#ifndef CHEBFI_FFT_DF
template <typename R>
bool fast_real_space(chebfi_ctx* ctx, const cplx<R>* Y, int64_t ldy, int64_t nb, cplx<R>* T, cplx<R>* out, bool planes,
                     cudaStream_t st) {
  switch (ctx->grid[0]) {
#define CHEBFI_X(n) \
  case n: real_launch<R, n>(ctx, Y, ldy, nb, T, out, planes, st); return true;
    CHEBFI_FFT_SIZES(CHEBFI_X)
#undef CHEBFI_X
    default: return false;
  }
}
#endif

}  // namespace chebfi
