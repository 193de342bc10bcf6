// Launches of the fixed-point plane passes of the FP64 path (fft_fixed.cuh).
#include "fft_fixed.cuh"
#include "fft_launch.cuh"

namespace chebfi {
namespace {

// A plane takes 16 bytes a point: from N = 90 it fills an SM, whose one block then takes 24
// warps; smaller planes run in smaller blocks so that several share an SM and fill each
// other's barriers.
template <int N> constexpr int fx_threads() { return N >= 90 ? 768 : N >= 48 ? 256 : 128; }

template <int N, typename C>
__global__ void __launch_bounds__(fx_threads<N>()) k_plane_fx(C* __restrict__ T, const int2* __restrict__ Vs,
                                                              const int* __restrict__ ve, fk::FastArgs fa) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx::plane_body<N, fx_threads<N>()>(T, Vs, ve[blockIdx.x], fa, blockIdx.x, blockIdx.y, smem_raw);
}

template <int N>
__global__ void __launch_bounds__(fx_threads<N>()) k_plane_real_fx(const double2* __restrict__ T, double2* __restrict__ out,
                                                                   fk::FastArgs fa) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx::plane_real_body<N, fx_threads<N>()>(T, out + ((int64_t)blockIdx.y * N + blockIdx.x) * N * N, fa, blockIdx.x, blockIdx.y,
                                          smem_raw);
}

template <int N> size_t prepare(const chebfi_ctx* ctx, const void* kernel) {
  CHEBFI_REQUIRE(ctx->sph.pitch == fk::plane_pitch(N), CHEBFI_ERR_STATE, "plane pitch of the compile-time path");
  const size_t bytes = (size_t)(N * fk::plane_pitch(N)) * sizeof(fx::cfx);
  CHEBFI_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return bytes;
}

template <int N, typename C> void launch(chebfi_ctx* ctx, int64_t nb, C* T, cudaStream_t st) {
  const size_t bytes = prepare<N>(ctx, (const void*)k_plane_fx<N, C>);
  const double col = (double)N * ctx->sph.ncol * (double)nb * sizeof(C);
  CHEBFI_LAUNCH_W("k_plane", st, 2.0 * col,
                  k_plane_fx<N, C><<<dim3(N, (unsigned)nb), fx_threads<N>(), bytes, st>>>(T, ctx->d_vsfx.p, ctx->d_vexp.p,
                                                                                      fk::fast_args(ctx)));
}
template <int N> void launch_real(chebfi_ctx* ctx, int64_t nb, const double2* T, double2* out, cudaStream_t st) {
  const size_t bytes = prepare<N>(ctx, (const void*)k_plane_real_fx<N>);
  CHEBFI_LAUNCH("k_plane_real", st,
                k_plane_real_fx<N><<<dim3(N, (unsigned)nb), fx_threads<N>(), bytes, st>>>(T, out, fk::fast_args(ctx)));
}

}  // namespace

void fixed_tables() {
  static fk::OncePerDevice once;
  once(fx::fill_twiddles);
}

bool fixed_planes(chebfi_ctx* ctx, int64_t nb, cdf* T, cudaStream_t st) {
  switch (ctx->grid[0]) {
#define CHEBFI_X(n) \
  case n: launch<n>(ctx, nb, T, st); return true;
    CHEBFI_FFT_DF_SIZES(CHEBFI_X)
#undef CHEBFI_X
    default: return false;
  }
}

bool fixed_planes(chebfi_ctx* ctx, int64_t nb, double2* T, cudaStream_t st) {
  if (ctx->fft64 != CHEBFI_FFT64_DOUBLE_FLOAT) return false;
  switch (ctx->grid[0]) {
#define CHEBFI_X(n) \
  case n: launch<n>(ctx, nb, T, st); return true;
    CHEBFI_FFT_FX_SIZES(CHEBFI_X)
#undef CHEBFI_X
    default: return false;
  }
}

bool fixed_planes_real(chebfi_ctx* ctx, int64_t nb, const double2* T, double2* out, cudaStream_t st) {
  switch (ctx->grid[0]) {
#define CHEBFI_X(n) \
  case n: launch_real<n>(ctx, nb, T, out, st); return true;
    CHEBFI_FFT_DF_SIZES(CHEBFI_X)
    CHEBFI_FFT_FX_SIZES(CHEBFI_X)
#undef CHEBFI_X
    default: return false;
  }
}

}  // namespace chebfi
