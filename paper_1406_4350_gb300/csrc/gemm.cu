// Complex GEMM on the CUDA cores (FP64 DFMA or FP32 FFMA), C = alpha op(A) op(B) + beta C.
//
// Used for the FP64 and FP32 forms of the projector products P^H psi and P W
// (Algorithm 1, Section 5.1), the Woodbury core products, and the subspace matrices and
// rotations of Algorithm 2.  FP32: 64 x 64 output tiles, 256 threads, 4 x 4 complex outputs
// per thread (gemm_tile.cuh).  FP64: 256 outputs per tile, one per thread (k_gemm_d).  Both split K, with a
// deterministic second pass, when the output has too few tiles to fill the SMs.
#include <algorithm>

#include "gemm_tile.cuh"
#include "internal.cuh"
#include "kernels.cuh"

namespace chebfi {
namespace {

template <typename C> __device__ __forceinline__ C ld_op(const C* p, bool conj_) {
  C v = *p;
  if (conj_) v.y = -v.y;
  return v;
}

// FP32: one tile of gemm_tile.cuh per block, blockIdx.z the K range.  Shapes with few tiles
// split K down to 64 products so that every SM gets blocks.  256 x 256 x 8217: 238 us with an
// unbuffered loop and ranges of 1024, now 106 us; 256^3: 52 us on 16 SMs, now 10 us.
template <int TM, int TN, bool CA, bool CB>
__global__ void __launch_bounds__(256, TN == 4 ? 3 : 4)
    k_gemm_f(int64_t M, int64_t N, int64_t K, float alpha, const float2* __restrict__ A, int64_t lda,
             const float2* __restrict__ B, int64_t ldb, float beta, float2* __restrict__ Cm, int64_t ldc, int64_t kchunk,
             float2* __restrict__ ws, int lower, int tiles_m, int tiles_n, int n_fastest) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int BM = 16 * TM, BN = 16 * TN;
  // n_fastest: consecutive blocks walk the column tiles, so blocks launched together share a
  // row tile of A (the large operand when M >> N) in L2
  const int64_t tile_i = n_fastest ? blockIdx.x / tiles_n : blockIdx.x % tiles_m;
  const int64_t tile_j = n_fastest ? blockIdx.x % tiles_n : blockIdx.x / tiles_m;
  const int64_t i0 = tile_i * BM, j0 = tile_j * BN, kbeg = (int64_t)blockIdx.z * kchunk;
  if (lower && i0 + BM - 1 < j0) return;  // tile strictly above the diagonal
  float accr[TM][TN], acci[TM][TN];
  gt::tile<float, TM, TN, CA, CB>(A, lda, B, ldb, M, N, i0, j0, kbeg, min(K, kbeg + kchunk), smem_raw, accr, acci);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll
  for (int b = 0; b < TN; ++b) {
    const int64_t gj = j0 + TN * ty + b;
    if (gj >= N) continue;
#pragma unroll
    for (int a = 0; a < TM; ++a) {
      const int64_t gi = i0 + gt::row_of<float>(tx, a);
      if (gi >= M || (lower && gi < gj)) continue;
      float2 r = make_float2(alpha * accr[a][b], alpha * acci[a][b]);
      if (ws) {
        ws[(int64_t)blockIdx.z * M * N + gi + gj * M] = r;
      } else {
        if (beta != 0.f) {
          const float2 c = Cm[gi + gj * ldc];
          r.x = fma(beta, c.x, r.x);
          r.y = fma(beta, c.y, r.y);
        }
        Cm[gi + gj * ldc] = r;
      }
    }
  }
}

// FP64: one output per thread, TM x TN = 256 outputs per block.  GB300 issues about two FP64
// FMAs per clock and SM, so a block's 16-step k tile keeps the unit busy for 8192 clocks on
// 8 KB of operands: reuse in registers gains nothing, and what counts is that no work is
// spent on padding and that every SM has blocks.  Small tiles (8 x 32, 16 x 16 or 32 x 8,
// whichever pads the output least) and a split of K down to 16 products do that; 64 x 64
// tiles spent 16 times the needed FMAs on an 8 x 32 product and ran it on one SM
// (8 x 32 x 1021: 4.13 ms, now 0.010 ms and 0.008 ms for its reduction; 256 x 256 x 256:
// 1.04 ms on 16 SMs, now 0.14 ms).
constexpr int KD = 16;
template <int TM, int TN, bool CA, bool CB>
__global__ void __launch_bounds__(256) k_gemm_d(int64_t M, int64_t N, int64_t K, double alpha,
                                                const double2* __restrict__ A, int64_t lda,
                                                const double2* __restrict__ B, int64_t ldb, double beta,
                                                double2* __restrict__ Cm, int64_t ldc, int64_t kchunk,
                                                double2* __restrict__ ws, int lower, int tiles_m, int tiles_n,
                                                int n_fastest) {
  static_assert(TM * TN == 256, "one output per thread");
  const int64_t tile_i = n_fastest ? blockIdx.x / tiles_n : blockIdx.x % tiles_m;
  const int64_t tile_j = n_fastest ? blockIdx.x % tiles_n : blockIdx.x / tiles_m;
  const int64_t i0 = tile_i * TM, j0 = tile_j * TN;
  if (lower && i0 + TM - 1 < j0) return;  // tile strictly above the diagonal
  __shared__ double2 As[KD][TM + 1];
  __shared__ double2 Bs[KD][TN + 1];
  const int tid = threadIdx.x, tx = tid % TM, ty = tid / TM;
  const int64_t kbeg = (int64_t)blockIdx.z * kchunk, kend = min(K, kbeg + kchunk);
  const double2 zero = make_double2(0.0, 0.0);
  double re = 0.0, im = 0.0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += KD) {
#pragma unroll
    for (int e = tid; e < TM * KD; e += 256) {
      const int i = CA ? e / KD : e % TM, k = CA ? e % KD : e / TM;
      const int64_t gi = i0 + i, gk = k0 + k;
      double2 v = zero;
      if (gi < M && gk < kend) v = CA ? ld_op(A + gk + gi * lda, true) : A[gi + gk * lda];
      As[k][i] = v;
    }
#pragma unroll
    for (int e = tid; e < TN * KD; e += 256) {
      const int j = CB ? e % TN : e / KD, k = CB ? e / TN : e % KD;
      const int64_t gj = j0 + j, gk = k0 + k;
      double2 v = zero;
      if (gj < N && gk < kend) v = CB ? ld_op(B + gj + gk * ldb, true) : B[gk + gj * ldb];
      Bs[k][j] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < KD; ++k) {
      const double2 a = As[k][tx], b = Bs[k][ty];
      re = fma(a.x, b.x, re);
      im = fma(a.x, b.y, im);
      re = fma(-a.y, b.y, re);
      im = fma(a.y, b.x, im);
    }
    __syncthreads();
  }
  const int64_t gi = i0 + tx, gj = j0 + ty;
  if (gi >= M || gj >= N || (lower && gi < gj)) return;
  double2 r = make_double2(alpha * re, alpha * im);
  if (ws) {
    ws[(int64_t)blockIdx.z * M * N + gi + gj * M] = r;
    return;
  }
  if (beta != 0.0) {
    const double2 c = Cm[gi + gj * ldc];
    r.x = fma(beta, c.x, r.x);
    r.y = fma(beta, c.y, r.y);
  }
  Cm[gi + gj * ldc] = r;
}

// C = sum_z ws[z] + beta C (lower: of the entries on and below the diagonal, the only ones that
// the products left in ws).  32 outputs per block; eight threads per output each add every
// eighth split, their partial sums are added in a fixed order: one thread per output is a
// chain of up to 64 dependent loads and slow FP64 additions (16 us at 64 splits of 8 x 32, now 8 us).
template <typename R>
__global__ void __launch_bounds__(256) k_splitk_reduce(int64_t M, int64_t N, int splits, const cplx<R>* __restrict__ ws,
                                                       R beta, cplx<R>* __restrict__ Cm, int64_t ldc, int lower) {
  __shared__ cplx<R> part[8][33];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const int64_t idx = (int64_t)blockIdx.x * 32 + tx;
  const bool in = idx < M * N && !(lower && idx % M < idx / M);
  cplx<R> r = cmake<cplx<R>>(0.0, 0.0);
  if (in) {
#pragma unroll 4
    for (int z = ty; z < splits; z += 8) {
      const cplx<R> v = ws[(int64_t)z * M * N + idx];
      r.x += v.x;
      r.y += v.y;
    }
  }
  part[ty][tx] = r;
  __syncthreads();
  if (ty != 0 || !in) return;
#pragma unroll
  for (int z = 1; z < 8; ++z) {
    r.x += part[z][tx].x;
    r.y += part[z][tx].y;
  }
  const int64_t i = idx % M, j = idx / M;
  if (beta != (R)0) {
    const cplx<R> c = Cm[i + j * ldc];
    r.x = fma(beta, c.x, r.x);
    r.y = fma(beta, c.y, r.y);
  }
  Cm[i + j * ldc] = r;
}

int sm_count() {
  int dev = 0, sms = 0;
  CHEBFI_CUDA(cudaGetDevice(&dev));
  CHEBFI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  return sms;
}

template <bool CA, bool CB>
void launch_f(int64_t M, int64_t N, int64_t K, double alpha, const float2* A, int64_t lda, const float2* B, int64_t ldb,
              double beta, float2* Cm, int64_t ldc, cudaStream_t st, DevBuf<float2>* ws, const char* tag, bool lower) {
  // 64 x 64 tiles (three blocks per SM) or 64 x 32 ones (four, about 10 % slower per output):
  // whichever leaves the shorter schedule; a shape with less than a round of tiles splits K
  // into ranges of at least 64 until it fills one.  8217 x 256 x 256: 516 and 1032 tiles, 125
  // us (a second round of 60 tiles) and 107 us.
  const int64_t tm = (M + 63) / 64;
  auto plan = [&](int64_t tn, int64_t per_round, int64_t& splits, int64_t& kchunk) {
    const int64_t tiles = tm * tn;
    splits = 1;
    if (ws && tiles < per_round) splits = std::max<int64_t>(1, std::min<int64_t>({per_round / tiles, K / 64, 64}));
    kchunk = std::max<int64_t>(gt::BK, ((K + splits - 1) / splits + gt::BK - 1) / gt::BK * gt::BK);
    splits = std::max<int64_t>(1, (K + kchunk - 1) / kchunk);
    return (double)((tiles * splits + per_round - 1) / per_round) * (double)kchunk;
  };
  const int64_t sms = sm_count();
  int64_t s4, c4, s2, c2;
  const double cost4 = 3.0 * plan((N + 63) / 64, 3 * sms, s4, c4), cost2 = 4.0 * 0.5 * 1.1 * plan((N + 31) / 32, 4 * sms, s2, c2);
  const bool narrow = cost2 < cost4;
  const int64_t tn = narrow ? (N + 31) / 32 : (N + 63) / 64, tiles = tm * tn, splits = narrow ? s2 : s4, kchunk = narrow ? c2 : c4;
  float2* wsp = nullptr;
  if (splits > 1) {
    ws->alloc((size_t)(splits * M * N));
    wsp = ws->p;
  }
  CHEBFI_REQUIRE(tiles < (1ll << 31), CHEBFI_ERR_ARG, "GEMM too large");
  static_assert(gt::smem_bytes<float, 4, 4>() <= 48 * 1024, "within the default shared memory limit");
  const double tiles_done = lower ? 0.5 * (1.0 + 1.0 / (double)tm) : 1.0;
  auto go = [&](auto kernel, size_t smem) {
    CHEBFI_LAUNCH_W(tag, st, 8.0 * (double)M * (double)N * (double)K * tiles_done,
                    kernel<<<dim3((unsigned)tiles, 1, (unsigned)splits), 256, smem, st>>>(
                        M, N, K, (float)alpha, A, lda, B, ldb, (float)beta, Cm, ldc, kchunk, wsp, lower ? 1 : 0, (int)tm,
                        (int)tn, tm > 4 * tn ? 1 : 0));
  };
  if (narrow) go(k_gemm_f<4, 2, CA, CB>, gt::smem_bytes<float, 4, 2>());
  else go(k_gemm_f<4, 4, CA, CB>, gt::smem_bytes<float, 4, 4>());
  if (splits > 1) {
    const int64_t tot = M * N;
    CHEBFI_LAUNCH("k_splitk_reduce", st,
                  k_splitk_reduce<float><<<(unsigned)((tot + 31) / 32), 256, 0, st>>>(M, N, (int)splits, wsp, (float)beta, Cm, ldc, lower ? 1 : 0));
  }
}

// the FP64 tile shape with the least padded output: 16 x 16, 8 x 32 (few rows), 32 x 8
template <bool CA, bool CB>
void launch_d(int64_t M, int64_t N, int64_t K, double alpha, const double2* A, int64_t lda, const double2* B,
              int64_t ldb, double beta, double2* Cm, int64_t ldc, cudaStream_t st, DevBuf<double2>* ws,
              const char* tag, bool lower) {
  auto padded = [&](int64_t tm, int64_t tn) { return (M + tm - 1) / tm * ((N + tn - 1) / tn); };
  int64_t TM = 16, TN = 16;
  if (padded(8, 32) < padded(TM, TN)) { TM = 8; TN = 32; }
  if (padded(32, 8) < padded(TM, TN)) { TM = 32; TN = 8; }
  const int64_t tm = (M + TM - 1) / TM, tn = (N + TN - 1) / TN, tiles = tm * tn;
  // two blocks per SM; a split is at least one k tile
  const int64_t blocks = 2 * sm_count();
  int64_t splits = 1;
  if (ws && tiles < blocks) splits = std::max<int64_t>(1, std::min<int64_t>((blocks + tiles - 1) / tiles, (K + KD - 1) / KD));
  int64_t kchunk = std::max<int64_t>(KD, ((K + splits - 1) / splits + KD - 1) / KD * KD);
  splits = std::max<int64_t>(1, (K + kchunk - 1) / kchunk);
  double2* wsp = nullptr;
  if (splits > 1) {
    ws->alloc((size_t)(splits * M * N));
    wsp = ws->p;
  }
  const bool n_fastest = tm > 4 * tn;
  CHEBFI_REQUIRE(tiles < (1ll << 31), CHEBFI_ERR_ARG, "GEMM too large");
  const dim3 grid((unsigned)tiles, 1, (unsigned)splits);
  const double tiles_done = lower ? 0.5 * (1.0 + 1.0 / (double)tm) : 1.0;
  auto go = [&](auto kernel) {
    CHEBFI_LAUNCH_W(tag, st, 8.0 * (double)M * (double)N * (double)K * tiles_done,
                    kernel<<<grid, 256, 0, st>>>(M, N, K, alpha, A, lda, B, ldb, beta, Cm, ldc, kchunk, wsp,
                                                 lower ? 1 : 0, (int)tm, (int)tn, n_fastest ? 1 : 0));
  };
  if (TM == 8) go(k_gemm_d<8, 32, CA, CB>);
  else if (TM == 32) go(k_gemm_d<32, 8, CA, CB>);
  else go(k_gemm_d<16, 16, CA, CB>);
  if (splits > 1) {
    const int64_t tot = M * N;
    CHEBFI_LAUNCH("k_splitk_reduce", st,
                  k_splitk_reduce<double><<<(unsigned)((tot + 31) / 32), 256, 0, st>>>(M, N, (int)splits, wsp, beta, Cm, ldc, lower ? 1 : 0));
  }
}

template <typename R, bool CA, bool CB, typename... Args> void route(Args... args) {
  if constexpr (sizeof(R) == 8) launch_d<CA, CB>(args...);
  else launch_f<CA, CB>(args...);
}

}  // namespace

template <typename R>
void gemm(bool conjA, bool conjB, int64_t M, int64_t N, int64_t K, double alpha, const cplx<R>* A, int64_t lda,
          const cplx<R>* B, int64_t ldb, double beta, cplx<R>* C, int64_t ldc, cudaStream_t st,
          DevBuf<cplx<R>>* ws, const char* tag, bool lower) {
  if (M <= 0 || N <= 0) return;
  CHEBFI_REQUIRE(!lower || M == N, CHEBFI_ERR_ARG, "lower-triangle GEMM needs a square result");
  if (conjA && conjB) route<R, true, true>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, st, ws, tag, lower);
  else if (conjA) route<R, true, false>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, st, ws, tag, lower);
  else if (conjB) route<R, false, true>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, st, ws, tag, lower);
  else route<R, false, false>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, st, ws, tag, lower);
}

template void gemm<double>(bool, bool, int64_t, int64_t, int64_t, double, const double2*, int64_t, const double2*,
                           int64_t, double, double2*, int64_t, cudaStream_t, DevBuf<double2>*, const char*, bool);
template void gemm<float>(bool, bool, int64_t, int64_t, int64_t, double, const float2*, int64_t, const float2*,
                          int64_t, double, float2*, int64_t, cudaStream_t, DevBuf<float2>*, const char*, bool);

}  // namespace chebfi
