// The complex GEMM tile of the CUDA cores, shared by the single (gemm.cu) and the batched
// k-point (batch.cu) kernels: a block of 256 threads accumulates a 16 TM x 16 TN tile of
// op(A) op(B) over [klo, khi), TM x TN outputs per thread.
//
// FP32 is bound by the FFMA issue: per k step a thread's TM TN complex products are 4 TM TN
// FFMAs, fed by (TM + TN) / 2 16-byte shared loads (pairs of neighbouring rows and columns).  The next BK-deep slices are fetched
// into registers while the current ones are multiplied (two shared buffers, one barrier a
// slice).
#pragma once

#include "internal.cuh"

namespace chebfi {
namespace gt {

constexpr int BK = 16;

// the rows of thread tx: groups of V = 16 / sizeof(complex) neighbours (one shared load), the
// groups 16 V apart so that the 16 threads' loads are contiguous (thread-contiguous rows, a
// 32-byte stride, doubled the shared wavefronts, which then bound the FP32 tile)
template <typename R> __device__ __forceinline__ int row_of(int tx, int a) {
  constexpr int V = 16 / (int)sizeof(cplx<R>);
  return (a / V) * (16 * V) + V * tx + a % V;
}

// row pitch of a slice: a multiple of 16 bytes
template <typename R, int T> constexpr int pitch() { return 16 * T + 16 / (int)sizeof(cplx<R>); }
template <typename R, int TM, int TN> constexpr size_t smem_bytes() {
  return (size_t)2 * BK * (pitch<R, TM>() + pitch<R, TN>()) * sizeof(cplx<R>);
}

// n neighbouring values at a 16-byte aligned address
template <typename C, int n> __device__ __forceinline__ void load_n(C* d, const C* s) {
  if constexpr (sizeof(C) == 8 && n % 2 == 0) {
#pragma unroll
    for (int i = 0; i < n; i += 2) {
      const float4 v = *reinterpret_cast<const float4*>(s + i);
      d[i].x = v.x;
      d[i].y = v.y;
      d[i + 1].x = v.z;
      d[i + 1].y = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < n; ++i) d[i] = s[i];
  }
}

// acc[a][b] = sum_k op(A)[i0 + row_of(tx, a), k] op(B)[k, j0 + TN ty + b], tx = tid % 16, ty = tid / 16;
// CA: op(A) = A^H, CB: op(B) = B^H.  Rows past M, columns past N and k past khi count as zeros.
// Every thread of the block must call; ends with a barrier.
template <typename R, int TM, int TN, bool CA, bool CB>
__device__ __forceinline__ void tile(const cplx<R>* __restrict__ A, int64_t lda, const cplx<R>* __restrict__ B, int64_t ldb,
                                     int64_t M, int64_t N, int64_t i0, int64_t j0, int64_t klo, int64_t khi,
                                     unsigned char* smem_raw, R (&accr)[TM][TN], R (&acci)[TM][TN]) {
  using C = cplx<R>;
  constexpr int V = 16 / (int)sizeof(C);  // TM is a multiple of V
  constexpr int BM = 16 * TM, BN = 16 * TN, PA = pitch<R, TM>(), PB = pitch<R, TN>();
  constexpr int LA = BM * BK / 256, LB = BN * BK / 256;
  static_assert(LA * 256 == BM * BK && LB * 256 == BN * BK, "tile slices must split evenly over 256 threads");
  C* As = reinterpret_cast<C*>(smem_raw);  // [2][BK][PA]
  C* Bs = As + 2 * BK * PA;                // [2][BK][PB]
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const C zero = cmake<C>(0.0, 0.0);
#pragma unroll
  for (int a = 0; a < TM; ++a)
#pragma unroll
    for (int b = 0; b < TN; ++b) accr[a][b] = acci[a][b] = (R)0;
  // entry l of this thread in a slice: row (column) r0 + l rs and k offset q0 + l qs; its address
  // is the thread's running pointer plus l times a uniform stride, its row check a bit of a mask
  const int ra0 = CA ? tid / BK : tid % BM, ras = CA ? 256 / BK : 0, qa0 = CA ? tid % BK : tid / BM, qas = CA ? 0 : 256 / BM;
  const int rb0 = CB ? tid % BN : tid / BK, rbs = CB ? 0 : 256 / BK, qb0 = CB ? tid / BN : tid % BK, qbs = CB ? 256 / BN : 0;
  static_assert(256 % BM == 0 || CA, "rows of a slice");
  const C* pa = A + (CA ? (klo + qa0) + (i0 + ra0) * lda : (i0 + ra0) + (klo + qa0) * lda);
  const C* pb = B + (CB ? (j0 + rb0) + (klo + qb0) * ldb : (klo + qb0) + (j0 + rb0) * ldb);
  const int64_t la = CA ? ras * lda : qas * lda, lb = CB ? qbs * ldb : rbs * ldb;
  const int64_t sa = CA ? BK : BK * lda, sb = CB ? BK * ldb : BK;
  unsigned ma = 0, mb = 0;
#pragma unroll
  for (int l = 0; l < LA; ++l) ma |= (i0 + ra0 + l * ras < M ? 1u : 0u) << l;
#pragma unroll
  for (int l = 0; l < LB; ++l) mb |= (j0 + rb0 + l * rbs < N ? 1u : 0u) << l;
  C ra[LA], rb[LB];
  auto fetch = [&](int64_t k0) {
    const int left = (int)min(khi - k0, (int64_t)BK);
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      ra[l] = zero;
      if ((ma >> l & 1u) && qa0 + l * qas < left) ra[l] = pa[l * la];
      if (CA) ra[l].y = -ra[l].y;
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      rb[l] = zero;
      if ((mb >> l & 1u) && qb0 + l * qbs < left) rb[l] = pb[l * lb];
      if (CB) rb[l].y = -rb[l].y;
    }
    pa += sa;
    pb += sb;
  };
  auto stash = [&](int buf) {
    C *as = As + buf * BK * PA, *bs = Bs + buf * BK * PB;
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int e = l * 256 + tid, i = CA ? e / BK : e % BM, k = CA ? e % BK : e / BM;
      as[k * PA + i] = ra[l];
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int e = l * 256 + tid, j = CB ? e % BN : e / BK, k = CB ? e / BN : e % BK;
      bs[k * PB + j] = rb[l];
    }
  };
  if (klo < khi) {
    fetch(klo);
    stash(0);
  }
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = klo; k0 < khi; k0 += BK) {
    const bool more = k0 + BK < khi;
    if (more) fetch(k0 + BK);  // in flight while the current slice is multiplied
    const C *as = As + buf * BK * PA, *bs = Bs + buf * BK * PB + TN * ty;
#pragma unroll 8
    for (int k = 0; k < BK; ++k) {
      C av[TM], bv[TN];
#pragma unroll
      for (int a = 0; a < TM; a += V) load_n<C, V>(av + a, as + k * PA + row_of<R>(tx, a));
      load_n<C, TN>(bv, bs + k * PB);
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TN; ++b) {
          accr[a][b] = fma(av[a].x, bv[b].x, accr[a][b]);
          acci[a][b] = fma(av[a].x, bv[b].y, acci[a][b]);
          accr[a][b] = fma(-av[a].y, bv[b].y, accr[a][b]);
          acci[a][b] = fma(av[a].y, bv[b].x, acci[a][b]);
        }
    }
    if (more) stash(buf ^ 1);  // that buffer was last read before the previous barrier
    __syncthreads();
    buf ^= 1;
  }
}

}  // namespace gt
}  // namespace chebfi
