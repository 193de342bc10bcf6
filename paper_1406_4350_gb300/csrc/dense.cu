// Dense FP64 linear algebra on the device for the Rayleigh-Ritz step of Algorithm 2 and
// the Woodbury core of Section 5.1: blocked Cholesky, triangular solve, and a cyclic
// Jacobi eigensolver for complex Hermitian matrices.
//
// Jacobi: each rotation removes one off-diagonal entry a_pq = |a_pq| e^{i phi} of the
// 2 x 2 block [[a_pp, a_pq], [conj(a_pq), a_qq]]: U = diag(1, e^{-i phi}) [[c, s], [-s, c]]
// with zeta = (a_qq - a_pp) / (2 |a_pq|), t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)),
// c = 1/sqrt(1 + t^2), s = t c (the symmetric Schur step of Golub & Van Loan, Section 8.5),
// applied as A <- U^H A U, V <- V U.  One step applies n/2 disjoint rotations chosen by the
// circle method (player 0 fixed, the others rotate), one sweep is n-1 steps.
#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.cuh"
#include "kernels.cuh"
#include "grid_barrier.cuh"

namespace chebfi {
namespace {

constexpr int NB = 32;

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

__device__ __forceinline__ void flag_error(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// Unblocked Cholesky of one nb x nb diagonal block (nb <= NB) in shared memory.  One block:
// the pivots are a serial chain, and GB300's FP64 unit (about two FMAs per clock) makes each
// square root and division ~10 dependent slow instructions.  Only 1 / sqrt(d) is on the
// chain, with one Newton step for the root itself; one warp forms the next column's while the
// others update the trailing triangle.  32 x 32: 66 us with sqrt and a division per entry on the
// chain, now 36.
// Each operation rounds once, as those did: an entry times the reciprocal is corrected by its
// residual to a / s, and a product of two complex entries is formed before it is subtracted.
// Without these (the reciprocal alone, two multiply-adds into the entry: 31 us) the rms of
// |A - L L^H| is 0.86-0.89 units of 2^-53 |L| |L|^H where it is 0.64.
__global__ void __launch_bounds__(256) k_chol_diag(double2* A, int64_t lda, int nb, int* status) {
  __shared__ double2 a[NB][NB + 1];
  __shared__ double2 piv;  // (sqrt(d), 1 / sqrt(d))
  const int tid = threadIdx.x;
  for (int e = tid; e < nb * nb; e += blockDim.x) {
    const int i = e % nb, j = e / nb;
    a[i][j] = A[i + j * lda];
  }
  __syncthreads();
  auto pivot = [&](int j) {  // by one thread; a pivot that is not positive (or NaN) counts as 1
    const double d = a[j][j].x;
    if (!(d > 0.0)) {
      flag_error(status, CHEBFI_ERR_NOT_SPD);
      a[j][j].x = 1.0;
    }
    // the root of the pivot, rounded to nearest but for rare ties: one Newton step on d rsqrt(d)
    const double p = a[j][j].x, r = rsqrt(p), s = p * r;
    piv = make_double2(fma(0.5 * r, fma(-s, s, p), s), r);
  };
  if (tid == 0) pivot(0);
  __syncthreads();
  for (int j = 0; j < nb; ++j) {
    const int i = j + 1 + tid % 32;
    if (tid < 64 && i < nb) {  // one warp a part: a / s rounded once
      double* v = &a[i][j].x + tid / 32;
      const double q = *v * piv.y;
      *v = fma(fma(-q, piv.x, *v), piv.y, q);
    }
    if (tid == 64) a[j][j] = make_double2(piv.x, 0.0);
    __syncthreads();
    // trailing update of the lower triangle: a[i][k] -= L[i][j] conj(L[k][j]) for i >= k > j.
    // Its m columns are folded in pairs (q, m - 1 - q) of m + 1 entries together, so that no
    // lane of the slow FP64 instructions is spent above the diagonal.
    const int m = nb - j - 1;
    auto update = [&](int i, int k) {
      const double2 li = a[i][j], lk = a[k][j];
      double2 v = a[i][k];
      v.x -= fma(li.y, lk.y, li.x * lk.x);
      v.y -= fma(li.y, lk.x, -(li.x * lk.y));
      a[i][k] = v;
    };
    if (tid < 32) {
      if (tid == 0 && m > 0) {
        const double2 l = a[j + 1][j];  // the diagonal is real
        a[j + 1][j + 1].x -= fma(l.y, l.y, l.x * l.x);
        pivot(j + 1);
      }
    } else {
      for (int e = tid - 32; e < (m + 1) * ((m + 1) / 2); e += blockDim.x - 32) {
        const int q = e / (m + 1), c = e - q * (m + 1);
        const bool first = c < m - q;
        if (!first && m - 1 - q == q) continue;  // the middle column of an odd m has no partner
        const int k = j + 1 + (first ? q : m - 1 - q), i = first ? k + c : k + c - (m - q);
        if (i != j + 1) update(i, k);  // (j + 1, j + 1) is the next pivot
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < nb * nb; e += blockDim.x) {
    const int i = e % nb, j = e / nb;
    A[i + j * lda] = i >= j ? a[i][j] : make_double2(0.0, 0.0);
  }
}

// The two triangular solves with an nb x nb lower L (diagonal real), one system per warp: the
// lanes hold its unknowns, and step k broadcasts x_k = s_k / L_kk to the lanes that still
// need it.  A system is a serial chain of nb slow FP64 steps, so systems are spread over the
// SMs (four warps a block) instead of one per thread, which kept 128 of them on one SM
// (224 x 32: 131 and 172 us with a thread per system, now 18 us).  The reciprocal is a pair of
// twice the precision and a complex product is formed before it is subtracted, so that each
// operation rounds once, as with a division (rms residual 0.50 units of 2^-53 |L| |x|; with the
// reciprocal alone and two multiply-adds 0.66, and 4 us less).
constexpr int kTrsmWarps = 4;
// x_l <- x_l - sum_{k < l} c_lk x_k solved forward; c_lk = L[l][k], or its conjugate
template <bool CONJ>
__device__ __forceinline__ double2 warp_forward(const double2 (*l)[NB + 1], const double2* rd, double2 x, int nb) {
  const int lane = threadIdx.x % 32;
  for (int k = 0; k < nb; ++k) {
    const double2 r = rd[k];
    const double sx = __shfl_sync(0xffffffffu, x.x, k), sy = __shfl_sync(0xffffffffu, x.y, k);
    const double2 xk = make_double2(fma(sx, r.x, sx * r.y), fma(sy, r.x, sy * r.y));
    double2 c = l[lane][k];  // L is lower triangular: zero above, and rows >= nb are zero
    if (CONJ) c.y = -c.y;
    if (lane == k) x = xk;
    else if (lane > k) {
      x.x -= fma(c.x, xk.x, -(c.y * xk.y));
      x.y -= fma(c.x, xk.y, c.y * xk.x);
    }
  }
  return x;
}
__device__ __forceinline__ void load_tri(const double2* __restrict__ L, int64_t ldl, int nb, double2 (*l)[NB + 1],
                                         double2* rd) {
  // one warp's lanes take the reciprocals side by side: a division in every warp's pass over its
  // column of the square, for the one lane on the diagonal, took 4 of 22 us
  if (threadIdx.x < NB) {
    const int i = threadIdx.x;
    const double d = i < nb ? L[i + i * ldl].x : 1.0, r = 1.0 / d;
    rd[i] = make_double2(r, r * fma(-r, d, 1.0));
  }
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
    const int i = e % NB, j = e / NB;
    l[i][j] = i < nb && j < nb ? L[i + j * ldl] : make_double2(0.0, 0.0);
  }
  __syncthreads();
}

// Panel: rows of B (m x nb) <- B L^{-H}; row r of X solves conj(L) x = b.
__global__ void __launch_bounds__(32 * kTrsmWarps) k_trsm_right_lh(const double2* __restrict__ L, int64_t ldl, double2* B, int64_t ldb, int64_t m,
                                                                  int nb) {
  __shared__ double2 l[NB][NB + 1];
  __shared__ double2 rd[NB];
  load_tri(L, ldl, nb, l, rd);
  const int lane = threadIdx.x % 32;
  const int64_t r = (int64_t)blockIdx.x * kTrsmWarps + threadIdx.x / 32;
  if (r >= m) return;
  double2 x = lane < nb ? B[r + lane * ldb] : make_double2(0.0, 0.0);
  x = warp_forward<true>(l, rd, x, nb);
  if (lane < nb) B[r + lane * ldb] = x;
}

// Columns of B (nb x m) <- L^{-1} B.
__global__ void __launch_bounds__(32 * kTrsmWarps) k_trsm_left_l(const double2* __restrict__ L, int64_t ldl, double2* B, int64_t ldb, int64_t m,
                                                                int nb) {
  __shared__ double2 l[NB][NB + 1];
  __shared__ double2 rd[NB];
  load_tri(L, ldl, nb, l, rd);
  const int lane = threadIdx.x % 32;
  const int64_t c = (int64_t)blockIdx.x * kTrsmWarps + threadIdx.x / 32;
  if (c >= m) return;
  double2 x = lane < nb ? B[lane + c * ldb] : make_double2(0.0, 0.0);
  x = warp_forward<false>(l, rd, x, nb);
  if (lane < nb) B[lane + c * ldb] = x;
}

__global__ void k_zero_upper(int64_t n, double2* A, int64_t lda) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * n) return;
  const int64_t i = idx % n, j = idx / n;
  if (i < j) A[i + j * lda] = make_double2(0.0, 0.0);
}

// ------------------------------------------------------------------ Jacobi
// In FP64; the refined eigensolver's first stage has its own FP32 form (blocked Jacobi, below).
constexpr double kEpsD = 1.1102230246251565e-16, kTinyD = 1e-300;
constexpr float kEpsF = 5.9604645e-8f;

__device__ __forceinline__ int64_t rr_player(int64_t pos, int64_t round, int64_t n) {
  return pos == 0 ? 0 : 1 + (pos - 1 + round) % (n - 1);
}

struct Rot {
  double c, s;
  double2 ph;  // e^{i phi}
};

// rotation parameters of pair t of the given round (p < q; q = -1 for the padding player)
__device__ __forceinline__ void jac_params_item(int64_t t, int64_t n0, int64_t n, int64_t round,
                                                const double2* __restrict__ A, int64_t lda, Rot* __restrict__ rot,
                                                int* __restrict__ pairs) {
  int64_t p = rr_player(t, round, n), q = rr_player(n - 1 - t, round, n);
  if (p > q) {
    const int64_t tmp = p;
    p = q;
    q = tmp;
  }
  Rot r;
  r.c = 1.0;
  r.s = 0.0;
  r.ph = make_double2(1.0, 0.0);
  if (q < n0) {
    const double2 h = A[p + q * lda];
    const double g = hypot(h.x, h.y);
    const double app = A[p + p * lda].x, aqq = A[q + q * lda].x;
    if (g > kTinyD && g > kEpsD * sqrt(fabs(app * aqq))) {
      const double zeta = (aqq - app) / (2.0 * g);
      const double t_ = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + hypot(1.0, zeta));
      r.c = 1.0 / sqrt(1.0 + t_ * t_);
      r.s = t_ * r.c;
      r.ph = make_double2(h.x / g, h.y / g);
    }
  } else {
    q = -1;
  }
  rot[t] = r;
  pairs[2 * t] = (int)p;
  pairs[2 * t + 1] = (int)q;
}

__global__ void k_jac_params(int64_t n0, int64_t n, int64_t round, const double2* __restrict__ A, int64_t lda,
                             Rot* __restrict__ rot, int* __restrict__ pairs) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n / 2) jac_params_item(t, n0, n, round, A, lda, rot, pairs);
}

// [a, b] <- [c a - s e^{i phi} b, s a + c e^{i phi} b] (rows, U^H from the left) and
// [a, b] <- [c a - s e^{-i phi} b, s a + c e^{-i phi} b] (columns, U from the right)
__device__ __forceinline__ void rot2(double2& a, double2& b, double c, double s, double2 ph) {
  double2 na, nb;
  na.x = c * a.x - s * (ph.x * b.x - ph.y * b.y);
  na.y = c * a.y - s * (ph.x * b.y + ph.y * b.x);
  nb.x = s * a.x + c * (ph.x * b.x - ph.y * b.y);
  nb.y = s * a.y + c * (ph.x * b.y + ph.y * b.x);
  a = na;
  b = nb;
}

// items of one round: h x h blocks of A, n rows x h column pairs of V
__host__ __device__ inline int64_t jac_items(int64_t h, int64_t n) { return h * h + n * h; }

// One round of rotations in one pass: item (t1, t2) maps the 2 x 2 block of A on rows
// {p1, q1} and columns {p2, q2} to U1^H A U2 (the pairs are disjoint, so every element of A
// belongs to exactly one block); the remaining items apply V <- V U2 on columns {p2, q2}.
__device__ __forceinline__ void jac_apply_item(int64_t idx, int64_t h, int64_t n, double2* A, int64_t lda,
                                               double2* V, int64_t ldv, const Rot* __restrict__ rot,
                                               const int* __restrict__ pairs) {
  const int64_t nblk_a = h * h;
  if (idx < nblk_a) {
    const int64_t t1 = idx % h, t2 = idx / h;
    const int q1 = pairs[2 * t1 + 1], q2 = pairs[2 * t2 + 1];
    const int p1 = pairs[2 * t1], p2 = pairs[2 * t2];
    const Rot r1 = rot[t1], r2 = rot[t2];
    const bool act1 = q1 >= 0 && r1.s != 0.0, act2 = q2 >= 0 && r2.s != 0.0;
    if (!act1 && !act2) return;
    const double2 cph2 = conjg(r2.ph);
    // the padding player (q < 0) owns no row or column of A: 1 x 2 or 2 x 1 blocks
    if (q1 < 0 || q2 < 0) {
      if (q1 < 0 && q2 < 0) return;
      if (q1 < 0) {  // row p1 alone, columns {p2, q2} rotate by U2
        double2 a = A[p1 + (int64_t)p2 * lda], b = A[p1 + (int64_t)q2 * lda];
        rot2(a, b, r2.c, r2.s, cph2);
        A[p1 + (int64_t)p2 * lda] = a;
        A[p1 + (int64_t)q2 * lda] = b;
      } else {  // column p2 alone, rows {p1, q1} rotate by U1^H
        double2 a = A[p1 + (int64_t)p2 * lda], b = A[q1 + (int64_t)p2 * lda];
        rot2(a, b, r1.c, r1.s, r1.ph);
        A[p1 + (int64_t)p2 * lda] = a;
        A[q1 + (int64_t)p2 * lda] = b;
      }
      return;
    }
    double2 m00 = A[p1 + (int64_t)p2 * lda], m10 = A[q1 + (int64_t)p2 * lda];
    double2 m01 = A[p1 + (int64_t)q2 * lda], m11 = A[q1 + (int64_t)q2 * lda];
    if (act1) {  // rows: [m0*; m1*] <- U1^H [m0*; m1*]
      rot2(m00, m10, r1.c, r1.s, r1.ph);
      rot2(m01, m11, r1.c, r1.s, r1.ph);
    }
    if (act2) {  // columns: [m*0, m*1] <- [m*0, m*1] U2
      rot2(m00, m01, r2.c, r2.s, cph2);
      rot2(m10, m11, r2.c, r2.s, cph2);
    }
    A[p1 + (int64_t)p2 * lda] = m00;
    A[q1 + (int64_t)p2 * lda] = m10;
    A[p1 + (int64_t)q2 * lda] = m01;
    A[q1 + (int64_t)q2 * lda] = m11;
    return;
  }
  const int64_t vidx = idx - nblk_a;
  if (vidx >= n * h) return;
  const int64_t i = vidx % n, t = vidx / n;
  const int q = pairs[2 * t + 1];
  if (q < 0) return;
  const Rot r = rot[t];
  if (r.s == 0.0) return;
  const int p = pairs[2 * t];
  double2 ap = V[i + (int64_t)p * ldv], aq = V[i + (int64_t)q * ldv];
  rot2(ap, aq, r.c, r.s, conjg(r.ph));
  V[i + (int64_t)p * ldv] = ap;
  V[i + (int64_t)q * ldv] = aq;
}

__global__ void k_jac_apply(int64_t h, int64_t n, double2* A, int64_t lda, double2* V, int64_t ldv,
                            const Rot* __restrict__ rot, const int* __restrict__ pairs) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  jac_apply_item(idx, h, n, A, lda, V, ldv, rot, pairs);
}

// All n-1 rounds of one Jacobi sweep in one cooperative launch: per round, the rotation
// parameters of the n/2 pairs, a grid barrier, the one-pass update of A and V, a barrier.
__global__ void k_jac_sweep(int64_t n0, int64_t n, double2* A, int64_t lda, double2* V, int64_t ldv, Rot* rot,
                            int* pairs, unsigned* bar, int* status) {
  const int64_t h = n / 2;
  const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t round = 0; round < n - 1; ++round) {
    for (int64_t t = tid; t < h; t += nthreads) jac_params_item(t, n0, n, round, A, lda, rot, pairs);
    grid_barrier(bar, bar + 1, gridDim.x, status);
    for (int64_t i = tid; i < jac_items(h, n0); i += nthreads) jac_apply_item(i, h, n0, A, lda, V, ldv, rot, pairs);
    grid_barrier(bar, bar + 1, gridDim.x, status);
  }
}

// Per-block partial sums of |off-diagonal|^2 and |A|^2 (FP64), then one block adds the
// partials in block order: deterministic.
template <typename R>
__global__ void k_offnorm_part(int64_t n, const cplx<R>* A, int64_t lda, double* part) {
  __shared__ double r0[256], r1[256];
  double s0 = 0, s1 = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % n, j = e / n;
    const cplx<R> a = A[i + j * lda];
    const double v = (double)a.x * a.x + (double)a.y * a.y;
    s1 += v;
    if (i != j) s0 += v;
  }
  r0[threadIdx.x] = s0;
  r1[threadIdx.x] = s1;
  __syncthreads();
  for (int hh = blockDim.x / 2; hh > 0; hh >>= 1) {
    if ((int)threadIdx.x < hh) {
      r0[threadIdx.x] += r0[threadIdx.x + hh];
      r1[threadIdx.x] += r1[threadIdx.x + hh];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = r0[0];
    part[2 * blockIdx.x + 1] = r1[0];
  }
}

__global__ void k_offnorm_sum(int nparts, const double* part, double* out) {
  if (threadIdx.x == 0) {
    double s0 = 0, s1 = 0;
    for (int b = 0; b < nparts; ++b) {
      s0 += part[2 * b];
      s1 += part[2 * b + 1];
    }
    out[0] = s0;
    out[1] = s1;
  }
}

// Sort eigenpairs ascending (stable): rank by counting, then permute w and the columns of V.
__global__ void k_eig_sort(int64_t n, const double2* __restrict__ A, int64_t lda, const double2* __restrict__ Vin,
                           int64_t ldvi, double* __restrict__ w, double2* __restrict__ Vout, int64_t ldvo) {
  const int64_t i = blockIdx.x;
  __shared__ int64_t rank;
  const double wi = A[i + i * lda].x;
  if (threadIdx.x == 0) rank = 0;
  __syncthreads();
  int64_t cnt = 0;
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
    const double wj = A[j + j * lda].x;
    if (wj < wi || (wj == wi && j < i)) ++cnt;
  }
  atomicAdd((unsigned long long*)&rank, (unsigned long long)cnt);
  __syncthreads();
  const int64_t r = rank;
  if (threadIdx.x == 0) w[r] = wi;
  for (int64_t k = threadIdx.x; k < n; k += blockDim.x) Vout[k + r * ldvo] = Vin[k + i * ldvi];
}

void jacobi_scalar(int64_t n0, double2* A, int64_t lda, double* w, double2* V, int64_t ldv, int* status, cudaStream_t st,
                   DevBuf<double2>* ws) {
  constexpr double tol_conv = 1e-15, tol_stall = 1e-12;
  if (n0 <= 0) return;
  const int64_t n = n0 + (n0 & 1);  // a padding player never paired for real
  // workspace (in double2 units): rotations, pair list, norm partials, barrier, a copy of V
  constexpr int kParts = 256;
  const size_t rot_c = (size_t)(n / 2) * sizeof(Rot) / sizeof(double2) + 1;
  const size_t pair_c = (size_t)n * sizeof(int) / sizeof(double2) + 1;
  const size_t part_c = kParts + 2;
  ws->alloc(rot_c + pair_c + part_c + 1 + (size_t)n0 * n0);
  Rot* rot = reinterpret_cast<Rot*>(ws->p);
  int* pairs = reinterpret_cast<int*>(ws->p + rot_c);
  double* part = reinterpret_cast<double*>(ws->p + rot_c + pair_c);
  double* nrm = part + 2 * kParts;
  unsigned* bar = reinterpret_cast<unsigned*>(ws->p + rot_c + pair_c + part_c);
  double2* Vtmp = reinterpret_cast<double2*>(ws->p + rot_c + pair_c + part_c + 1);
  if (n0 == 1) {
    set_identity(1, Vtmp, 1, st);
    CHEBFI_LAUNCH("k_eig_sort", st, k_eig_sort<<<1, 32, 0, st>>>(1, A, lda, Vtmp, 1, w, V, ldv));
    return;
  }
  CHEBFI_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st));
  // one cooperative launch per sweep when the device allows it (all blocks resident)
  int dev = 0, coop = 0, sms = 0, per_sm = 0;
  CHEBFI_CUDA(cudaGetDevice(&dev));
  CHEBFI_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  CHEBFI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  CHEBFI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_jac_sweep, 256, 0));
  const int coop_blocks = sms * std::min(per_sm, 8);
  set_identity(n0, Vtmp, n0, st);
  const int max_sweeps = 40;
  const unsigned parts = (unsigned)std::min<int64_t>(kParts, std::max<int64_t>(1, n0 * n0 / 4096));
  double prev_off = INFINITY;
  bool done = false, report = true;
  for (int sweep = 0; sweep <= max_sweeps && !done; ++sweep) {
    CHEBFI_LAUNCH("k_offnorm", st, k_offnorm_part<double><<<parts, 256, 0, st>>>(n0, A, lda, part));
    CHEBFI_LAUNCH("k_offnorm", st, k_offnorm_sum<<<1, 32, 0, st>>>((int)parts, part, nrm));
    double hn[2];
    CHEBFI_CUDA(cudaMemcpyAsync(hn, nrm, sizeof(hn), cudaMemcpyDeviceToHost, st));
    CHEBFI_CUDA(cudaStreamSynchronize(st));
    const double off = std::sqrt(hn[0]), tot = std::sqrt(hn[1]);
    if (!std::isfinite(tot)) {  // Inf or NaN in the matrix: no sweep can help
      int code = CHEBFI_ERR_NONFINITE;
      CHEBFI_CUDA(cudaMemcpyAsync(status, &code, sizeof(int), cudaMemcpyHostToDevice, st));
      CHEBFI_CUDA(cudaStreamSynchronize(st));
      report = false;
      break;
    }
    // converged: off-diagonal at the rounding level, or no longer decreasing near it
    if (off <= tol_conv * tot || off == 0.0 || (sweep > 2 && off > 0.5 * prev_off && off <= tol_stall * tot)) {
      done = true;
      break;
    }
    if (sweep == max_sweeps) break;
    prev_off = off;
    if (coop && coop_blocks > 0) {
      int64_t n0a = n0, na = n, ldaa = lda, ldva = n0;
      double2* Aa = A;
      double2* Va = Vtmp;
      void* args[] = {&n0a, &na, &Aa, &ldaa, &Va, &ldva, &rot, &pairs, &bar, &status};
      // work: per round every entry of A gets two rotations and every entry of V one, about
      // 11 real flops per complex entry per rotation: 33 n^3 per sweep
      CHEBFI_LAUNCH_W("k_jac_sweep", st, 33.0 * (double)n0 * (double)n0 * (double)n0,
                      CHEBFI_CUDA(cudaLaunchCooperativeKernel((const void*)k_jac_sweep, dim3(coop_blocks),
                                                              dim3(256), args, 0, st)));
    } else {
      for (int64_t round = 0; round < n - 1; ++round) {
        CHEBFI_LAUNCH("k_jac_params", st,
                      k_jac_params<<<nblk(n / 2), 256, 0, st>>>(n0, n, round, A, lda, rot, pairs));
        const int64_t h = n / 2;
        CHEBFI_LAUNCH("k_jac_apply", st,
                      k_jac_apply<<<nblk(jac_items(h, n0)), 256, 0, st>>>(h, n0, A, lda, Vtmp, n0, rot, pairs));
      }
    }
  }
  if (!done && report) {
    int code = CHEBFI_ERR_NO_CONVERGENCE;
    // record on the device flag as well so chebfi_sync_status sees it
    CHEBFI_CUDA(cudaMemcpyAsync(status, &code, sizeof(int), cudaMemcpyHostToDevice, st));
    CHEBFI_CUDA(cudaStreamSynchronize(st));
  }
  CHEBFI_LAUNCH("k_eig_sort", st, k_eig_sort<<<(unsigned)n0, 128, 0, st>>>(n0, A, lda, Vtmp, n0, w, V, ldv));
}


// ------------------------------------------------------------------ refinement of eigenvectors
// One step of the iterative refinement of Ogita & Aishima (2018) for a Hermitian A and
// approximate eigenvectors X, from G = X^H X (= I - R) and S = X^H A X:
//   lambda_i = S_ii / G_ii,
//   E_ij = (S_ij - lambda_j G_ij) / (lambda_j - lambda_i)   (i != j; = (s_ij + lambda_j r_ij)/(...)),
//   E_ii = (1 - G_ii) / 2,
// and X <- X (I + E).  A pair whose gap is not large against its numerator (|gap| <=
// 16 |num|, below 1e-13 |A|, or a numerator at rounding level that still turns the pair by more
// than 1e-8) is treated as a cluster: E_ij = -G_ij / 2 only restores orthogonality, and the
// pair is listed for a dense solve of the cluster.
__global__ void k_oa_lambda(int64_t n, const double2* __restrict__ G, int64_t ldg, const double2* __restrict__ S,
                            int64_t lds, double* __restrict__ lam, unsigned long long* __restrict__ amax) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double l = S[i + i * lds].x / G[i + i * ldg].x;
  lam[i] = l;
  atomicMax(amax, (unsigned long long)__double_as_longlong(fabs(l)));
}

__global__ void k_oa_update(int64_t n, const double2* __restrict__ G, int64_t ldg, const double2* __restrict__ S,
                            int64_t lds, const double* __restrict__ lam, const unsigned long long* __restrict__ amax,
                            double2* __restrict__ M, int64_t ldm, unsigned long long* __restrict__ emax,
                            int* __restrict__ npairs, int2* __restrict__ pairs, int cap) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = idx < n * n;
  const int64_t i = in ? idx % n : 0, j = in ? idx / n : 0;
  const double2 g = in ? G[i + j * ldg] : make_double2(1.0, 0.0);
  double2 e;
  double mag = 0.0;
  bool quiet = false;
  if (!in) {
    e = make_double2(0.0, 0.0);
  } else if (i == j) {
    e = make_double2(0.5 * (1.0 - g.x), 0.0);
    mag = fabs(e.x);
  } else {
    const double2 s = S[i + j * lds];
    const double lj = lam[j], gap = lj - lam[i];
    const double2 num = make_double2(s.x - lj * g.x, s.y - lj * g.y);
    const double anum = hypot(num.x, num.y);
    const double top = __longlong_as_double((long long)*amax);
    // the numerator of exact eigenvectors is rounding noise of S (about 2^-53 |A| times a small
    // constant); an update of that size is no sign of missing convergence
    const bool noise = anum <= 2e-15 * top;
    if (fabs(gap) > 16.0 * anum && fabs(gap) > 1e-13 * top && !(noise && anum > 1e-8 * fabs(gap))) {
      e = make_double2(num.x / gap, num.y / gap);
      quiet = noise;
    } else {
      e = make_double2(-0.5 * g.x, -0.5 * g.y);
      if (i < j) {
        const int k = atomicAdd(npairs, 1);
        if (k < cap) pairs[k] = make_int2((int)i, (int)j);
      }
    }
    if (!quiet) mag = hypot(e.x, e.y);
  }
  // max |E| over the warp first (the bits of non-negative doubles order like their values,
  // a NaN above all), then one atomic per warp: one per element serialises on the word
  unsigned long long bits = (unsigned long long)__double_as_longlong(mag);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xffffffffu, bits, o);
    bits = other > bits ? other : bits;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(emax, bits);
  if (in) M[i + j * ldm] = make_double2((i == j ? 1.0 : 0.0) + e.x, e.y);
}

// ascending order of w (stable), columns of X permuted alike
__global__ void k_sort_pairs(int64_t n, const double* __restrict__ win, const double2* __restrict__ Xin, int64_t ldi,
                             double* __restrict__ wout, double2* __restrict__ Xout, int64_t ldo) {
  const int64_t i = blockIdx.x;
  __shared__ unsigned long long rank;
  const double wi = win[i];
  if (threadIdx.x == 0) rank = 0;
  __syncthreads();
  unsigned long long cnt = 0;
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
    const double wj = win[j];
    if (wj < wi || (wj == wi && j < i)) ++cnt;
  }
  atomicAdd(&rank, cnt);
  __syncthreads();
  const int64_t r = (int64_t)rank;
  if (threadIdx.x == 0) wout[r] = wi;
  for (int64_t k = threadIdx.x; k < n; k += blockDim.x) Xout[k + r * ldo] = Xin[k + i * ldi];
}

// sub[a, b] = A[idx[a], idx[b]] (k x k); cols: sub[:, b] = X[:, idx[b]] or the reverse
__global__ void k_gather_sub(int k, const int* __restrict__ idx, const double2* __restrict__ A, int64_t lda,
                             double2* __restrict__ sub) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= k * k) return;
  const int a = e % k, b = e / k;
  sub[e] = A[idx[a] + (int64_t)idx[b] * lda];
}
__global__ void k_cols(int64_t m, int k, const int* __restrict__ idx, double2* X, int64_t ldx, double2* Y,
                       int64_t ldy, int to_y) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m * k) return;
  const int64_t r = e % m;
  const int b = (int)(e / m);
  if (to_y) Y[r + b * ldy] = X[r + idx[b] * ldx];
  else X[r + idx[b] * ldx] = Y[r + b * ldy];
}
__global__ void k_scatter_vals(int k, const int* __restrict__ idx, const double* __restrict__ src, double* dst) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < k) dst[idx[b]] = src[b];
}

// ------------------------------------------------------------------ clusters (FP64)
// Small dense problems of the refinement's clusters: one block per cluster c of k <= kMaxCluster
// listed columns idx[off[c]..off[c + 1]).  The block S[idx, idx] is diagonalised in shared
// memory by the cyclic Jacobi method above; lam[idx] gets its eigenvalues and
// X[:, idx] <- X[:, idx] Z.  With G (inside the refinement, X^H X not yet the identity, lam the
// step's values): the block of the basis that the step's -G / 2 orthogonalises, to first order
// S_ij - (lam_i + lam_j) G_ij / 2 beside lam on the diagonal.  A symmetric crystal has dozens of 2- and 3-fold shells: one
// launch for all of them instead of a cooperative eigensolve, three copies and a host
// synchronisation each (about 0.2 ms apiece).
constexpr int kMaxCluster = 32;
__global__ void __launch_bounds__(256) k_cluster_solve(int64_t n, const int* __restrict__ off, const int* __restrict__ idx,
                                                       const double2* __restrict__ S, const double2* __restrict__ G,
                                                       double2* X, double* __restrict__ lam, int* status) {
  constexpr int P = kMaxCluster + 1;
  __shared__ double2 A[kMaxCluster * P], Z[kMaxCluster * P];
  __shared__ Rot rot[kMaxCluster / 2];
  __shared__ int pairs[kMaxCluster];
  __shared__ double norms[2];
  const int* id = idx + off[blockIdx.x];
  const int k = off[blockIdx.x + 1] - off[blockIdx.x], kp = k + (k & 1), tid = threadIdx.x;
  for (int e = tid; e < k * k; e += blockDim.x) {
    const int i = e % k, j = e / k;
    // the Hermitian part
    const double2 u = S[id[i] + id[j] * n], v = S[id[j] + id[i] * n];
    double2 h = make_double2(0.5 * (u.x + v.x), 0.5 * (u.y - v.y));
    if (G && i == j) h = make_double2(lam[id[i]], 0.0);
    if (G && i != j) {
      const double2 g = G[id[i] + id[j] * n];
      const double l = 0.5 * (lam[id[i]] + lam[id[j]]);
      h = make_double2(h.x - l * g.x, h.y - l * g.y);
    }
    A[i + P * j] = h;
    Z[i + P * j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  double prev = INFINITY;
  bool done = false;
  for (int sweep = 0; sweep <= 40; ++sweep) {
    if (tid < 32) {
      double o = 0.0, t = 0.0;
      for (int e = tid; e < k * k; e += 32) {
        const double2 v = A[e % k + P * (e / k)];
        const double m = v.x * v.x + v.y * v.y;
        t += m;
        if (e % k != e / k) o += m;
      }
#pragma unroll
      for (int h = 16; h > 0; h >>= 1) {
        o += __shfl_xor_sync(0xffffffffu, o, h);
        t += __shfl_xor_sync(0xffffffffu, t, h);
      }
      if (tid == 0) {
        norms[0] = sqrt(o);
        norms[1] = sqrt(t);
      }
    }
    __syncthreads();
    const double o = norms[0], t = norms[1];
    __syncthreads();
    if (o <= 1e-15 * t || o == 0.0 || (sweep > 2 && o > 0.5 * prev && o <= 1e-12 * t)) {
      done = true;
      break;
    }
    if (sweep == 40 || !(t < INFINITY)) break;
    prev = o;
    for (int r = 0; r < kp - 1; ++r) {
      if (tid < kp / 2) jac_params_item(tid, k, kp, r, A, P, rot, pairs);
      __syncthreads();
      for (int i = tid; i < (int)jac_items(kp / 2, k); i += blockDim.x)
        jac_apply_item(i, kp / 2, k, A, P, Z, P, rot, pairs);
      __syncthreads();
    }
  }
  if (!done && tid == 0) flag_error(status, CHEBFI_ERR_NO_CONVERGENCE);
  if (tid < k) lam[id[tid]] = A[tid + P * tid].x;
  // rows of X in steps of the block: a thread holds its row's k entries
  for (int64_t row = tid; row < n; row += blockDim.x) {
    double2 x[kMaxCluster];
    for (int j = 0; j < k; ++j) x[j] = X[row + id[j] * n];
    for (int j = 0; j < k; ++j) {
      double2 y = make_double2(0.0, 0.0);
      for (int l = 0; l < k; ++l) {
        const double2 z = Z[l + P * j];
        y.x = fma(x[l].x, z.x, fma(-x[l].y, z.y, y.x));
        y.y = fma(x[l].x, z.y, fma(x[l].y, z.x, y.y));
      }
      X[row + id[j] * n] = y;
    }
  }
}

// ------------------------------------------------------------------ blocked Jacobi (FP32)
// The two-sided cyclic Jacobi method on blocks: the n columns form n / 32 blocks, paired by
// the round-robin tournament (n / 32 - 1 rounds per sweep, n / 64 disjoint pairs per round).
// For a pair (I, J) the 64 x 64 subproblem A[IJ, IJ] is swept once in shared memory by the
// scalar method (same rotations as above; the pairs within I and within J only in the first
// round, so that a sweep meets every pair of columns once) giving a unitary W, then A <- W^H A W on rows and
// columns I u J and V <- V W: each round is one pass over A and V as small dense products
// instead of 63 passes of scalar rotations, which the scalar method spends in grid barriers
// and load latency.
//
// Two launches a round.  k_bj_update forms the tile W1^H A W2 of each pair of pairs in one
// go and only for the lower triangle of A, writing the conjugate tile beside it (2080 64^3
// products a round at n = 2048 where column and row passes take 3072).  The subproblems are a
// chain of 63 short steps on n / 64 SMs, so k_bj_solve's other blocks meanwhile apply the
// round before's W to V, which nobody waits for.  n = 2048: 233 us a round (93 + 140) with
// one kernel each for solve, columns and rows, now 121 us.
namespace bj {
constexpr int B = 32, S2 = 64, PS = S2 + 1;  // block, subproblem, shared pitch

__device__ __forceinline__ int player(int pos, int round, int m) {
  if (pos == 0) return 0;
  const int p = pos - 1 + round;  // round < m - 1, pos < m
  return 1 + (p >= m - 1 ? p - (m - 1) : p);
}
__device__ __forceinline__ void blocks_of(int pair, int round, int nbk, int& I, int& J) {
  I = player(pair, round, nbk);
  J = player(nbk - 1 - pair, round, nbk);
  if (I > J) {
    const int t = I;
    I = J;
    J = t;
  }
}
__device__ __forceinline__ int gidx(int l, int I, int J) { return l < B ? I * B + l : J * B + (l - B); }

// acc(r, c) = sum_l X(r, l) W(l, c), or with CONJ sum_l conj(X(l, r)) W(l, c), of 64 x 64 tiles
// in shared memory (X[i + PS j] = element (i, j)); thread: rows ri + 16 k, columns ci + 16 m
template <bool CONJ>
__device__ __forceinline__ void mul64(const float2* X, const float2* W, float2 (&acc)[4][4]) {
  const int ri = threadIdx.x % 16, ci = threadIdx.x % 256 / 16;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[k][m] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int l = 0; l < S2; ++l) {
    float2 x[4], y[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[k] = CONJ ? X[l + PS * (ri + 16 * k)] : X[ri + 16 * k + PS * l];
      if (CONJ) x[k].y = -x[k].y;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) y[m] = W[l + PS * (ci + 16 * m)];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        acc[k][m].x = fmaf(x[k].x, y[m].x, fmaf(-x[k].y, y[m].y, acc[k][m].x));
        acc[k][m].y = fmaf(x[k].x, y[m].y, fmaf(x[k].y, y[m].x, acc[k][m].y));
      }
  }
}
__device__ __forceinline__ void put64(float2* X, const float2 (&acc)[4][4]) {
  const int ri = threadIdx.x % 16, ci = threadIdx.x / 16;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int m = 0; m < 4; ++m) X[ri + 16 * k + PS * (ci + 16 * m)] = acc[k][m];
}

// [a, b] <- [c a - s ph b, s a + c ph b] as packed (Re, Im) operations
__device__ __forceinline__ void rot2p(float2& a, float2& b, float c, float s, float2 ph) {
  const float2 pb = __ffma2_rn(make_float2(ph.x, ph.x), b, __fmul2_rn(make_float2(-ph.y, ph.y), make_float2(b.y, b.x)));
  const float2 na = __ffma2_rn(make_float2(c, c), a, __fmul2_rn(make_float2(-s, -s), pb));
  b = __ffma2_rn(make_float2(s, s), a, __fmul2_rn(make_float2(c, c), pb));
  a = na;
}

// Diagonalise the SS x SS Hermitian S (in shared memory, S[i + (SS + 1) j]) by up to `sweeps`
// cyclic sweeps, or until its off-diagonal part is below tol of its norm; W (same layout,
// the identity on entry) collects the rotations.  A sweep is a chain of SS - 1 short rounds,
// bound by latency: lane l of every warp computes the rotation of pair l from the same
// entries (no hand-over through shared memory, one barrier less) with the fast reciprocal
// square root (2 ulp there cost nothing, the vectors are refined), takes the 2 x 2 blocks of
// row pair l and of its warp's column pairs, and gets the latter's rotations by shuffles.
// One 64 x 64 sweep: 93 us with 1024 threads and rotations through shared memory, now 86 us,
// and 45 us for the 32 x 32 pairs across the blocks.
template <int SS> struct SolveThreads { static constexpr int v = SS == 64 ? 512 : 256; };
// CROSS: only the pairs of one index below SS / 2 and one above (SS / 2 rounds).
template <int SS, bool CROSS>
__device__ void solve_shared(float2* S, float2* W, int sweeps, float tol) {
  constexpr int P = SS + 1, NP = SS / 2, NT = SolveThreads<SS>::v, NW = NT / 32;
  static_assert(NP * NP % NT == 0 && (NP == 32 || 2 * NW == NP), "items of a round");
  __shared__ float red[2][NW];
  const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
  const unsigned all = 0xffffffffu;
  for (int sw = 0; sw < sweeps; ++sw) {
    float o = 0.f, t = 0.f;
    for (int e = tid; e < SS * SS; e += NT) {
      const int i = e % SS, j = e / SS;
      const float2 v = S[i + P * j];
      const float m = v.x * v.x + v.y * v.y;
      t += m;
      if (i != j) o += m;
    }
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
      o += __shfl_xor_sync(all, o, h);
      t += __shfl_xor_sync(all, t, h);
    }
    if (lane == 0) {
      red[0][warp] = o;
      red[1][warp] = t;
    }
    __syncthreads();
    o = t = 0.f;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      o += red[0][i];
      t += red[1][i];
    }
    __syncthreads();
    if (!(o > tol * tol * t)) break;
    for (int r = 0; r < (CROSS ? NP : SS - 1); ++r) {
      int p = lane % NP, q = NP + (p + r) % NP;
      if (!CROSS) {
        p = player(lane % NP, r, SS);
        q = player(SS - 1 - lane % NP, r, SS);
        if (p > q) {
          const int x = p;
          p = q;
          q = x;
        }
      }
      const float2 h = S[p + P * q];
      const float app = S[p + P * p].x, aqq = S[q + P * q].x;
      const float g2 = h.x * h.x + h.y * h.y;
      float c = 1.f, s = 0.f, px = 1.f, py = 0.f;
      if (g2 > 1e-36f && g2 > kEpsF * kEpsF * fabsf(app * aqq)) {
        const float rg = rsqrtf(g2), zeta = 0.5f * (aqq - app) * rg;
        const float tt = __fdividef(copysignf(1.f, zeta), fabsf(zeta) + __fsqrt_rn(fmaf(zeta, zeta, 1.f)));
        c = rsqrtf(fmaf(tt, tt, 1.f));
        s = tt * c;
        px = h.x * rg;
        py = h.y * rg;
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < NP * NP / NT; ++i) {
        // block of row pair t1 = lane % NP and column pair t2: U1^H S U2
        const int t2 = NP == 32 ? warp + NW * i : 2 * warp + lane / 16;
        const int p2 = CROSS ? t2 : __shfl_sync(all, p, t2), q2 = CROSS ? NP + (t2 + r) % NP : __shfl_sync(all, q, t2);
        const float c2 = __shfl_sync(all, c, t2), s2 = __shfl_sync(all, s, t2);
        const float2 ph2 = make_float2(__shfl_sync(all, px, t2), -__shfl_sync(all, py, t2));
        const float2 ph1 = make_float2(px, py);
        float2 m00 = S[p + P * p2], m10 = S[q + P * p2], m01 = S[p + P * q2], m11 = S[q + P * q2];
        rot2p(m00, m10, c, s, ph1);
        rot2p(m01, m11, c, s, ph1);
        rot2p(m00, m01, c2, s2, ph2);
        rot2p(m10, m11, c2, s2, ph2);
        S[p + P * p2] = m00;
        S[q + P * p2] = m10;
        S[p + P * q2] = m01;
        S[q + P * q2] = m11;
        // W <- W U2 on columns {p2, q2}
        if (NP == 32) {
#pragma unroll
          for (int row = lane; row < SS; row += 32) {
            float2 a = W[row + P * p2], b = W[row + P * q2];
            rot2p(a, b, c2, s2, ph2);
            W[row + P * p2] = a;
            W[row + P * q2] = b;
          }
        } else {  // SS = 32: the half-warp's own column pair, both halves of its rows
#pragma unroll
          for (int row = lane % 16; row < SS; row += 16) {
            float2 a = W[row + P * p2], b = W[row + P * q2];
            rot2p(a, b, c2, s2, ph2);
            W[row + P * p2] = a;
            W[row + P * q2] = b;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Blocks [0, nsolve) (all pairs, or none): gather the pair's subproblem, one sweep, write its
// rotation W (64 x 64, column-major) to Wout[pair].  The others: V <- V W of the round before
// (Wprev), a block per 128 rows and pair, 64 rows for each half of its threads.
__global__ void __launch_bounds__(512) k_bj_solve(const float2* __restrict__ A, float2* __restrict__ V, int64_t ld,
                                                  int nbk, int nsolve, int round, int round_prev, float2* __restrict__ Wout,
                                                  const float2* __restrict__ Wprev, float tol) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2* W = reinterpret_cast<float2*>(smem);
  float2* S = W + S2 * PS;
  const int tid = threadIdx.x, npairs = nbk / 2;
  int I, J;
  if ((int)blockIdx.x < nsolve) {
    blocks_of(blockIdx.x, round, nbk, I, J);
    for (int e = tid; e < S2 * S2; e += 512) {
      const int i = e % S2, j = e / S2;
      S[i + PS * j] = A[gidx(i, I, J) + (int64_t)gidx(j, I, J) * ld];
      W[i + PS * j] = make_float2(i == j ? 1.f : 0.f, 0.f);
    }
    __syncthreads();
    // the pairs within a block meet once a sweep, in its first round
    if (round == 0) solve_shared<S2, false>(S, W, 1, tol);
    else solve_shared<S2, true>(S, W, 1, tol);
    float2* wo = Wout + (int64_t)blockIdx.x * S2 * S2;
    for (int e = tid; e < S2 * S2; e += 512) wo[e] = W[(e % S2) + PS * (e / S2)];
    return;
  }
  const int u = blockIdx.x - nsolve, pair = u % npairs, half = tid / 256, t = tid % 256;
  const int64_t r0 = (int64_t)(u / npairs) * 2 * S2 + half * S2;
  const bool rows = r0 < ld;  // an odd number of 64-row tiles leaves the last half idle
  blocks_of(pair, round_prev, nbk, I, J);
  const float2* w = Wprev + (int64_t)pair * S2 * S2;
  S += half * S2 * PS;
  for (int e = tid; e < S2 * S2; e += 512) W[e % S2 + PS * (e / S2)] = w[e];
  if (rows)
    for (int e = t; e < S2 * S2; e += 256) S[e % S2 + PS * (e / S2)] = V[r0 + e % S2 + (int64_t)gidx(e / S2, I, J) * ld];
  __syncthreads();
  if (!rows) return;
  float2 acc[4][4];
  mul64<false>(S, W, acc);
  const int ri = t % 16, ci = t / 16;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int m = 0; m < 4; ++m) V[r0 + ri + 16 * k + (int64_t)gidx(ci + 16 * m, I, J) * ld] = acc[k][m];
}

// A <- W^H A W, one block per tile (pair t1, pair t2), t1 >= t2: the rows of pair t1 and the
// columns of pair t2, and the conjugate tile across the diagonal
__global__ void __launch_bounds__(256) k_bj_update(float2* A, int64_t ld, int nbk, int round, const float2* __restrict__ Win) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2* X = reinterpret_cast<float2*>(smem);
  float2* W = X + S2 * PS;
  const int tid = threadIdx.x;
  // block -> (t1, t2) of the lower triangle, row by row
  int t1 = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((t1 + 1) * (t1 + 2) / 2 <= (int)blockIdx.x) ++t1;
  while (t1 * (t1 + 1) / 2 > (int)blockIdx.x) --t1;
  const int t2 = (int)blockIdx.x - t1 * (t1 + 1) / 2;
  int I1, J1, I2, J2;
  blocks_of(t1, round, nbk, I1, J1);
  blocks_of(t2, round, nbk, I2, J2);
  const float2 *w1 = Win + (int64_t)t1 * S2 * S2, *w2 = Win + (int64_t)t2 * S2 * S2;
  for (int e = tid; e < S2 * S2; e += 256) {
    const int a = e % S2, b = e / S2;
    W[a + PS * b] = w2[e];
    X[a + PS * b] = A[gidx(a, I1, J1) + (int64_t)gidx(b, I2, J2) * ld];
  }
  __syncthreads();
  float2 acc[4][4];
  mul64<false>(X, W, acc);
  __syncthreads();
  put64(X, acc);
  for (int e = tid; e < S2 * S2; e += 256) W[e % S2 + PS * (e / S2)] = w1[e];
  __syncthreads();
  mul64<true>(W, X, acc);
  __syncthreads();
  put64(X, acc);
  __syncthreads();
  for (int e = tid; e < S2 * S2; e += 256) {
    const int a = e % S2, b = e / S2;
    A[gidx(a, I1, J1) + (int64_t)gidx(b, I2, J2) * ld] = X[a + PS * b];
  }
  if (t1 == t2) return;
  for (int e = tid; e < S2 * S2; e += 256) {
    const int b = e % S2, a = e / S2;
    const float2 v = X[a + PS * b];
    A[gidx(b, I2, J2) + (int64_t)gidx(a, I1, J1) * ld] = make_float2(v.x, -v.y);
  }
}

// the whole problem in one block, n <= SS (padded with decoupled zero rows): V's n x n block
template <int SS>
__global__ void __launch_bounds__(SolveThreads<SS>::v) k_bj_small(int n, const float2* __restrict__ A, int64_t lda, float2* __restrict__ V,
                                                  int64_t ldv, float tol) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2* S = reinterpret_cast<float2*>(smem);
  float2* W = S + SS * (SS + 1);
  for (int e = threadIdx.x; e < SS * SS; e += SolveThreads<SS>::v) {
    const int i = e % SS, j = e / SS;
    S[i + (SS + 1) * j] = i < n && j < n ? A[i + j * lda] : make_float2(0.f, 0.f);
    W[i + (SS + 1) * j] = make_float2(i == j ? 1.f : 0.f, 0.f);
  }
  __syncthreads();
  solve_shared<SS, false>(S, W, 16, tol);
  for (int e = threadIdx.x; e < n * n; e += SolveThreads<SS>::v) V[e % n + (e / n) * ldv] = W[e % n + (SS + 1) * (e / n)];
}

// The largest biased exponent of A's components (A dense, n2 entries), and A times the power of
// two that brings them below 2 in FP32: the rotations square entries, and a matrix in other units
// of energy must not lose them to float's range.  A non-finite A stays so.
__global__ void __launch_bounds__(256) k_bj_exponent(int64_t n2, const double2* __restrict__ A, int* __restrict__ emax) {
  int e = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = A[i];
    e = max(e, max((__double2hiint(v.x) >> 20) & 0x7FF, (__double2hiint(v.y) >> 20) & 0x7FF));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if (threadIdx.x % 32 == 0) atomicMax(emax, e);
}
__global__ void __launch_bounds__(256) k_bj_scale(int64_t n2, const double2* __restrict__ A, const int* __restrict__ emax,
                                                  float2* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n2) return;
  const double f = ldexp(1.0, 1023 - *emax);
  out[i] = make_float2((float)(A[i].x * f), (float)(A[i].y * f));
}

__global__ void k_bj_identity(int64_t n, float2* V) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n * n) V[e] = make_float2(e % (n + 1) == 0 ? 1.f : 0.f, 0.f);
}

// zero-padded copy
__global__ void k_bj_pad(int64_t n0, int64_t np, const float2* __restrict__ A, int64_t lda, float2* __restrict__ Ap) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= np * np) return;
  const int64_t i = e % np, j = e / np;
  Ap[e] = (i < n0 && j < n0) ? A[i + j * lda] : make_float2(0.f, 0.f);
}
}  // namespace bj

}  // namespace

void oa_step(int64_t n, const double2* G, const double2* S, double* lam, double2* M, unsigned long long* stats,
             int* npairs, int2* pairs, int cap, cudaStream_t st) {
  CHEBFI_CUDA(cudaMemsetAsync(stats, 0, 2 * sizeof(unsigned long long), st));
  CHEBFI_CUDA(cudaMemsetAsync(npairs, 0, sizeof(int), st));
  CHEBFI_LAUNCH("k_oa_lambda", st, k_oa_lambda<<<nblk(n), 256, 0, st>>>(n, G, n, S, n, lam, stats));
  CHEBFI_LAUNCH("k_oa_update", st,
                k_oa_update<<<nblk(n * n), 256, 0, st>>>(n, G, n, S, n, lam, stats, M, n, stats + 1, npairs, pairs, cap));
}

void sort_eigpairs(int64_t n, const double* win, const double2* Xin, double* wout, double2* Xout, cudaStream_t st) {
  CHEBFI_LAUNCH("k_sort_pairs", st, k_sort_pairs<<<(unsigned)n, 128, 0, st>>>(n, win, Xin, n, wout, Xout, n));
}

void gather_sub(int k, const int* idx, const double2* A, int64_t lda, double2* sub, cudaStream_t st) {
  CHEBFI_LAUNCH("k_gather_sub", st, k_gather_sub<<<nblk((int64_t)k * k), 256, 0, st>>>(k, idx, A, lda, sub));
}
void gather_cols(int64_t m, int k, const int* idx, const double2* X, int64_t ldx, double2* Y, int64_t ldy,
                 cudaStream_t st) {
  CHEBFI_LAUNCH("k_cols", st, k_cols<<<nblk(m * k), 256, 0, st>>>(m, k, idx, const_cast<double2*>(X), ldx, Y, ldy, 1));
}
void scatter_cols(int64_t m, int k, const int* idx, double2* X, int64_t ldx, const double2* Y, int64_t ldy,
                  cudaStream_t st) {
  CHEBFI_LAUNCH("k_cols", st, k_cols<<<nblk(m * k), 256, 0, st>>>(m, k, idx, X, ldx, const_cast<double2*>(Y), ldy, 0));
}
void scatter_vals(int k, const int* idx, const double* src, double* dst, cudaStream_t st) {
  CHEBFI_LAUNCH("k_scatter_vals", st, k_scatter_vals<<<nblk(k), 256, 0, st>>>(k, idx, src, dst));
}

void cholesky(int64_t n, double2* A, int64_t lda, int* status, cudaStream_t st, DevBuf<double2>* ws) {
  for (int64_t k0 = 0; k0 < n; k0 += NB) {
    const int nb = (int)std::min<int64_t>(NB, n - k0);
    CHEBFI_LAUNCH("k_chol_diag", st, k_chol_diag<<<1, 256, 0, st>>>(A + k0 + k0 * lda, lda, nb, status));
    const int64_t m2 = n - k0 - nb;
    if (m2 > 0) {
      double2* L21 = A + (k0 + nb) + k0 * lda;
      CHEBFI_LAUNCH("k_trsm_right_lh", st, k_trsm_right_lh<<<nblk(m2, kTrsmWarps), 32 * kTrsmWarps, 0, st>>>(A + k0 + k0 * lda, lda, L21, lda, m2, nb));
      gemm<double>(false, true, m2, m2, nb, -1.0, L21, lda, L21, lda, 1.0, A + (k0 + nb) + (k0 + nb) * lda, lda, st,
                   ws, "k_gemm", true);
    }
  }
  CHEBFI_LAUNCH("k_zero_upper", st, k_zero_upper<<<nblk(n * n), 256, 0, st>>>(n, A, lda));
}

void trsm_lower(int64_t n, int64_t m, const double2* L, int64_t ldl, double2* B, int64_t ldb, cudaStream_t st,
                DevBuf<double2>* ws) {
  for (int64_t k0 = 0; k0 < n; k0 += NB) {
    const int nb = (int)std::min<int64_t>(NB, n - k0);
    CHEBFI_LAUNCH("k_trsm_left_l", st, k_trsm_left_l<<<nblk(m, kTrsmWarps), 32 * kTrsmWarps, 0, st>>>(L + k0 + k0 * ldl, ldl, B + k0, ldb, m, nb));
    const int64_t m2 = n - k0 - nb;
    if (m2 > 0)
      gemm<double>(false, false, m2, m, nb, -1.0, L + (k0 + nb) + k0 * ldl, ldl, B + k0, ldb, 1.0, B + k0 + nb, ldb, st,
                   ws);
  }
}

void jacobi_eigh(int64_t n0, double2* A, int64_t lda, double* w, double2* V, int64_t ldv, int* status, cudaStream_t st,
                 DevBuf<double2>* ws) {
  jacobi_scalar(n0, A, lda, w, V, ldv, status, st, ws);
}

void scaled_to_f32(int64_t n, const double2* A, float2* out, int* emax, cudaStream_t st) {
  const int64_t n2 = n * n;
  CHEBFI_CUDA(cudaMemsetAsync(emax, 0, sizeof(int), st));
  CHEBFI_LAUNCH("k_bj_scale", st, bj::k_bj_exponent<<<(unsigned)std::min<int64_t>(nblk(n2), 1024), 256, 0, st>>>(n2, A, emax));
  CHEBFI_LAUNCH("k_bj_scale", st, bj::k_bj_scale<<<nblk(n2), 256, 0, st>>>(n2, A, emax, out));
}

// The FP32 Jacobi (bj:: kernels) on A (n0 x n0), components below about 2 (scaled_to_f32): approximate eigenvectors in V (ld ldv), in
// no particular order.  One block for n0 <= 64, the block tournament above.  The matrix is
// padded with decoupled zero rows and columns, which no rotation touches (a rotation needs a
// non-zero off-diagonal entry).  False if A is not finite in FP32 (V is not written).
bool jacobi_eigh_f32(int64_t n0, const float2* A, int64_t lda, float2* V, int64_t ldv, cudaStream_t st,
                     DevBuf<double2>* ws) {
  // off-diagonal entries of rms 1e-5 |A|_F / n turn a pair of typical gap by about 1e-3, which
  // the refinement squares in each step; FP32 sweeps past this level mostly stir rounding noise
  constexpr double tol_conv = 1e-5;
  const int64_t np = n0 <= 64 ? 0 : (n0 + bj::S2 - 1) / bj::S2 * bj::S2;
  const int nbk = (int)(np / bj::B), npairs = nbk / 2;
  constexpr int kParts = 256;
  // workspace in float2 slots: Ap and Vp (np^2 each), two sets of W (npairs x 64^2), norm
  // partials and sums (2 kParts + 2 doubles)
  const size_t nn = (size_t)np * np, nw = (size_t)npairs * bj::S2 * bj::S2;
  ws->alloc((2 * nn + 2 * nw + 2 * kParts + 2) / 2 + 1);
  float2* Ap = reinterpret_cast<float2*>(ws->p);
  float2* Vp = Ap + nn;
  float2* Wb[2] = {Vp + nn, Vp + nn + nw};
  double* part = reinterpret_cast<double*>(Vp + nn + 2 * nw);
  double* nrm = part + 2 * kParts;
  auto norms = [&](const float2* M, int64_t n, int64_t ld, double& off, double& tot) {
    const unsigned parts = (unsigned)std::min<int64_t>(kParts, std::max<int64_t>(1, n * n / 4096));
    CHEBFI_LAUNCH("k_offnorm", st, k_offnorm_part<float><<<parts, 256, 0, st>>>(n, M, ld, part));
    CHEBFI_LAUNCH("k_offnorm", st, k_offnorm_sum<<<1, 32, 0, st>>>((int)parts, part, nrm));
    double hn[2];
    CHEBFI_CUDA(cudaMemcpyAsync(hn, nrm, sizeof(hn), cudaMemcpyDeviceToHost, st));
    CHEBFI_CUDA(cudaStreamSynchronize(st));
    off = std::sqrt(hn[0]);
    tot = std::sqrt(hn[1]);
  };
  double off = 0.0, tot = 0.0;
  norms(A, n0, lda, off, tot);
  if (!std::isfinite(tot)) return false;
  if (n0 <= 64) {
    auto small = [&](auto kernel, int ss, int threads) {
      const size_t bytes = (size_t)2 * ss * (ss + 1) * sizeof(float2);
      CHEBFI_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
      CHEBFI_LAUNCH("k_bj_small", st, kernel<<<1, threads, bytes, st>>>((int)n0, A, lda, V, ldv, (float)tol_conv));
    };
    if (n0 <= 32) small(bj::k_bj_small<32>, 32, bj::SolveThreads<32>::v);
    else small(bj::k_bj_small<64>, 64, bj::SolveThreads<64>::v);
    return true;
  }
  CHEBFI_LAUNCH("k_bj_pad", st, bj::k_bj_pad<<<nblk((int64_t)nn), 256, 0, st>>>(n0, np, A, lda, Ap));
  CHEBFI_LAUNCH("k_identity", st, bj::k_bj_identity<<<nblk((int64_t)nn), 256, 0, st>>>(np, Vp));
  const size_t bytes = (size_t)2 * bj::S2 * bj::PS * sizeof(float2);
  const size_t sbytes = (size_t)3 * bj::S2 * bj::PS * sizeof(float2);
  CHEBFI_CUDA(cudaFuncSetAttribute(bj::k_bj_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sbytes));
  CHEBFI_CUDA(cudaFuncSetAttribute(bj::k_bj_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  const unsigned vtiles = (unsigned)((np / bj::S2 + 1) / 2) * npairs, atiles = (unsigned)npairs * (npairs + 1) / 2;
  const double prod = 8.0 * bj::S2 * bj::S2 * bj::S2;  // flops of one 64^3 complex product
  double prev_off = INFINITY;
  int w = 0, last_round = -1;  // W of round last_round, in Wb[w ^ 1], is still to be applied to V
  for (int sweep = 0; sweep <= 40; ++sweep) {
    if (sweep > 0) {
      double t;
      norms(Ap, np, np, off, t);
      if (!std::isfinite(t)) return false;
    }
    if (off <= tol_conv * tot || off == 0.0 || (sweep > 2 && off > 0.5 * prev_off && off <= 1e-3 * tot)) break;
    if (sweep == 40) break;
    prev_off = off;
    for (int round = 0; round < nbk - 1; ++round) {
      const unsigned extra = last_round >= 0 ? vtiles : 0;
      CHEBFI_LAUNCH_W("k_bj_solve", st, prod * 2.0 * extra,
                      bj::k_bj_solve<<<npairs + extra, 512, sbytes, st>>>(Ap, Vp, np, nbk, npairs, round, last_round, Wb[w],
                                                                         Wb[w ^ 1], 1e-7f));
      CHEBFI_LAUNCH_W("k_bj_update", st, prod * 2.0 * atiles,
                      bj::k_bj_update<<<atiles, 256, bytes, st>>>(Ap, np, nbk, round, Wb[w]));
      last_round = round;
      w ^= 1;
    }
  }
  if (last_round >= 0) {  // the last W: nothing is left to solve
    CHEBFI_LAUNCH_W("k_bj_solve", st, prod * 2.0 * vtiles,
                    bj::k_bj_solve<<<vtiles, 512, sbytes, st>>>(Ap, Vp, np, nbk, 0, 0, last_round, Wb[w], Wb[w ^ 1], 1e-7f));
  }
  CHEBFI_CUDA(cudaMemcpy2DAsync(V, ldv * sizeof(float2), Vp, np * sizeof(float2), n0 * sizeof(float2), n0,
                                cudaMemcpyDeviceToDevice, st));
  return true;
}

int max_cluster() { return kMaxCluster; }
void cluster_solve(int64_t n, int ncl, const int* off, const int* idx, const double2* S, const double2* G, double2* X,
                   double* lam, int* status, cudaStream_t st) {
  CHEBFI_LAUNCH("k_cluster_solve", st, k_cluster_solve<<<ncl, 256, 0, st>>>(n, off, idx, S, G, X, lam, status));
}

}  // namespace chebfi
