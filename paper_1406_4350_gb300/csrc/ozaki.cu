// FP64-accurate complex GEMM on the tcgen05 tensor cores by modular arithmetic.
//
// GB300 runs FP64 FMAs at about 2 per clock per SM, so the subspace matrices, rotations and
// projector products of Algorithm 2 (Section 4.2) in FP64 would be bound by that unit.
// This file emulates them on the bf16 tensor pipe with the integer-modular scheme of Ozaki,
// Uchino and Imamura ("Ozaki scheme II", 2025), written here from its mathematics:
//
//  1. each row r of op(A) and each column n of op(B) is scaled by a power of two 2^s so
//     that its 2-norm lies in [2^(E-1), 2^E), and rounded to integers: A_int, B_int;
//     by Cauchy-Schwarz every entry of C_int = A_int B_int then satisfies |C_int| < 2^(2E);
//  2. for pairwise coprime moduli m_1..m_n <= 256 with M = prod m_i >= 2^(2E+3), the
//     symmetric residues of A_int and B_int (|r| <= 128) are exact in bf16 and their
//     products exact in FP32; one tensor-core GEMM per modulus sums them in FP32 in chunks
//     of 512 products (|partial| <= 2^23, so every partial sum is an exact integer), and the
//     epilogue reduces each chunk modulo m_i on the FP32 units;
//  3. C_int mod M follows from the n residue matrices by the Chinese remainder theorem,
//     evaluated exactly in 128-bit integers, and C = 2^-(s_r + s_n) C_int.
// The only rounding is step 1's: each scaled entry is within 1/2 of its integer, so an
// entry of C is within about 2^-E ||a_r|| ||b_n|| (times a small constant) of the exact
// product - with 14 moduli E = 53, the order of an FP64 dot product's error (1.3 to 6 times what
// the FP64 units give on products of middle size), with all 15 E = 57, below it.
//
// Complex products take three real ones per modulus instead of four (Gauss): with
//   T1 = Re a Re b,  T2 = Im a Im b,  T3 = (Re a + Im a)(Re b + Im b),
// Re = T1 - T2 and Im = T3 - T1 - T2.  In floating point the form loses accuracy in Im; modulo
// m it is exact, so the result's bits are those of the four products at 3/4 of their work.
// An operand is therefore three residue matrices per modulus: Re, Im and (Re + Im) mod m.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.cuh"
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace chebfi {
namespace oz {

// pairwise coprime moduli, largest first; a set uses the first n of them
constexpr int kMods[kOzMaxMod] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197};

// A CTA pair (cta_group::2) computes a 256 x BN tile: each CTA loads 128 rows of A and BN / 2
// rows of B per k-tile, half of what one CTA's 128 x BN tile would need, and each operand
// byte in shared memory feeds the tensor cores of both SMs.  With one CTA per 128 x 128 tile
// the loads (128 bytes per clock and SM at full rate) bound the kernel at 0.61 of the
// sustained bf16 rate; now a 2048 x 2048 x 20000 product runs 1.61 PFLOP/s of bf16 (0.95 of
// it, at the card's power limit; 153 TFLOP/s FP64-equivalent), 16384 x 2048 x 2048 1.53.
// BN = 128 serves products of at most 128 columns.
constexpr int BM = 256, BK = 64, STAGES = 6;
constexpr int CHUNK = 8;                      // k-tiles (512 products) per exact TMEM accumulation
constexpr int A_BYTES = 128 * BK * 2;         // 16 KB per CTA
constexpr int THREADS = 320;                  // TMA, MMA and eight epilogue warps
constexpr int NACC = 2;
constexpr int kMaxSplit = 16;
template <int BN> constexpr int stage_bytes() { return A_BYTES + BN / 2 * BK * 2; }
template <int BN> constexpr int smem_bytes() { return STAGES * stage_bytes<BN>() + 1024 + 256; }

struct GemmArgs {
  int M, N, num_k;  // complex rows and columns, k-tiles of one product
  int nplanes;      // 3 nmod
  int lower;        // lower triangle only: tiles that reach the diagonal
  int tiles_m, tiles_n, tiles;  // tiles = valid tiles per plane
  int splits, kt_split;         // K ranges of kt_split k-tiles (whole chunks), summed by the reconstruction
  signed char* R;   // residues: R[(split * nplanes + plane) * rstride + n * ldr + m]
  int64_t ldr, rstride;
  int* status;
  float m[kOzMaxMod], inv[kOzMaxMod];
};

// number of BN-column tiles of the 256-row tile tm that touch the lower triangle
__host__ __device__ __forceinline__ int lower_count(int tm, int bn, int tiles_n) { return min(tiles_n, (BM * tm + BM - 1) / bn + 1); }

template <int BN> __device__ __forceinline__ void unit_tile(const GemmArgs& a, int t, int& tm, int& tn) {
  if (!a.lower) {
    tm = t / a.tiles_n;
    tn = t % a.tiles_n;
    return;
  }
  int cum = 0;
  for (tm = 0; tm < a.tiles_m; ++tm) {
    const int c = lower_count(tm, BN, a.tiles_n);
    if (t < cum + c) break;
    cum += c;
  }
  tn = t - cum;
}

// unit u -> its plane (of plane-major units, so that the pairs in flight share operand
// k-slices in L2), tile and k-tile range
struct Unit {
  int plane, split, tm, tn, kt0, kt1;
};
template <int BN> __device__ __forceinline__ Unit unit_of(const GemmArgs& a, int u) {
  Unit r;
  const int per = a.tiles * a.splits;
  r.plane = u / per;
  const int v = u - r.plane * per;
  r.split = v / a.tiles;
  unit_tile<BN>(a, v - r.split * a.tiles, r.tm, r.tn);
  r.kt0 = r.split * a.kt_split;
  r.kt1 = min(a.num_k, r.kt0 + a.kt_split);
  return r;
}

// One persistent CTA pair per two SMs over (plane, split, tile) units.  Warp 0 of each CTA: TMA
// loads of its halves of the residue tiles (6-stage ring, bytes counted on the leader's
// barriers); warp 1 of the leader: one tcgen05 MMA chain per k-tile into one of two TMEM
// accumulators (one per 512-product chunk); warps 2-9: per chunk, add the exact FP32 sums
// into register accumulators reduced modulo m, then store the tile's residues as int8.
template <int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    k_oz_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const __grid_constant__ GemmArgs args) {
  using namespace tc;
  constexpr int SB = stage_bytes<BN>(), HN = BN / 2;
  constexpr uint32_t TMEM_COLS = NACC * BN;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * SB);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;
  uint64_t* acc_empty = acc_full + NACC;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + NACC);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int rank = (int)cluster_rank();
  const int pair = blockIdx.x / 2, npairs = gridDim.x / 2;
  const int units = args.tiles * args.splits * args.nplanes;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int q = 0; q < NACC; ++q) {
      mbar_init(&acc_full[q], 1);
      mbar_init(&acc_empty[q], 16);  // eight epilogue warps in each CTA
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int u = pair; u < units && ok; u += npairs) {
        const Unit un = unit_of<BN>(args, u);
        const int ra = un.tm * BM + 128 * rank, rb = un.tn * BN + HN * rank;
        for (int kt = un.kt0; kt < un.kt1; ++kt, ++g) {
          const int s = g % STAGES;
          const uint32_t par = (g / STAGES) & 1;
          if (g >= STAGES && !mbar_wait(&empty[s], par ^ 1)) {
            flag(args.status, CHEBFI_ERR_CUDA);
            ok = false;
            break;
          }
          uint8_t* st = smem + s * SB;
          if (rank == 0) mbar_expect_tx(&full[s], 2 * SB);
          const uint32_t bar = leader_addr(&full[s]);
          tma_load_3d_pair(st, &tmA, kt * BK, ra, un.plane, bar);
          tma_load_3d_pair(st + A_BYTES, &tmB, kt * BK, rb, un.plane, bar);
        }
      }
      // the last signals of every stage have landed before this CTA may leave
      for (int i = 0; i < STAGES && ok; ++i, ++g) {
        if (g >= STAGES && !mbar_wait(&empty[g % STAGES], ((g / STAGES) & 1) ^ 1)) {
          flag(args.status, CHEBFI_ERR_CUDA);
          ok = false;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(BM, BN);
      bool ok = true;
      int g = 0, gch = 0;
      for (int u = pair; u < units && ok; u += npairs) {
        const Unit un = unit_of<BN>(args, u);
        for (int kc = un.kt0; kc < un.kt1 && ok; kc += CHUNK, ++gch) {
          const int acc = gch % NACC;
          if (gch >= NACC && !mbar_wait(&acc_empty[acc], ((gch / NACC) - 1) & 1)) {
            flag(args.status, CHEBFI_ERR_CUDA);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(acc * BN);
          const int kend = min(un.kt1, kc + CHUNK);
          for (int kt = kc; kt < kend; ++kt, ++g) {
            const int s = g % STAGES;
            const uint32_t par = (g / STAGES) & 1;
            if (!mbar_wait(&full[s], par)) {
              flag(args.status, CHEBFI_ERR_CUDA);
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t base = smem_u32(smem + s * SB);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {
              const uint32_t off = kk * 32;  // 16 bf16 along K
              mma_bf16_pair(d, sw128_desc(base + off), sw128_desc(base + A_BYTES + off), idesc,
                            (kt == kc && kk == 0) ? 0u : 1u);
            }
            mma_commit_pair(&empty[s]);
          }
          if (ok) mma_commit_pair(&acc_full[acc]);
        }
      }
    }
  } else {
    const int lane_base = 32 * (warp % 4), col0 = HN * ((warp - 2) / 4);
    bool ok = true;
    int gch = 0;
    for (int u = pair; u < units && ok; u += npairs) {
      const Unit un = unit_of<BN>(args, u);
      const int mod = un.plane / 3;
      const float mm = args.m[mod], inv = args.inv[mod];
      const int m = un.tm * BM + 128 * rank + lane_base + lane;
      float racc[HN];
#pragma unroll
      for (int j = 0; j < HN; ++j) racc[j] = 0.f;
      for (int kc = un.kt0; kc < un.kt1; kc += CHUNK, ++gch) {
        const int acc = gch % NACC;
        // every lane's wait: the warp's collective loads and shuffles need one decision
        if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], (gch / NACC) & 1))) {
          flag(args.status, CHEBFI_ERR_CUDA);
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < HN; c += 32) {
          float v[32];
          tmem_ld32(tmem + ((uint32_t)lane_base << 16) + (uint32_t)(acc * BN + col0 + c), v);
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            // exact: |racc| < m and |v| <= 2^23, so the sum s and the product q m are integers
            // below 2^24; q = round(s / m) by adding and subtracting 1.5 2^23 (|s / m| < 2^16)
            const float s = __fadd_rn(racc[c + j], v[j]);
            const float q = __fsub_rn(__fmaf_rn(s, inv, 12582912.f), 12582912.f);
            racc[c + j] = __fmaf_rn(-mm, q, s);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_leader(leader_addr(&acc_empty[acc]));
      }
      if (!ok) break;
      // store: four columns at a time, a 4 x 4 byte transpose among groups of four lanes, so that
      // each lane writes four rows of one column (byte stores of single rows left the tensor
      // pipe idle at the end of short-K units: 16384 x 2048 x 2048 4.98 ms, now 3.78 ms).
      // The rounding and the conversion to bytes go through 1.5 2^23 (+128 wraps to -128).
      const int n0 = un.tn * BN + col0, q = lane & 3;
      const int m4 = un.tm * BM + 128 * rank + lane_base + (lane & ~3);
      signed char* out =
          args.R + (int64_t)(un.split * args.nplanes + un.plane) * args.rstride + (int64_t)(n0 + q) * args.ldr + m4;
#pragma unroll
      for (int j = 0; j < HN; j += 4) {
        unsigned w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float x = racc[j + e], k = __fsub_rn(__fmaf_rn(x, inv, 12582912.f), 12582912.f);
          w[e] = (unsigned)__float_as_int(__fadd_rn(__fmaf_rn(-mm, k, x), 12582912.f));  // |r| <= m / 2 in the low bits
        }
        // this row's columns j..j+3, lowest byte first
        unsigned v = __byte_perm(__byte_perm(w[0], w[1], 0x0040), __byte_perm(w[2], w[3], 0x0040), 0x5410);
        // transpose 2 x 2 blocks of bytes across lane bit 0, then of byte pairs across lane bit 1
        unsigned o = __shfl_xor_sync(0xffffffffu, v, 1);
        v = (q & 1) ? __byte_perm(o, v, 0x7351) : __byte_perm(v, o, 0x6240);
        o = __shfl_xor_sync(0xffffffffu, v, 2);
        v = (q & 2) ? __byte_perm(o, v, 0x7632) : __byte_perm(v, o, 0x5410);
        // lane q now holds rows m4..m4+3 of column j + q (rows past M are zero: padded tile rows)
        if (n0 + j + q < args.N && m4 < args.M) *reinterpret_cast<unsigned*>(out + (int64_t)j * args.ldr) = v;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // no CTA leaves while its peer may still signal its barriers or use its tiles
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
}

// ---------------------------------------------------------------- operand preparation
// 2-norm of each row of op(X) -> scale exponent s with ||row|| 2^s in [2^(E-1), 2^E);
// 0 for a zero row, kOzBadShift for a non-finite one (its products come out NaN).
__device__ __forceinline__ int shift_for(double sumsq, int E) {
  return E - 1 - (ilogb(sumsq) >> 1);  // floor(log2 sqrt(x)) = floor(floor(log2 x) / 2)
}
// Whether the plain sum of squares is as good as it looks: squares below FP64's range have not
// mattered, none has overflowed.  Other rows (zero, beyond 2^-450 or 2^511, or not finite) are
// summed again, scaled by their largest component.
__device__ __forceinline__ bool sum_in_range(double sumsq) { return sumsq >= 0x1p-900 && sumsq < INFINITY; }
constexpr int kAgain = 0x40000000;  // no shift yet
__device__ __forceinline__ int exponent_of(double2 v) {
  return max((__double2hiint(v.x) >> 20) & 0x7FF, (__double2hiint(v.y) >> 20) & 0x7FF);
}
// the power of two that brings components of largest biased exponent e to [1, 2)
__device__ __forceinline__ double scale_of(int e) { return ldexp(1.0, 1023 - e); }
__device__ __forceinline__ double add_scaled(double s, double2 v, double f) {
  const double x = v.x * f, y = v.y * f;
  return fma(x, x, fma(y, y, s));
}
// shift of a row of largest biased exponent e whose scaled squares sum to s
__device__ __forceinline__ int shift_scaled(int e, double s, int E) {
  return e == 0x7FF ? kOzBadShift : e == 0 ? 0 : shift_for(s, E) + (1023 - e);  // e = 0: zero or dropped (scaled_int)
}
// the scaled sum of a column x of X by the whole block; the result in every thread
__device__ __noinline__ int column_shift_scaled(const double2* __restrict__ x, int64_t K, int E) {
  __shared__ int se[32];
  __shared__ double ss[32];
  const int tid = threadIdx.x, nw = blockDim.x / 32;
  int e = 0;
  for (int64_t k = tid; k < K; k += blockDim.x) e = max(e, exponent_of(x[k]));
  e = __reduce_max_sync(0xffffffffu, e);
  if (tid % 32 == 0) se[tid / 32] = e;
  __syncthreads();
  for (int i = 0; i < nw; ++i) e = max(e, se[i]);
  double s = 0.0;
  const double f = scale_of(e);
  for (int64_t k = tid; k < K; k += blockDim.x) s = add_scaled(s, x[k], f);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (tid % 32 == 0) ss[tid / 32] = s;
  __syncthreads();
  s = 0.0;
  for (int i = 0; i < nw; ++i) s += ss[i];
  return shift_scaled(e, s, E);
}

// rows of op(X) are the columns of X (contiguous): one block per row
__global__ void k_oz_norm_cols(int64_t nrows, int64_t K, const double2* __restrict__ X, int64_t ldx, int E,
                               int* __restrict__ shift) {
  __shared__ double red[256];
  const int64_t r = blockIdx.x;
  const double2* x = X + r * ldx;
  double s = 0.0;
  for (int64_t k = threadIdx.x; k < K; k += blockDim.x) {
    const double2 v = x[k];
    s = fma(v.x, v.x, fma(v.y, v.y, s));
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (sum_in_range(red[0])) {
    if (threadIdx.x == 0) shift[r] = shift_for(red[0], E);
    return;
  }
  const int sh = column_shift_scaled(x, K, E);
  if (threadIdx.x == 0) shift[r] = sh;
}

// rows of op(X) are the rows of X (strided): 32 rows per block, eight threads per row
// summing every eighth column, their partial sums added in a fixed order
__global__ void __launch_bounds__(256) k_oz_norm_rows(int64_t nrows, int64_t K, const double2* __restrict__ X,
                                                      int64_t ldx, int E, int* __restrict__ shift) {
  __shared__ double part[8][33];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const int64_t r = (int64_t)blockIdx.x * 32 + tx;
  double s = 0.0;
  if (r < nrows) {
    for (int64_t k = ty; k < K; k += 8) {
      const double2 v = X[r + k * ldx];
      s = fma(v.x, v.x, fma(v.y, v.y, s));
    }
  }
  part[ty][tx] = s;
  __syncthreads();
  bool again = false;
  if (ty == 0 && r < nrows) {
    double t = part[0][tx];
#pragma unroll
    for (int j = 1; j < 8; ++j) t += part[j][tx];
    if (sum_in_range(t)) shift[r] = shift_for(t, E);
    else again = true;
  }
  if (!__syncthreads_or(again)) return;
  // a row of this block is out of range: all of them again
  __shared__ int pe[8][33];
  int e = 0;
  if (r < nrows)
    for (int64_t k = ty; k < K; k += 8) e = max(e, exponent_of(X[r + k * ldx]));
  pe[ty][tx] = e;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 8; ++j) e = max(e, pe[j][tx]);
  const double f = scale_of(e);
  s = 0.0;
  if (r < nrows)
    for (int64_t k = ty; k < K; k += 8) s = add_scaled(s, X[r + k * ldx], f);
  part[ty][tx] = s;
  __syncthreads();
  if (ty == 0 && r < nrows) {
#pragma unroll
    for (int j = 1; j < 8; ++j) s += part[j][tx];
    shift[r] = shift_scaled(e, s, E);
  }
}

// round(x 2^s) for |x 2^s| <= 2^62 by integer operations on the bits (ties to even)
__device__ __forceinline__ long long scaled_int(double x, int s) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF);
  if (e == 0 || e == 0x7FF) return 0;  // zero, subnormal (below 2^-1022: dropped), non-finite (flagged by the norm)
  const long long mant = (long long)((b & 0xFFFFFFFFFFFFFull) | (1ull << 52));
  const int sh = e - 1075 + s;  // x 2^s = mant 2^sh
  long long q;
  if (sh >= 0) {
    q = mant << min(sh, 10);
  } else if (sh < -63) {
    q = 0;
  } else {
    const int k = -sh;
    q = mant >> k;
    const unsigned long long rem = (unsigned long long)mant & ((1ull << k) - 1), half = 1ull << (k - 1);
    if (rem > half || (rem == half && (q & 1))) ++q;
  }
  return (b >> 63) ? -q : q;
}

// Symmetric residue of v modulo kMods[I] from its 19-bit limbs v = a 2^38 + b 2^19 + c
// (|v| <= 2^57; a signed, b and c unsigned): v is congruent to
//   x = a (2^38 mod m) + b (2^19 mod m) + c + (a multiple of m that makes it positive) < 2^30,
// and x - m floor((x + h) / m) with h = floor((m - 1) / 2) is its representative in
// [-h, m - 1 - h], within [-128, 128]: one 32-bit quotient by a constant per modulus.
template <int I> __device__ __forceinline__ int sres_limbs(int a, unsigned b, unsigned c) {
  constexpr unsigned m = (unsigned)kMods[I], h = (m - 1) / 2;
  constexpr unsigned c38 = (unsigned)((1ull << 38) % m), c19 = (unsigned)((1ull << 19) % m);
  constexpr unsigned up = (1u << 28) / m * m + m;  // >= |a| c38: |a| <= 2^19 + 1, c38 < 2^8
  const unsigned x = (unsigned)(a * (int)c38) + b * c19 + (c + up + h);
  return (int)(x % m) - (int)h;
}

// the 19-bit limbs of v, the highest one with its sign
struct Limbs {
  int a;
  unsigned b, c;
};
__device__ __forceinline__ Limbs limbs_of(long long v) {
  return Limbs{(int)(v >> 38), (unsigned)(v >> 19) & 0x7FFFFu, (unsigned)v & 0x7FFFFu};
}

// the float bits of a small integer (|n| < 2^22) without a conversion instruction: 1.5 2^23 + n
// has n in its low mantissa bits, and subtracting 1.5 2^23 is exact
__device__ __forceinline__ unsigned small_int_float_bits(int n) {
  return (unsigned)__float_as_int(__fsub_rn(__int_as_float(0x4B400000 + n), 12582912.0f));
}
// two residues (|r| <= 128, exact in bf16) as a bf16 pair: the high halves of their float bits
__device__ __forceinline__ unsigned bf16_pair(unsigned lo_bits, unsigned hi_bits) {
  return __byte_perm(lo_bits, hi_bits, 0x7632);
}

// Writes the residues of four consecutive complex entries a_e = op(X)[r][k + e] (after the
// optional conjugation) for moduli I.. into their planes (Re, Im, Re + Im), one modulus at a
// time so that no residue outlives its store.  o: entry k of row r in modulus I's first plane.
template <int I>
__device__ __forceinline__ void put_mods(const Limbs (&re)[4], const Limbs (&im)[4], int nmod, __nv_bfloat16* o,
                                         int64_t pstride) {
  if constexpr (I < kOzMaxMod) {
    if (I < nmod) {
      constexpr int m = kMods[I];
      unsigned fr[4], fi[4], fs[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = sres_limbs<I>(re[e].a, re[e].b, re[e].c);
        const int i = sres_limbs<I>(im[e].a, im[e].b, im[e].c);
        int s = r + i;  // |s| <= m: one correction gives a residue of magnitude <= m / 2
        if (s > m / 2) s -= m;
        else if (s < -(m / 2)) s += m;
        fr[e] = small_int_float_bits(r);
        fi[e] = small_int_float_bits(i);
        fs[e] = small_int_float_bits(s);
      }
      *reinterpret_cast<uint2*>(o) = make_uint2(bf16_pair(fr[0], fr[1]), bf16_pair(fr[2], fr[3]));
      *reinterpret_cast<uint2*>(o + pstride) = make_uint2(bf16_pair(fi[0], fi[1]), bf16_pair(fi[2], fi[3]));
      *reinterpret_cast<uint2*>(o + 2 * pstride) = make_uint2(bf16_pair(fs[0], fs[1]), bf16_pair(fs[2], fs[3]));
      put_mods<I + 1>(re, im, nmod, o + 3 * pstride, pstride);
    }
  }
}

// the residues of entries a[0..4) = op(X)[r][k..k+4) with row shift s; k is a multiple of 4
// and entries past K are zeros, so the 8-byte stores are aligned and end within the padded row
__device__ __forceinline__ void put_entries(const double2 (&a)[4], bool conj, int s, int nmod,
                                            __nv_bfloat16* __restrict__ out, int64_t pstride, int64_t ld, int64_t r,
                                            int64_t k) {
  Limbs re[4], im[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    re[e] = limbs_of(s == kOzBadShift ? 0ll : scaled_int(a[e].x, s));
    im[e] = limbs_of(s == kOzBadShift ? 0ll : scaled_int(conj ? -a[e].y : a[e].y, s));
  }
  put_mods<0>(re, im, nmod, out + r * ld + k, pstride);
}

// rows of op(X) = columns of X: grid (k blocks, rows); four consecutive entries per thread
// (ld and the plane stride are multiples of 8 bf16 values)
__global__ void __launch_bounds__(256) k_oz_res_cols(int64_t K, const double2* __restrict__ X, int64_t ldx,
                                                     const int* __restrict__ shift, int conj, int nmod,
                                                     __nv_bfloat16* __restrict__ out, int64_t pstride, int64_t ld) {
  const int64_t r = blockIdx.y;
  const int64_t k = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  if (k >= K) return;
  const double2* x = X + r * ldx + k;
  double2 a[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) a[e] = k + e < K ? x[e] : make_double2(0.0, 0.0);
  put_entries(a, conj != 0, shift[r], nmod, out, pstride, ld, r, k);
}

// The norm and the residues of a short row (a column of X, K <= 2048) in one block that holds
// it in registers, four entries a thread and group: one launch instead of two, which is what
// the small products of the projection space cost (256 x 256: 22 us, now 12 us).
template <int G>
__global__ void __launch_bounds__(256) k_oz_prep_cols(int64_t K, const double2* __restrict__ X, int64_t ldx, int E,
                                                      int* __restrict__ shift, int conj, int nmod,
                                                      __nv_bfloat16* __restrict__ out, int64_t pstride, int64_t ld) {
  __shared__ double red[8];
  __shared__ int s_shift;
  const int64_t r = blockIdx.x;
  const double2* x = X + r * ldx;
  const int tid = threadIdx.x, nt = blockDim.x;
  double2 a[G][4];
  double s = 0.0;
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t k = 4 * ((int64_t)g * nt + tid) + e;
      a[g][e] = k < K ? x[k] : make_double2(0.0, 0.0);
      s = fma(a[g][e].x, a[g][e].x, fma(a[g][e].y, a[g][e].y, s));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (tid % 32 == 0) red[tid / 32] = s;
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < nt / 32; ++i) s += red[i];
    s_shift = sum_in_range(s) ? shift_for(s, E) : kAgain;
  }
  __syncthreads();
  int sh = s_shift;
  if (sh == kAgain) sh = column_shift_scaled(x, K, E);
  if (tid == 0) shift[r] = sh;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int64_t k = 4 * ((int64_t)g * nt + tid);
    if (k < K) put_entries(a[g], conj != 0, sh, nmod, out, pstride, ld, r, k);
  }
}

// rows of op(X) = rows of X: 32-row x 64-k tiles through shared memory so that both the
// reads (along rows of X) and the writes (along k, four entries per thread) are coalesced
__global__ void __launch_bounds__(256) k_oz_res_rows(int64_t nrows, int64_t K, const double2* __restrict__ X,
                                                     int64_t ldx, const int* __restrict__ shift, int conj, int nmod,
                                                     __nv_bfloat16* __restrict__ out, int64_t pstride, int64_t ld) {
  __shared__ double2 t[32][65];  // [row][k], odd pitch
  const int64_t r0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 64;
  {
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;  // 256 threads: 8 rows of 32
    for (int j = ty; j < 64; j += 8) {
      const int64_t r = r0 + tx, k = k0 + j;
      t[tx][j] = (r < nrows && k < K) ? X[r + k * ldx] : make_double2(0.0, 0.0);
    }
  }
  __syncthreads();
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  for (int j = ty; j < 32; j += 16) {
    const int64_t r = r0 + j, k = k0 + 4 * tx;
    if (r >= nrows || k >= K) continue;
    const double2 a[4] = {t[j][4 * tx], t[j][4 * tx + 1], t[j][4 * tx + 2], t[j][4 * tx + 3]};
    put_entries(a, conj != 0, shift[r], nmod, out, pstride, ld, r, k);
  }
}

// ---------------------------------------------------------------- reconstruction
struct CrtArgs {
  int nmod;
  float m[kOzMaxMod], inv[kOzMaxMod], y[kOzMaxMod];  // y_i = (M / m_i)^-1 mod m_i
  int L[kOzMaxMod][4];                               // M / m_i in 30-bit limbs, least significant first
  int ML[4];                                         // M in 30-bit limbs
};

// M < 2^120 for every modulus count: four 30-bit limbs hold M and each M / m_i
constexpr bool mods_fit_limbs() {
  unsigned __int128 M = 1;
  for (int i = 0; i < kOzMaxMod; ++i) M *= (unsigned)kMods[i];
  return (M >> 120) == 0;
}
static_assert(mods_fit_limbs(), "CRT modulus too large for four 30-bit limbs");

// 1.5 2^23: for |x| < 2^22, x + kMagic rounds x to an integer held in the low mantissa bits
constexpr float kMagic = 12582912.0f;

// one modulus' term of the CRT sum for r (|r| <= 3 128 16, a sum of residues): t = r y_i
// mod m_i (symmetric, exact in float), its share t / m_i of S / M added to f.  The float conversions go through kMagic
// (one integer and one float addition each) instead of conversion instructions.
__device__ __forceinline__ int crt_term(int r, float y, float m, float inv, float& f) {
  const float p = __fmul_rn(__fsub_rn(__int_as_float(0x4B400000 + r), kMagic), y);  // r y, exact (< 2^21)
  const float q = __fsub_rn(__fmaf_rn(p, inv, kMagic), kMagic);                     // round(p / m_i)
  const float t = __fmaf_rn(-m, q, p);                                               // exact, |t| <= m_i / 2 + 1
  f = __fmaf_rn(t, inv, f);
  return __float_as_int(__fadd_rn(t, kMagic)) - 0x4B400000;
}

// sum_j a_j 2^(30 j) in 128-bit two's complement (the true sum fits)
__device__ __forceinline__ __int128 limb_sum(const long long (&a)[4]) {
  using u128 = unsigned __int128;
  const u128 u = (u128)(__int128)a[0] + ((u128)(__int128)a[1] << 30) + ((u128)(__int128)a[2] << 60) +
                 ((u128)(__int128)a[3] << 90);
  return (__int128)u;
}

// C_int of Re and Im from the residues t1, t2, t3 of the three products: Re = T1 - T2 and
// Im = T3 - T1 - T2 modulo each m_i, t_i = r_i y_i mod m_i, S = sum t_i (M / m_i) = C_int
// (mod M), and C_int = S - M round(S / M) with S / M = sum t_i / m_i (FP32 suffices:
// |C_int| <= M / 8 keeps S / M at least 3/8 away from a half-integer).  The products
// t_i (M / m_i) accumulate per 30-bit limb of M / m_i in 64-bit integers (one 32 x 32 ->
// 64-bit multiply-add each, sums below 2^43), combined once into 128 bits: exact.
struct CrtSum {
  long long a0[4] = {0, 0, 0, 0}, a1[4] = {0, 0, 0, 0};
  float f0 = 0.f, f1 = 0.f;
  __device__ __forceinline__ void add(int i, int t1, int t2, int t3, const CrtArgs& c) {
    const int u0 = crt_term(t1 - t2, c.y[i], c.m[i], c.inv[i], f0);
    const int u1 = crt_term(t3 - t1 - t2, c.y[i], c.m[i], c.inv[i], f1);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      a0[j] += (long long)u0 * (long long)c.L[i][j];
      a1[j] += (long long)u1 * (long long)c.L[i][j];
    }
  }
  __device__ __forceinline__ void finish(const CrtArgs& c, __int128& S0, __int128& S1) {
    const int k0 = __float_as_int(__fadd_rn(f0, kMagic)) - 0x4B400000;
    const int k1 = __float_as_int(__fadd_rn(f1, kMagic)) - 0x4B400000;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      a0[j] -= (long long)k0 * (long long)c.ML[j];
      a1[j] -= (long long)k1 * (long long)c.ML[j];
    }
    S0 = limb_sum(a0);
    S1 = limb_sum(a1);
  }
};

// S 2^-sh as the nearest double (ties to even), by integer operations on the bits: GB300's
// FP64 pipe is its slowest, and a conversion plus a scaling there per value bound this
// kernel.  Results outside the normal range go through ldexp.
__device__ __forceinline__ double scaled_double(__int128 S, int sh) {
  if (S == 0) return 0.0;
  const bool neg = S < 0;
  unsigned __int128 u = neg ? (unsigned __int128)(-S) : (unsigned __int128)S;
  const unsigned long long h = (unsigned long long)(u >> 64), l = (unsigned long long)u;
  const int lz = h ? __clzll((long long)h) : 64 + __clzll((long long)l);
  u <<= lz;  // leading one at bit 127
  const unsigned long long top = (unsigned long long)(u >> 64), rest = (unsigned long long)u;
  unsigned long long mant = top >> 11;  // 53 bits, bit 52 set
  const unsigned long long rb = top & 0x7FFull;
  if (rb > 0x400ull || (rb == 0x400ull && (rest != 0 || (mant & 1ull)))) ++mant;
  int e = 127 - lz;
  if (mant >> 53) {
    mant >>= 1;
    ++e;
  }
  e -= sh;
  if (e < -1022 || e > 1023) {  // subnormal or overflow: the library's ldexp
    const double v = __longlong_as_double((long long)((1023ull << 52) | (mant & ((1ull << 52) - 1))));
    return ldexp(neg ? -v : v, e);
  }
  const unsigned long long bits =
      ((unsigned long long)neg << 63) | ((unsigned long long)(e + 1023) << 52) | (mant & ((1ull << 52) - 1));
  return __longlong_as_double((long long)bits);
}

// C[m, n] = alpha 2^-(s1 + s2) C_int + beta C[m, n]
__device__ __forceinline__ void put_entry(__int128 S0, __int128 S1, int s1, int s2, double alpha, double beta,
                                          double2* c) {
  double re, im;
  if (s1 == kOzBadShift || s2 == kOzBadShift) {
    re = im = __longlong_as_double(0x7FF8000000000000ll);
  } else {
    re = scaled_double(S0, s1 + s2);
    im = scaled_double(S1, s1 + s2);
  }
  double2 v = alpha == 1.0 ? make_double2(re, im) : make_double2(alpha * re, alpha * im);
  if (beta != 0.0) {
    const double2 o = *c;
    v.x = fma(beta, o.x, v.x);
    v.y = fma(beta, o.y, v.y);
  }
  *c = v;
}

struct ReconArgs {
  int64_t M, N, M4;  // M4 = ceil(M / 4)
  const signed char* R;
  int64_t ldr, rstride;
  const int *sa, *sb;
  double alpha, beta;
  double2* C;
  int64_t ldc;
  int lower, splits;
};

// One thread per four consecutive rows of a column: four residues per 4-byte load, all 3 NM
// loads in flight (NM = crt.nmod, a compile-time count).
template <int NM>
__global__ void __launch_bounds__(128) k_oz_recon(const __grid_constant__ ReconArgs a, const __grid_constant__ CrtArgs crt) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = idx / a.M4, m0 = 4 * (idx - n * a.M4);
  if (n >= a.N || (a.lower && m0 + 3 < n)) return;
  const signed char* r = a.R + n * a.ldr + m0;
  unsigned v[3 * NM];
#pragma unroll
  for (int i = 0; i < 3 * NM; ++i) v[i] = *reinterpret_cast<const unsigned*>(r + i * a.rstride);
  const int s2 = a.sb[n];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int64_t m = m0 + e;
    if (m >= a.M || (a.lower && m < n)) continue;
    CrtSum s;
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      const int t1 = (int)(signed char)(v[3 * i] >> (8 * e)), t2 = (int)(signed char)(v[3 * i + 1] >> (8 * e)),
                t3 = (int)(signed char)(v[3 * i + 2] >> (8 * e));
      s.add(i, t1, t2, t3, crt);
    }
    __int128 S0, S1;
    s.finish(crt, S0, S1);
    put_entry(S0, S1, a.sa[m], s2, a.alpha, a.beta, a.C + m + n * a.ldc);
  }
}

// the same for K-split products (few outputs): one thread per entry, its residues added over
// the splits first
template <int NM>
__global__ void __launch_bounds__(128) k_oz_recon_split(const __grid_constant__ ReconArgs a,
                                                        const __grid_constant__ CrtArgs crt) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = idx / a.M, m = idx - n * a.M;
  if (n >= a.N || (a.lower && m < n)) return;
  const signed char* r = a.R + n * a.ldr + m;
  CrtSum s;
#pragma unroll
  for (int i = 0; i < NM; ++i) {
    int t1 = 0, t2 = 0, t3 = 0;
    for (int z = 0; z < a.splits; ++z) {
      const signed char* p = r + (int64_t)(z * 3 * NM + 3 * i) * a.rstride;
      t1 += p[0];
      t2 += p[a.rstride];
      t3 += p[2 * a.rstride];
    }
    s.add(i, t1, t2, t3, crt);
  }
  __int128 S0, S1;
  s.finish(crt, S0, S1);
  put_entry(S0, S1, a.sa[m], a.sb[n], a.alpha, a.beta, a.C + m + n * a.ldc);
}

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

// 3-D bf16 map over the residue planes [3 nmod][rows][ld], boxes of 64 x box_rows x 1, 128-byte swizzle
CUtensorMap make_map3(const OzOperand& o, int box_rows) {
  CHEBFI_REQUIRE(o.ld % 8 == 0 && o.pstride % 8 == 0 && (reinterpret_cast<uintptr_t>(o.res.p) % 16) == 0,
                 CHEBFI_ERR_ARG, "residue operand must be 16-byte aligned with strides multiple of 8 elements");
  CUtensorMap mp;
  cuuint64_t dims[3] = {(cuuint64_t)o.K, (cuuint64_t)o.rows, (cuuint64_t)(3 * o.nmod)};
  cuuint64_t strides[2] = {(cuuint64_t)(o.ld * 2), (cuuint64_t)(o.pstride * 2)};
  cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = tc::encode_fn()(&mp, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)o.res.p, dims, strides, box, estr,
                               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  CHEBFI_REQUIRE(r == CUDA_SUCCESS, CHEBFI_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return mp;
}

struct ModSet {
  int n = 0, E = 0;
  CrtArgs crt;
};

// moduli, E and the CRT constants of the first n moduli (host, 128-bit arithmetic)
ModSet make_modset(int n) {
  ModSet s{};
  unsigned __int128 M = 1;
  double l2 = 0.0;
  for (int i = 0; i < n; ++i) {
    M *= (unsigned)kMods[i];
    l2 += std::log2((double)kMods[i]);
  }
  s.crt.nmod = n;
  for (int i = 0; i < n; ++i) {
    const int m = kMods[i];
    const unsigned __int128 Mi = M / (unsigned)m;
    const int a = (int)(Mi % (unsigned)m);
    int y = 1;
    while ((a * y) % m != 1) ++y;  // m <= 256: direct search of the inverse
    s.crt.m[i] = (float)m;
    s.crt.inv[i] = 1.0f / (float)m;
    s.crt.y[i] = (float)y;
    for (int j = 0; j < 4; ++j) s.crt.L[i][j] = (int)((Mi >> (30 * j)) & ((1u << 30) - 1));
  }
  for (int j = 0; j < 4; ++j) s.crt.ML[j] = (int)((M >> (30 * j)) & ((1u << 30) - 1));
  s.E = std::min(62, (int)std::floor((l2 - 3.0) / 2.0));
  s.n = n;
  return s;
}
// built once, whichever thread comes first
const ModSet& modset(int n) {
  static const std::vector<ModSet> sets = [] {
    std::vector<ModSet> v(kOzMaxMod + 1);
    for (int k = kOzMinMod; k <= kOzMaxMod; ++k) v[k] = make_modset(k);
    return v;
  }();
  return sets[n];
}

}  // namespace oz

int oz_precision_bits(int nmod) {
  CHEBFI_REQUIRE(nmod >= kOzMinMod && nmod <= kOzMaxMod, CHEBFI_ERR_ARG, "modulus count out of range");
  return oz::modset(nmod).E;
}

void oz_prepare(const double2* X, int64_t ldx, int64_t nrows, int64_t K, bool rows_are_columns, bool conj, int nmod,
                OzOperand& out, cudaStream_t st) {
  const oz::ModSet& ms = oz::modset(nmod);
  out.nmod = 0;  // not prepared until the last launch: a failed allocation must not leave it marked
  out.rows = nrows;
  out.K = K;
  out.ld = (K + 7) / 8 * 8;
  out.pstride = out.rows * out.ld;
  out.res.alloc((size_t)3 * nmod * out.pstride);
  out.shift.alloc((size_t)std::max<int64_t>(nrows, 1));
  if (nrows == 0 || K == 0) {
    out.nmod = nmod;
    return;
  }
  if (rows_are_columns && K <= 2048) {
    const int nt = (int)std::min<int64_t>(256, (K + 127) / 128 * 32);
    auto prep = [&](auto kernel) {
      CHEBFI_LAUNCH("k_oz_res", st, kernel<<<(unsigned)nrows, nt, 0, st>>>(K, X, ldx, ms.E, out.shift.p, conj ? 1 : 0, nmod,
                                                                          out.res.p, out.pstride, out.ld));
    };
    if (K <= 1024) prep(oz::k_oz_prep_cols<1>);
    else prep(oz::k_oz_prep_cols<2>);
  } else if (rows_are_columns) {
    CHEBFI_LAUNCH("k_oz_norm", st, oz::k_oz_norm_cols<<<(unsigned)nrows, 256, 0, st>>>(nrows, K, X, ldx, ms.E, out.shift.p));
    const unsigned kb = (unsigned)((K + 1023) / 1024);  // four entries per thread
    CHEBFI_REQUIRE(nrows <= 65535, CHEBFI_ERR_ARG, "too many rows for the residue kernel");
    CHEBFI_LAUNCH("k_oz_res", st,
                  oz::k_oz_res_cols<<<dim3(kb, (unsigned)nrows), 256, 0, st>>>(K, X, ldx, out.shift.p, conj ? 1 : 0,
                                                                               nmod, out.res.p, out.pstride, out.ld));
  } else {
    CHEBFI_LAUNCH("k_oz_norm", st, oz::k_oz_norm_rows<<<oz::nblk(nrows, 32), 256, 0, st>>>(nrows, K, X, ldx, ms.E, out.shift.p));
    CHEBFI_REQUIRE((K + 63) / 64 <= 65535, CHEBFI_ERR_ARG, "inner dimension too large for the residue kernel");
    CHEBFI_LAUNCH("k_oz_res", st,
                  oz::k_oz_res_rows<<<dim3((unsigned)((nrows + 31) / 32), (unsigned)((K + 63) / 64)), 256, 0, st>>>(
                      nrows, K, X, ldx, out.shift.p, conj ? 1 : 0, nmod, out.res.p, out.pstride, out.ld));
  }
  out.nmod = nmod;
}

namespace {
// The product's GEMM with BN output columns per CTA pair.
template <int BN>
void oz_gemm_bn(const OzOperand& A, const OzOperand& B, oz::GemmArgs& a, DevBuf<signed char>& R, int pairs,
                cudaStream_t st) {
  const int nplanes = a.nplanes;
  a.tiles_m = (a.M + oz::BM - 1) / oz::BM;
  a.tiles_n = (a.N + BN - 1) / BN;
  int64_t tiles = (int64_t)a.tiles_m * a.tiles_n;
  if (a.lower) {
    tiles = 0;
    for (int tm = 0; tm < a.tiles_m; ++tm) tiles += oz::lower_count(tm, BN, a.tiles_n);
  }
  CHEBFI_REQUIRE(tiles * nplanes * oz::kMaxSplit < (1ll << 31), CHEBFI_ERR_ARG, "GEMM too large");
  a.tiles = (int)tiles;
  // K ranges: the split with the fewest chunk steps on the busiest pair, when the units of one
  // range leave pairs idle; every range costs about one more chunk (fill, drain, its residues)
  const int chunks = (a.num_k + oz::CHUNK - 1) / oz::CHUNK;
  const int64_t units1 = tiles * nplanes;
  int best = 1;
  if (units1 < 4 * pairs) {
    int64_t cost1 = 0;
    for (int s = 1; s <= std::min(oz::kMaxSplit, chunks); ++s) {
      const int per = (chunks + s - 1) / s;
      const int64_t cost = (units1 * s + pairs - 1) / pairs * (per + 1);
      if (s == 1 || cost < cost1) {
        cost1 = cost;
        best = s;
      }
    }
  }
  a.kt_split = (chunks + best - 1) / best * oz::CHUNK;
  a.splits = std::max(1, (a.num_k + a.kt_split - 1) / a.kt_split);
  a.ldr = ((int64_t)a.M + 31) / 32 * 32;
  a.rstride = a.ldr * a.N;
  R.alloc((size_t)a.splits * nplanes * a.rstride);
  a.R = R.p;
  const CUtensorMap ta = oz::make_map3(A, 128), tb = oz::make_map3(B, BN / 2);
  CHEBFI_CUDA(cudaFuncSetAttribute(oz::k_oz_gemm<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::smem_bytes<BN>()));
  const unsigned blocks = 2 * (unsigned)std::min<int64_t>(units1 * a.splits, pairs);
  // recorded work: the FP64 product's algorithmic flops (8 M N K complex); the tensor pipe
  // executes 3/4 nmod times as many (three bf16 GEMMs per modulus for four real products)
  const double tiles_done = (double)tiles / ((double)a.tiles_m * a.tiles_n);
  CHEBFI_LAUNCH_W("k_oz_gemm", st, 8.0 * (double)a.M * (double)a.N * (double)A.K * tiles_done,
                  oz::k_oz_gemm<BN><<<blocks, oz::THREADS, oz::smem_bytes<BN>(), st>>>(ta, tb, a));
}
}  // namespace

void oz_gemm(const OzOperand& A, const OzOperand& B, double alpha, double beta, double2* C, int64_t ldc, bool lower,
             DevBuf<signed char>& R, int* status, cudaStream_t st, const char* tag) {
  const int64_t M = A.rows, N = B.rows;
  if (M <= 0 || N <= 0) return;
  CHEBFI_REQUIRE(A.K == B.K && A.nmod == B.nmod, CHEBFI_ERR_ARG, "modular GEMM operands do not match");
  CHEBFI_REQUIRE(!lower || M == N, CHEBFI_ERR_ARG, "lower-triangle GEMM needs a square result");
  CHEBFI_REQUIRE(M < (1ll << 30) && N < (1ll << 30) && A.K < (1ll << 30), CHEBFI_ERR_ARG, "GEMM too large");
  const int nmod = A.nmod;
  const oz::ModSet& ms = oz::modset(nmod);
  oz::GemmArgs a;
  a.M = (int)M;
  a.N = (int)N;
  a.num_k = (int)((A.K + oz::BK - 1) / oz::BK);
  a.nplanes = 3 * nmod;
  a.lower = lower ? 1 : 0;
  a.status = status;
  for (int i = 0; i < kOzMaxMod; ++i) {
    a.m[i] = ms.crt.m[i];
    a.inv[i] = ms.crt.inv[i];
  }
  int dev = 0, sms = 0;
  CHEBFI_CUDA(cudaGetDevice(&dev));
  CHEBFI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int pairs = std::max(1, sms / 2);
  (void)tag;  // every modular GEMM is timed under one name, so its engine is unambiguous
  if (N <= 128) oz_gemm_bn<128>(A, B, a, R, pairs, st);
  else oz_gemm_bn<256>(A, B, a, R, pairs, st);
  oz::ReconArgs ra;
  ra.M = M;
  ra.N = N;
  ra.M4 = (M + 3) / 4;
  ra.R = R.p;
  ra.ldr = a.ldr;
  ra.rstride = a.rstride;
  ra.sa = A.shift.p;
  ra.sb = B.shift.p;
  ra.alpha = alpha;
  ra.beta = beta;
  ra.C = C;
  ra.ldc = ldc;
  ra.lower = lower ? 1 : 0;
  ra.splits = a.splits;
  const int64_t threads = (a.splits > 1 ? M : ra.M4) * N;
  CHEBFI_REQUIRE((threads + 127) / 128 < (1ll << 31), CHEBFI_ERR_ARG, "GEMM too large");
  auto recon = [&](auto whole, auto split) {
    CHEBFI_LAUNCH("k_oz_recon", st, (a.splits > 1 ? split : whole)<<<oz::nblk(threads, 128), 128, 0, st>>>(ra, ms.crt));
  };
  static_assert(kOzMinMod == 8 && kOzMaxMod == 15, "one reconstruction kernel per modulus count");
  switch (nmod) {
    case 8: recon(oz::k_oz_recon<8>, oz::k_oz_recon_split<8>); break;
    case 9: recon(oz::k_oz_recon<9>, oz::k_oz_recon_split<9>); break;
    case 10: recon(oz::k_oz_recon<10>, oz::k_oz_recon_split<10>); break;
    case 11: recon(oz::k_oz_recon<11>, oz::k_oz_recon_split<11>); break;
    case 12: recon(oz::k_oz_recon<12>, oz::k_oz_recon_split<12>); break;
    case 13: recon(oz::k_oz_recon<13>, oz::k_oz_recon_split<13>); break;
    case 14: recon(oz::k_oz_recon<14>, oz::k_oz_recon_split<14>); break;
    default: recon(oz::k_oz_recon<15>, oz::k_oz_recon_split<15>); break;
  }
}

}  // namespace chebfi
