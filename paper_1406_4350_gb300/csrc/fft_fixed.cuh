// The plane pass of the FP64 form in 64-bit fixed point.
//
// GB300 issues FP64 FMAs at 1/64 of its FP32 rate; double-float sums (11 packed FP32
// instructions per complex sum) bound the plane pass instead.  A complex sum of 64-bit
// integers is four integer instructions, and a transform is mostly sums.  So the planes are
// transformed as integers with one power-of-two scale per plane (block floating point):
//
//  * a component is an integer below 2^61.5 in magnitude.  Every intermediate value of an
//    unnormalised transform is a sum of inputs with unit weights, so the sum of the inputs'
//    magnitudes bounds them all: the inverse transforms' scale makes sum |c| <= 2^61;
//  * products with constants |c| <= 1 (twiddles, V_loc / 2^e) keep 62-bit constants as two
//    31-bit parts, c = (h 2^31 + l) 2^-62, and give x c / 2 from three 32 x 32 -> 64-bit
//    multiply-adds per real product: with x = xh 2^32 + 2 xm (+ the dropped lowest bit),
//      x c / 2 = xh h + (xh l + xm h) 2^-31, rounded.
//    The halving at each twiddle is headroom that the sums after it use;
//  * before the forward x and y transforms the plane's largest component, taken while the
//    plane is stored, sets a new common shift, so the forward passes also start with their
//    full word length, whatever V_loc's range;
//  * sums that could pass the word length shift their inputs first, by compile-time amounts.
//
// Against the double-float planes: rounding is 1 part in 2^61 of the plane's scale instead of
// 2^-48 of each value.  A complex sum issues in 5 clocks per warp and scheduler (double-float:
// 24), a twiddle product in 87 (55), so the pass is now bound by its products; per
// 256-band application at 48^3 0.86 -> 0.60 ms, per 2048 at 96^3 48.5 -> 41 ms.
// Against FP64 planes (lengths with FP64 z passes, normalised planes below), per 512 bands:
// 36^3 2.27 -> 0.57 ms, 60^3 12.5 -> 3.1 ms, 54^3 9.7 -> 2.3 ms; 108^3, 256 bands 42 -> 10 ms.
#pragma once

#include <cmath>
#include <type_traits>

#include "dfloat.cuh"
#include "fft_fast.cuh"
#include "fft_fast_kernels.cuh"

namespace chebfi {
namespace fx {

using ll = long long;
struct cfx {
  ll x, y;
};

// c = (h 2^31 + l) 2^-62, |c| <= 1 (1 itself as the largest representable value)
struct Cst {
  int h, l;
};
// c + c2: a constant as its double and the rest (a double alone is off by up to 2^-54, more than
// the transforms round)
__host__ __device__ constexpr Cst make_cst(double c, double c2) {
  const double s = c * 2147483648.0;
  ll h = (ll)(s + (s >= 0 ? 0.5 : -0.5));
  if (h > 2147483647) h = 2147483647;
  if (h < -2147483647) h = -2147483647;
  const double r = (s - (double)h) * 2147483648.0 + c2 * 4611686018427387904.0;
  ll l = (ll)(r + (r >= 0 ? 0.5 : -0.5));
  if (l > 2147483647) l = 2147483647;
  if (l < -2147483647) l = -2147483647;
  return Cst{(int)h, (int)l};
}

__device__ __forceinline__ int hi32(ll v) { return (int)(v >> 32); }
__device__ __forceinline__ int mid31(ll v) { return (int)((unsigned)v >> 1); }
__device__ __forceinline__ ll mad(int a, int b, ll c) { return (ll)a * (ll)b + c; }
constexpr ll kHalfUlp = 1ll << 30;

// x c / 2
__device__ __forceinline__ ll mulh(ll x, Cst c) {
  ll u = mad(hi32(x), c.l, kHalfUlp);
  u = mad(mid31(x), c.h, u);
  return mad(hi32(x), c.h, u >> 31);
}
__device__ __forceinline__ cfx operator+(cfx a, cfx b) { return cfx{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cfx operator-(cfx a, cfx b) { return cfx{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cfx sar(cfx a, int s) { return cfx{a.x >> s, a.y >> s}; }
// a (c + i s) / 2: the two products of a component share their carry chain (|c| + |s| <= sqrt 2)
__device__ __forceinline__ cfx cmulh(cfx a, Cst c, Cst s) {
  const int xh = hi32(a.x), xm = mid31(a.x), yh = hi32(a.y), ym = mid31(a.y);
  ll u = mad(xh, c.l, kHalfUlp), v = mad(xh, s.l, kHalfUlp);
  u = mad(xm, c.h, u);
  v = mad(xm, s.h, v);
  u = mad(yh, -s.l, u);
  v = mad(yh, c.l, v);
  u = mad(ym, -s.h, u);
  v = mad(ym, c.h, v);
  cfx r;
  r.x = mad(yh, -s.h, mad(xh, c.h, u >> 31));
  r.y = mad(yh, c.h, mad(xh, s.h, v >> 31));
  return r;
}
// SIGN i a
template <int SIGN> __device__ __forceinline__ cfx rot(cfx a) { return SIGN > 0 ? cfx{-a.y, a.x} : cfx{a.y, -a.x}; }

// In-register transforms, natural order in and out (fast::dft on integers).
template <int L, int SIGN> __device__ __forceinline__ void dft(cfx* x) {
  if constexpr (L == 1) {
  } else if constexpr (L == 2) {
    const cfx a = x[0], b = x[1];
    x[0] = a + b;
    x[1] = a - b;
  } else if constexpr (L == 3) {
    constexpr Cst h = make_cst(0.86602540378443864676, 5.0175421109034514e-17);
    const cfx s = x[1] + x[2], d = x[1] - x[2];
    const cfx t = x[0] - sar(s, 1);
    cfx u{mulh(d.y, h), mulh(d.x, h)};  // half of sqrt(3)/2 (d.y, d.x)
    u = cfx{u.x + u.x, u.y + u.y};
    x[0] = x[0] + s;
    if (SIGN > 0) {
      x[1] = cfx{t.x - u.x, t.y + u.y};
      x[2] = cfx{t.x + u.x, t.y - u.y};
    } else {
      x[1] = cfx{t.x + u.x, t.y - u.y};
      x[2] = cfx{t.x - u.x, t.y + u.y};
    }
  } else if constexpr (L == 4) {
    const cfx a = x[0] + x[2], b = x[0] - x[2], c = x[1] + x[3], d = x[1] - x[3];
    x[0] = a + c;
    x[2] = a - c;
    if (SIGN > 0) {
      x[1] = cfx{b.x - d.y, b.y + d.x};
      x[3] = cfx{b.x + d.y, b.y - d.x};
    } else {
      x[1] = cfx{b.x + d.y, b.y - d.x};
      x[3] = cfx{b.x - d.y, b.y + d.x};
    }
  } else if constexpr (L == 5) {
    // cosine parts x0 - (a + b) / 4 +- sqrt(5)/4 (a - b), sine parts s1 c + s2 d and
    // s2 c - s1 d (s1, s2 = sin(2 pi / 5), sin(4 pi / 5)) from three products
    constexpr Cst g = make_cst(0.55901699437494742410, -2.716057601841253e-17);
    constexpr Cst s1 = make_cst(0.95105651629515357212, 4.0934500900087295e-17);
    constexpr Cst dif = make_cst(0.36327126400268044295, -6.641899492980514e-18);  // s1 - s2
    constexpr Cst sum1 = make_cst(0.53884176858762670129, 3.299975006189727e-17);  // s1 + s2 - 1
    const cfx a = x[1] + x[4], b = x[2] + x[3], c = x[1] - x[4], d = x[2] - x[3];
    const cfx r = a + b, q = a - b, e = c + d;
    const cfx m = x[0] - sar(r, 2), qh{mulh(q.x, g), mulh(q.y, g)}, eh{mulh(e.x, s1), mulh(e.y, s1)};
    const cfx t = qh + qh, t1 = m + t, t2 = m - t;
    const cfx uh = eh - cfx{mulh(d.x, dif), mulh(d.y, dif)}, vh = cfx{mulh(c.x, sum1), mulh(c.y, sum1)} - eh;
    const cfx u = rot<SIGN>(uh + uh), v = rot<SIGN>(vh + vh + c);
    x[0] = x[0] + r;
    x[1] = t1 + u;
    x[4] = t1 - u;
    x[2] = t2 + v;
    x[3] = t2 - v;
  } else if constexpr (L == 9) {
    constexpr Cst c1 = make_cst(0.76604444311897803520, 2.1750711742081045e-17);
    constexpr Cst s1 = make_cst(SIGN * 0.64278760968653932632, SIGN * -3.659607900790949e-17);
    constexpr Cst c2 = make_cst(0.17364817766693034885, -1.0090493350843633e-17);
    constexpr Cst s2 = make_cst(SIGN * 0.98480775301220805937, SIGN * 3.905108875799298e-17);
    constexpr Cst c4 = make_cst(-0.93969262078590838405, 4.3850932840020416e-17);
    constexpr Cst s4 = make_cst(SIGN * 0.34202014332566873304, SIGN * 2.0136016534644645e-17);
    cfx y[9];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      cfx t[3] = {x[n], x[3 + n], x[6 + n]};
      dft<3, SIGN>(t);
#pragma unroll
      for (int k = 0; k < 3; ++k) y[3 * k + n] = t[k];
    }
    y[4] = cmulh(y[4], c1, s1);
    y[5] = cmulh(y[5], c2, s2);
    y[7] = cmulh(y[7], c2, s2);
    y[8] = cmulh(y[8], c4, s4);
    y[4] = y[4] + y[4];
    y[5] = y[5] + y[5];
    y[7] = y[7] + y[7];
    y[8] = y[8] + y[8];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      dft<3, SIGN>(y + 3 * k);
#pragma unroll
      for (int n = 0; n < 3; ++n) x[k + 3 * n] = y[3 * k + n];
    }
  } else if constexpr (L == 8) {
    constexpr Cst h = make_cst(0.70710678118654752440, -4.833646656726457e-17);
    cfx e[4], o[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      e[n] = x[n] + x[n + 4];
      o[n] = x[n] - x[n + 4];
    }
    // o[1] w, o[3] w^3, w = exp(SIGN i pi / 4): (1 + SIGN i) / sqrt 2 and (-1 + SIGN i) / sqrt 2
    const cfx p = o[1] + rot<SIGN>(o[1]), q = rot<SIGN>(o[3]) - o[3];
    const cfx ph{mulh(p.x, h), mulh(p.y, h)}, qh{mulh(q.x, h), mulh(q.y, h)};
    o[1] = cfx{ph.x + ph.x, ph.y + ph.y};
    o[2] = rot<SIGN>(o[2]);
    o[3] = cfx{qh.x + qh.x, qh.y + qh.y};
    dft<4, SIGN>(e);
    dft<4, SIGN>(o);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[2 * k] = e[k];
      x[2 * k + 1] = o[k];
    }
  } else {
    constexpr int A = fast::Split<L>::A, B = fast::Split<L>::B;
    static_assert(fast::gcd(A, B) == 1, "coprime factors only");
    constexpr int ea = B * fast::inv_mod(B % A, A), eb = A * fast::inv_mod(A % B, B);
    cfx y[L];
#pragma unroll
    for (int nb = 0; nb < B; ++nb) {
      cfx t[A];
#pragma unroll
      for (int na = 0; na < A; ++na) t[na] = x[(B * na + A * nb) % L];
      dft<A, SIGN>(t);
#pragma unroll
      for (int ka = 0; ka < A; ++ka) y[ka * B + nb] = t[ka];
    }
#pragma unroll
    for (int ka = 0; ka < A; ++ka) {
      dft<B, SIGN>(y + ka * B);
#pragma unroll
      for (int kb = 0; kb < B; ++kb) x[(ea * ka + eb * kb) % L] = y[ka * B + kb];
    }
  }
}

// upper bounds of 8 log2 n, the bits by which an n-point transform can grow
constexpr int grow8(int n) {
  return n <= 1 ? 0 : n == 2 ? 8 : n == 3 ? 13 : n == 4 ? 16 : n == 5 ? 19 : n == 6 ? 21 : n <= 8 ? 24 : n <= 9 ? 26 : n <= 10 ? 27 : n <= 12 ? 29 : 32;
}
constexpr int kTop8 = 8 * 61 + 4;  // magnitudes stay below 2^61.5
// shift before an n-point transform of values below 2^(b8 / 8), and the bound after it
constexpr int pre_shift(int b8, int n) {
  int s = 0;
  while (b8 - 8 * s + grow8(n) > kTop8) ++s;
  return s;
}
// bits that an n-point transform's inputs may have
constexpr int pass_bits(int n) { return (kTop8 - grow8(n)) / 8; }
constexpr int after(int b8, int n) { return b8 - 8 * pre_shift(b8, n) + grow8(n); }

// Twiddles (cos, -sin)(2 pi e / N) of the compiled lengths as (c.h, c.l, s.h, s.l); filled as
// the other passes' tables are (fft_fast_kernels.cuh).
static __constant__ int4 c_twfx[fk::kTwTotal];
template <int N, int SIGN> __device__ __forceinline__ void twiddle(int e, Cst& c, Cst& s) {
  const int4 w = c_twfx[fk::TwOff<N>::v + e];
  c = Cst{w.x, w.y};
  s = SIGN > 0 ? Cst{-w.z, -w.w} : Cst{w.z, w.w};
}
static inline void fill_twiddles() {
  std::vector<int4> t;
  for (int n : fk::kTwLens)
    for (int k = 0; k < n; ++k) {
      const long double a = 2.0L * 3.14159265358979323846264338327950288L * k / n;
      // the two parts from the extended-precision value: 62 bits
      auto part = [](long double v) {
        const long double s = v * 2147483648.0L;
        ll h = std::llround(s);
        h = std::max(-2147483647ll, std::min(2147483647ll, h));
        ll l = std::llround((s - (long double)h) * 2147483648.0L);
        l = std::max(-2147483647ll, std::min(2147483647ll, l));
        return std::make_pair((int)h, (int)l);
      };
      const auto c = part(std::cos(a)), s = part(-std::sin(a));
      t.push_back(make_int4(c.first, c.second, s.first, s.second));
    }
  CHEBFI_CUDA(cudaMemcpyToSymbol(c_twfx, t.data(), sizeof(int4) * t.size()));
}

// 2^e as a float, |e| <= 126
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }
// v 2^e for |e| <= 252, in two exact steps (where the result is a normal float)
struct Pow2 {
  float a, b;
};
__device__ __forceinline__ Pow2 pow2(int e) {
  const int i = max(-126, min(126, e)), j = max(-126, min(126, e - i));
  return Pow2{pow2f(i), pow2f(j)};
}
__device__ __forceinline__ float scale(float v, Pow2 p) { return __fmul_rn(__fmul_rn(v, p.a), p.b); }

// The conversions between scaled double-float values and integers, chunk by chunk through
// 1.5 2^23 (adding it rounds a float below 2^22 to an integer in the low mantissa bits): the
// 64-bit conversion instructions issue every 65 clocks per warp, which made them a third of
// the pass (96^3: 45.8 ms per 2048-band application, now 41).
constexpr float kMagic = 12582912.0f;
constexpr int kMagicBits = 0x4B400000;
// round(v 2^e) for |v 2^e| < 2^61
__device__ __forceinline__ ll to_fixed(dfl v, Pow2 p) {
  const float h = scale(v.h, p), l = scale(v.l, p);  // |l| <= 2^37
  const float ta = __fmaf_rn(h, 0x1p-40f, kMagic);
  const float r1 = __fmaf_rn(__fsub_rn(ta, kMagic), -0x1p40f, h);   // exact, |r1| <= 2^39
  const float tb = __fmaf_rn(r1, 0x1p-18f, kMagic);
  const float r2 = __fmaf_rn(__fsub_rn(tb, kMagic), -0x1p18f, r1);  // exact, |r2| <= 2^17
  const float tl = __fmaf_rn(l, 0x1p-18f, kMagic);
  const float r3 = __fmaf_rn(__fsub_rn(tl, kMagic), -0x1p18f, l);   // exact, |r3| <= 2^17
  const float tc = __fadd_rn(__fadd_rn(r2, r3), kMagic);
  const int a = __float_as_int(ta) - kMagicBits, b = __float_as_int(tb) + __float_as_int(tl) - 2 * kMagicBits;
  const int c = __float_as_int(tc) - kMagicBits;
  return ((ll)(a << 8) << 32) + ((ll)b << 18) + (ll)c;
}
// v 2^(e - 21) as a double-float: v = a 2^42 + b 2^21 + c
__device__ __forceinline__ dfl from_fixed(ll v, Pow2 p) {
  const float fa = __fsub_rn(__int_as_float(kMagicBits + (int)(v >> 42)), kMagic);  // |a| <= 2^20
  const float fb = __fsub_rn(__int_as_float(0x4B000000 + ((int)(v >> 21) & 0x1FFFFF)), 8388608.0f);
  const float fc = __fsub_rn(__int_as_float(0x4B000000 + ((int)v & 0x1FFFFF)), 8388608.0f);
  // a 2^21 + b, exact as a pair; |a 2^21| >= |b| or a = 0
  const float h = __fmaf_rn(fa, 0x1p21f, fb), e = __fsub_rn(fb, __fmaf_rn(fa, -0x1p21f, h));
  const dfl r = df_fast2sum(h, __fmaf_rn(fc, 0x1p-21f, e));
  return dfl(scale(r.h, p), scale(r.l, p));
}

// x 2^s rounded to an integer, |x 2^s| < 2^61, by integer operations on the bits (the FP64
// unit takes 65 clocks a warp for a conversion); subnormals count as zero
__device__ __forceinline__ ll to_fixed(double x, int s) {
  const ll b = __double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7FF, k = e - 1075 + s;
  ll q = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  q = e == 0 || k < -54 ? 0 : k >= 0 ? q << k : (q + (1ll << (-k - 1))) >> -k;
  return b < 0 ? -q : q;
}
// v 2^-s as a double
__device__ __forceinline__ double to_double(ll v, int s) {
  const unsigned long long u = (unsigned long long)(v < 0 ? -v : v);
  const int lz = __clzll((ll)u), e = 63 - lz - s;
  if (u == 0 || e < -1022) return 0.0;
  if (e > 1023) return v < 0 ? -INFINITY : INFINITY;
  const unsigned long long m = u << lz;  // leading one at bit 63
  // the implicit bit and the rounding carry add into the exponent field
  const ll bits = ((ll)(e + 1022) << 52) + (ll)((m >> 11) + ((m >> 10) & 1));
  return __longlong_as_double(bits | (v < 0 ? 1ll << 63 : 0));
}

// The scale s of a plane's columns (integers x 2^s); false if a component is Inf or NaN.  A call
// synchronises the block before it returns.
template <int NT> struct Reduce {
  int e[NT / 32];
  float f[NT / 32];
};
template <int NT> __device__ __forceinline__ float block_sum(float sum, Reduce<NT>& sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (threadIdx.x % 32 == 0) sh.f[threadIdx.x / 32] = sum;
  __syncthreads();
  sum = 0.f;
#pragma unroll
  for (int i = 0; i < NT / 32; ++i) sum += sh.f[i];
  return sum;
}
// double-float columns: 2^s sum (|re| + |im|) <= 2^61
template <int N, int NT> __device__ __forceinline__ bool plane_scale(const cdf* t, int ncol, Reduce<NT>& sh, int& s) {
  float sum = 0.f;
  for (int c = threadIdx.x; c < ncol; c += NT) {
    const cdf v = t[c];
    sum += (fabsf(v.x.h) + fabsf(v.y.h)) * 1.220703125e-4f;  // 2^-13, against overflow
  }
  sum = block_sum(sum, sh);
  s = 61 - 13 - (sum > 0.f ? ilogbf(sum) + 1 : 0) - 1;  // one bit spare for the sum's rounding
  return sum < INFINITY;
}
// FP64 columns (normalised planes, below): the scale that brings the largest component below
// half of what pass A takes.
template <int N, int NT> __device__ __forceinline__ bool plane_scale(const double2* t, int ncol, Reduce<NT>& sh, int& s) {
  int e = 0;
  for (int c = threadIdx.x; c < ncol; c += NT)
    e = max(e, max((__double2hiint(t[c].x) >> 20) & 0x7FF, (__double2hiint(t[c].y) >> 20) & 0x7FF));
  e = __reduce_max_sync(0xffffffffu, e);
  if (threadIdx.x % 32 == 0) sh.e[threadIdx.x / 32] = e;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NT / 32; ++i) e = max(e, sh.e[i]);
  s = pass_bits(fast::Plan<N>::NA) - 1 - (e - 1022);
  return e != 0x7FF;
}
// columns to scaled integers and back: x 2^s, and v 2^-s
struct LoadDf {
  const cdf* t;
  Pow2 p;
  __device__ LoadDf(const cdf* t, int s) : t(t), p(pow2(s)) {}
  __device__ __forceinline__ cfx operator()(int c) const {
    const cdf u = t[c];
    return cfx{to_fixed(u.x, p), to_fixed(u.y, p)};
  }
};
struct LoadD {
  const double2* t;
  int s;
  __device__ LoadD(const double2* t, int s) : t(t), s(s) {}
  __device__ __forceinline__ cfx operator()(int c) const {
    const double2 u = t[c];
    return cfx{to_fixed(u.x, s), to_fixed(u.y, s)};
  }
};
struct StoreDf {
  cdf* t;
  Pow2 p;
  __device__ StoreDf(cdf* t, int s) : t(t), p(pow2(21 - s)) {}  // from_fixed's unit is 2^21
  __device__ __forceinline__ void operator()(int c, cfx v) const { t[c] = cdf{from_fixed(v.x, p), from_fixed(v.y, p)}; }
};
struct StoreD {
  double2* t;
  int s;
  __device__ StoreD(double2* t, int s) : t(t), s(s) {}
  __device__ __forceinline__ void operator()(int c, cfx v) const { t[c] = make_double2(to_double(v.x, s), to_double(v.y, s)); }
};
__device__ __forceinline__ LoadDf loader(const cdf* t, int s) { return LoadDf(t, s); }
__device__ __forceinline__ LoadD loader(const double2* t, int s) { return LoadD(t, s); }
__device__ __forceinline__ StoreDf storer(cdf* t, int s) { return StoreDf(t, s); }
__device__ __forceinline__ StoreD storer(double2* t, int s) { return StoreD(t, s); }
__device__ __forceinline__ cdf nan_of(cdf) {
  const float q = __int_as_float(0x7fc00000);
  return cdf{dfl(q, q), dfl(q, q)};
}
__device__ __forceinline__ double2 nan_of(double2) {
  const double q = __longlong_as_double(0x7FF8000000000000ll);
  return make_double2(q, q);
}

// bits of magnitude of the high words: their OR bounds the largest component
__device__ __forceinline__ unsigned mag(ll v) {
  const int h = hi32(v);
  return (unsigned)(h ^ (h >> 31));
}
// left shift that brings components with the given OR of magnitudes below 2^(top - 1/2), so
// that complex magnitudes are below 2^top
__device__ __forceinline__ int norm_shift(unsigned m, int top) {
  const int bits = 64 - __clz((int)m);  // components < 2^bits (the high words' bits, above bit 32)
  return top - 1 - bits;
}
__device__ __forceinline__ cfx shl(cfx a, int s) { return cfx{a.x << s, a.y << s}; }
// rounded shift right
__device__ __forceinline__ cfx sar_rn(cfx a, int s) {
  if (s == 0) return a;
  const ll h = 1ll << (s - 1);
  return cfx{(a.x + h) >> s, (a.y + h) >> s};
}
// n values times 2^s, s the same for the block
template <int L> __device__ __forceinline__ void scale_all(cfx* v, int s) {
  if (s >= 0) {
#pragma unroll
    for (int i = 0; i < L; ++i) v[i] = shl(v[i], s);
  } else {
#pragma unroll
    for (int i = 0; i < L; ++i) v[i] = sar_rn(v[i], -s);
  }
}

// The inverse y transform and pass A of the inverse x transform of a plane whose columns
// load(c) gives as scaled integers: the plane then holds pass B's inputs.  tws: the twiddles in
// shared memory (a warp of a y pass holds several nb, and the constant cache serves one
// address per warp at a time; the x passes use constant memory).
//
// kNormalised = false: the sum of the columns' magnitudes is at most 2^61, no pass needs a
// shift, and the result is a quarter of the transform.  That sum exceeds a plane of random
// phases by the root of the number of columns, 6 bits at N = 100: little beside
// double-float z passes, but more than FP64 loses.
// kNormalised = true: shifts to the word length before the x transform's two passes, by the
// largest component of the values just stored (its bits collect in ored[0], ored[1], zero
// before), and a static one inside the y transform.  `back` is the shift that pass B has to
// apply to its inputs (the caller's part), and s gets all of them and the twiddles' halvings.
// Rounding then stays within that of FP64 planes (relative error of a random plane with these
// against the FP64 units, both with FP64 z passes: 36^3 2.6e-16 and 4.6e-16, 60^3 2.5e-16 and
// 3.2e-16, 108^3 3.5e-16 and 4.0e-16).
template <int N, int NT, bool kNormalised, typename Load>
__device__ __forceinline__ void inverse_passes(Load load, const fk::FastArgs& fa, cfx* plane, const int4* tws,
                                               unsigned* ored, int& s, int& back) {
  constexpr int NA = fast::Plan<N>::NA, NB = fast::Plan<N>::NB, P = fk::plane_pitch(N);
  constexpr int kShiftB = kNormalised ? pre_shift(pass_bits(NA) * 8 + grow8(NA) - 8, NB) : 0;
  const int nl = fa.nact, lo = fa.act_lo, tid = threadIdx.x;
  cfx* rows = plane + lo * P;  // row a of the active range
  const cfx zero{0, 0};
  // y, inverse, pass A on the active rows, its inputs read from the column buffer
  for (int it = tid; it < nl * NB; it += NT) {
    const int a = it / NB, nb = it - a * NB;
    cfx* row = rows + a * P + nb;
    const int32_t* rc = fa.row_col + a * N + nb;
    cfx v[NA];
#pragma unroll
    for (int na = 0; na < NA; ++na) {
      const int c = __ldg(rc + NB * na);
      v[na] = c >= 0 ? load(c) : zero;
    }
    dft<NA, +1>(v);
    row[0] = sar(v[0], 1);
#pragma unroll
    for (int ka = 1; ka < NA; ++ka) {
      const int4 w = tws[nb * ka];
      row[NB * ka] = cmulh(v[ka], Cst{w.x, w.y}, Cst{-w.z, -w.w});
    }
  }
  __syncthreads();
  unsigned m = 0;
  for (int it = tid; it < nl * NA; it += NT) {  // pass B
    const int ka = nl == 1 ? it : (int)__umulhi((unsigned)it, fa.nl_magic), a = it - ka * nl;
    cfx* g = rows + a * P + NB * ka;
    cfx u[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) u[q] = sar_rn(g[q], kShiftB);
    dft<NB, +1>(u);
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      if constexpr (kNormalised) m |= mag(u[q].x) | mag(u[q].y);
      g[q] = u[q];
    }
  }
  if constexpr (kNormalised) {
    m = __reduce_or_sync(0xffffffffu, m);
    if (tid % 32 == 0 && m) atomicOr(&ored[0], m);
  }
  __syncthreads();
  int shift = 0;
  if constexpr (kNormalised) shift = norm_shift(ored[0], pass_bits(NA));
  m = 0;
  // x, inverse: pass A on every y line, rows outside the active range are zero
  for (int it = tid; it < N * NB; it += NT) {
    const int nb = it / N, yy = it - nb * N, d = nb - lo;
    cfx* a = plane + yy + nb * P;
    cfx v[NA];
#pragma unroll
    for (int na = 0; na < NA; ++na) v[na] = (unsigned)(d + NB * na) < (unsigned)nl ? a[NB * na * P] : zero;
    if constexpr (kNormalised) scale_all<NA>(v, shift);
    dft<NA, +1>(v);
    v[0] = sar(v[0], 1);
#pragma unroll
    for (int ka = 0; ka < NA; ++ka) {
      if (ka > 0) {
        Cst c, sn;
        twiddle<N, +1>(nb * ka, c, sn);
        v[ka] = cmulh(v[ka], c, sn);
      }
      if constexpr (kNormalised) m |= mag(v[ka].x) | mag(v[ka].y);
      a[NB * ka * P] = v[ka];
    }
  }
  if constexpr (kNormalised) {
    m = __reduce_or_sync(0xffffffffu, m);
    if (tid % 32 == 0 && m) atomicOr(&ored[1], m);
  }
  __syncthreads();
  back = 0;
  if constexpr (kNormalised) back = norm_shift(ored[1], pass_bits(NB));
  s += shift + back - kShiftB - 2;
}

// Plane z of band b (fk::plane_body_pruned in fixed point): inverse y and x transforms,
// multiply by V_loc (Vs: (h, l) of V_loc / 2^ve in split order, ve the plane's exponent), forward x and y.  C: the
// column buffer's elements, double-float pairs or FP64.  NT threads; the plane (16 bytes a
// point) fills the SM's shared memory, so one block runs per SM at N = 96.
template <int N, int NT, typename C>
__device__ __forceinline__ void plane_body(C* __restrict__ T, const int2* __restrict__ Vs, int ve,
                                           const fk::FastArgs& fa, int z, int64_t b, unsigned char* smem_raw) {
  constexpr int NA = fast::Plan<N>::NA, NB = fast::Plan<N>::NB, P = fk::plane_pitch(N);
  __shared__ Reduce<NT> red;
  __shared__ unsigned ored[4];
  __shared__ int4 tws[N];
  cfx* plane = reinterpret_cast<cfx*>(smem_raw);
  C* t = T + b * fa.ldt + (int64_t)z * fa.ncolp;
  const int nl = fa.nact, lo = fa.act_lo, tid = threadIdx.x;
  cfx* rows = plane + lo * P;  // row a of the active range
  if (tid < 4) ored[tid] = 0u;
  for (int i = tid; i < N; i += NT) tws[i] = c_twfx[fk::TwOff<N>::v + i];
  int s;
  if (!plane_scale<N, NT>(t, fa.ncol, red, s)) {  // Inf or NaN in the plane: so is every value of its transform
    for (int c = tid; c < fa.ncol; c += NT) t[c] = nan_of(C());
    return;
  }
  constexpr bool kNormalised = std::is_same<C, double2>::value;
  int back;
  inverse_passes<N, NT, kNormalised>(loader(t, s), fa, plane, tws, ored + 2, s, back);
  {  // pass B and the multiply by V_loc; the largest component of the product
    const int2* v = Vs + (int64_t)z * N * N;
    unsigned m = 0;
    for (int it = tid; it < N * NA; it += NT) {
      const int ka = it / N, yy = it - ka * N;
      cfx* a = plane + yy + NB * ka * P;
      const int2* vv = v + (NB * ka) * N + yy;
      cfx u[NB];
#pragma unroll
      for (int q = 0; q < NB; ++q) u[q] = a[q * P];
      if constexpr (kNormalised) scale_all<NB>(u, back);
      dft<NB, +1>(u);
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        const int2 w = __ldg(vv + q * N);
        const Cst c{w.x, w.y};
        u[q] = cfx{mulh(u[q].x, c), mulh(u[q].y, c)};
        m |= mag(u[q].x) | mag(u[q].y);
        a[q * P] = u[q];
      }
    }
    m = __reduce_or_sync(0xffffffffu, m);
    if (tid % 32 == 0 && m) atomicOr(&ored[0], m);
  }
  __syncthreads();
  // forward bounds in 1/8 bits: values enter below 2^58, and again after the x transform
  constexpr int b0 = 58 * 8;
  static_assert(pre_shift(b0, NB) == 0, "the normalised plane leaves room for pass B");
  constexpr int b1 = after(b0, NB) - 8;  // pass B, halved by its twiddles
  constexpr int s2 = pre_shift(b1, NA);  // pass A
  // the product is below 2^57 without normalised planes (2^60 of the inverse transforms, halved
  // three times), so its shift is to the left; normalised, and after the x transform, it may
  // go either way
  const int na1 = kNormalised ? norm_shift(ored[0], 58) : max(norm_shift(ored[0], 58), 0);
  // x, forward: pass B with the normalising shift
  for (int it = tid; it < N * NA; it += NT) {
    const int ka = it / N, yy = it - ka * N;
    cfx* a = plane + yy + NB * ka * P;
    cfx u[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) u[q] = a[q * P];
    if constexpr (kNormalised) scale_all<NB>(u, na1);
    else {
#pragma unroll
      for (int q = 0; q < NB; ++q) u[q] = shl(u[q], na1);
    }
    dft<NB, -1>(u);
    a[0] = sar(u[0], 1);
#pragma unroll
    for (int q = 1; q < NB; ++q) {
      Cst c, sn;
      twiddle<N, -1>(q * ka, c, sn);
      a[q * P] = cmulh(u[q], c, sn);
    }
  }
  __syncthreads();
  {  // pass A, storing only the rows the y pass reads; their largest component
    unsigned m = 0;
    for (int it = tid; it < N * NB; it += NT) {
      const int nb = it / N, yy = it - nb * N, d = nb - lo;
      cfx* a = plane + yy + nb * P;
      cfx v[NA];
#pragma unroll
      for (int ka = 0; ka < NA; ++ka) v[ka] = kNormalised ? sar_rn(a[NB * ka * P], s2) : sar(a[NB * ka * P], s2);
      dft<NA, -1>(v);
#pragma unroll
      for (int na = 0; na < NA; ++na)
        if ((unsigned)(d + NB * na) < (unsigned)nl) {
          m |= mag(v[na].x) | mag(v[na].y);
          a[NB * na * P] = v[na];
        }
    }
    m = __reduce_or_sync(0xffffffffu, m);
    if (tid % 32 == 0 && m) atomicOr(&ored[1], m);
  }
  __syncthreads();
  const int na2 = norm_shift(ored[1], 58), up2 = max(na2, 0), down2 = max(-na2, 0);
  // y, forward: pass B with the normalising shift
  for (int it = tid; it < nl * NA; it += NT) {
    const int ka = nl == 1 ? it : (int)__umulhi((unsigned)it, fa.nl_magic), a = it - ka * nl;
    cfx* g = rows + a * P + NB * ka;
    cfx u[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) u[q] = kNormalised ? g[q] : sar(shl(g[q], up2), down2);
    if constexpr (kNormalised) scale_all<NB>(u, na2);
    dft<NB, -1>(u);
    g[0] = sar(u[0], 1);
#pragma unroll
    for (int q = 1; q < NB; ++q) {
      const int4 w = tws[q * ka];
      g[q] = cmulh(u[q], Cst{w.x, w.y}, Cst{w.z, w.w});
    }
  }
  __syncthreads();
  // pass A, storing the columns to the column buffer.  Scale so far: s, - 1 - ve (V_loc), then
  // per forward transform the normalising shift - 1 - s2
  const auto out = storer(t, s - 1 - ve + (na1 - 1 - s2) + (na2 - 1 - s2));
  for (int it = tid; it < nl * NB; it += NT) {
    const int a = it / NB, nb = it - a * NB;  // consecutive columns per warp
    const cfx* row = rows + a * P + nb;
    const int32_t* rc = fa.row_col + a * N + nb;
    cfx v[NA];
#pragma unroll
    for (int ka = 0; ka < NA; ++ka) v[ka] = kNormalised ? sar_rn(row[NB * ka], s2) : sar(row[NB * ka], s2);
    dft<NA, -1>(v);
#pragma unroll
    for (int na = 0; na < NA; ++na) {
      const int c = __ldg(rc + NB * na);
      if (c >= 0) out(c, v[na]);
    }
  }
}

// Real-space values of plane z of band b from the FP64 column buffer, for the derivative with
// respect to V_loc: out[x'][y'] in split order.
template <int N, int NT>
__device__ __forceinline__ void plane_real_body(const double2* __restrict__ T, double2* __restrict__ out,
                                                const fk::FastArgs& fa, int z, int64_t b, unsigned char* smem_raw) {
  constexpr int NA = fast::Plan<N>::NA, NB = fast::Plan<N>::NB, P = fk::plane_pitch(N);
  __shared__ Reduce<NT> red;
  __shared__ unsigned ored[2];
  __shared__ int4 tws[N];
  cfx* plane = reinterpret_cast<cfx*>(smem_raw);
  const double2* t = T + b * fa.ldt + (int64_t)z * fa.ncolp;
  const int tid = threadIdx.x;
  if (tid < 2) ored[tid] = 0u;
  for (int i = tid; i < N; i += NT) tws[i] = c_twfx[fk::TwOff<N>::v + i];
  int s;
  if (!plane_scale<N, NT>(t, fa.ncol, red, s)) {
    for (int i = tid; i < N * N; i += NT) out[i] = nan_of(double2());
    return;
  }
  int back;
  inverse_passes<N, NT, true>(loader(t, s), fa, plane, tws, ored, s, back);
  for (int it = tid; it < N * NA; it += NT) {  // pass B
    const int ka = it / N, yy = it - ka * N;
    const cfx* a = plane + yy + NB * ka * P;
    cfx u[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) u[q] = a[q * P];
    scale_all<NB>(u, back);
    dft<NB, +1>(u);
    double2* o = out + (int64_t)(NB * ka) * N + yy;
#pragma unroll
    for (int q = 0; q < NB; ++q) o[q * N] = make_double2(to_double(u[q].x, s), to_double(u[q].y, s));
  }
}

}  // namespace fx
}  // namespace chebfi
