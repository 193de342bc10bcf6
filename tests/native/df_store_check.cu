// The conversions between FP64 and double-float pairs against the FP64 unit's: df_to(h, l) is
// the double nearest to h + l, df_from(v) the pair (float(v), float(v - float(v))).  Prints the
// number of pairs and of values and the mismatches of each.
#include <cstdio>
#include <cstring>
#include <vector>

#include "dfloat.cuh"

using namespace chebfi;

__global__ void k_to(const float2* a, double* got, double* want, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  got[i] = df_to(dfl(a[i].x, a[i].y));
  want[i] = __dadd_rn((double)a[i].x, (double)a[i].y);
}
__global__ void k_from(const double* v, float2* got, float2* want, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const dfl d = df_from(v[i]);
  got[i] = make_float2(d.h, d.l);
  const float h = __double2float_rn(v[i]);
  want[i] = make_float2(h, __double2float_rn(__dadd_rn(v[i], -(double)h)));
}

static unsigned long long seed = 0x9E3779B97F4A7C15ull;
static unsigned rnd() {
  seed = seed * 6364136223846793005ull + 1442695040888963407ull;
  return (unsigned)(seed >> 32);
}
static float bits(unsigned b) {
  float f;
  memcpy(&f, &b, 4);
  return f;
}

int main() {
  std::vector<float2> p;
  std::vector<double> v;
  for (int e = 60; e <= 250; e += 5)
    for (int i = 0; i < 4096; ++i) {
      // high parts: powers of two, their neighbours, random; low parts: within half an ulp of h,
      // of every size down to where they no longer count, with few and with many bits
      const unsigned m = i % 4 == 0 ? 0u : i % 4 == 1 ? 0x7FFFFFu : i % 4 == 2 ? 1u : rnd() & 0x7FFFFF;
      const float h = bits((rnd() & 0x80000000u) | (unsigned)e << 23 | m);
      const int down = 25 + (int)(rnd() % 34);  // |l| < 2^(e - down + 1) <= ulp(h) / 2
      const unsigned lm = rnd() % 3 ? rnd() & 0x7FFFFF : (rnd() & 7u) << 20;
      const float l = e - down > 0 ? bits((rnd() & 0x80000000u) | (unsigned)(e - down) << 23 | lm) : 0.f;
      p.push_back(make_float2(h, l));
      v.push_back((double)h + (double)l);
      v.push_back((double)h * (1.0 + rnd() * 0x1p-32 * 0x1p-20));
    }
  for (unsigned e : {25u, 30u, 58u, 251u, 253u}) p.push_back(make_float2(bits(e << 23), 0.f));
  for (double d : {0.0, 1.0, -1.0, 1e-45, 1e38, 3.4e38, 1e300, -1e-300}) v.push_back(d);
  const int n = (int)p.size(), nv = (int)v.size();
  DevBuf<float2> dp, g2, w2;
  DevBuf<double> got, want, dv;
  dp.upload(p.data(), n);
  dv.upload(v.data(), nv);
  got.alloc(n);
  want.alloc(n);
  g2.alloc(nv);
  w2.alloc(nv);
  k_to<<<(n + 255) / 256, 256>>>(dp.p, got.p, want.p, n);
  k_from<<<(nv + 255) / 256, 256>>>(dv.p, g2.p, w2.p, nv);
  std::vector<double> hg(n), hw(n);
  std::vector<float2> fg(nv), fw(nv);
  CHEBFI_CUDA(cudaMemcpy(hg.data(), got.p, n * 8, cudaMemcpyDeviceToHost));
  CHEBFI_CUDA(cudaMemcpy(hw.data(), want.p, n * 8, cudaMemcpyDeviceToHost));
  CHEBFI_CUDA(cudaMemcpy(fg.data(), g2.p, nv * 8, cudaMemcpyDeviceToHost));
  CHEBFI_CUDA(cudaMemcpy(fw.data(), w2.p, nv * 8, cudaMemcpyDeviceToHost));
  int bad = 0, badv = 0;
  for (int i = 0; i < n; ++i) bad += memcmp(&hg[i], &hw[i], 8) != 0;
  for (int i = 0; i < nv; ++i) {
    const bool same = memcmp(&fg[i].x, &fw[i].x, 4) == 0 && fg[i].y == fw[i].y;
    const bool nans = fg[i].y != fg[i].y && fw[i].y != fw[i].y && fg[i].x == fw[i].x;  // past float's range
    badv += !(same || nans);
  }
  printf("%d %d %d %d\n", n, nv, bad, badv);
  return 0;
}
