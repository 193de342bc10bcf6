// A lower-triangle product whose K is split: the entries above the diagonal keep what they
// held, whatever the workspace holds, and the lower ones match a plain sum.  Prints the
// number of entries that changed above the diagonal and the largest error below it, for each
// precision and size.
#include <cmath>
#include <cstdio>
#include <limits>
#include <vector>

#include "internal.cuh"
#include "kernels.cuh"

using namespace chebfi;

template <typename R> static void run(int n, int k) {
  using C = cplx<R>;
  std::vector<C> a((size_t)n * k), c((size_t)n * n), got(c.size());
  for (size_t i = 0; i < a.size(); ++i) a[i] = cmake<C>(std::sin(0.1 + i), std::cos(0.3 * i));
  for (size_t i = 0; i < c.size(); ++i) c[i] = cmake<C>(1.0 + i, 0.5);
  DevBuf<C> dA, dC, ws;
  dA.upload(a.data(), a.size());
  dC.upload(c.data(), c.size());
  ws.alloc((size_t)512 * n * n);
  CHEBFI_CUDA(cudaMemset(ws.p, 0xFF, ws.n * sizeof(C)));  // NaN
  gemm<R>(false, true, n, n, k, -1.0, dA.p, n, dA.p, n, 1.0, dC.p, n, 0, &ws, "check", true);
  CHEBFI_CUDA(cudaMemcpy(got.data(), dC.p, got.size() * sizeof(C), cudaMemcpyDeviceToHost));
  int changed = 0;
  double err = 0.0;
  for (int j = 0; j < n; ++j)
    for (int i = 0; i < n; ++i) {
      const C g = got[i + (size_t)j * n], o = c[i + (size_t)j * n];
      if (i < j) {
        changed += !(g.x == o.x && g.y == o.y);
        continue;
      }
      double re = o.x, im = o.y;
      for (int l = 0; l < k; ++l) {
        const C u = a[i + (size_t)l * n], v = a[j + (size_t)l * n];
        re -= (double)u.x * v.x + (double)u.y * v.y;
        im -= (double)u.y * v.x - (double)u.x * v.y;
      }
      const double d = std::hypot(g.x - re, g.y - im) / (std::hypot((double)o.x, (double)o.y) + k);
      if (!(d <= err)) err = std::isnan(d) ? std::numeric_limits<double>::infinity() : d;
    }
  printf("%d %d %d %d %.3e\n", (int)sizeof(R), n, k, changed, err);
}

int main() {
  const int sizes[][2] = {{40, 32}, {100, 32}, {65, 200}, {130, 3000}};
  for (auto& s : sizes) {
    run<double>(s[0], s[1]);
    run<float>(s[0], s[1]);
  }
  return 0;
}
