// The Cholesky factor and the triangular solve entry by entry, where each value can be told
// exactly: a quotient is rounded once, and so is the subtraction of a small product from a value of
// order one.  Cholesky of 32 x 32: the first column is small, so L_i0 = a_i0 / sqrt(a_00) and
// L_ij = (a_ij - L_i0 conj(L_j0)) / L_jj for the entries (i odd, j = i - 1) that the others do not
// touch.  Solve: the first column of L is small, the rest diagonal, so x_0 = b_0 / L_00 and
// x_i = (b_i - L_i0 x_0) / L_ii.  Prints the number of values and of those that are not what
// these formulas give, of each.
#include <cmath>
#include <cstdio>
#include <vector>

#include "internal.cuh"
#include "kernels.cuh"

using namespace chebfi;
typedef long double ld;

static unsigned long long seed = 12345;
static double rnd() {
  seed = seed * 6364136223846793005ull + 1442695040888963407ull;
  return (double)(seed >> 11) * 0x1p-53 - 0.5;
}
static double part(double b, ld p, double d) { return (double)(b - p) / d; }

int main() {
  const int n = 32;
  const double tiny = 0x1p-24;
  int nq = 0, bad = 0, nt = 0, badt = 0;
  for (int rep = 0; rep < 200; ++rep) {
    std::vector<double2> A(n * n, make_double2(0.0, 0.0)), L(n * n), B(n * n), X(n * n);
    for (int i = 0; i < n; ++i) A[i + i * n].x = 2.0 + std::exp(2.0 * rnd());
    for (int i = 1; i < n; ++i) A[i] = make_double2(tiny * rnd(), tiny * rnd());
    for (int i = 3; i < n; i += 2) A[i + (i - 1) * n] = make_double2(rnd(), rnd());
    for (int j = 0; j < n; ++j)
      for (int i = j + 1; i < n; ++i) A[j + i * n] = make_double2(A[i + j * n].x, -A[i + j * n].y);
    DevBuf<double2> dA, dB, ws;
    DevBuf<int> status;
    const int zero = 0;
    status.upload(&zero, 1);
    dA.upload(A.data(), n * n);
    cholesky(n, dA.p, n, status.p, 0, &ws);
    CHEBFI_CUDA(cudaMemcpy(L.data(), dA.p, n * n * 16, cudaMemcpyDeviceToHost));
    auto count = [](int& all, int& wrong, double got, double want) {
      ++all;
      wrong += got != want;
    };
    count(nq, bad, L[0].x, std::sqrt(A[0].x));
    for (int i = 1; i < n; ++i) {
      count(nq, bad, L[i].x, A[i].x / L[0].x);
      count(nq, bad, L[i].y, A[i].y / L[0].x);
    }
    for (int i = 3; i < n; i += 2) {
      const int j = i - 1;
      const double2 u = L[i], v = L[j], a = A[i + j * n];
      count(nq, bad, L[i + j * n].x, part(a.x, (ld)u.x * v.x + (ld)u.y * v.y, L[j + j * n].x));
      count(nq, bad, L[i + j * n].y, part(a.y, (ld)u.y * v.x - (ld)u.x * v.y, L[j + j * n].x));
    }
    for (int i = 0; i < n * n; ++i) L[i] = make_double2(0.0, 0.0);
    for (int i = 0; i < n; ++i) {
      if (i > 0) L[i] = make_double2(tiny * rnd(), tiny * rnd());
      L[i + i * n].x = std::exp(4.0 * rnd());
    }
    for (auto& b : B) b = make_double2(rnd(), rnd());
    dA.upload(L.data(), n * n);
    dB.upload(B.data(), n * n);
    trsm_lower(n, n, dA.p, n, dB.p, n, 0, &ws);
    CHEBFI_CUDA(cudaMemcpy(X.data(), dB.p, n * n * 16, cudaMemcpyDeviceToHost));
    for (int j = 0; j < n; ++j) {
      const double2 x = X[j * n];
      count(nt, badt, x.x, B[j * n].x / L[0].x);
      count(nt, badt, x.y, B[j * n].y / L[0].x);
      for (int i = 1; i < n; ++i) {
        const double2 l = L[i], b = B[i + j * n];
        count(nt, badt, X[i + j * n].x, part(b.x, (ld)l.x * x.x - (ld)l.y * x.y, L[i + i * n].x));
        count(nt, badt, X[i + j * n].y, part(b.y, (ld)l.x * x.y + (ld)l.y * x.x, L[i + i * n].x));
      }
    }
  }
  printf("%d %d %d %d\n", nq, bad, nt, badt);
  return 0;
}
