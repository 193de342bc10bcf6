// The host-side check of the two-pass line FFTs (fft_fast_check.cu) at every length that has
// compiled kernels.
#define main fixed_list
#include "fft_fast_check.cu"
#undef main

int main() {
#define CHEBFI_X(n) row<n>();
  CHEBFI_FFT_SIZES(CHEBFI_X)
#undef CHEBFI_X
  return 0;
}
