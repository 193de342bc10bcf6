// A modular GEMM operand whose planes cannot be allocated is not marked as prepared: the next
// call on the same data would otherwise read planes that were never written.
// Prints the allocation's error code and the operand's modulus count afterwards.
#include <cstdio>

#include "internal.cuh"
#include "kernels.cuh"

int main() {
  chebfi::OzOperand o;
  int code = 0;
  try {  // 2^52 bytes: no device has them (and no device at all fails the same way)
    chebfi::oz_prepare(nullptr, 1 << 20, (int64_t)1 << 25, (int64_t)1 << 20, true, false, 14, o, 0);
  } catch (const chebfi::Error& e) {
    code = e.code;
  }
  printf("%d %d\n", code, o.nmod);
  return 0;
}
