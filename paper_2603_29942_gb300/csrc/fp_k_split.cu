// fp_k_split.cu -- tensor-core enumeration kernels for one code with p = 3,
// 5 or 7 (n - k up to 128 for p = 3, 42 for p = 5 and 7: split_k).
#include "fp_split_kernel.cuh"
#include "fp_kernels.h"

namespace fpk {
const void *kernel_split(int p, int W) {
  if (p == 3) {
    switch (W) {
      case 1: return (const void *)split_kernel<3, 2, 1>;
      case 2: return (const void *)split_kernel<3, 2, 2>;
      case 3: return (const void *)split_kernel<3, 2, 3>;
      case 4: return (const void *)split_kernel<3, 2, 4>;
      default: return nullptr;
    }
  }
  if (p == 5) return W == 1 ? (const void *)split_kernel<5, 3, 1> : W == 2 ? (const void *)split_kernel<5, 3, 2> : nullptr;
  if (p == 7) return W == 1 ? (const void *)split_kernel<7, 3, 1> : W == 2 ? (const void *)split_kernel<7, 3, 2> : nullptr;
  return nullptr;
}
}  // namespace fpk
