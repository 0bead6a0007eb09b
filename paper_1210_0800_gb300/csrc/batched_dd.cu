// Instantiations of the batched solve and its adjoint in double-double (batched_wide.cuh, adjoint_wide.cuh).
#include "adjoint_wide.cuh"
#include "batched_wide.cuh"

namespace mgs {
const void* batched_kernel_dd(int T, int S) {
  if (T == 128)
    return S == 4   ? (const void*)mgs_batched_wide_kernel<2, 128, 4>
           : S == 2 ? (const void*)mgs_batched_wide_kernel<2, 128, 2>
                    : (const void*)mgs_batched_wide_kernel<2, 128, 1>;
  return S == 4   ? (const void*)mgs_batched_wide_kernel<2, 256, 4>
         : S == 2 ? (const void*)mgs_batched_wide_kernel<2, 256, 2>
                  : (const void*)mgs_batched_wide_kernel<2, 256, 1>;
}
const void* adjoint_kernel_dd(int T) {
  return T == 128 ? (const void*)mgs_adjoint_wide_kernel<2, 128> : (const void*)mgs_adjoint_wide_kernel<2, 256>;
}
}  // namespace mgs
