// Instantiations of the batched solve and its adjoint in quad-double (batched_wide.cuh, adjoint_wide.cuh).
#include "adjoint_wide.cuh"
#include "batched_wide.cuh"

namespace mgs {
const void* batched_kernel_qd(int T, int S) {
  if (T == 128)
    return S == 4   ? (const void*)mgs_batched_wide_kernel<4, 128, 4>
           : S == 2 ? (const void*)mgs_batched_wide_kernel<4, 128, 2>
                    : (const void*)mgs_batched_wide_kernel<4, 128, 1>;
  return S == 4   ? (const void*)mgs_batched_wide_kernel<4, 256, 4>
         : S == 2 ? (const void*)mgs_batched_wide_kernel<4, 256, 2>
                  : (const void*)mgs_batched_wide_kernel<4, 256, 1>;
}
const void* adjoint_kernel_qd(int T) {
  return T == 128 ? (const void*)mgs_adjoint_wide_kernel<4, 128> : (const void*)mgs_adjoint_wide_kernel<4, 256>;
}
}  // namespace mgs
