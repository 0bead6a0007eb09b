// Instantiations and launch of the column kernel (mgs_column.cuh).
#include "launch.cuh"
#include "mgs_column.cuh"

namespace mgs {
namespace {
const void* column_kernel(int L) {
  return L == 2 ? (const void*)mgs_column_kernel<2> : (const void*)mgs_column_kernel<4>;
}
}  // namespace

// Resident CTAs per SM with `smem` bytes (0: the kernel does not fit).
int column_capacity(int L, int threads, size_t smem) {
  const void* kern = column_kernel(L);
  if (ensure_smem(kern, smem) != cudaSuccess) return 0;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess) return 0;
  return per_sm;
}

int launch_column(int L, const ColParams& pr, int threads, size_t smem, cudaStream_t stream) {
  const void* kern = column_kernel(L);
  cudaError_t e = ensure_smem(kern, smem);
  if (e != cudaSuccess) return (int)e;
  ColParams copy = pr;
  void* args[] = {&copy};
  return (int)cudaLaunchCooperativeKernel(kern, dim3(pr.Bc), dim3(threads), args, smem, stream);
}

}  // namespace mgs
