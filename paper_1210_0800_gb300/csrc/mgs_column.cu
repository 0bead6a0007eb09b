// Instantiations and launch of the column kernel (mgs_column.cuh).
#include "launch.cuh"
#include "mgs_column.cuh"

namespace mgs {
namespace {
const void* column_kernel(int L) {
  return L == 1   ? (const void*)mgs_column_kernel<1>
         : L == 2 ? (const void*)mgs_column_kernel<2>
                  : (const void*)mgs_column_kernel<4>;
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

// How many clusters of `cl` CTAs can be resident at once.
int column_clusters(int L, int cl, int threads, size_t smem) {
  const void* kern = column_kernel(L);
  if (ensure_smem(kern, smem) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cl);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = cl;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

int launch_column(int L, const ColParams& pr, int threads, size_t smem, cudaStream_t stream) {
  const void* kern = column_kernel(L);
  cudaError_t e = ensure_smem(kern, smem);
  if (e != cudaSuccess) return (int)e;
  ColParams copy = pr;
  void* args[] = {&copy};
  const int grid = (pr.Bc + pr.CL - 1) / pr.CL * pr.CL;
  if (pr.CL == 1) return (int)cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(threads), args, smem, stream);
  return launch_clusters(kern, args, grid, pr.CL, threads, smem, stream);
}

}  // namespace mgs
