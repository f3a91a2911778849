// Register annealer, strict acceptance, Delta E within int32 (see
// moda_reg_body.cuh), and the launch of every variant.
#include "moda_reg_body.cuh"

namespace moda {

const void *reg_kernel_strict(int K, bool narrow) {
  if (!narrow) return reg_kernel_strict_wide(K);
  return K == 1    ? reinterpret_cast<const void *>(reg_anneal_kernel<1, false, false, false, false>)
         : K == 2  ? reinterpret_cast<const void *>(reg_anneal_kernel<2, false, false, false, false>)
         : K == 4  ? reinterpret_cast<const void *>(reg_anneal_kernel<4, false, false, true, false>)
         : K == 8  ? reinterpret_cast<const void *>(reg_anneal_kernel<8, false, false, true, false>)
         : K == 16 ? reinterpret_cast<const void *>(reg_anneal_kernel<16, false, false, true, false>)
         : K == 24 ? reinterpret_cast<const void *>(reg_anneal_kernel<24, false, false, true, false>)
                   : nullptr;
}

cudaError_t reg_function(int K, bool narrow, bool lenient, bool ext, int optin,
                         const void **func) {
  const void *f = ext       ? reg_kernel_ext(K)
                  : lenient ? reg_kernel_lenient(K, narrow)
                            : reg_kernel_strict(K, narrow);
  if (f == nullptr) return cudaErrorInvalidValue;
  // the device's limit, always: launches of one kernel with other sizes may
  // be under way in a graph or on another thread
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) *func = f;
  return e;
}

cudaError_t reg_occupancy(const void *func, int warps, size_t smem, int *blocks) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, func, 32 * warps, smem);
}

cudaError_t launch_reg(const RegLaunch &L, const void *func, int grid, size_t smem,
                       cudaStream_t stream) {
  void *args[1] = {const_cast<RegLaunch *>(&L)};
  cudaError_t e =
      cudaLaunchKernel(func, dim3((unsigned)grid),
                       dim3((unsigned)(32 * (L.workers + L.draws + 2))), args, smem, stream);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace moda
