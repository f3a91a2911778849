// Register annealer with normalisation, the offset escape and snapshots (see
// moda_reg_body.cuh).
#include "moda_reg_body.cuh"

namespace moda {

const void *reg_kernel_ext(int K) {
  return K == 1    ? reinterpret_cast<const void *>(reg_anneal_kernel<1, true, false, false, true>)
         : K == 2  ? reinterpret_cast<const void *>(reg_anneal_kernel<2, true, false, false, true>)
         : K == 4  ? reinterpret_cast<const void *>(reg_anneal_kernel<4, true, false, true, true>)
         : K == 8  ? reinterpret_cast<const void *>(reg_anneal_kernel<8, true, false, true, true>)
         : K == 16 ? reinterpret_cast<const void *>(reg_anneal_kernel<16, true, false, true, true>)
         : K == 24 ? reinterpret_cast<const void *>(reg_anneal_kernel<24, true, false, true, true>)
                   : nullptr;
}

}  // namespace moda
