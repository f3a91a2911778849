// Register annealer, lenient acceptance, Delta E beyond int32 (see
// moda_reg_body.cuh).
#include "moda_reg_body.cuh"

namespace moda {

const void *reg_kernel_lenient_wide(int K) {
  return K == 4    ? reinterpret_cast<const void *>(reg_anneal_kernel<4, true, true, true, false>)
         : K == 8  ? reinterpret_cast<const void *>(reg_anneal_kernel<8, true, true, true, false>)
         : K == 16 ? reinterpret_cast<const void *>(reg_anneal_kernel<16, true, true, true, false>)
         : K == 24 ? reinterpret_cast<const void *>(reg_anneal_kernel<24, true, true, true, false>)
                   : nullptr;
}

}  // namespace moda
