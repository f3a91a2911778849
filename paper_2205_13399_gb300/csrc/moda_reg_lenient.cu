// Register annealer, lenient acceptance, Delta E within int32 (see
// moda_reg_body.cuh).
#include "moda_reg_body.cuh"

namespace moda {

const void *reg_kernel_lenient(int K, bool narrow) {
  if (!narrow) return reg_kernel_lenient_wide(K);
  return K == 1    ? reinterpret_cast<const void *>(reg_anneal_kernel<1, false, true, false, false>)
         : K == 2  ? reinterpret_cast<const void *>(reg_anneal_kernel<2, false, true, false, false>)
         : K == 4  ? reinterpret_cast<const void *>(reg_anneal_kernel<4, false, true, true, false>)
         : K == 8  ? reinterpret_cast<const void *>(reg_anneal_kernel<8, false, true, true, false>)
         : K == 16 ? reinterpret_cast<const void *>(reg_anneal_kernel<16, false, true, true, false>)
         : K == 24 ? reinterpret_cast<const void *>(reg_anneal_kernel<24, false, true, true, false>)
                   : nullptr;
}

}  // namespace moda
