// Mixed-precision instantiations of the dense kernel for one and two atoms per cell.
#include "fp_dense_kernel.cuh"

namespace fp {
const void* dense_kernel_f32(int nb, int maxt) {
  switch (nb * 100 + maxt) {
    case 301: return reinterpret_cast<const void*>(dense_kernel<3, 1>);
    case 308: return reinterpret_cast<const void*>(dense_kernel<3, kMaxT>);
    case 601: return reinterpret_cast<const void*>(dense_kernel<6, 1>);
    case 608: return reinterpret_cast<const void*>(dense_kernel<6, kMaxT>);
    default: return nullptr;
  }
}
}  // namespace fp
