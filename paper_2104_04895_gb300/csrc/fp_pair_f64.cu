// FP64 instantiations of the pair kernel for 1, 2 and 4 atoms per cell.
#include "fp_pair_kernel.cuh"

namespace fp {
// sliced: the contractions on the tensor cores (6 and 12 branches)
const void* pair_kernel_f64(int nb, int maxt, bool sliced) {
  switch (nb * 1000 + maxt * 10 + (sliced ? 1 : 0)) {
    case 3010: return reinterpret_cast<const void*>(pair_kernel<3, 1, false, false>);
    case 3020: return reinterpret_cast<const void*>(pair_kernel<3, 2, false, false>);
    case 3080: return reinterpret_cast<const void*>(pair_kernel<3, kMaxT, false, false>);
    case 6010: return reinterpret_cast<const void*>(pair_kernel<6, 1, false, false>);
    case 6020: return reinterpret_cast<const void*>(pair_kernel<6, 2, false, false>);
    case 6080: return reinterpret_cast<const void*>(pair_kernel<6, kMaxT, false, false>);
    case 12010: return reinterpret_cast<const void*>(pair_kernel<12, 1, false, false>);
    case 12020: return reinterpret_cast<const void*>(pair_kernel<12, 2, false, false>);
    case 12080: return reinterpret_cast<const void*>(pair_kernel<12, kMaxT, false, false>);
    case 6011: return reinterpret_cast<const void*>(pair_kernel<6, 1, false, true>);
    case 6021: return reinterpret_cast<const void*>(pair_kernel<6, 2, false, true>);
    case 6081: return reinterpret_cast<const void*>(pair_kernel<6, kMaxT, false, true>);
    case 12011: return reinterpret_cast<const void*>(pair_kernel<12, 1, false, true>);
    case 12021: return reinterpret_cast<const void*>(pair_kernel<12, 2, false, true>);
    case 12081: return reinterpret_cast<const void*>(pair_kernel<12, kMaxT, false, true>);
    default: return nullptr;
  }
}
}  // namespace fp
