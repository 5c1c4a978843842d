// Double-float instantiations of the pair kernel (FP_PREC_DOUBLE_FLOAT) for 1, 2 and 4 atoms per cell.
#include "fp_pair_kernel.cuh"

namespace fp {
const void* pair_kernel_df(int nb, int maxt) {
  switch (nb * 100 + maxt) {
    case 301: return reinterpret_cast<const void*>(pair_kernel<3, 1, true, false>);
    case 302: return reinterpret_cast<const void*>(pair_kernel<3, 2, true, false>);
    case 308: return reinterpret_cast<const void*>(pair_kernel<3, kMaxT, true, false>);
    case 601: return reinterpret_cast<const void*>(pair_kernel<6, 1, true, false>);
    case 602: return reinterpret_cast<const void*>(pair_kernel<6, 2, true, false>);
    case 608: return reinterpret_cast<const void*>(pair_kernel<6, kMaxT, true, false>);
    case 1201: return reinterpret_cast<const void*>(pair_kernel<12, 1, true, false>);
    case 1202: return reinterpret_cast<const void*>(pair_kernel<12, 2, true, false>);
    case 1208: return reinterpret_cast<const void*>(pair_kernel<12, kMaxT, true, false>);
    default: return nullptr;
  }
}
}  // namespace fp
