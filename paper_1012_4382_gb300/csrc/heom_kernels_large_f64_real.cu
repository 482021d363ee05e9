// Instantiations of the large-N engine (9..24 sites): FP64, real Hamiltonian.
#include "heom_internal.h"
#include "heom_large.cuh"

namespace heom {

const void* large_kernel_f64_real(int N) {
  switch (N) {
    case 9: return (const void*)heom_large_kernel<9, double, false, false>;
    case 10: return (const void*)heom_large_kernel<10, double, false, false>;
    case 11: return (const void*)heom_large_kernel<11, double, false, false>;
    case 12: return (const void*)heom_large_kernel<12, double, false, false>;
    case 13: return (const void*)heom_large_kernel<13, double, false, false>;
    case 14: return (const void*)heom_large_kernel<14, double, false, false>;
    case 15: return (const void*)heom_large_kernel<15, double, false, false>;
    case 16: return (const void*)heom_large_kernel<16, double, false, false>;
    case 17: return (const void*)heom_large_kernel<17, double, false, false>;
    case 18: return (const void*)heom_large_kernel<18, double, false, false>;
    case 19: return (const void*)heom_large_kernel<19, double, false, false>;
    case 20: return (const void*)heom_large_kernel<20, double, false, false>;
    case 21: return (const void*)heom_large_kernel<21, double, false, false>;
    case 22: return (const void*)heom_large_kernel<22, double, false, false>;
    case 23: return (const void*)heom_large_kernel<23, double, false, false>;
    case 24: return (const void*)heom_large_kernel<24, double, false, false>;
    default: return nullptr;
  }
}

}  // namespace heom
