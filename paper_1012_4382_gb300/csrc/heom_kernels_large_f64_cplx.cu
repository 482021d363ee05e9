// Instantiations of the large-N engine (9..24 sites): FP64, complex Hamiltonian.
#include "heom_internal.h"
#include "heom_large.cuh"

namespace heom {

const void* large_kernel_f64_cplx(int N) {
  switch (N) {
    case 9: return (const void*)heom_large_kernel<9, double, false, true>;
    case 10: return (const void*)heom_large_kernel<10, double, false, true>;
    case 11: return (const void*)heom_large_kernel<11, double, false, true>;
    case 12: return (const void*)heom_large_kernel<12, double, false, true>;
    case 13: return (const void*)heom_large_kernel<13, double, false, true>;
    case 14: return (const void*)heom_large_kernel<14, double, false, true>;
    case 15: return (const void*)heom_large_kernel<15, double, false, true>;
    case 16: return (const void*)heom_large_kernel<16, double, false, true>;
    case 17: return (const void*)heom_large_kernel<17, double, false, true>;
    case 18: return (const void*)heom_large_kernel<18, double, false, true>;
    case 19: return (const void*)heom_large_kernel<19, double, false, true>;
    case 20: return (const void*)heom_large_kernel<20, double, false, true>;
    case 21: return (const void*)heom_large_kernel<21, double, false, true>;
    case 22: return (const void*)heom_large_kernel<22, double, false, true>;
    case 23: return (const void*)heom_large_kernel<23, double, false, true>;
    case 24: return (const void*)heom_large_kernel<24, double, false, true>;
    default: return nullptr;
  }
}

}  // namespace heom
