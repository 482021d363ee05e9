// Instantiations of the large-N engine (9..24 sites): mixed precision, complex Hamiltonian.
#include "heom_internal.h"
#include "heom_large.cuh"

namespace heom {

const void* large_kernel_f32_cplx(int N) {
  switch (N) {
    case 9: return (const void*)heom_large_kernel<9, float, true, true>;
    case 10: return (const void*)heom_large_kernel<10, float, true, true>;
    case 11: return (const void*)heom_large_kernel<11, float, true, true>;
    case 12: return (const void*)heom_large_kernel<12, float, true, true>;
    case 13: return (const void*)heom_large_kernel<13, float, true, true>;
    case 14: return (const void*)heom_large_kernel<14, float, true, true>;
    case 15: return (const void*)heom_large_kernel<15, float, true, true>;
    case 16: return (const void*)heom_large_kernel<16, float, true, true>;
    case 17: return (const void*)heom_large_kernel<17, float, true, true>;
    case 18: return (const void*)heom_large_kernel<18, float, true, true>;
    case 19: return (const void*)heom_large_kernel<19, float, true, true>;
    case 20: return (const void*)heom_large_kernel<20, float, true, true>;
    case 21: return (const void*)heom_large_kernel<21, float, true, true>;
    case 22: return (const void*)heom_large_kernel<22, float, true, true>;
    case 23: return (const void*)heom_large_kernel<23, float, true, true>;
    case 24: return (const void*)heom_large_kernel<24, float, true, true>;
    default: return nullptr;
  }
}

}  // namespace heom
