// Instantiations of the N <= 8 engine kernel: FP64, complex Hamiltonian.
// (One translation unit per precision and Hamiltonian kind so they compile in parallel.)
#include "heom_engine.cuh"
#include "heom_internal.h"

namespace heom {

const void* engine_kernel_f64_cplx(int N) {
  switch (N) {
    case 1: return (const void*)heom_engine_kernel<1, double, false, true>;
    case 2: return (const void*)heom_engine_kernel<2, double, false, true>;
    case 3: return (const void*)heom_engine_kernel<3, double, false, true>;
    case 4: return (const void*)heom_engine_kernel<4, double, false, true>;
    case 5: return (const void*)heom_engine_kernel<5, double, false, true>;
    case 6: return (const void*)heom_engine_kernel<6, double, false, true>;
    case 7: return (const void*)heom_engine_kernel<7, double, false, true>;
    case 8: return (const void*)heom_engine_kernel<8, double, false, true>;
    default: return nullptr;
  }
}

}  // namespace heom
