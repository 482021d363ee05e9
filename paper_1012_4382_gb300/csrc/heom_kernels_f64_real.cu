// Instantiations of the N <= 8 engine kernel: FP64, real Hamiltonian.
// (One translation unit per precision and Hamiltonian kind so they compile in parallel.)
#include "heom_engine.cuh"
#include "heom_internal.h"

namespace heom {

const void* engine_kernel_f64_real(int N) {
  switch (N) {
    case 1: return (const void*)heom_engine_kernel<1, double, false, false>;
    case 2: return (const void*)heom_engine_kernel<2, double, false, false>;
    case 3: return (const void*)heom_engine_kernel<3, double, false, false>;
    case 4: return (const void*)heom_engine_kernel<4, double, false, false>;
    case 5: return (const void*)heom_engine_kernel<5, double, false, false>;
    case 6: return (const void*)heom_engine_kernel<6, double, false, false>;
    case 7: return (const void*)heom_engine_kernel<7, double, false, false>;
    case 8: return (const void*)heom_engine_kernel<8, double, false, false>;
    default: return nullptr;
  }
}

}  // namespace heom
