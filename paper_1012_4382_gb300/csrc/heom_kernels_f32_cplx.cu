// Instantiations of the N <= 8 engine kernel: FP32 auxiliaries with FP64 root, complex Hamiltonian.
// (One translation unit per precision and Hamiltonian kind so they compile in parallel.)
#include "heom_engine.cuh"
#include "heom_internal.h"

namespace heom {

const void* engine_kernel_f32_cplx(int N) {
  switch (N) {
    case 1: return (const void*)heom_engine_kernel<1, float, true, true>;
    case 2: return (const void*)heom_engine_kernel<2, float, true, true>;
    case 3: return (const void*)heom_engine_kernel<3, float, true, true>;
    case 4: return (const void*)heom_engine_kernel<4, float, true, true>;
    case 5: return (const void*)heom_engine_kernel<5, float, true, true>;
    case 6: return (const void*)heom_engine_kernel<6, float, true, true>;
    case 7: return (const void*)heom_engine_kernel<7, float, true, true>;
    case 8: return (const void*)heom_engine_kernel<8, float, true, true>;
    default: return nullptr;
  }
}

}  // namespace heom
