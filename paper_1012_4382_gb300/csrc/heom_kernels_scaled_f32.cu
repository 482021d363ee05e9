// Instantiations of the N <= 8 engine kernel for scaled hierarchies (HEOM_FLAG_SCALED):
// FP32 auxiliaries with FP64 root, load views only (node_threads >= 3), real and complex Hamiltonians.
#include "heom_engine.cuh"
#include "heom_internal.h"

namespace heom {

const void* engine_kernel_scaled_f32(int N, bool cplx) {
  switch (N) {
    case 1: return cplx ? (const void*)heom_engine_kernel<1, float, true, true, true>
                     : (const void*)heom_engine_kernel<1, float, true, false, true>;
    case 2: return cplx ? (const void*)heom_engine_kernel<2, float, true, true, true>
                     : (const void*)heom_engine_kernel<2, float, true, false, true>;
    case 3: return cplx ? (const void*)heom_engine_kernel<3, float, true, true, true>
                     : (const void*)heom_engine_kernel<3, float, true, false, true>;
    case 4: return cplx ? (const void*)heom_engine_kernel<4, float, true, true, true>
                     : (const void*)heom_engine_kernel<4, float, true, false, true>;
    case 5: return cplx ? (const void*)heom_engine_kernel<5, float, true, true, true>
                     : (const void*)heom_engine_kernel<5, float, true, false, true>;
    case 6: return cplx ? (const void*)heom_engine_kernel<6, float, true, true, true>
                     : (const void*)heom_engine_kernel<6, float, true, false, true>;
    case 7: return cplx ? (const void*)heom_engine_kernel<7, float, true, true, true>
                     : (const void*)heom_engine_kernel<7, float, true, false, true>;
    case 8: return cplx ? (const void*)heom_engine_kernel<8, float, true, true, true>
                     : (const void*)heom_engine_kernel<8, float, true, false, true>;
    default: return nullptr;
  }
}

}  // namespace heom
