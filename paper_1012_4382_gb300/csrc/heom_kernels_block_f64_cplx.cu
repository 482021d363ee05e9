// Instantiations of the throughput engine (heom_block.cuh): FP64, complex Hamiltonian.
#include "heom_block.cuh"
#include "heom_internal.h"

namespace heom {

const void* block_kernel_f64_cplx(int N) {
  switch (N) {
    case 1: return (const void*)heom_block_kernel<1, double, false, true>;
    case 2: return (const void*)heom_block_kernel<2, double, false, true>;
    case 3: return (const void*)heom_block_kernel<3, double, false, true>;
    case 4: return (const void*)heom_block_kernel<4, double, false, true>;
    case 5: return (const void*)heom_block_kernel<5, double, false, true>;
    case 6: return (const void*)heom_block_kernel<6, double, false, true>;
    case 7: return (const void*)heom_block_kernel<7, double, false, true>;
    case 8: return (const void*)heom_block_kernel<8, double, false, true>;
    default: return nullptr;
  }
}

}  // namespace heom
