// Instantiations of the throughput engine (heom_block.cuh): FP64, real Hamiltonian.
#include "heom_block.cuh"
#include "heom_internal.h"

namespace heom {

const void* block_kernel_f64_real(int N) {
  switch (N) {
    case 1: return (const void*)heom_block_kernel<1, double, false, false>;
    case 2: return (const void*)heom_block_kernel<2, double, false, false>;
    case 3: return (const void*)heom_block_kernel<3, double, false, false>;
    case 4: return (const void*)heom_block_kernel<4, double, false, false>;
    case 5: return (const void*)heom_block_kernel<5, double, false, false>;
    case 6: return (const void*)heom_block_kernel<6, double, false, false>;
    case 7: return (const void*)heom_block_kernel<7, double, false, false>;
    case 8: return (const void*)heom_block_kernel<8, double, false, false>;
    default: return nullptr;
  }
}

}  // namespace heom
