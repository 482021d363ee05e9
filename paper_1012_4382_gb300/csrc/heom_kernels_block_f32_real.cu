// Instantiations of the throughput engine (heom_block.cuh): mixed precision (float auxiliaries, float-float root), real Hamiltonian.
#include "heom_block.cuh"
#include "heom_internal.h"

namespace heom {

const void* block_kernel_f32_real(int N) {
  switch (N) {
    case 1: return (const void*)heom_block_kernel<1, float, true, false>;
    case 2: return (const void*)heom_block_kernel<2, float, true, false>;
    case 3: return (const void*)heom_block_kernel<3, float, true, false>;
    case 4: return (const void*)heom_block_kernel<4, float, true, false>;
    case 5: return (const void*)heom_block_kernel<5, float, true, false>;
    case 6: return (const void*)heom_block_kernel<6, float, true, false>;
    case 7: return (const void*)heom_block_kernel<7, float, true, false>;
    case 8: return (const void*)heom_block_kernel<8, float, true, false>;
    default: return nullptr;
  }
}

}  // namespace heom
