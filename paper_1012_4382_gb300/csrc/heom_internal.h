// Private declarations shared by the translation units of libheom.
#pragma once

#include <cstdint>
#include <vector>

namespace heom {

// Load-view engine for N = 1..8 (nullptr otherwise): any number of unit groups.
const void* engine_kernel_f64_real(int N);
const void* engine_kernel_f64_cplx(int N);
const void* engine_kernel_f32_real(int N);
const void* engine_kernel_f32_cplx(int N);
// Throughput engine for N = 1..8 (nullptr otherwise), scaled hierarchies included.
const void* block_kernel_f64_real(int N);
const void* block_kernel_f64_cplx(int N);
const void* block_kernel_f32_real(int N);
const void* block_kernel_f32_cplx(int N);
// Scaled hierarchies (HEOM_FLAG_SCALED), N = 1..8, load views.
const void* engine_kernel_scaled_f64(int N, bool cplx);
const void* engine_kernel_scaled_f32(int N, bool cplx);
// Large-N engine for N = 9..24 (nullptr otherwise), scaled hierarchies included.
const void* large_kernel_f64_real(int N);
const void* large_kernel_f64_cplx(int N);
const void* large_kernel_f32_real(int N);
const void* large_kernel_f32_cplx(int N);
inline const void* large_kernel(bool fp64, bool cplx, int N) {
  if (fp64) return cplx ? large_kernel_f64_cplx(N) : large_kernel_f64_real(N);
  return cplx ? large_kernel_f32_cplx(N) : large_kernel_f32_real(N);
}
// Dataflow engine (launch mode 3, one hierarchy on the whole GPU), N = 1..8,
// npt nodes per thread (nullptr where that count is not built).
const void* flow_kernel_f32(int N, bool cplx, int npt);
const void* flow_kernel_f64(int N, bool cplx, int npt);
inline const void* flow_kernel(bool fp64, bool cplx, int N, int npt = 1) {
  return fp64 ? flow_kernel_f64(N, cplx, npt) : flow_kernel_f32(N, cplx, npt);
}
// One CTA with a thread per real of the hierarchy, N = 1..8 (mode 3 on small hierarchies).
const void* small_kernel_f32(int N, bool cplx);
const void* small_kernel_f64(int N, bool cplx);
inline const void* small_kernel(bool fp64, bool cplx, int N) {
  return fp64 ? small_kernel_f64(N, cplx) : small_kernel_f32(N, cplx);
}
// Distributed-shared-memory engine (mixed precision only).
const void* smem_kernel_f32_real(int N, bool reg);
const void* smem_kernel_f32_cplx(int N, bool reg);
inline const void* smem_kernel(bool cplx, bool reg, int N) {
  return cplx ? smem_kernel_f32_cplx(N, reg) : smem_kernel_f32_real(N, reg);
}
inline const void* block_kernel(bool fp64, bool cplx, int N) {
  if (fp64) return cplx ? block_kernel_f64_cplx(N) : block_kernel_f64_real(N);
  return cplx ? block_kernel_f32_cplx(N) : block_kernel_f32_real(N);
}
// Kernel of launch modes 0 and 1 for node_threads G: the throughput engine for
// 1, 2 and 4, the load views otherwise; scaled hierarchies refuse 1 and 2.
// nullptr where there is no such kernel.
inline const void* engine_kernel(bool fp64, bool cplx, int G, int N, bool scaled = false) {
  if (scaled && G <= 2) return nullptr;
  if (G == 1 || G == 2 || G == 4) return block_kernel(fp64, cplx, N);
  if (scaled) return fp64 ? engine_kernel_scaled_f64(N, cplx) : engine_kernel_scaled_f32(N, cplx);
  if (fp64) return cplx ? engine_kernel_f64_cplx(N) : engine_kernel_f64_real(N);
  return cplx ? engine_kernel_f32_cplx(N) : engine_kernel_f32_real(N);
}

// Hierarchy index builder (heom_index.cpp).
int64_t num_nodes(int N, int K);  // -1 on overflow beyond int64
struct Index {
  int N = 0, K = 0;
  int64_t M = 0;
  std::vector<int32_t> multi;  // [M][N]
  std::vector<int32_t> up;     // [M][N]
  std::vector<int32_t> down;   // [M][N]
};
void build_index(int N, int K, Index& out);
int64_t rank_of(const int32_t* n, int N, int K);
// Writes the element-major tables up[j*Mpad + i] and the packed down links
// (n_j << 24 | index) without allocating; returns the number of nodes.
int64_t write_packed_tables(int N, int K, int Mpad, int32_t* up, int32_t* dn);

}  // namespace heom
