// heom_block.cuh -- the throughput engine for N <= 8 sites (launch modes 0 and
// 1 with node_threads 1, 2 or 4): 32 consecutive nodes (one lane each) are
// computed by a set of N warps of one CTA, one warp per site.
//
// Same method as heom_engine.cuh.  The right-hand side of a Hermitian node is
// D = P + P^+ + (local terms), where column b of P needs only column b of the
// node and the links of site b:
//   P_ab = -i (H' sigma)_ab + [down link b] n_b (beta_b - i alpha_b) sigma_{n-e_b, ab}
//          - i [up link b] sigma_{n+e_b, ab},         H' = H off the diagonal
// (the Hermitian conjugate supplies the terms of row a).  So warp b reads 2N - 1
// reals of its node, 2N - 2 of n + e_b and 2N - 1 of n - e_b, multiplies by the
// couplings, hands the elements it does not own to their owners through shared
// memory, and finishes its own N elements: the diagonal b and the pairs (b, b+d)
// at cyclic distance d = 1..N/2 above it, with the site-energy differences and
// the damping.  Each of the N(N-1) products of the commutator is computed once,
// as in a pair-by-pair form, but a thread holds one column instead of a whole
// matrix, a stage is one round of independent loads, and a warp needs two links.
//
// All warps run the same code: sites are counted relative to the warp's own
// (r = a - b mod N), with the couplings rotated accordingly in shared memory,
// and the state is in cyclic order during a call (see cyc_pair), so that every
// element is at a compile-time offset from one of 2 + N/2 addresses and the two
// reals of a pair are one load.  N bodies
// with compile-time columns were 43 KB of code at N = 7 and waited on
// instruction fetch (no_instruction 5.5 of 23 cycles per issue).
//
// Bound and measured (us per RK4 step, whole grid, FMO-like N = 7 models; in
// brackets the pair-by-pair kernels this engine took the place of): mixed
// precision depth 8 13.2 [17.5], depth 10 18 [65], depth 12 35.5 [92]; FP64
// depth 8 74 [76], depth 10 143 [184].  In mixed precision a stage costs about
// 2.4 us (grid barrier 1.2, one trip to L2 and the exchange) plus 0.52 us per
// node block of an SM, where the SM issues about half of its slots;
// FP64 is bound by the FP64 pipe: about 980 double-precision instructions per
// 32 nodes at 64 cycles on four sub-partitions, 8.1 us per block.  Tried and
// dropped: the whole matrix or half of it per thread (168 registers, 12 warps:
// 34.6 us at depth 12), neighbours staged through cp.async (38), node blocks
// resident in shared memory (46), and counters per block in place of the grid
// barrier (44.8: every block pays a release and an acquire).
//
// The state is stored in blocks of 32 nodes (node_col); lanes without a link
// read the zero block that ends every state array.  The Markov terminator is
// a shift of the leaf node's site energies and damping: i V_j^x of
// (n_j+1)/(ngam+gamma_j) theta_j sigma_n multiplies element (a, b) by
// -(c_a alpha_a + c_b alpha_b) + i (c_a beta_a - c_b beta_b), c_j =
// (n_j+1)/(ngam+gamma_j).
#pragma once

#include "heom_engine.cuh"

namespace heom {

// Sets (N warps each) of the largest CTA, and the threads the kernels are
// compiled for.  FP32: three sets at N = 7 (80 registers a thread, of which 136 bytes
// spill and 156 are read back), two at N = 8 (128, no spills).  With up to 28 warps (72
// registers, 212 bytes of spills read back at N = 7, 172 at N = 8) depth 8 took 15.3 us
// per step against 13.2, depth 12 37.5 against 35.5, a scan of 256 hierarchies 29.6 ms
// against 28.6, a serving burst 46.0 ms against 41.8; with 24 the burst 46.0 (three sets
// at N = 8), with 18 the scan 33.2.  FP64: two sets, 128 registers, with 148 bytes of spill
// stores and 220 of loads at N = 7 (complex H 124 and 136), 388 and 448 at N = 8.
__host__ __device__ constexpr int block_max_sets(int N, int rsize) {
  const int warps = rsize == 8 ? 16 : 21;
  return warps / N < 1 ? 1 : (warps / N > 14 ? 14 : warps / N);
}
__host__ __device__ constexpr int block_max_threads(int N, int rsize) { return 32 * N * block_max_sets(N, rsize); }
// Sets of a CTA for a launch of `block` threads (heom_set_launch): its threads
// are about twice that, since a node has more, lighter threads here.
__host__ __device__ constexpr int block_sets(int N, int rsize, int block) {
  const int s = 2 * block / (32 * N);
  return s < 1 ? 1 : (s < block_max_sets(N, rsize) ? s : block_max_sets(N, rsize));
}

template <typename R>
struct Vec2;
template <>
struct Vec2<float> {
  typedef float2 type;
};
template <>
struct Vec2<double> {
  typedef double2 type;
};
// Bytes of a set's exchange area (two buffers: items alternate): the two reals
// of every pair.
__host__ __device__ constexpr int exch_bytes(int N, int rsize) { return 2 * N * (N - 1) * 32 * rsize; }
__host__ __device__ constexpr int block_exch_bytes(int N, int rsize, int sets) { return sets * exch_bytes(N, rsize); }
// Bytes of the cached links of one block: up and down, per site and lane.
__host__ __device__ constexpr int block_link_bytes(int N) { return 2 * N * 32 * 4; }

// Root state of the CTA that runs the root's block (shared memory): float-float
// y, wa, wb of the mixed path, in the order of root_index.
template <int N>
struct BlockRoot {
  FF w[3][N * N];
  float acc[N * N];  // the root's right-hand side, from lane 0
};

// Coefficients in each column's own site order (r = 0: the column's site).
template <int N, typename R, bool CPLX>
struct BlockCoef {
  static constexpr int JS = CoefLayout<R>::JS(N);
  alignas(16) R J[N][N][JS];                 // [b][r][r'] = J(b + r, b + r')
  alignas(16) R Ji[CPLX ? N : 1][N][JS];
  alignas(16) R site[2 * N][4];              // eps, goff, alpha, beta of site b + r at [b + r]
  R gam[N], gd[N];
};

// Loop state of an instance that only single lanes need, kept in shared memory
// so that the stage code has the registers: the output row under way, the rows'
// bookkeeping (lead) and the running sums of each site (its owner lane).
template <int N, typename R>
struct BlockRows {
  OutStep os;
  EtaRows rows;
  EtaAcc<R> ea[N];
};

// What a stage's items share.
template <typename R>
struct StageArgs {
  const R* win;
  R* wout;
  const R* yv;
  const R* ngam;
  unsigned zero;  // the zero block: its first element (N > 8: its index)
  R h;
  float hl;       // low part of h (mixed)
  int s, in_sel, out_sel;
  bool terminator;
  const R* wsc;   // scaled hierarchy: link weights (see scaled_up), else null
  int wstride;
};

// One RK4 stage of column b of the 32 nodes of block nb.  up, dn: this lane's
// links of site b as in the node tables; ex: this lane's pair of the set's
// exchange buffer; bar: the set's barrier.
template <int N, typename R, bool MIXED, bool CPLX>
__device__ __forceinline__ void column_stage(const Inst& I, const BlockCoef<N, R, CPLX>& cf,
                                             const double* __restrict__ cfd, const StageArgs<R>& A, int nb, int lane,
                                             int b, int up, int dn, BlockRows<N, R>& rw, BlockRoot<N>& br,
                                             typename Vec2<R>::type* ex, int bar) {
  typedef typename Vec2<R>::type R2;
  constexpr int NN = N * N;
  constexpr int JS = CoefLayout<R>::JS(N);
  constexpr int D = (N - 1) / 2;          // distances whose pairs every column owns one of
  constexpr bool EVEN = N % 2 == 0 && N > 1;  // the pairs at distance N/2: owned by their lower site
  // offsets (pairs of reals) of this column's forward pairs, of the pairs (b - d, b), and of the pair at distance N/2
  const unsigned ob = b * 32;
  unsigned om[D + 1];
#pragma unroll
  for (int d = 1; d <= D; ++d) om[d] = (b >= d ? b - d : b - d + N) * 32;
  const bool low = 2 * b < N;
  const unsigned oh = (low ? b : b - N / 2) * 32;
  // column b of the node in lane l of the block at q: r = d is pair (b, b+d), Im sigma_{b+d,b} = -(its imaginary part)
  auto column = [&](unsigned q, unsigned l, R* re, R* im) {
    re[0] = A.win[(size_t)(q + ob + l)];
    const R2* pw = reinterpret_cast<const R2*>(A.win) + (size_t)((q >> 1) + N * 16 + l);
    const R2* pb = pw + ob;
    static_for<1, D + 1>([&](auto dc) {
      constexpr int d = decltype(dc)::value;
      const R2 f = pb[cyc_pair(N, d) * 32];
      re[d] = f.x;
      im[d] = -f.y;
      const R2 g = pw[om[d] + cyc_pair(N, d) * 32];
      re[N - d] = g.x;
      im[N - d] = g.y;
    });
    if constexpr (EVEN) {
      const R2 f = pw[oh + cyc_pair(N, N / 2) * 32];
      re[N / 2] = f.x;
      im[N / 2] = low ? -f.y : f.y;
    }
  };
  auto block_of = [](int m) -> unsigned { return (unsigned)(m >> 5) * (NN * 32); };
  R sr[N], si[N], gr[N], gi[N], ur[N], ui[N];
  const unsigned self = nb * (NN * 32);
  column(self, lane, sr, si);
  column(dn >= 0 ? block_of(dn & 0xFFFFFF) : A.zero, dn & 31, gr, gi);
  column(up >= 0 ? block_of(up) : A.zero, up & 31, ur, ui);
  const R ng = A.ngam[nb * 32 + lane];

  // P = -i H' sigma
  R p_r[N], p_i[N];
  static_for<0, N>([&](auto ac) {
    constexpr int a = decltype(ac)::value;
    R jr[JS], ir[CPLX ? JS : 1];
    load_row<JS>(cf.J[b][a], jr);
    if constexpr (CPLX) load_row<JS>(cf.Ji[b][a], ir);
    p_r[a] = p_i[a] = R(0);
    static_for<0, N>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (k != a) {
        if constexpr (k != 0) p_r[a] += jr[k] * si[k];
        if constexpr (a != 0) p_i[a] -= jr[k] * sr[k];
        if constexpr (CPLX) {
          p_r[a] += ir[k] * sr[k];
          if constexpr (k != 0 && a != 0) p_i[a] += ir[k] * si[k];
        }
      }
    });
  });
  R sb[4];
  load_row<4>(cf.site[b], sb);
  // the arithmetic of a link no lane has is skipped in FP64 (a double-precision instruction costs 64 cycles)
  R w_dn = R((dn >> 24) & 0xFF), w_up = R(1);  // lanes without the link read zeros
  if (A.wsc) {
    const R n_b = dn < 0 ? R(0) : w_dn;
    w_up = scaled_up(A.wsc, A.wstride, b, n_b);
    w_dn = scaled_dn(A.wsc, A.wstride, b, n_b);
  }
  if (sizeof(R) == 4 || __any_sync(0xFFFFFFFFu, dn >= 0)) {
    const R al = w_dn * sb[2], be = w_dn * sb[3];
    p_r[0] += be * gr[0];
    static_for<1, N>([&](auto ac) {
      constexpr int a = decltype(ac)::value;
      p_r[a] += be * gr[a];
      p_r[a] += al * gi[a];
      p_i[a] += be * gi[a];
      p_i[a] -= al * gr[a];
    });
  }
  if (sizeof(R) == 4 || __any_sync(0xFFFFFFFFu, up >= 0)) {
    static_for<1, N>([&](auto ac) {
      constexpr int a = decltype(ac)::value;
      p_r[a] += w_up * ui[a];
      p_i[a] -= w_up * ur[a];
    });
  }
  // terminator of a leaf node, column part (the conjugate supplies the row part)
  if (A.terminator) {
    const R nj = dn < 0 ? R(0) : R(dn >> 24);
    const R c = up < 0 ? (nj + R(1)) / (ng + cf.gam[b]) : R(0);
    const R ca = c * sb[2], cb = c * sb[3];
    static_for<1, N>([&](auto ac) {
      constexpr int a = decltype(ac)::value;
      p_r[a] -= ca * sr[a];
      p_r[a] += cb * si[a];
      p_i[a] -= ca * si[a];
      p_i[a] -= cb * sr[a];
    });
  }
  // y of the owned elements (stage 0: the stage input is y)
  R y0;
  R2 y[N / 2 + 1];
  const unsigned pcol = (self >> 1) + N * 16 + lane + ob;  // (the pair at distance N/2 of its lower site: oh = ob)
  if (A.s != 0) {
    y0 = A.yv[(size_t)(self + lane + ob)];
    const R2* yo = reinterpret_cast<const R2*>(A.yv) + (size_t)pcol;
    static_for<1, N / 2 + 1>([&](auto dc) {
      constexpr int d = decltype(dc)::value;
      if (2 * d < N || low) y[d] = yo[cyc_pair(N, d) * 32];
    });
  } else {
    y0 = sr[0];
    static_for<1, N / 2 + 1>([&](auto dc) {
      constexpr int d = decltype(dc)::value;
      y[d].x = sr[d];
      y[d].y = -si[d];
    });
  }

  // hand over the elements of the pairs (b - d, b) to column b - d, take those of (b, b + d)
  if constexpr (N > 1) {
    static_for<1, D + 1>([&](auto dc) {
      constexpr int d = decltype(dc)::value;
      ex[om[d] + cyc_pair(N, d) * 32] = R2{p_r[N - d], p_i[N - d]};
    });
    if constexpr (EVEN) {
      if (!low) ex[oh + cyc_pair(N, N / 2) * 32] = R2{p_r[N / 2], p_i[N / 2]};
    }
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(32 * N) : "memory");
  }
  const bool root = MIXED && nb == 0 && lane == 0;
  R* wd = A.wout + (size_t)(self + lane + ob);
  {
    const R d = (p_r[0] + p_r[0]) - (ng + R(2) * cf.gd[b]) * sr[0];
    if (root) br.acc[b] = (float)d;
    *wd = y0 + A.h * d;
  }
  R2* wo = reinterpret_cast<R2*>(A.wout) + (size_t)pcol;
  static_for<1, N / 2 + 1>([&](auto dc) {
    constexpr int d = decltype(dc)::value;
    if (2 * d < N || low) {
      R sa[4];
      load_row<4>(cf.site[b + d], sa);
      const R w = sa[0] - sb[0], c = ng + (sa[1] + sb[1]);
      const R2 o = ex[ob + cyc_pair(N, d) * 32];
      R re = p_r[d] + o.x;
      R im = o.y - p_i[d];  // of sigma_{b, b+d}
      re += w * si[d];
      re -= c * sr[d];
      im += w * sr[d];
      im += c * si[d];
      if (root) {
        br.acc[N + 2 * (cyc_pair(N, d) + b)] = (float)re;
        br.acc[N + 2 * (cyc_pair(N, d) + b) + 1] = (float)im;
      }
      wo[cyc_pair(N, d) * 32] = R2{y[d].x + A.h * re, y[d].y + A.h * im};
    }
  });

  if (nb == 0) {
    __syncwarp();
    if constexpr (MIXED) {
      // float-float update of the root's owned elements, their hi parts to column 0 for the neighbours: lane 0 the
      // diagonal, lanes 2d-1 and 2d the pair at distance d
      const int d = (lane + 1) / 2;
      if (lane <= N && (lane == 0 || 2 * d < N || (2 * d == N && low))) {
        const int p = lane == 0 ? b : N + 2 * (cyc_pair(N, d) + b) + ((lane + 1) & 1);
        const FF w = ff_axpy(br.w[0][p], (float)A.h, A.hl, br.acc[p]);
        if (lane == 0) {
          // the eta, loss and xi rows of site b
          if (A.s == 2) {
            rw.ea[b].add_xi(I, b, br.w[A.in_sel][p]);
            rw.ea[b].step_xi(I);
          }
          if (A.s == 3) {
            rw.ea[b].add(I, b, br.w[A.in_sel][p]);
            static_cast<FF*>(I.y0)[b * (N + 1)] = w;  // for the stop rule
            if (rw.os.now && I.out_pops) I.out_pops[rw.os.row * N + b] = ff_to_double(w);
          }
        }
        br.w[A.out_sel][p] = w;
        A.wout[lane == 0 ? b * 32 : N * 32 + 64 * (cyc_pair(N, d) + b) + ((lane + 1) & 1)] = w.h;
      }
    } else {
      if (lane == 0) {
        if (A.s == 2) {
          rw.ea[b].add_xi(I, cfd, b, (double)sr[0]);
          rw.ea[b].step_xi(I);
        }
        if (A.s == 3) {
          rw.ea[b].add(I, cfd, N, b, (double)sr[0]);
          if (rw.os.now && I.out_pops) I.out_pops[rw.os.row * N + b] = (double)*wd;
        }
      }
    }
  }
}

// Reorders a block of 32 nodes in place: packed to cyclic order, or back (all lanes of a warp).
template <int N, typename R, bool TO_CYCLIC>
__device__ __forceinline__ void reorder_block(R* q, int lane) {
  R v[N * N];
  static_for<0, N * N>([&](auto pc) {
    constexpr int p = decltype(pc)::value;
    bool neg;
    const int c = cyc_index(N, p / N, p % N, lane, &neg);
    v[p] = q[TO_CYCLIC ? p * 32 + lane : c];
    if (neg) v[p] = -v[p];
  });
  __syncwarp();
  static_for<0, N * N>([&](auto pc) {
    constexpr int p = decltype(pc)::value;
    bool neg;
    q[TO_CYCLIC ? cyc_index(N, p / N, p % N, lane, &neg) : p * 32 + lane] = v[p];
  });
}

// link_cache: node blocks whose links a CTA's dynamic shared memory holds (all
// of the CTA's blocks, or none).
template <int N, typename R, bool MIXED, bool CPLX>
__global__ void __launch_bounds__(block_max_threads(N, (int)sizeof(R)), 1) heom_block_kernel(EngineArgs A, int link_cache) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ __align__(16) unsigned char s_coef[CoefLayout<R>::bytes(kMaxSmallN) + 64];
  __shared__ BlockRoot<N> s_root;
  __shared__ BlockRows<N, R> s_rows;
  __shared__ BlockCoef<N, R, CPLX> s_bc;
  __shared__ Inst s_inst;
  __shared__ int s_stop;
  constexpr int NN = N * N;

  int team, rank, team_size;
  if (A.mode == 0) {
    team = blockIdx.x / A.team_ctas;
    rank = blockIdx.x - team * A.team_ctas;
    team_size = A.team_ctas;
  } else {
    team = 0;
    rank = blockIdx.x;
    team_size = gridDim.x;
  }
  const int wid = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int sets = (blockDim.x >> 5) / N;
  const int set = wid / N, col = wid - set * N;
  // Blocks are dealt to the CTAs in turn (block k runs on CTA k % team_size), a CTA's blocks to its sets in turn.
  const bool lead = rank == 0 && threadIdx.x == 0;
  // the root's block runs on set 0 of rank 0; lane 0 of its warp b keeps the eta, loss and xi sums of site b
  const bool owner = rank == 0 && set == 0 && lane == 0;
  unsigned epoch = 0;
  typedef typename Vec2<R>::type R2;
  R2* const ex0 = reinterpret_cast<R2*>(dsm + (size_t)set * exch_bytes(N, (int)sizeof(R))) + lane;
  int32_t* const s_lk = reinterpret_cast<int32_t*>(dsm + (size_t)sets * exch_bytes(N, (int)sizeof(R)));
  int parity = 0;

  for (int li = A.team_first[team]; li < A.team_first[team + 1]; ++li) {
    load_instance<R>(A, li, s_inst, s_coef);
    const Inst& I = s_inst;
    const R* cf = reinterpret_cast<const R*>(s_coef);
    const double* cfd = reinterpret_cast<const double*>(s_coef + CoefLayout<R>::dbl_offset(N));
    const int nblk = (I.M + 31) >> 5;
    const int nloc = nblk > rank ? (nblk - rank + team_size - 1) / team_size : 0;
    const bool cached = nloc <= link_cache;
    if (cached)
      for (int i = threadIdx.x; i < nloc * N * 32; i += blockDim.x) {
        const int lb = i / (N * 32), j = (i >> 5) % N;
        const int n = ((lb * team_size + rank) << 5) + (i & 31);
        s_lk[i] = I.up[j * I.Mpad + n];
        s_lk[nloc * N * 32 + i] = I.dn[j * I.Mpad + n];
      }
    if (lead) {
      s_rows.os = OutStep{I.out_every == 1, 1};
      s_rows.rows.pending = -1;
      s_rows.rows.acc0 = I.acc[0];
      s_rows.rows.acc1 = I.acc[1];
      write_row0<N, R, MIXED>(I);
      for (int k = 0; k < N; ++k) {  // zero the running sums of every site
        s_rows.ea[k] = EtaAcc<R>{};
        s_rows.ea[k].store(I, k);
      }
    }
    for (int i = threadIdx.x; i < N * N * BlockCoef<N, R, CPLX>::JS; i += blockDim.x) {
      using L = CoefLayout<R>;
      constexpr int JS = BlockCoef<N, R, CPLX>::JS;
      const int k = i % JS, r = i / JS % N, c = i / (JS * N);
      s_bc.J[c][r][k] = k < N ? cf[L::J(N) + (c + r) % N * JS + (c + k) % N] : R(0);
      if constexpr (CPLX) s_bc.Ji[c][r][k] = k < N ? cf[L::Ji(N) + (c + r) % N * JS + (c + k) % N] : R(0);
      if (i < 8 * N) s_bc.site[i / 4][i % 4] = cf[L::site(N) + 4 * (i / 4 % N) + i % 4];
      if (i < N) {
        s_bc.gam[i] = cf[L::gam(N) + i];
        s_bc.gd[i] = cf[L::gd(N) + i];
      }
    }
    __syncthreads();  // row 0 before the reordering
    if constexpr (MIXED) {
      for (int p = threadIdx.x; p < NN; p += blockDim.x) {
        bool neg;
        const int q = root_index(N, p / N, p % N, &neg);
        const FF w = static_cast<const FF*>(I.y0)[p];
        s_root.w[0][q] = neg ? FF{-w.h, -w.l} : w;
      }
    }
    for (int lb = wid; lb < nloc; lb += blockDim.x >> 5)
      reorder_block<N, R, true>(static_cast<R*>(I.y) + (size_t)(lb * team_size + rank) * (NN * 32), lane);
    if (!team_barrier(A, epoch)) return;

    int64_t done = I.nsteps;
    for (int64_t t = 0; t < I.nsteps; ++t) {
#pragma unroll 1
      for (int s = 0; s < 4; ++s) {
        if (s == 0 && lead && s_rows.rows.pending >= 0) {
          eta_write_row<R>(I, N, s_rows.rows.acc0, s_rows.rows.acc1, s_rows.rows.pending, A.status);
          s_rows.rows.pending = -1;
        }
        int in_sel, out_sel;
        stage_buffers(s, in_sel, out_sel);
        StageArgs<R> S;
        S.win = static_cast<const R*>(in_sel == 0 ? I.y : (in_sel == 1 ? I.wa : I.wb));
        S.wout = static_cast<R*>(out_sel == 0 ? I.y : (out_sel == 1 ? I.wa : I.wb));
        S.yv = static_cast<const R*>(I.y);
        S.ngam = static_cast<const R*>(I.ngam);
        S.zero = (unsigned)(I.Mpad >> 5) * (NN * 32);
        S.h = sizeof(R) == 8 ? (R)I.hd[s] : (R)I.hh[s];
        S.hl = I.hl[s];
        S.s = s;
        S.in_sel = in_sel;
        S.out_sel = out_sel;
        S.terminator = I.terminator != 0;
        S.wsc = static_cast<const R*>(I.wsc);
        S.wstride = I.wstride;
#pragma unroll 1
        for (int lb = set; lb < nloc; lb += sets) {
          const int nb = lb * team_size + rank;
          int up, dn;
          if (cached) {
            up = s_lk[(lb * N + col) * 32 + lane];
            dn = s_lk[((nloc + lb) * N + col) * 32 + lane];
          } else {
            up = I.up[col * I.Mpad + nb * 32 + lane];
            dn = I.dn[col * I.Mpad + nb * 32 + lane];
          }
          column_stage<N, R, MIXED, CPLX>(I, s_bc, cfd, S, nb, lane, col, up, dn, s_rows, s_root,
                                          ex0 + parity * (N * (N - 1) / 2 * 32), 1 + set);
          parity ^= 1;
        }
        if (s == 3 && owner && (s_rows.os.now || t + 1 == I.nsteps)) s_rows.ea[col].store(I, col);
        if (!team_barrier(A, epoch)) return;
      }
      if (lead) {
        if (s_rows.os.now) s_rows.rows.pending = s_rows.os.row++;
        s_rows.os.now = t + 2 == I.out_every * s_rows.os.row;
      }
      if (I.stop_trace > 0.0 && t + 1 < I.nsteps && stop_now<R, MIXED>(I, N, &s_stop, 32)) {
        if (owner) s_rows.ea[col].store(I, col);
        done = t + 1;
        if (!team_barrier(A, epoch)) return;
        break;
      }
    }
    // back to packed order
    for (int lb = wid; lb < nloc; lb += blockDim.x >> 5)
      reorder_block<N, R, false>(static_cast<R*>(I.y) + (size_t)(lb * team_size + rank) * (NN * 32), lane);
    if constexpr (MIXED) {
      if (rank == 0)
        for (int p = threadIdx.x; p < NN; p += blockDim.x) {
          bool neg;
          const FF w = s_root.w[0][root_index(N, p / N, p % N, &neg)];
          static_cast<FF*>(I.y0)[p] = neg ? FF{-w.h, -w.l} : w;
        }
    }
    if (!team_barrier(A, epoch)) return;
    if (lead) finish_instance<R>(I, N, s_rows.rows, done, s_rows.os.row, N, A.status);
    if (!team_barrier(A, epoch)) return;
    if (lead) signal_done(I);
  }
}

}  // namespace heom
