// heom_large.cuh -- the engine for hierarchies with 9..24 sites.  Shares the
// descriptors, coefficient layout, barriers, eta sums and stop rule of
// heom_engine.cuh and the column form and cyclic order of heom_block.cuh:
//
//   D = P + P^+ + (local terms),  P = -i Q, column b of Q from column b of the
//   node and the links of site b:
//   Q_ab = (H' sigma)_ab + w_b sigma_{n+e_b, ab} + n_b (alpha_b + i beta_b) sigma_{n-e_b, ab}
//
// 32 consecutive nodes (one lane each) are computed by a set of warps of one
// CTA, a warp taking whole columns.  The state stays in cyclic order (state_elem),
// where pair (b, b+d) belongs to column b.  A block is done in two phases: the
// lower half of every column (its pairs (b-d, b), which their other column
// finishes) goes to the exchange area in shared memory; after a barrier the
// upper half (the diagonal and the pairs (b, b+d)) is computed, completed with
// the exchanged elements and the local terms, and stored.  So a thread holds
// the accumulators of half a column (26 registers in FP32, 52 in FP64 at N =
// 24), and every coupling read from shared memory (a broadcast) serves two
// multiply-adds, in FP32 packed two rows to an instruction (fma.rn.f32x2).
//
// FP32 first brings the block's stage input (74 KB at N = 24) into shared
// memory, since the two phases and the two columns of a pair read every element
// four times; FP64, bound by its pipe, reads it through L1.  Links that no lane
// of the warp has (most: a node of depth 4 has at most four nonzero n_j) are
// skipped by a vote, with their arithmetic.
//
// Bound and measured (24 sites, depth 4, 20 475 nodes, whole grid; in brackets
// the kernel this one took the place of, 4x4 blocks of 16 nodes with two lanes
// a node): mixed precision 70 us per stage [148], bound by issue slots, shared
// memory and the barriers between the phases of the one block an SM holds; FP64
// 1119 us [1800], bound by the FP64 pipe (the algorithm's multiply-adds alone
// 1000 us).  16 sites, mixed: 9.2 us [21] at depth 4, 27.3 [66] at depth 5.
// What made the difference in FP32, us per stage: y of a column read in one
// batch (a load between two stores waits for its own round trip) and the stage's
// arguments in shared memory instead of registers, 92 -> 80; two rows instead of
// the two parts of one row per packed multiply-add, which halves the bytes of
// couplings read (a broadcast 16-byte read takes two passes of the shared-memory
// pipe), 80 -> 70.  Tried and dropped: two columns a warp with absolute rows and
// a table of places 117 to 136, two columns with relative rows 105, the same
// with the staged block 99.5, rows in halves 102.
#pragma once

#include "heom_block.cuh"

namespace heom {

// Columns a warp takes, sets of a CTA, warps of a set.  FP32: a warp per column
// and 18 to 24 warps; FP64: two columns a warp (168 or 128 registers a thread).
__host__ __device__ constexpr int large_cols(int rsize) { return rsize == 8 ? 2 : 1; }
__host__ __device__ constexpr int large_set_warps(int N, int rsize) { return (N + large_cols(rsize) - 1) / large_cols(rsize); }
__host__ __device__ constexpr int large_sets(int N, int rsize) { return N <= (rsize == 8 ? 16 : 12) ? 2 : 1; }
__host__ __device__ constexpr int large_threads(int N, int rsize) {
  return 32 * large_set_warps(N, rsize) * large_sets(N, rsize);
}
// Coupling table [copy][N][jrow]: one copy per entry of a 16-byte word, each
// shifted by one entry more, so that a row's part starts a word in one of them
// from any column.
__host__ __device__ constexpr int large_jcopies(int rsize) { return 16 / rsize; }
__host__ __device__ constexpr int large_jrow(int N, int rsize) {
  const int w = large_jcopies(rsize);
  return (2 * N + 2 * w + w - 1) / w * w;  // columns to 2N - 2, the shift and the last word's rest
}
__host__ __device__ constexpr int large_jbytes(int N, int rsize) {
  return large_jcopies(rsize) * N * large_jrow(N, rsize) * rsize;
}
__host__ __device__ constexpr int large_stage_bytes(int N, int rsize) { return rsize == 4 ? N * N * 32 * 4 : 0; }
__host__ __device__ constexpr int large_exch_bytes(int N, int rsize) { return N * (N - 1) * 32 * rsize; }
__host__ __device__ constexpr int large_smem_bytes(int N, int rsize, bool cplx) {
  return (cplx ? 2 : 1) * large_jbytes(N, rsize) +
         large_sets(N, rsize) * (large_stage_bytes(N, rsize) + large_exch_bytes(N, rsize));
}

// Parts in which a team of `team` CTAs with `sets` sets each computes its last `rest` < sets * team blocks, at least three
// columns a part: those that make the largest share of a block on one CTA smallest.  A CTA's sets share its FP64 pipe, so
// sharing must save a CTA 5 % to be worth its extra reads (16 sites depth 4, 152 blocks on 152 CTAs, in halves 407 us a
// step against 370), but of two counts with the same share the larger keeps more sets busy (12 sites depth 4, 57 blocks:
// a half per CTA 122 us, two quarters 107).
__host__ __device__ constexpr int large_parts(int N, int sets, int team, int rest) {
  int best = 1, most = rest > 0 ? (rest + team - 1) / team : 1;  // parts, and those of the fullest CTA
  for (int p = 2; p <= N / 3 && p * rest <= sets * team; ++p) {
    const int m = (rest * p + team - 1) / team;
    if (best == 1 ? 20 * m < 19 * most * p : m * best <= most * p) {
      best = p;
      most = m;
    }
  }
  return best;
}

// The sum over k of J(k, row) sigma_k for NR rows: j holds NR couplings (and
// what fills the last 16-byte word), x and y multiply them into the real and
// imaginary sums.
template <typename R, int NR>
struct ColumnSum;
template <int NR>
struct ColumnSum<double, NR> {
  double re[NR], im[NR];
  __device__ __forceinline__ ColumnSum() {
#pragma unroll
    for (int i = 0; i < NR; ++i) re[i] = im[i] = 0.0;
  }
  __device__ __forceinline__ void add(const double* j, double x, double y) {
#pragma unroll
    for (int i = 0; i < NR; i += 2) {
      const double2 w = *reinterpret_cast<const double2*>(j + i);
      re[i] = fma(w.x, x, re[i]);
      im[i] = fma(w.x, y, im[i]);
      if (i + 1 < NR) {
        re[i + 1] = fma(w.y, x, re[i + 1]);
        im[i + 1] = fma(w.y, y, im[i + 1]);
      }
    }
  }
  __device__ __forceinline__ double2 get(int i) const { return double2{re[i], im[i]}; }
};
// FP32: two rows per packed multiply-add, so that a 16-byte read serves eight of them.
template <int NR>
struct ColumnSum<float, NR> {
  static constexpr int NQ = (NR + 1) / 2;
  unsigned long long re[NQ], im[NQ];  // rows 2q (low half) and 2q + 1
  __device__ __forceinline__ ColumnSum() {
#pragma unroll
    for (int i = 0; i < NQ; ++i) re[i] = im[i] = 0;
  }
  static __device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long j, unsigned long long v) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(j), "l"(v));
  }
  __device__ __forceinline__ void add(const float* j, float x, float y) {
    unsigned long long xx, yy;
    asm("mov.b64 %0, {%1, %1};" : "=l"(xx) : "f"(x));
    asm("mov.b64 %0, {%1, %1};" : "=l"(yy) : "f"(y));
#pragma unroll
    for (int q = 0; q < NQ; q += 2) {
      const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(j + 2 * q);
      fma2(re[q], w.x, xx);
      fma2(im[q], w.x, yy);
      if (q + 1 < NQ) {
        fma2(re[q + 1], w.y, xx);
        fma2(im[q + 1], w.y, yy);
      }
    }
  }
  static __device__ __forceinline__ float half(unsigned long long v, int i) {
    return __uint_as_float((unsigned)(i & 1 ? v >> 32 : v));
  }
  __device__ __forceinline__ float2 get(int i) const { return float2{half(re[i / 2], i), half(im[i / 2], i)}; }
};

// Barrier of `threads` threads (a set's warps).
__device__ __forceinline__ void set_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void copy16_async(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

template <int N, typename R>
struct LargeCoef {
  alignas(16) R site[2 * N][4];  // eps, goff, alpha, beta of site a at [a] and [a + N]
  R gam[N], gd[N];
};

// What the columns of one item share.
template <typename R>
struct LargeItem {
  const StageArgs<R>& S;  // in shared memory, so that the columns have the registers
  const R* win;    // the block's stage input: in shared memory (FP32) or device memory
  int nb, lane;
  R ng;
};

// Half of column b of Q: rows r0..r0+NR-1 (sites b + r).  BACK: the pairs (b-d, b), r = N-D..N-1; else the diagonal
// and the pairs (b, b+d), r = 0..D.  HALF (even N): with the pair at distance N/2.
template <int N, typename R, bool CPLX, bool BACK, bool HALF>
struct HalfColumn {
  typedef typename Vec2<R>::type R2;
  static constexpr int D = (N - 1) / 2;
  static constexpr int NR = (BACK ? D : D + 1) + (HALF ? 1 : 0);
  static constexpr int r0 = BACK ? (HALF ? N / 2 : N - D) : 0;
  R2 acc[NR];

  // place of the pair {b, b + r} (times 32), and whether its stored imaginary part is that of sigma_{b, b+r}
  static __device__ __forceinline__ int place(int r, int b) {
    if (2 * r < N) return (r - 1) * N + b;
    if (2 * r == N) return (N / 2 - 1) * N + (2 * b < N ? b : b - N / 2);
    const int d = N - r;
    return (d - 1) * N + (b >= d ? b - d : b - d + N);
  }
  static __device__ __forceinline__ bool forward(int r, int b) { return 2 * r < N || (2 * r == N && 2 * b < N); }

  // sum += J(b + k, b + r) v over the rows r
  static __device__ __forceinline__ void couple(ColumnSum<R, NR>& sum, const R* jt, const R* jti, int b, int site_k, R2 v) {
    constexpr int W = large_jcopies((int)sizeof(R));
    const int c0 = b + r0, copy = -c0 & (W - 1);
    const int at = (copy * N + site_k) * large_jrow(N, (int)sizeof(R)) + c0 + copy;
    sum.add(jt + at, v.x, v.y);
    // the table holds Ji(b + k, b + r) = -Ji(b + r, b + k); stored with that sign turned
    if constexpr (CPLX) sum.add(jti + at, -v.y, v.x);
  }

  __device__ __forceinline__ void compute(const LargeItem<R>& it, const LargeCoef<N, R>& cf, const R* jt, const R* jti,
                                          int b, int up, int dn) {
    const StageArgs<R>& S = it.S;
    ColumnSum<R, NR> sum;
    const R* diag = it.win + it.lane;
    const R2* pairs = reinterpret_cast<const R2*>(it.win + N * 32) + it.lane;
    // H' sigma, column entry by column entry
    couple(sum, jt, jti, b, b, R2{diag[b * 32], R(0)});
    {
      const R2* p = pairs + b * 32;
      int site = b;
#pragma unroll 4
      for (int k = 1; k <= D; ++k, p += N * 32) {
        site = site + 1 == N ? 0 : site + 1;
        const R2 v = *p;
        couple(sum, jt, jti, b, site, R2{v.x, -v.y});
      }
    }
    if constexpr (N % 2 == 0) {
      const bool low = 2 * b < N;
      const R2 v = pairs[((N / 2 - 1) * N + (low ? b : b - N / 2)) * 32];
      couple(sum, jt, jti, b, low ? b + N / 2 : b - N / 2, R2{v.x, low ? -v.y : v.y});
    }
    {
      int site = b;
      const R2* p = pairs;
#pragma unroll 4
      for (int d = 1; d <= D; ++d, p += N * 32) {
        site = site == 0 ? N - 1 : site - 1;
        couple(sum, jt, jti, b, site, p[site * 32]);
      }
    }
#pragma unroll
    for (int i = 0; i < NR; ++i) acc[i] = sum.get(i);
    // links of site b
    const R* sb = cf.site[b];
    R w_dn = R((dn >> 24) & 0xFF), w_up = R(1);
    if (S.wsc) {
      const R n_b = dn < 0 ? R(0) : w_dn;
      w_up = scaled_up(S.wsc, S.wstride, b, n_b);
      w_dn = scaled_dn(S.wsc, S.wstride, b, n_b);
    }
    // (the elements of a state may pass 2^32: 24 sites from depth 8)
    auto linked = [&](int l) { return S.win + (size_t)(l >= 0 ? (unsigned)(l >> 5) : S.zero) * (N * N * 32); };
    if (__any_sync(0xFFFFFFFFu, dn >= 0)) {
      const int m = dn < 0 ? -1 : (dn & 0xFFFFFF);
      const R* g0 = linked(m) + (m & 31);
      const R2* g = reinterpret_cast<const R2*>(linked(m) + N * 32) + (m & 31);
      const R al = w_dn * sb[2], be = w_dn * sb[3];
      static_for<0, NR>([&](auto ic) {
        constexpr int i = decltype(ic)::value, r = r0 + i;
        if constexpr (r == 0) {
          acc[i].y += be * g0[b * 32];
        } else {
          const R2 v = g[place(r, b) * 32];
          const R vi = forward(r, b) ? -v.y : v.y;
          acc[i].x += al * v.x;
          acc[i].x -= be * vi;
          acc[i].y += al * vi;
          acc[i].y += be * v.x;
        }
      });
    }
    if (__any_sync(0xFFFFFFFFu, up >= 0)) {
      const R2* g = reinterpret_cast<const R2*>(linked(up) + N * 32) + (up & 31);
      static_for<0, NR>([&](auto ic) {
        constexpr int i = decltype(ic)::value, r = r0 + i;
        if constexpr (r != 0) {
          const R2 v = g[place(r, b) * 32];
          acc[i].x += w_up * v.x;
          if (forward(r, b)) acc[i].y -= w_up * v.y;
          else acc[i].y += w_up * v.y;
        }
      });
    }
    // Markov terminator of a leaf node (see heom_block.cuh)
    if (S.terminator) {
      const R nj = dn < 0 ? R(0) : R(dn >> 24);
      const R c = up < 0 ? (nj + R(1)) / (it.ng + cf.gam[b]) : R(0);
      const R ca = c * sb[2], cb = c * sb[3];
      static_for<0, NR>([&](auto ic) {
        constexpr int i = decltype(ic)::value, r = r0 + i;
        if constexpr (r != 0) {
          const R2 v = pairs[place(r, b) * 32];
          const R vi = forward(r, b) ? -v.y : v.y;
          acc[i].x += cb * v.x;
          acc[i].x += ca * vi;
          acc[i].y += cb * vi;
          acc[i].y -= ca * v.x;
        }
      });
    }
  }
};

// First phase: the elements of column b that other columns finish.
template <int N, typename R, bool CPLX, bool HALF>
__device__ __forceinline__ void large_hand_over(const LargeItem<R>& it, const LargeCoef<N, R>& cf,
                                                const R* jt,
                                                const R* jti, int b, int up, int dn,
                                                typename Vec2<R>::type* ex) {
  typedef HalfColumn<N, R, CPLX, true, HALF> C;
  C c;
  c.compute(it, cf, jt, jti, b, up, dn);
  static_for<0, C::NR>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    ex[C::place(C::r0 + i, b) * 32] = typename Vec2<R>::type{c.acc[i].y, -c.acc[i].x};  // P = -i Q
  });
}

// What column c = b + d hands over to the pair (b, b+d), alone: for a block whose columns are shared out among CTAs.
// The same terms in the same order as in HalfColumn.
template <int N, typename R, bool CPLX>
__device__ __forceinline__ void large_hand_over_one(const Inst& I, const LargeItem<R>& it, const LargeCoef<N, R>& cf,
                                                    const R* jt, const R* jti, int b, int d,
                                                    typename Vec2<R>::type* ex) {
  typedef typename Vec2<R>::type R2;
  constexpr int D = (N - 1) / 2, JR = large_jrow(N, (int)sizeof(R));
  const StageArgs<R>& S = it.S;
  const int c = b + d < N ? b + d : b + d - N, at = ((d - 1) * N + b) * 32;
  const R2* pairs = reinterpret_cast<const R2*>(it.win + N * 32) + it.lane;
  R re = R(0), im = R(0);
  auto add = [&](int site, R x, R y) {
    const R j = jt[site * JR + b];
    re = fma(j, x, re);
    im = fma(j, y, im);
    if constexpr (CPLX) {
      const R ji = jti[site * JR + b];
      re = fma(ji, -y, re);
      im = fma(ji, x, im);
    }
  };
  add(c, it.win[c * 32 + it.lane], R(0));
  {
    const R2* p = pairs + c * 32;
    int site = c;
#pragma unroll 4
    for (int k = 1; k <= D; ++k, p += N * 32) {
      site = site + 1 == N ? 0 : site + 1;
      const R2 v = *p;
      add(site, v.x, -v.y);
    }
  }
  if constexpr (N % 2 == 0) {
    const bool low = 2 * c < N;
    const R2 v = pairs[((N / 2 - 1) * N + (low ? c : c - N / 2)) * 32];
    add(low ? c + N / 2 : c - N / 2, v.x, low ? -v.y : v.y);
  }
  {
    int site = c;
    const R2* p = pairs;
#pragma unroll 4
    for (int k = 1; k <= D; ++k, p += N * 32) {
      site = site == 0 ? N - 1 : site - 1;
      const R2 v = p[site * 32];
      add(site, v.x, v.y);
    }
  }
  const int up = I.up[c * I.Mpad + it.nb * 32 + it.lane], dn = I.dn[c * I.Mpad + it.nb * 32 + it.lane];
  const R* sb = cf.site[c];
  const R n_c = dn < 0 ? R(0) : R(dn >> 24);
  auto linked = [&](int l) {
    return reinterpret_cast<const R2*>(S.win + (size_t)(l >= 0 ? (unsigned)(l >> 5) : S.zero) * (N * N * 32) + N * 32);
  };
  if (__any_sync(0xFFFFFFFFu, dn >= 0)) {
    const int m = dn < 0 ? -1 : (dn & 0xFFFFFF);
    const R w = S.wsc ? scaled_dn(S.wsc, S.wstride, c, n_c) : n_c;
    const R al = w * sb[2], be = w * sb[3];
    const R2 v = linked(m)[(m & 31) + at];
    re += al * v.x;
    re -= be * v.y;
    im += al * v.y;
    im += be * v.x;
  }
  if (__any_sync(0xFFFFFFFFu, up >= 0)) {
    const R w = S.wsc ? scaled_up(S.wsc, S.wstride, c, n_c) : R(1);
    const R2 v = linked(up)[(up & 31) + at];
    re += w * v.x;
    im += w * v.y;
  }
  if (S.terminator) {
    const R q = up < 0 ? (n_c + R(1)) / (it.ng + cf.gam[c]) : R(0);
    const R ca = q * sb[2], cb = q * sb[3];
    const R2 v = pairs[at];
    re += cb * v.x;
    re += ca * v.y;
    im += cb * v.y;
    im -= ca * v.x;
  }
  ex[at] = R2{im, -re};  // P = -i Q
}

// Second phase: the diagonal b and the pairs (b, b+d), the Horner update and the stores.
template <int N, typename R, bool MIXED, bool CPLX, bool HALF>
__device__ __forceinline__ void large_finish(const Inst& I, const LargeItem<R>& it, const LargeCoef<N, R>& cf,
                                             const R* jt,
                                             const R* jti, const double* __restrict__ cfd,
                                             int b, int up, int dn, const typename Vec2<R>::type* ex,
                                             BlockRows<N, R>& rw, BlockRoot<MIXED ? N : 1>& br) {
  typedef typename Vec2<R>::type R2;
  typedef HalfColumn<N, R, CPLX, false, HALF> C;
  const StageArgs<R>& S = it.S;
  const int lane = it.lane;
  const size_t self = (size_t)it.nb * (N * N * 32);
  C c;
  c.compute(it, cf, jt, jti, b, up, dn);
  const R* sb = cf.site[b];
  const bool root = MIXED && it.nb == 0 && lane == 0;
  const R* yd = S.yv + self;
  const R2* yp = reinterpret_cast<const R2*>(yd + N * 32) + lane;
  R* wd = S.wout + self + b * 32 + lane;
  R2* wp = reinterpret_cast<R2*>(S.wout + self + N * 32) + lane;
  const R2* pairs = reinterpret_cast<const R2*>(it.win + N * 32) + lane;
  const R s0 = it.win[b * 32 + lane], y0 = yd[b * 32 + lane];
  // every y of the column before the first store: one trip to memory, not one per pair (the compiler keeps the order
  // of loads and stores that may meet)
  R2 y[C::NR];
  static_for<1, C::NR>([&](auto ic) {
    constexpr int r = decltype(ic)::value;
    y[r] = yp[((r - 1) * N + b) * 32];
  });
  {
    R d = R(2) * c.acc[0].y;
    d -= (it.ng + R(2) * cf.gd[b]) * s0;
    if (root) br.acc[b] = (float)d;
    *wd = y0 + S.h * d;
  }
  static_for<1, C::NR>([&](auto ic) {
    constexpr int r = decltype(ic)::value;
    const int k = (r - 1) * N + b;
    const R2 o = ex[k * 32], v = pairs[k * 32];
    const R* sa = cf.site[b + r];
    const R w = sa[0] - sb[0], g = it.ng + (sa[1] + sb[1]);
    R re = c.acc[r].y + o.x;
    R im = o.y + c.acc[r].x;  // of sigma_{b, b+r}
    re -= w * v.y;
    re -= g * v.x;
    im += w * v.x;
    im -= g * v.y;
    if (root) {
      br.acc[N + 2 * k] = (float)re;
      br.acc[N + 2 * k + 1] = (float)im;
    }
    c.acc[r] = R2{re, im};
  });
  static_for<1, C::NR>([&](auto ic) {
    constexpr int r = decltype(ic)::value;
    wp[((r - 1) * N + b) * 32] = R2{y[r].x + S.h * c.acc[r].x, y[r].y + S.h * c.acc[r].y};
  });
  if (it.nb == 0) {
    __syncwarp();
    if constexpr (MIXED) {
      // float-float update of the root's elements (lane 0 the diagonal, lanes 2d-1 and 2d the pair at distance d),
      // their hi parts to column 0 for the neighbours
      const int d = (lane + 1) / 2;
      if (lane <= 2 * (C::NR - 1)) {
        const int p = lane == 0 ? b : N + 2 * ((d - 1) * N + b) + ((lane + 1) & 1);
        const FF w = ff_axpy(br.w[0][p], (float)S.h, S.hl, br.acc[p]);
        if (lane == 0) {
          if (S.s == 2) {
            rw.ea[b].add_xi(I, b, br.w[S.in_sel][p]);
            rw.ea[b].step_xi(I);
          }
          if (S.s == 3) {
            rw.ea[b].add(I, b, br.w[S.in_sel][p]);
            static_cast<FF*>(I.y0)[b * (N + 1)] = w;  // for the stop rule
            if (rw.os.now && I.out_pops) I.out_pops[rw.os.row * N + b] = ff_to_double(w);
          }
        }
        br.w[S.out_sel][p] = w;
        S.wout[lane == 0 ? b * 32 : N * 32 + 64 * ((d - 1) * N + b) + ((lane + 1) & 1)] = w.h;
      }
    } else {
      if (lane == 0) {
        if (S.s == 2) {
          rw.ea[b].add_xi(I, cfd, b, (double)s0);
          rw.ea[b].step_xi(I);
        }
        if (S.s == 3) {
          rw.ea[b].add(I, cfd, N, b, (double)s0);
          if (rw.os.now && I.out_pops) I.out_pops[rw.os.row * N + b] = (double)*wd;
        }
      }
    }
  }
}

template <int N, typename R, bool MIXED, bool CPLX>
__global__ void __launch_bounds__(large_threads(N, (int)sizeof(R)), 1) heom_large_kernel(EngineArgs A) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ LargeCoef<N, R> s_cf;
  __shared__ double s_rates[2 * N];
  __shared__ BlockRoot<MIXED ? N : 1> s_root;
  __shared__ BlockRows<N, R> s_rows;
  __shared__ Inst s_inst;
  __shared__ StageArgs<R> s_stage;
  __shared__ int s_stop;
  typedef typename Vec2<R>::type R2;
  constexpr int NN = N * N;
  constexpr int RS = (int)sizeof(R);
  constexpr int SW = large_set_warps(N, RS), SETS = large_sets(N, RS);
  constexpr bool STAGED = RS == 4, EVEN = N % 2 == 0, SHARE = RS == 8;

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
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int set = wid / SW, sw = wid - set * SW;
  const bool lead = rank == 0 && threadIdx.x == 0;
  R* const jt = reinterpret_cast<R*>(dsm);
  R* const jti = reinterpret_cast<R*>(dsm + (CPLX ? large_jbytes(N, RS) : 0));
  unsigned char* const area = dsm + (CPLX ? 2 : 1) * large_jbytes(N, RS) +
                              (size_t)set * (large_stage_bytes(N, RS) + large_exch_bytes(N, RS));
  R* const stage = reinterpret_cast<R*>(area);
  R2* const ex = reinterpret_cast<R2*>(area + large_stage_bytes(N, RS)) + lane;
  unsigned epoch = 0;

  for (int li = A.team_first[team]; li < A.team_first[team + 1]; ++li) {
    __syncthreads();
    if (threadIdx.x == 0) s_inst = A.insts[A.team_list[li]];
    __syncthreads();
    const Inst& I = s_inst;
    {
      using L = CoefLayout<R>;
      const R* cf = static_cast<const R*>(I.coef);
      const double* rates = reinterpret_cast<const double*>(static_cast<const unsigned char*>(I.coef) + L::dbl_offset(N));
      constexpr int JR = large_jrow(N, RS);
      for (int i = threadIdx.x; i < large_jcopies(RS) * N * JR; i += blockDim.x) {
        const int copy = i / (N * JR), a = i / JR % N, c = i % JR - copy;
        const int col = c < 0 ? 0 : c % N;  // entries outside 0..2N-1 are never used, only read
        jt[i] = cf[L::J(N) + a * L::JS(N) + col];
        // Ji(b + r, b + k), read from row b + k
        if constexpr (CPLX) jti[i] = -cf[L::Ji(N) + a * L::JS(N) + col];
      }
      for (int i = threadIdx.x; i < 8 * N; i += blockDim.x) s_cf.site[i / 4][i % 4] = cf[L::site(N) + 4 * (i / 4 % N) + i % 4];
      for (int i = threadIdx.x; i < N; i += blockDim.x) {
        s_cf.gam[i] = cf[L::gam(N) + i];
        s_cf.gd[i] = cf[L::gd(N) + i];
        s_rates[i] = rates[i];
        s_rates[N + i] = rates[N + i];
      }
    }
    const int nblk = (I.M + 31) >> 5;
    // FP64: rounds in which every set has a block of its own, and the parts of each block of the round after them (the
    // only one of a small hierarchy).  With fewer blocks left than sets, several sets take a share of the columns of one,
    // and compute the elements that other columns would hand over themselves: more reads, the same arithmetic, and
    // fewer idle CTAs (see large_parts).  24 sites, depth 4 (640 blocks, 152 CTAs): 1300 -> 1119 us per stage; depth 1 (one
    // block, 8 CTAs): 273 -> 49.  FP32, bound by issue slots, shared memory and barriers, gained 2 % on the former and
    // lost 3 to 5 % where nothing is shared.
    const int slots = SETS * team_size, full = nblk / slots, rest = nblk - full * slots;
    const int parts = SHARE ? large_parts(N, SETS, team_size, rest) : 1;
    // the columns of the root's block this set runs: they keep its output rows and sums
    const int slot0 = set * team_size + rank;
    const bool root_shared = SHARE && full == 0;
    const int rc0 = root_shared ? min(slot0, parts) * N / parts : 0;
    const int rc1 = root_shared ? min(slot0 + 1, parts) * N / parts : (slot0 == 0 ? N : 0);
    if (threadIdx.x == 0) {
      s_rows.os = OutStep{I.out_every == 1, 1};
      s_rows.rows.pending = -1;
      s_rows.rows.acc0 = I.acc[0];
      s_rows.rows.acc1 = I.acc[1];
      for (int k = 0; k < N; ++k) s_rows.ea[k] = EtaAcc<R>{};
    }
    if (lead) {
      write_row0<N, R, MIXED>(I);
      for (int k = 0; k < N; ++k) s_rows.ea[k].store(I, k);  // zero the running sums of every site
    }
    if constexpr (MIXED) {
      for (int p = threadIdx.x; p < NN; p += blockDim.x) {
        bool neg;
        const int q = root_index(N, p / N, p % N, &neg);
        const FF w = static_cast<const FF*>(I.y0)[p];
        s_root.w[0][q] = neg ? FF{-w.h, -w.l} : w;
      }
    }
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
        __syncthreads();
        if (threadIdx.x == 0) {
          s_stage.win = static_cast<const R*>(in_sel == 0 ? I.y : (in_sel == 1 ? I.wa : I.wb));
          s_stage.wout = static_cast<R*>(out_sel == 0 ? I.y : (out_sel == 1 ? I.wa : I.wb));
          s_stage.yv = static_cast<const R*>(I.y);
          s_stage.ngam = static_cast<const R*>(I.ngam);
          s_stage.zero = (unsigned)(I.Mpad >> 5);
          s_stage.h = RS == 8 ? (R)I.hd[s] : (R)I.hh[s];
          s_stage.hl = I.hl[s];
          s_stage.s = s;
          s_stage.in_sel = in_sel;
          s_stage.out_sel = out_sel;
          s_stage.terminator = I.terminator != 0;
          s_stage.wsc = static_cast<const R*>(I.wsc);
          s_stage.wstride = I.wstride;
        }
        __syncthreads();
        const StageArgs<R>& S = s_stage;
        LargeItem<R> it{s_stage, nullptr, 0, lane, R(0)};
#pragma unroll 1
        for (int lb = set;; lb += SETS) {
          it.nb = lb * team_size + rank;
          int b0 = 0, b1 = N;
          if constexpr (SHARE) {
            if (lb >= full * SETS) {
              // the blocks of the last round, each in `parts` parts of its columns
              if (lb >= (full + 1) * SETS) break;
              const int part = slot0 % parts;
              it.nb = full * slots + slot0 / parts;
              b0 = part * N / parts;
              b1 = (part + 1) * N / parts;
            }
          }
          if (it.nb >= nblk) break;
          const R* src = S.win + (size_t)it.nb * (NN * 32);
          if constexpr (STAGED) {
            const int tid = sw * 32 + lane;
            for (int i = tid; i < NN * 8; i += SW * 32) copy16_async(stage + 4 * i, src + 4 * i);
            // the set's next block and this block's y on their way to L2
            const int next = it.nb + SETS * team_size;
            const char* pn = reinterpret_cast<const char*>(S.win + (size_t)next * (NN * 32));
            const char* py = reinterpret_cast<const char*>(S.yv + (size_t)it.nb * (NN * 32));
            for (int i = tid; i < NN; i += SW * 32) {
              if (next < nblk) prefetch_l2(pn + 128 * i);
              if (s != 0) prefetch_l2(py + 128 * i);
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            set_sync(1 + set, 32 * SW);
            it.win = stage;
          } else {
            it.win = src;
          }
          it.ng = S.ngam[it.nb * 32 + lane];
          if (!SHARE || b1 - b0 == N) {
#pragma unroll 1
            for (int b = sw; b < N; b += SW) {
              const int up = I.up[b * I.Mpad + it.nb * 32 + lane], dn = I.dn[b * I.Mpad + it.nb * 32 + lane];
              if (EVEN && 2 * b >= N) large_hand_over<N, R, CPLX, EVEN>(it, s_cf, jt, jti, b, up, dn, ex);
              else large_hand_over<N, R, CPLX, false>(it, s_cf, jt, jti, b, up, dn, ex);
            }
          } else if constexpr (SHARE) {
            constexpr int H = N / 2;
#pragma unroll 1
            for (int i = sw; i < (b1 - b0) * H; i += SW) {
              const int b = b0 + i / H, d = 1 + i % H;
              if (!EVEN || d < H || 2 * b < N) large_hand_over_one<N, R, CPLX>(I, it, s_cf, jt, jti, b, d, ex);
            }
          }
          set_sync(1 + set, 32 * SW);
#pragma unroll 1
          for (int b = b0 + sw; b < b1; b += SW) {
            const int up = I.up[b * I.Mpad + it.nb * 32 + lane], dn = I.dn[b * I.Mpad + it.nb * 32 + lane];
            if (EVEN && 2 * b < N)
              large_finish<N, R, MIXED, CPLX, EVEN>(I, it, s_cf, jt, jti, s_rates, b, up, dn, ex, s_rows, s_root);
            else
              large_finish<N, R, MIXED, CPLX, false>(I, it, s_cf, jt, jti, s_rates, b, up, dn, ex, s_rows, s_root);
          }
          set_sync(1 + set, 32 * SW);  // the set's areas are free again
        }
        // lane 0 of the warps that run the root's block keep the sums of their columns
        if (s == 3 && lane == 0 && (s_rows.os.now || t + 1 == I.nsteps))
          for (int b = rc0 + sw; b < rc1; b += SW) s_rows.ea[b].store(I, b);
        if (!team_barrier(A, epoch)) return;
      }
      if (threadIdx.x == 0) {
        if (s_rows.os.now) s_rows.rows.pending = s_rows.os.row++;
        s_rows.os.now = t + 2 == I.out_every * s_rows.os.row;
      }
      if (I.stop_trace > 0.0 && t + 1 < I.nsteps && stop_now<R, MIXED>(I, N, &s_stop)) {
        if (lane == 0)
          for (int b = rc0 + sw; b < rc1; b += SW) s_rows.ea[b].store(I, b);
        done = t + 1;
        if (!team_barrier(A, epoch)) return;
        break;
      }
    }
    if constexpr (MIXED) {
      if (rank == 0)
        for (int p = threadIdx.x; p < NN; p += blockDim.x) {
          bool neg;
          const FF w = s_root.w[0][root_index(N, p / N, p % N, &neg)];
          static_cast<FF*>(I.y0)[p] = neg ? FF{-w.h, -w.l} : w;
        }
      if (!team_barrier(A, epoch)) return;
    }
    if (lead) finish_instance<R>(I, N, s_rows.rows, done, s_rows.os.row, N, A.status);
    if (!team_barrier(A, epoch)) return;
    if (lead) signal_done(I);
  }
}

}  // namespace heom
