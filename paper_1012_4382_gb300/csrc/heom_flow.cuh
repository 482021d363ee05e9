// heom_flow.cuh -- the dataflow engine for one hierarchy with N <= 8 sites
// (launch mode 3): the whole GPU, no grid-wide barrier.
//
// Method: the same right-hand side and Horner-form RK4 as heom_engine.cuh
// (App. A2 Eqs. labsevena/lab8, App. A1, App. B), with trapping as the
// anti-Hermitian part of H_eff.
//
// Decomposition.  CTA c owns the SL = S * NPT consecutive nodes
// [c*SL, c*SL + SL) and keeps their three stage arrays (y, wa, wb) in shared
// memory for the whole call, node-major: element p of local node l at
// l*N*N + p.  Thread (u, l) of the CTA computes unit u (an off-diagonal pair
// (a, b), two packed reals, or a diagonal a) of the local nodes k*S + l,
// k = 0..NPT-1, in every stage (NPT nodes per thread, 1 by default).  The part of a unit's right-hand side
// that involves its own node -- the commutator with H_eff, the site-energy
// differences, the trap/decay and low-temperature damping -- is a fixed
// linear form in at most NRE (real part) and NIM (imaginary part) packed
// elements of the node; the host evaluates it once per unit and the thread
// keeps the nonzero coefficients and element indices in registers.  The
// node-dependent parts (the hierarchy damping -sum_j n_j gamma_j, the
// terminator at the last level, the up and down link weights, including the
// scaled hierarchy's) are folded into the same registers at the start of the
// call.  A stage is then a short sparse dot product over shared memory plus
// at most four neighbour pairs.
//
// Exchange.  Neighbour values go through global memory as 64-bit words that
// carry the stage they belong to: (tag << 32 | float bits) in FP32, two such
// words (low and high halves of the double) in FP64.  A thread gathers the
// words of its links n +- e_a, n +- e_b and waits (bounded) until every tag is
// the one of the previous stage, so it waits exactly for the values it reads,
// and no flag, fence or barrier crosses CTAs.  The dependence is symmetric
// (unit (a, b) of n reads element (a, b) of n +- e_a, n +- e_b, and unit (a, b)
// of each of those reads element (a, b) of n), so a writer of stage s + 1 has
// always seen every reader of its stage-s value finish: three tagged buffers
// (y, wa, wb) in the Horner rotation are enough.  Diagonal units also wait on
// their up link, whose weight is zero, to keep that symmetry.  Within a CTA
// the stages are separated by __syncthreads.
//
// Tags: the call starts at tag0; the initial y carries tag0 + 1 and the output
// of step t, stage s carries tag0 + 4t + s + 2, so stage s of step t waits for
// tag0 + 4t + s + 1.  The host advances tag0 by 4 nsteps + 2 per call and
// clears the buffers before the 32-bit tags would wrap, so a stale word never
// carries an expected tag.
#pragma once

#include "heom_engine.cuh"

namespace heom {

constexpr int kFlowMaxE = 28;   // 4N - 4 at N = 8
constexpr int kFlowRing = 64;   // stop-rule decisions kept in flight
// Threads per CTA the kernels are compiled for: at most 168 registers a thread,
// so that a CTA of 13 nodes at N = 7 (364 threads) fits one SM; real-H kernels
// do not spill at this budget.
constexpr int kFlowMaxThreads = 384;
// Threads per CTA of the kernels whose threads carry several nodes (NPT > 1):
// eight warps, two per SM sub-partition, so that a thread may hold 255
// registers (with ten or twelve warps some sub-partition holds three, and its
// register file allows 168).
constexpr int kFlowMaxThreadsMulti = 256;
constexpr int kFlowMaxNpt = 6;       // accepted by the launch shape
// built; more nodes per thread run the throughput engine (see launch_flow)
__host__ __device__ constexpr int flow_built_npt(int N) { return N == 8 ? 2 : 3; }

// One unit's own-node linear form (host-built).  Slot 0 of both lists is the
// unit's own real element x = P[a*N + b]; for a pair, slot 1 is its imaginary
// element yi = P[b*N + a] (the node-dependent terms are added to these two
// slots); the other slots hold the remaining elements with a nonzero weight,
// and unused slots have weight 0.
struct FlowUnit {
  uint8_t ire[kFlowMaxE];
  uint8_t iim[kFlowMaxE];
  uint8_t a, b, pad[6];
  double cre[kFlowMaxE];
  double cim[kFlowMaxE];
};
// Per-site bath data in double (host-built, after the units).
struct FlowSite {
  double alpha, beta, gamma, scale;  // 2 lambda k_B T, lambda gamma, gamma, s_j of the scaled hierarchy
};

struct FlowArgs {
  const Inst* inst;                  // the one instance
  const FlowUnit* units;             // [U] then FlowSite[N]
  unsigned long long* tags;          // tagged y, wa, wb, one after the other: [N*N][Mpad] words each
                                     // (FP64: pairs of words)
  long long tag_stride;              // words from one tagged buffer to the next
  unsigned long long* ring;          // [kFlowRing] stop decisions
  int* status;
  int S;                             // nodes per CTA
  unsigned tag0;
};

__host__ __device__ constexpr int flow_nre(int N, bool cplx) {
  return (cplx ? 4 * N - 4 : 2 * N - 2) < 2 ? 2 : (cplx ? 4 * N - 4 : 2 * N - 2);
}
__host__ __device__ constexpr int flow_nim(int N, bool cplx) {
  return (cplx ? 4 * N - 4 : 2 * N) < 2 ? 2 : (cplx ? 4 * N - 4 : 2 * N);
}
// Dynamic shared memory of a CTA whose slice holds S nodes.
__host__ __device__ constexpr int flow_smem_bytes(int N, int S, int rsize) { return 3 * S * N * N * rsize; }

// ------------------------------------------------------------ tagged words

__device__ __forceinline__ void flow_store(unsigned long long* p, float v, unsigned tag) {
  const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w));
}
__device__ __forceinline__ void flow_store(unsigned long long* p, double v, unsigned tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | (b & 0xFFFFFFFFull)),
               "l"(t | (b >> 32)));
}

// A gathered word (FP32) or pair of words (FP64) and its check.
template <typename R>
struct FlowWord;
template <>
struct FlowWord<float> {
  unsigned long long w = 0;
  __device__ __forceinline__ void load(const unsigned long long* p) {
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p));
  }
  __device__ __forceinline__ bool ok(unsigned tag) const { return (unsigned)(w >> 32) == tag; }
  __device__ __forceinline__ float value() const { return __uint_as_float((unsigned)w); }
};
template <>
struct FlowWord<double> {
  unsigned long long lo = 0, hi = 0;
  __device__ __forceinline__ void load(const unsigned long long* p) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(p));
  }
  __device__ __forceinline__ bool ok(unsigned tag) const {
    return (unsigned)(lo >> 32) == tag && (unsigned)(hi >> 32) == tag;
  }
  __device__ __forceinline__ double value() const {
    return __hiloint2double((int)(unsigned)hi, (int)(unsigned)lo);
  }
};
template <typename R>
__host__ __device__ constexpr int flow_words() {
  return sizeof(R) == 8 ? 2 : 1;
}

// The eta and loss row `row` from the diagonal owners' running sums in shared
// memory (the same sums, in the same order, as eta_total reads from the parts
// slots), and the check of the row for NaN or infinity; the population row
// is the root's diagonal of the step's y, also in shared memory.
template <typename R, bool MIXED>
__device__ __forceinline__ void flow_eta_row(const Inst& I, const EtaAcc<R>* ea, const FF* trace_ff,
                                             const double* trace_d, int N, double acc0, double acc1, int64_t row,
                                             int* status) {
  double e, l;
  if constexpr (sizeof(R) == 4) {
    FF se{0.f, 0.f}, sl{0.f, 0.f};
    for (int k = 0; k < N; ++k) {
      se = ff_add(se, ea[k].e);
      sl = ff_add(sl, ea[k].l);
    }
    e = acc0 + ff_to_double(se);
    l = acc1 + ff_to_double(sl);
  } else {
    double se = 0.0, sl = 0.0;
    for (int k = 0; k < N; ++k) {
      se += ea[k].e;
      sl += ea[k].l;
    }
    e = acc0 + se;
    l = acc1 + sl;
  }
  flag_nonfinite(status, e);
  flag_nonfinite(status, l);
  for (int k = 0; k < N; ++k) flag_nonfinite(status, MIXED ? ff_to_double(trace_ff[k]) : trace_d[k]);
  if (!I.out_el) return;
  I.out_el[2 * row] = e;
  I.out_el[2 * row + 1] = l;
}

// ------------------------------------------------------------------ kernel
//
// NPT nodes per thread: thread (u, l) of CTA c computes unit u of the nodes
// c*S*NPT + k*S + l, k = 0..NPT-1 (the lanes of a warp stay consecutive nodes
// of one unit for every k, so the exchange keeps its coalescing).  A thread
// first runs the own-node parts and issues the gathers of all its nodes
// (independent chains the compiler interleaves), then waits for and updates
// them node by node, so one exchange latency covers all of its nodes.
// NPT = 1 runs the steps in the same order as a plain one-node-per-thread
// kernel.
template <int N, typename R, bool MIXED, bool CPLX, int NPT = 1>
__global__ void __launch_bounds__(NPT == 1 ? kFlowMaxThreads : kFlowMaxThreadsMulti) heom_flow_kernel(FlowArgs A) {
  constexpr int NN = N * N;
  constexpr int NP = N * (N - 1) / 2;
  constexpr int U = NP + N;
  constexpr int NRE = flow_nre(N, CPLX);
  constexpr int NIM = flow_nim(N, CPLX);
  constexpr int WD = flow_words<R>();
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ Inst s_inst;
  __shared__ int s_abort, s_stop;
  // the root node (CTA 0, local node 0): float-float y and stage outputs of the
  // mixed path, and the eta/loss/xi running sums of its diagonal owners
  __shared__ FF s_ry[kMaxSmallN * kMaxSmallN], s_rw[kMaxSmallN];
  __shared__ EtaAcc<R> s_ea[kMaxSmallN];
  __shared__ FF s_trace_ff[kMaxSmallN];
  __shared__ double s_trace_d[kMaxSmallN];

  const int S = A.S;        // threads per unit: nodes of one row of the slice
  const int SL = S * NPT;   // nodes of the CTA's slice
  const int u = threadIdx.x / S;
  const int l = threadIdx.x - u * S;
  if (threadIdx.x == 0) {
    s_inst = *A.inst;
    s_abort = 0;
    s_stop = 0;
  }
  __syncthreads();
  const Inst& I = s_inst;
  const int M = I.M, Mp = I.Mpad;
  int nd[NPT];
  bool valid[NPT];
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    nd[k] = blockIdx.x * SL + k * S + l;
    valid[k] = u < U && nd[k] < M;
  }
  const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
  R* const sb = reinterpret_cast<R*>(dsm);  // stage buffer k at sb + k * SL * NN

  // ---- the thread's unit and its linear form (shared by its nodes); per node
  // the slots 0 and 1 of both forms (where the node's damping and terminator
  // enter), the links and the link weights
  int a = 0, b = 0, pab = 0, pba = 0;
  uint32_t ire4[(NRE + 3) / 4], iim4[(NIM + 3) / 4];
  R cre[NRE], cim[NIM];
  R c0r[NPT], c1r[NPT], c0i[NPT], c1i[NPT];
  int hl[NPT][4];  // up a, up b, down a, down b
  R cu_a[NPT], cu_b[NPT], pd_a[NPT], qd_a[NPT], pd_b[NPT], qd_b[NPT];
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    c0r[k] = c1r[k] = c0i[k] = c1i[k] = R(0);
    cu_a[k] = cu_b[k] = pd_a[k] = qd_a[k] = pd_b[k] = qd_b[k] = R(0);
#pragma unroll
    for (int j = 0; j < 4; ++j) hl[k][j] = -1;
  }
  const bool root = valid[0] && nd[0] == 0;  // only node 0 of a thread can be the root
  if (valid[0]) {
    const FlowUnit& fu = A.units[u];
    const FlowSite* fs = reinterpret_cast<const FlowSite*>(A.units + U);
    a = fu.a;
    b = fu.b;
    pab = a * N + b;
    pba = b * N + a;
#pragma unroll
    for (int i = 0; i < (NRE + 3) / 4; ++i) {
      uint32_t w = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * i + k < NRE) w |= (uint32_t)fu.ire[4 * i + k] << (8 * k);
      ire4[i] = w;
    }
#pragma unroll
    for (int i = 0; i < (NIM + 3) / 4; ++i) {
      uint32_t w = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (4 * i + k < NIM) w |= (uint32_t)fu.iim[4 * i + k] << (8 * k);
      iim4[i] = w;
    }
    double dre[NRE], dim[NIM];
#pragma unroll
    for (int i = 0; i < NRE; ++i) dre[i] = fu.cre[i];
#pragma unroll
    for (int i = 0; i < NIM; ++i) dim[i] = fu.cim[i];
#pragma unroll
    for (int i = 0; i < NRE; ++i) cre[i] = (R)dre[i];
#pragma unroll
    for (int i = 0; i < NIM; ++i) cim[i] = (R)dim[i];
    const FlowSite sa = fs[a], sbs = fs[b];
    const bool scaled = I.wsc != nullptr;
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      if (!valid[k]) continue;
      const int n = nd[k];
      // node data: links, n_a, n_b, sum_j n_j gamma_j, last level
      const int ra = I.dn[a * Mp + n], rb = I.dn[b * Mp + n];
      const int ua = I.up[a * Mp + n], ub = I.up[b * Mp + n];
      const double na = ra < 0 ? 0.0 : (double)(ra >> 24), nb = rb < 0 ? 0.0 : (double)(rb >> 24);
      const double ng = (double)static_cast<const R*>(I.ngam)[n];
      const bool leaf = I.up[n] < 0;
      double x0r = dre[0], x1r = dre[1], x0i = dim[0], x1i = dim[1];
      x0r -= ng;  // hierarchy damping -sum_j n_j gamma_j on x (and on yi below)
      if (a != b) {
        x1i -= ng;
        if (I.terminator && leaf) {
          // sigma_{n+e_j} ~ (n_j+1)/(ngam+gamma_j) theta_j sigma_n, then i V_j^x of it (j = a, b)
          const double ca = (na + 1.0) / (ng + sa.gamma), cb = (nb + 1.0) / (ng + sbs.gamma);
          x0r += -ca * sa.alpha - cb * sbs.alpha;
          x1r += -ca * sa.beta + cb * sbs.beta;
          x0i += ca * sa.beta - cb * sbs.beta;
          x1i += -ca * sa.alpha - cb * sbs.alpha;
        }
        // up links i V_j^x sigma_{n+e_j}: re += cu Im(up), im -= cu Re(up); weight 1, or
        // sqrt((n_j+1) s_j) in the scaled hierarchy
        hl[k][0] = ua;
        hl[k][1] = ub;
        cu_a[k] = (R)(-(scaled ? sqrt((na + 1.0) * sa.scale) : 1.0));
        cu_b[k] = (R)(scaled ? sqrt((nb + 1.0) * sbs.scale) : 1.0);
        // down links n_j theta_j sigma_{n-e_j}: re += p Re - q Im, im += q Re + p Im
        hl[k][2] = ra < 0 ? -1 : (ra & 0xFFFFFF);
        hl[k][3] = rb < 0 ? -1 : (rb & 0xFFFFFF);
        const double wa = scaled ? sqrt(na / sa.scale) : na, wb = scaled ? sqrt(nb / sbs.scale) : nb;
        pd_a[k] = (R)(wa * sa.beta);
        qd_a[k] = (R)(wa * sa.alpha);
        pd_b[k] = (R)(wb * sbs.beta);
        qd_b[k] = (R)(-wb * sbs.alpha);
      } else {
        // the up link carries no weight for a diagonal; it is still waited on (see above)
        hl[k][0] = ua;
        hl[k][2] = ra < 0 ? -1 : (ra & 0xFFFFFF);
        const double wa = scaled ? sqrt(na / sa.scale) : na;
        pd_a[k] = (R)(2.0 * wa * sa.beta);
      }
      c0r[k] = (R)x0r;
      c1r[k] = (R)x1r;
      c0i[k] = (R)x0i;
      c1i[k] = (R)x1i;
    }
  }
  const bool pair = a != b;

  // ---- the state: own elements in registers (the Horner base), slice in shared memory
  R y_r[NPT], y_i[NPT];
  // Element o = p * Mpad + n of the tagged buffers in the blocked state array.  Derived from o, which the step loop needs
  // anyway: with the blocked index computed from p and n the compiler kept addresses of both alive over the loop, in
  // registers that the FP64 and complex kernels do not have (us per step, FP64, complex H: 8 sites depth 4 19.3 against
  // 14.9, seven sites depth 6 25.9 against 25.2; mixed: seven sites depth 6 complex 5.9 against 5.2, 5 sites depth 12 10.4
  // against 8.2).  Three sites with real H in mixed precision do have them: depth 9 4.6 us a step that way, 4.85 this way.
  auto blocked = [&I](int o, int p, int n) {
    if constexpr (!(MIXED && !CPLX && N == 3)) {
      p = o / I.Mpad;
      n = o - p * I.Mpad;
    }
    return node_col<N>(n) + p * 32;
  };
  const R* gy = static_cast<const R*>(I.y);
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    y_r[k] = y_i[k] = R(0);
    if (!valid[k]) continue;
    const int oab = pab * Mp + nd[k], oba = pba * Mp + nd[k];
    y_r[k] = gy[blocked(oab, pab, nd[k])];
    y_i[k] = pair ? gy[blocked(oba, pba, nd[k])] : R(0);
    R* own = sb + (k * S + l) * NN;
    own[pab] = y_r[k];
    if (pair) own[pba] = y_i[k];
    flow_store(A.tags + WD * oab, y_r[k], A.tag0 + 1);
    if (pair) flow_store(A.tags + WD * oba, y_i[k], A.tag0 + 1);
  }
  if constexpr (MIXED) {
    if (root) {
      const FF* y0 = static_cast<const FF*>(I.y0);
      s_ry[pab] = y0[pab];
      if (pair) s_ry[pba] = y0[pba];
    }
  }
  if (root && !pair) s_ea[a] = EtaAcc<R>{};
  EtaRows rows;
  rows.acc0 = I.acc[0];
  rows.acc1 = I.acc[1];
  const bool diag_root = root && !pair;  // owner of the root's diagonal a: eta slot a, sums in s_ea[a]
  const double* cfd = reinterpret_cast<const double*>(static_cast<const unsigned char*>(I.coef) +
                                                      CoefLayout<R>::dbl_offset(N));
  if (lead) {
    write_row0<N, R, MIXED>(I);
    const EtaAcc<R> zero{};
    for (int k = 0; k < N; ++k) zero.store(I, k);  // zero every running-sum slot
  }
  __syncthreads();

  int64_t next_out = I.out_every, orow = 1, done = I.nsteps;
  for (int64_t t = 0; t < I.nsteps; ++t) {
    const OutStep os{t + 1 == next_out, orow};
    if (os.now) {
      next_out += I.out_every;
      ++orow;
    }
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      if (s == 0 && rows.pending >= 0) {
        if (lead) flow_eta_row<R, MIXED>(I, s_ea, s_trace_ff, s_trace_d, N, rows.acc0, rows.acc1, rows.pending, A.status);
        rows.pending = -1;
      }
      const int in_sel = (s == 0) ? 0 : (s == 2 ? 2 : 1);
      const int out_sel = (s == 1) ? 2 : (s == 3 ? 0 : 1);
      const unsigned want = A.tag0 + 4u * (unsigned)t + (unsigned)s + 1u;
      const unsigned long long* tin = A.tags + in_sel * A.tag_stride;
      R re[NPT], im[NPT];
      FlowWord<R> gr[NPT][4], gi[NPT][4];
      bool aborted = false;
      // the own-node part (shared memory), then the neighbours: by the time the
      // gathers reach L2 their producers have mostly stored (measured: equal in
      // FP32, 15 % faster in FP64 than gathering first)
      auto own_and_gather = [&](auto kc) {
        constexpr int k = decltype(kc)::value;
        re[k] = R(0);
        im[k] = R(0);
        if (!valid[k]) return;
        const R* sin = sb + in_sel * SL * NN + (k * S + l) * NN;
#pragma unroll
        for (int i = 0; i < NRE; ++i)
          re[k] += (i == 0 ? c0r[k] : (i == 1 ? c1r[k] : cre[i])) * sin[(ire4[i / 4] >> (8 * (i % 4))) & 0xFF];
        if (pair) {  // a diagonal has no imaginary part; its units fill the last warps of a CTA
#pragma unroll
          for (int i = 0; i < NIM; ++i)
            im[k] += (i == 0 ? c0i[k] : (i == 1 ? c1i[k] : cim[i])) * sin[(iim4[i / 4] >> (8 * (i % 4))) & 0xFF];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (hl[k][j] >= 0) {
            gr[k][j].load(tin + WD * (pab * Mp + hl[k][j]));
            gi[k][j].load(tin + WD * (pba * Mp + hl[k][j]));
          }
      };
      // wait, bounded, until every gathered word of node k carries the previous stage's tag
      auto wait_words = [&](auto kc) -> bool {
        constexpr int k = decltype(kc)::value;
        bool ready = true;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (hl[k][j] >= 0) ready = ready & gr[k][j].ok(want) & gi[k][j].ok(want);
        if (ready) return true;
        uint64_t t0 = 0;
        for (unsigned spins = 1;; ++spins) {
          // reload every word that is not there yet, then check them all
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (hl[k][j] >= 0) {
              if (!gr[k][j].ok(want)) gr[k][j].load(tin + WD * (pab * Mp + hl[k][j]));
              if (!gi[k][j].ok(want)) gi[k][j].load(tin + WD * (pba * Mp + hl[k][j]));
            }
          ready = true;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (hl[k][j] >= 0) ready = ready & gr[k][j].ok(want) & gi[k][j].ok(want);
          if (ready) return true;
          if ((spins & 255u) == 0) {
            if (ld_volatile(A.status) & kStatusTimeout) {
              s_abort = 1;
              return false;
            }
            const uint64_t now = global_timer_ns();
            if (t0 == 0) {
              t0 = now;
            } else if (now - t0 > kBarrierLimitNs) {
              atomicOr(A.status, kStatusTimeout);
              s_abort = 1;
              return false;
            }
          }
        }
      };
      // the neighbour terms, the Horner update and the stores of node k
      auto finish = [&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const R ur = gr[k][0].value(), ui = gi[k][0].value(), vr = gr[k][1].value(), vi = gi[k][1].value();
        const R dr = gr[k][2].value(), di = gi[k][2].value(), er = gr[k][3].value(), ei = gi[k][3].value();
        // absent links were never loaded and read as 0
        R rr = re[k], mm = im[k];
        rr += cu_a[k] * ui + cu_b[k] * vi + pd_a[k] * dr - qd_a[k] * di + pd_b[k] * er - qd_b[k] * ei;
        mm += -cu_a[k] * ur - cu_b[k] * vr + qd_a[k] * dr + pd_a[k] * di + qd_b[k] * er + pd_b[k] * ei;
        R w_r, w_i;
        const unsigned tag_out = want + 1u;
        const bool rt = k == 0 && root;
        if (MIXED && rt) {
          if constexpr (MIXED) {
            const float hh = I.hh[s], hlo = I.hl[s];
            if (!pair) {
              // eta, loss and xi rows of the augmented system: the float-float stage input
              if (s == 3) s_ea[a].add(I, a, s_rw[a]);
              if (s == 2) s_ea[a].add_xi(I, a, s_rw[a]);
            }
            const FF fr = ff_axpy(s_ry[pab], hh, hlo, rr);
            const FF fi = pair ? ff_axpy(s_ry[pba], hh, hlo, mm) : FF{0.f, 0.f};
            w_r = fr.h;
            w_i = fi.h;
            if (!pair) s_rw[a] = fr;
            if (s == 3) {
              s_ry[pab] = fr;
              if (pair) s_ry[pba] = fi;
              if (!pair && os.now && I.out_pops) I.out_pops[os.row * N + a] = ff_to_double(fr);
            }
          }
        } else {
          if constexpr (!MIXED) {
            if (rt && !pair) {
              const R* sin = sb + in_sel * SL * NN + (k * S + l) * NN;
              if (s == 3) s_ea[a].add(I, cfd, N, a, (double)sin[pab]);
              if (s == 2) s_ea[a].add_xi(I, cfd, a, (double)sin[pab]);
            }
          }
          const R h = sizeof(R) == 8 ? (R)I.hd[s] : (R)I.hh[s];
          w_r = y_r[k] + h * rr;
          w_i = y_i[k] + h * mm;
          if (s == 3 && rt && !pair && os.now && I.out_pops) I.out_pops[os.row * N + a] = (double)w_r;
        }
        R* sout = sb + out_sel * SL * NN + (k * S + l) * NN;
        unsigned long long* tout = A.tags + out_sel * A.tag_stride;
        const int oab = pab * Mp + nd[k], oba = pba * Mp + nd[k];
        sout[pab] = w_r;
        flow_store(tout + WD * oab, w_r, tag_out);
        if (pair) {
          sout[pba] = w_i;
          flow_store(tout + WD * oba, w_i, tag_out);
        }
        if (s == 3) {
          y_r[k] = w_r;
          y_i[k] = w_i;
        }
        if (k == 0 && diag_root) {
          if (s == 2) s_ea[a].step_xi(I);
          if (s == 3) {
            if (os.now || t + 1 == I.nsteps) s_ea[a].store(I, a);
            if constexpr (MIXED) s_trace_ff[a] = s_ry[pab];
            else s_trace_d[a] = (double)w_r;
          }
        }
      };
      // every node's own-node part and gathers first (independent chains the
      // compiler interleaves), then the waits and updates node by node
      static_for<0, NPT>([&](auto kc) { own_and_gather(kc); });
      static_for<0, NPT>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        if (valid[k] && !aborted) {
          if (wait_words(kc)) finish(kc);
          else aborted = true;
        }
      });
      __syncthreads();
      if (s_abort) return;
    }
    if (os.now) rows.pending = os.row;
    if (I.stop_trace > 0.0 && t + 1 < I.nsteps) {
      // the stop rule: CTA 0 holds the root and decides; every CTA waits for the decision of this step
      const unsigned dtag = A.tag0 + (unsigned)t + 1u;
      unsigned long long* slot = A.ring + (t % kFlowRing);
      if (threadIdx.x == 0) {
        if (blockIdx.x == 0) {
          double tr = 0.0;
          if constexpr (MIXED) {
            FF sum{0.f, 0.f};
            for (int k = 0; k < N; ++k) sum = ff_add(sum, s_trace_ff[k]);
            tr = ff_to_double(sum);
          } else {
            for (int k = 0; k < N; ++k) tr += s_trace_d[k];
          }
          const unsigned long long w = ((unsigned long long)dtag << 32) | (tr < I.stop_trace ? 1ull : 0ull);
          asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(slot), "l"(w));
          s_stop = (int)(w & 1ull);
        } else {
          unsigned long long w = 0;
          uint64_t t0 = 0;
          for (unsigned spins = 1;; ++spins) {
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(slot));
            if ((unsigned)(w >> 32) == dtag) break;
            if ((spins & 255u) == 0) {
              if (ld_volatile(A.status) & kStatusTimeout) {
                s_abort = 1;
                break;
              }
              const uint64_t now = global_timer_ns();
              if (t0 == 0) {
                t0 = now;
              } else if (now - t0 > kBarrierLimitNs) {
                atomicOr(A.status, kStatusTimeout);
                s_abort = 1;
                break;
              }
            }
          }
          s_stop = (int)(w & 1ull);
        }
      }
      __syncthreads();
      if (s_abort) return;
      if (s_stop) {
        if (diag_root) s_ea[a].store(I, a);
        done = t + 1;
        break;
      }
    }
  }
  // the state back to device memory (packed, see node_col; the root also in float-float)
  R* gyw = static_cast<R*>(I.y);
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    if (!valid[k]) continue;
    const int oab = pab * Mp + nd[k], oba = pba * Mp + nd[k];
    gyw[blocked(oab, pab, nd[k])] = y_r[k];
    if (pair) gyw[blocked(oba, pba, nd[k])] = y_i[k];
  }
  if constexpr (MIXED) {
    if (root) {
      FF* y0 = static_cast<FF*>(I.y0);
      y0[pab] = s_ry[pab];
      if (pair) y0[pba] = s_ry[pba];
    }
  }
  __syncthreads();
  if (lead) finish_instance<R>(I, N, rows, done, orow, N, A.status);
}

// ------------------------------------------------------- one CTA, all on chip
//
// Hierarchies whose N*N*M reals fit the threads of one CTA (flow_small_fits):
// one thread per real, all three stage arrays in shared memory ([N*N][M], so a
// warp reads consecutive words), the right-hand side of the thread's element
// -- own-node terms and the six neighbour terms alike -- as one list of (place,
// coefficient) in registers, and a __syncthreads per stage.  Nothing leaves the
// SM during a call but the output rows.  The bound is latency: a dependent chain
// of shared-memory loads and multiply-adds and the barrier; in FP64 the pipe (64
// cycles per instruction and warp), which is why the real and imaginary parts
// of a pair are separate threads, terms that are zero in a whole warp are
// skipped, and the output rows (sums and conversions in double) are left to one
// more warp.  us per step with a row every step, two sites, depth 4, FP64: 10.2 as
// a cluster launch of the load views, 8.4 of the throughput engine, 3.4 here.  Without
// rows, load views before and here: two sites depth 19 (840 reals) mixed 6.6, 2.6; four
// sites depth 3 (560) mixed 8.6, 2.5; seven sites depth 1 (392) mixed 20.2, 3.2; two sites
// depth 9 (220) FP64 9.0, 4.5.
template <int N, typename R, bool CPLX>
__host__ __device__ constexpr int flow_small_terms() {
  return (flow_nre(N, CPLX) > flow_nim(N, CPLX) ? flow_nre(N, CPLX) : flow_nim(N, CPLX)) + 6;
}
// In FP64 the CTA's FP64 units soon cost more than an exchange through L2.
__host__ __device__ constexpr int flow_small_max(int rsize) { return rsize == 8 ? 480 : 992; }
__host__ __device__ constexpr bool flow_small_fits(int N, int rsize, int64_t M) { return M * N * N <= flow_small_max(rsize); }

template <int N, typename R, bool MIXED, bool CPLX>
__global__ void __launch_bounds__(flow_small_max((int)sizeof(R)) + 32, 1) heom_small_kernel(FlowArgs A) {
  constexpr int NN = N * N;
  constexpr int NP = N * (N - 1) / 2;
  constexpr int U = NP + N;
  constexpr int NRE = flow_nre(N, CPLX), NIM = flow_nim(N, CPLX);
  constexpr int NT = NRE > NIM ? NRE : NIM;
  constexpr int T = NT + 6;
  __shared__ R s_st[3][flow_small_max((int)sizeof(R))];  // y, wa, wb
  __shared__ Inst s_inst;
  __shared__ int s_stop;
  __shared__ EtaAcc<R> s_ea[kMaxSmallN];
  __shared__ FF s_trace_ff[kMaxSmallN];
  __shared__ double s_trace_d[kMaxSmallN];
  if (threadIdx.x == 0) {
    s_inst = *A.inst;
    s_stop = 0;
  }
  __syncthreads();
  const Inst& I = s_inst;
  const int M = I.M, Mp = I.Mpad;
  const int t_el = threadIdx.x;  // p * M + n
  const bool valid = t_el < NN * M;
  const int p = valid ? t_el / M : 0, n = valid ? t_el - p * M : 0;
  const int er = p / N, ec = p - er * N;
  const int a = min(er, ec), b = max(er, ec);
  const bool im = er > ec, pair = er != ec, root = valid && n == 0, diag_root = root && !pair;
  const bool lead = threadIdx.x == blockDim.x - 32;  // of the warp without elements
  // FP64: this owner's step factors of eta, loss and xi
  double fe = 0.0, fl = 0.0, fx = 0.0;

  // the element's list: NT own terms, then n + e_a, n + e_b, n - e_a (two), n - e_b (two)
  R co[T];
  unsigned pl[(T + 1) / 2];  // places, 16 bits each
#pragma unroll
  for (int i = 0; i < T; ++i) co[i] = R(0);
#pragma unroll
  for (int i = 0; i < (T + 1) / 2; ++i) pl[i] = (unsigned)t_el | ((unsigned)t_el << 16);
  auto put = [&](auto ic, double w, int place) {
    constexpr int i = decltype(ic)::value;
    co[i] = (R)w;
    pl[i / 2] = i % 2 ? (pl[i / 2] & 0xFFFFu) | ((unsigned)place << 16) : (pl[i / 2] & 0xFFFF0000u) | (unsigned)place;
  };
  if (!valid) {
#pragma unroll
    for (int i = 0; i < (T + 1) / 2; ++i) pl[i] = 0;
  } else {
    const int u = pair ? a * (2 * N - a - 1) / 2 + b - a - 1 : NP + a;
    const FlowUnit& fu = A.units[u];
    const FlowSite* fs = reinterpret_cast<const FlowSite*>(A.units + U);
    const FlowSite sa = fs[a], sb = fs[b];
    const bool scaled = I.wsc != nullptr;
    const int pab = a * N + b, pba = b * N + a;
    const int ra = I.dn[a * Mp + n], rb = I.dn[b * Mp + n], ua = I.up[a * Mp + n], ub = I.up[b * Mp + n];
    const double na = ra < 0 ? 0.0 : (double)(ra >> 24), nb = rb < 0 ? 0.0 : (double)(rb >> 24);
    const double ng = (double)static_cast<const R*>(I.ngam)[n];
    // terms of the node itself on x (slot 0) and, for a pair, yi (slot 1): hierarchy damping and the terminator (see
    // heom_flow_kernel)
    double x0 = im ? 0.0 : -ng, x1 = im ? -ng : 0.0;
    if (pair && I.terminator && I.up[n] < 0) {
      const double ca = (na + 1.0) / (ng + sa.gamma), cb = (nb + 1.0) / (ng + sb.gamma);
      const double re = -ca * sa.alpha - cb * sb.alpha, ro = -ca * sa.beta + cb * sb.beta;
      x0 += im ? -ro : re;
      x1 += im ? re : ro;
    }
    static_for<0, NT>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      const bool in = im ? i < NIM : i < NRE;
      if (!in) return;
      double w = im ? fu.cim[i < NIM ? i : 0] : fu.cre[i < NRE ? i : 0];
      if (i == 0) w += x0;
      if (i == 1 && pair) w += x1;
      put(ic, w, (im ? fu.iim[i < NIM ? i : 0] : fu.ire[i < NRE ? i : 0]) * M + n);
    });
    const double wua = scaled ? sqrt((na + 1.0) * sa.scale) : 1.0, wub = scaled ? sqrt((nb + 1.0) * sb.scale) : 1.0;
    const double wa = scaled ? sqrt(na / sa.scale) : na, wb = scaled ? sqrt(nb / sb.scale) : nb;
    const int da = ra & 0xFFFFFF, db = rb & 0xFFFFFF;
    if (pair) {
      // re: -wu_a Im(up a) + wu_b Im(up b); im: wu_a Re(up a) - wu_b Re(up b)
      if (ua >= 0) put(std::integral_constant<int, NT>{}, im ? wua : -wua, (im ? pab : pba) * M + ua);
      if (ub >= 0) put(std::integral_constant<int, NT + 1>{}, im ? -wub : wub, (im ? pab : pba) * M + ub);
      // n_j theta_j: re: beta Re -+ alpha Im, im: beta Im +- alpha Re (upper sign for j = a)
      if (ra >= 0) {
        put(std::integral_constant<int, NT + 2>{}, wa * sa.beta, p * M + da);
        put(std::integral_constant<int, NT + 3>{}, im ? wa * sa.alpha : -wa * sa.alpha, (im ? pab : pba) * M + da);
      }
      if (rb >= 0) {
        put(std::integral_constant<int, NT + 4>{}, wb * sb.beta, p * M + db);
        put(std::integral_constant<int, NT + 5>{}, im ? -wb * sb.alpha : wb * sb.alpha, (im ? pab : pba) * M + db);
      }
    } else if (ra >= 0) {
      put(std::integral_constant<int, NT + 2>{}, 2.0 * wa * sa.beta, p * M + da);
    }
  }
  uint64_t terms = 0;  // terms some lane of the warp has
#pragma unroll
  for (int i = 0; i < T; ++i) terms |= __any_sync(0xFFFFFFFFu, co[i] != R(0)) ? 1ull << i : 0ull;

  R y = R(0);
  FF ry{0.f, 0.f}, rw{0.f, 0.f};  // the root's element in float-float: y and the last stage output (mixed)
  if (valid) {
    y = static_cast<const R*>(I.y)[node_col<N>(n) + p * 32];
    s_st[0][t_el] = y;
    if constexpr (MIXED) {
      if (root) ry = static_cast<const FF*>(I.y0)[p];
    }
  }
  if (diag_root) s_ea[a] = EtaAcc<R>{};
  EtaRows rows;
  rows.acc0 = I.acc[0];
  rows.acc1 = I.acc[1];
  const double* cfd = reinterpret_cast<const double*>(static_cast<const unsigned char*>(I.coef) +
                                                      CoefLayout<R>::dbl_offset(N));
  if (diag_root) {
    fe = I.dt * cfd[a];
    fl = I.dt * cfd[N + a];
    fx = 0.5 * I.dt * I.dt * cfd[a];
  }
  if (lead) {
    write_row0<N, R, MIXED>(I);
    const EtaAcc<R> zero{};
    for (int k = 0; k < N; ++k) zero.store(I, k);
  }
  __syncthreads();

  int64_t next_out = I.out_every, orow = 1, done = I.nsteps;
  for (int64_t t = 0; t < I.nsteps; ++t) {
    const OutStep os{t + 1 == next_out, orow};
    if (os.now) {
      next_out += I.out_every;
      ++orow;
    }
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      if (s == 0 && rows.pending >= 0) {
        if (lead) flow_eta_row<R, MIXED>(I, s_ea, s_trace_ff, s_trace_d, N, rows.acc0, rows.acc1, rows.pending, A.status);
        rows.pending = -1;
      }
      const R* sin = s_st[s == 0 ? 0 : (s == 2 ? 2 : 1)];
      R* sout = s_st[s == 1 ? 2 : (s == 3 ? 0 : 1)];
      R r0 = R(0), r1 = R(0);
#pragma unroll
      for (int i = 0; i < T; ++i) {
        if (sizeof(R) == 8 && !((terms >> i) & 1)) continue;
        const R v = sin[(pl[i / 2] >> (16 * (i % 2))) & 0xFFFFu];
        if (i % 2) r1 += co[i] * v;
        else r0 += co[i] * v;
      }
      const R r = r0 + r1;
      if (valid) {
        R w;
        if (MIXED && root) {
          if constexpr (MIXED) {
            if (diag_root) {
              if (s == 3) s_ea[a].add(I, a, rw);
              if (s == 2) s_ea[a].add_xi(I, a, rw);
            }
            rw = ff_axpy(ry, I.hh[s], I.hl[s], r);
            w = rw.h;
            if (s == 3) {
              ry = rw;
              if (diag_root && os.now && I.out_pops) I.out_pops[os.row * N + a] = ff_to_double(rw);
            }
          }
        } else {
          if constexpr (!MIXED) {
            if (diag_root && s == 3) {
              s_ea[a].e += fe * sin[t_el];
              s_ea[a].l += fl * sin[t_el];
            }
            if (diag_root && s == 2) s_ea[a].x += fx * sin[t_el];
          }
          w = y + (sizeof(R) == 8 ? (R)I.hd[s] : (R)I.hh[s]) * r;
          if (diag_root && s == 3 && os.now && I.out_pops) I.out_pops[os.row * N + a] = (double)w;
        }
        sout[t_el] = w;
        if (s == 3) y = w;
        if (diag_root) {
          if (s == 2) s_ea[a].step_xi(I);
          if (s == 3) {
            if (os.now || t + 1 == I.nsteps) s_ea[a].store(I, a);
            if constexpr (MIXED) s_trace_ff[a] = ry;
            else s_trace_d[a] = (double)w;
          }
        }
      }
      __syncthreads();
    }
    if (os.now) rows.pending = os.row;
    if (I.stop_trace > 0.0 && t + 1 < I.nsteps) {
      if (lead) {
        double tr = 0.0;
        if constexpr (MIXED) {
          FF sum{0.f, 0.f};
          for (int k = 0; k < N; ++k) sum = ff_add(sum, s_trace_ff[k]);
          tr = ff_to_double(sum);
        } else {
          for (int k = 0; k < N; ++k) tr += s_trace_d[k];
        }
        s_stop = tr < I.stop_trace;
      }
      __syncthreads();
      if (s_stop) {
        if (diag_root) s_ea[a].store(I, a);
        done = t + 1;
        break;
      }
    }
  }
  if (valid) static_cast<R*>(I.y)[node_col<N>(n) + p * 32] = y;
  if constexpr (MIXED) {
    if (root) static_cast<FF*>(I.y0)[p] = ry;
  }
  __syncthreads();
  if (lead) finish_instance<R>(I, N, rows, done, orow, N, A.status);
}

}  // namespace heom
