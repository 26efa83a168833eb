// Coarse-cycle launch: the levels with few nodes as one thread-block cluster
// per right-hand side.
//
// The small levels of the hierarchy (all levels from `lc` down to the
// coarsest grid) cost little arithmetic but a long serial chain: every
// smoothing step is four operator applications with global sums between
// them.  As grid-wide kernels each link of that chain is a launch (5 to 20
// us); in one thread block (the form this kernel replaces) one SM does all
// the work, and its FP64 pipe (two multiply-adds per clock) and L2 round
// trips set the time.  Here a cluster of C blocks (C <= 16, one per SM)
// walks the host-recorded V/W schedule of those levels (the recursion of the
// grid-wide driver, Sec. 3 of the paper):
//
//  * every block owns a slab of consecutive rows of each level and keeps all
//    vectors of its slab in shared memory for the whole visit;
//  * an operator application exchanges what its neighbours need through
//    distributed shared memory: on Kronecker-form levels the row sums G_x v
//    and W_x v of the first and last R own rows (so that no row sum is formed
//    twice: 12 (2R + 1) FMAs per node instead of OpK::apply's 6 (2R + 1)^2),
//    on the other levels the rows of v.  Slabs have at least three rows
//    (the largest radius), so only the two adjacent blocks exchange;
//  * a global sum is a block sum pushed to every block of the cluster, which
//    all add the C partial sums in the same order (reproducible, no
//    broadcast) and run the scalar step redundantly;
//  * the phases are separated by the hardware cluster barrier; exchange and
//    sum buffers alternate between two copies, so one barrier per phase is
//    enough (a block can be at most one phase ahead of its neighbours);
//  * stored stencils sit in shared memory as far as they fit, the coarsest
//    level's first, copied once per launch.
//
// GMRES(3): complex128 in the Arnoldi form of the grid-wide kernels
// (gmres.cuh).  complex64 in the s-step form of sstep.cuh: the basis r, B r,
// B^2 r, B^3 r without sums in between, one sum of its Gram matrix, and the
// 3 x 3 normal equations: four barriers per step instead of nine (five where
// the residual is formed afresh).
//
// The chain is latency-bound in complex64 (a phase is a barrier of about 0.3
// us and a few hundred clocks of work) and bound by the SMs' FP64 pipes in
// complex128.  Measured on whole solves, one block per right-hand side and
// one launch per kernel above 1100 nodes -> this kernel: omega-Jacobi V(1,1)
// FP64 on 65^2 46.0 -> 13.4 ms, W(2,2) FP64 on 161^2 298 -> 87.6 ms, V(2,2)
// complex64 on 81^2 8.4 -> 3.0 ms and on 1025^2 112 -> 78.9 ms (one
// right-hand side), FP64 8 x 513^2 521 -> 392 ms, 16 ragged problems
// 182 -> 117 ms.
// Carrying the residual between complex64 steps (16 -> 10 applications per
// V(2,2) cycle and level): one 1025^2 right-hand side 48.2 -> 46.0 ms, 81^2
// 3.02 -> 2.94 ms, 16 ragged problems 71.5 -> 68.8 ms.
// Against one block per right-hand side, complex64 Jacobi cycles on small grids
// were slower until the zero iterate's sweep skipped its exchange, the transfers
// issued their remote loads together and the stencils moved on chip: us per
// cycle, one block / cluster before / now: V(1,1) on 65^2 81 / 89 / 65, variable k
// 88 / 94 / 68; W(1,1) on 65^2 272 / 332 / 250, variable k 274 / 447 / 285.  W-cycles
// on 17^2 and 33^2 stay up to 15 % slower, by one to two cluster barriers per visit
// of a level: giving such levels to one block alone made them quicker, but its
// code cost the large levels 4 % (the loads of the stencils lost registers).
#pragma once
#include <algorithm>
#include <mutex>

#include "gmres.cuh"
#include "internal.h"
#include "ragged.cuh"
#include "ragged_api.h"
#include "sstep.cuh"

namespace hmg {
namespace {

// ------------------------------------------------------------ cluster PTX

__device__ __forceinline__ unsigned cl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cl_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// Barrier over every thread of the cluster (a hardware barrier, like
// __syncthreads: no polling); orders shared and distributed shared memory.
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of this block's shared location p in block `cta` of the cluster.
__device__ __forceinline__ unsigned cl_map(const void* p, unsigned cta) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(cta));
  return r;
}
__device__ __forceinline__ void cl_st(unsigned a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cl_st(unsigned a, double2 v) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void cl_st(unsigned a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_st(unsigned a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ float2 cl_ld(unsigned a, float2) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ double2 cl_ld(unsigned a, double2) {
  double2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
  return v;
}

// The same where p holds, else zero: a predicated load, so that the loads of a
// node's neighbours are issued one behind the other without a branch.
__device__ __forceinline__ float2 cl_ld_if(unsigned a, bool p, float2) {
  float2 v;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.s32 q, %3, 0;\n mov.f32 %0, 0f00000000;\n mov.f32 %1, 0f00000000;\n"
      " @q ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n}"
      : "=f"(v.x), "=f"(v.y) : "r"(a), "r"((int)p) : "memory");
  return v;
}
__device__ __forceinline__ double2 cl_ld_if(unsigned a, bool p, double2) {
  double2 v;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.s32 q, %3, 0;\n mov.f64 %0, 0d0000000000000000;\n mov.f64 %1, 0d0000000000000000;\n"
      " @q ld.shared::cluster.v2.f64 {%0, %1}, [%2];\n}"
      : "=d"(v.x), "=d"(v.y) : "r"(a), "r"((int)p) : "memory");
  return v;
}

// ------------------------------------------------------------- block state

template <class T> struct Blk {
  const ClArgs<T>* a;
  const ClLev<T>* lev;   // level table (shared memory)
  cx<T>* m;              // shared memory in elements of cx<T>
  T* red;                // [2][C][CL_NV] partial sums pushed by the blocks
  T* tot;                // [CL_NV] totals
  T* wsum;               // [CL_NV][warps] block-sum scratch
  T* S;                  // GMRES(3) scalars
  int rank, C, tid, par, rpar;
};

// The slab of one level: rows [r0, r0 + nr), nodes in row-major order.
template <class T> struct Slab {
  const ClLev<T>* L;
  int r0, nr, n1, nodes;
  __device__ __forceinline__ Slab(const Blk<T>& B, int l) {
    L = B.lev + l;
    n1 = L->n1;
    r0 = min(B.rank * L->rp, L->ny + 1);
    nr = min(L->rp, L->ny + 1 - r0);
    nodes = nr * n1;
  }
};

#define CL_NODES(s)                                                                      \
  for (int q = B.tid, jl = __umulhi(B.tid, (s).L->magic), i = q - jl * (s).n1; q < (s).nodes; \
       q += NT, jl = __umulhi(q, (s).L->magic), i = q - jl * (s).n1)

// Sums the NV per-thread values over the cluster: lane_sum within the warps,
// the warps' sums in warp order, and the blocks' sums pushed to every block.
// After the caller's next cl_sync(), cl_totals() gives the totals.
template <int NV, int NT, class T>
__device__ __forceinline__ void cl_push_sum(Blk<T>& B, T (&v)[NV]) {
  static_assert(NV <= CL_NV, "record");
  const int lane = B.tid & 31, warp = B.tid >> 5;
  constexpr int W = NT / 32;
  const T t = lane_sum<NV, T>(v, lane);
  if ((lane & (32 / NV - 1)) == 0) B.wsum[lane_value<NV>(lane) * W + warp] = t;
  __syncthreads();
  if (warp == 0) {
    T s = T(0);
    if (lane < NV) {
      s = B.wsum[lane * W];
#pragma unroll
      for (int w = 1; w < W; ++w) s += B.wsum[lane * W + w];
    }
    T* mine = B.red + (B.rpar * B.C + B.rank) * CL_NV;
    for (int e0 = 0; e0 < NV * B.C; e0 += 32) {   // the whole warp takes part in every exchange
      const int e = e0 + lane, k = e % NV;
      const T sv = __shfl_sync(0xffffffffu, s, k);
      if (e < NV * B.C) cl_st(cl_map(mine + k, e / NV), sv);
    }
  }
}
template <int NV, int NT, class T> __device__ __forceinline__ void cl_totals(Blk<T>& B) {
  if (B.tid < 32) {
    const T* q = B.red + B.rpar * B.C * CL_NV;
    T v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = B.tid < B.C ? q[B.tid * CL_NV + k] : T(0);
    const T t = lane_sum<NV, T>(v, B.tid);
    if ((B.tid & (32 / NV - 1)) == 0) B.tot[lane_value<NV>(B.tid)] = t;
    __syncwarp();
  }
  B.rpar ^= 1;
}

// --------------------------------------------------------- operator phases

// K: operator kind (1 fine level, 2 / 3 stored stencil, 4 / 5 Kronecker form);
// CHIP: the stored stencil is on chip (ClLev::ost; a variant of its own, because
// the grouped loads of the other one need all the registers)
template <int K, bool CHIP = false> struct KindOf {
  static constexpr int kind = K;
  static constexpr bool chip = CHIP;
  static constexpr int R = K == 1 ? 1 : (K == 2 || K == 4) ? 2 : 3;
  static constexpr bool kron = K >= 4;
};

// First half of A v: what the combination needs of this block's rows, into
// the exchange buffer here and, for the first and last R rows, in the
// adjacent blocks (rows above and below the slab).  Reads v of whole rows:
// the caller has synchronised the block after writing v (Kronecker kinds).
// The following cl_sync() completes it.
template <class KT, int NT, class T>
__device__ __forceinline__ void exchange(Blk<T>& B, const Slab<T>& s, const cx<T>* v) {
  constexpr int R = KT::R;
  const ClLev<T>& L = *s.L;
  const int n1 = s.n1, plane = (L.rp + 2 * R) * n1;
  cx<T>* X = B.m + B.a->oX + B.par * B.a->nX;
  const bool up = s.nr > 0 && B.rank > 0, down = s.r0 + s.nr <= L.ny;
  const unsigned pu = up ? cl_map(X, B.rank - 1) : 0u, pd = down ? cl_map(X, B.rank + 1) : 0u;
  CL_NODES(s) {
    cx<T> g, w;
    if constexpr (KT::kron) {
      const cx<T>* gx = B.m + L.ogx;
      const T* wx = reinterpret_cast<const T*>(B.m + L.owx);
      g = w = mk<T>(0, 0);
#pragma unroll
      for (int d = -R; d <= R; ++d) {
        if ((unsigned)(i + d) < (unsigned)n1) {
          const cx<T> e = v[q + d];
          const T c = wx[(d + R) * n1 + i];
          g = fma_c<T>(gx[(d + R) * n1 + i], e, g);
          w = mk<T>(fma(c, e.x, w.x), fma(c, e.y, w.y));
        }
      }
    } else {
      g = v[q];
    }
    const int o = (jl + R) * n1 + i;
    X[o] = g;
    if constexpr (KT::kron) X[plane + o] = w;
    if (up && jl < R) {   // the block above holds rp rows: its halo row R + rp + jl
      const unsigned t = pu + (unsigned)sizeof(cx<T>) * (unsigned)((L.rp + R + jl) * n1 + i);
      cl_st(t, g);
      if constexpr (KT::kron) cl_st(t + (unsigned)sizeof(cx<T>) * (unsigned)plane, w);
    }
    if (down && jl >= s.nr - R) {
      const unsigned t = pd + (unsigned)sizeof(cx<T>) * (unsigned)((jl - s.nr + R) * n1 + i);
      cl_st(t, g);
      if constexpr (KT::kron) cl_st(t + (unsigned)sizeof(cx<T>) * (unsigned)plane, w);
    }
  }
}

// Second half: (A v) at node (i, r0 + jl), from the exchange buffer.
template <class KT, class T>
__device__ __forceinline__ cx<T> combine(const Blk<T>& B, const Slab<T>& s, int jl, int i) {
  constexpr int R = KT::R;
  const ClLev<T>& L = *s.L;
  const int n1 = s.n1, j = s.r0 + jl;
  const cx<T>* X = B.m + B.a->oX + B.par * B.a->nX + (jl + R) * n1 + i;
  if constexpr (KT::kron) {
    const int plane = (L.rp + 2 * R) * n1;
    const cx<T>* hy = B.m + L.ohy + jl * (2 * R + 1);
    const T* wy = reinterpret_cast<const T*>(B.m + L.owy) + jl * (2 * R + 1);
    cx<T> acc = mk<T>(0, 0);
#pragma unroll
    for (int d = -R; d <= R; ++d) {
      if ((unsigned)(j + d) <= (unsigned)L.ny) {
        const cx<T> g = X[d * n1], w = X[plane + d * n1];
        const T c = wy[d + R];
        acc = mk<T>(fma(c, g.x, acc.x), fma(c, g.y, acc.y));
        acc = fma_c<T>(hy[d + R], w, acc);
      }
    }
    return acc;
  } else if constexpr (KT::kind == 1) {
    const cx<T> z = mk<T>(0, 0);
    const cx<T> xe = i < L.nx ? X[1] : z, xw = i > 0 ? X[-1] : z;
    const cx<T> xn = j < L.ny ? X[n1] : z, xs = j > 0 ? X[-n1] : z;
    return L.c0.abc2 ? Op0<T, true>{L.c0, L.kf, L.nx, L.ny}.apply5(X[0], xe, xw, xn, xs, i, j)
                     : Op0<T>{L.c0, L.kf, L.nx, L.ny}.apply5(X[0], xe, xw, xn, xs, i, j);
  } else if constexpr (KT::chip) {
    constexpr int K = 2 * R + 1;
    const int np = L.rp * n1;
    const cx<T>* cs = B.m + L.ost + jl * n1 + i;
    cx<T> acc = mk<T>(0, 0);
#pragma unroll
    for (int e = 0; e < K * K; ++e, cs += np) {
      const int dy = e / K - R, dx = e % K - R;
      if ((unsigned)(j + dy) <= (unsigned)L.ny && (unsigned)(i + dx) < (unsigned)n1)
        acc = fma_c<T>(*cs, X[dy * n1 + dx], acc);
    }
    return acc;
  } else {
    // Stored stencil.  A slab's coefficients that do not fit on chip come from L2
    // at every application: the loads are then issued in groups of rows before
    // the multiply-adds that wait for them (one load at a time was the chain that
    // took 446 us of a layered 1281 x 449 cycle).  A coupling off the grid has a
    // stored coefficient, and its node value is taken as zero.
    constexpr int K = 2 * R + 1, G = sizeof(T) == 8 ? 2 : R == 2 ? 5 : 4;
    cx<T> acc = mk<T>(0, 0);
    const cx<T>* st = L.st + (long long)j * n1 + i;
#pragma unroll
    for (int d0 = 0; d0 < K; d0 += G) {
      cx<T> c[G * K];
#pragma unroll
      for (int e = 0; e < G * K && d0 * K + e < K * K; ++e) c[e] = __ldg(st + (d0 * K + e) * L.plane);
#pragma unroll
      for (int e = 0; e < G * K && d0 * K + e < K * K; ++e) {
        const int dy = d0 + e / K - R, dx = e % K - R;
        if ((unsigned)(j + dy) <= (unsigned)L.ny && (unsigned)(i + dx) < (unsigned)n1)
          acc = fma_c<T>(c[e], X[dy * n1 + dx], acc);
      }
    }
    return acc;
  }
}

template <class KT, int NT, class T>
__device__ __forceinline__ void start_apply(Blk<T>& B, const Slab<T>& s, const cx<T>* v) {
  B.par ^= 1;
  exchange<KT, NT>(B, s, v);
}

// --------------------------------------------------------------- smoothers

// r = b - A x of the slab into u0
template <class KT, int NT, class T>
__device__ __forceinline__ void residual(Blk<T>& B, const Slab<T>& s, cx<T>* r) {
  const cx<T>* x = B.m + s.L->ox;
  const cx<T>* b = B.m + s.L->ob;
  start_apply<KT, NT>(B, s, x);
  cl_sync();
  CL_NODES(s) r[q] = sub<T>(b[q], combine<KT>(B, s, jl, i));
}

// nu weighted-Jacobi sweeps; z: x is zero on entry, so that the first is x = d b
// (no exchange, no barrier of the cluster)
template <class KT, int NT, class T>
__device__ __forceinline__ void jacobi(Blk<T>& B, const Slab<T>& s, int nu, bool z) {
  cx<T>* x = B.m + s.L->ox;
  const cx<T>* b = B.m + s.L->ob;
  const cx<T>* d = B.m + s.L->od;
  if (z) {
    CL_NODES(s) x[q] = fma_c<T>(d[q], b[q], mk<T>(0, 0));
    __syncthreads();
  }
  for (int it = z ? 1 : 0; it < nu; ++it) {
    start_apply<KT, NT>(B, s, x);
    cl_sync();
    CL_NODES(s) x[q] = fma_c<T>(d[q], sub<T>(b[q], combine<KT>(B, s, jl, i)), x[q]);
    __syncthreads();
  }
}

// Arnoldi step J, complex128: w = s_J A u_J, the Gram-form MGS coefficients
// (fin_a), u_{J+1} and its norm and Gram entries (fin_b), as the grid-wide
// kernels (gmres.cuh).  False once the process has stopped (the same in
// every block: all hold the same scalars).
template <int J, class KT, int NT, class T>
__device__ __forceinline__ bool arnoldi(Blk<T>& B, const Slab<T>& s, cx<T>* const (&u)[3], cx<T>* w) {
  if (B.S[G_BRK] != T(0) || B.S[G_M] < T(J)) return false;
  const T sJ = B.S[G_S + J];
  constexpr int ND = J == 0 ? 2 : J == 1 ? 4 : 8;
  T dt[ND];
#pragma unroll
  for (int l = 0; l < ND; ++l) dt[l] = T(0);
  CL_NODES(s) {   // the exchange of u_J completed at the last barrier
    const cx<T> a = scl<T>(sJ, combine<KT>(B, s, jl, i));
    w[q] = a;
#pragma unroll
    for (int l = 0; l <= J; ++l) {
      add_cmul<T>(dt[2 * l], dt[2 * l + 1], u[l][q], a);
    }
  }
  cl_push_sum<ND, NT>(B, dt);
  cl_sync();
  cl_totals<ND, NT>(B);
  if (B.tid == 0) fin_a<J, T, T, T>(B.S, B.tot);
  __syncthreads();
  cx<T> c[J + 1];
#pragma unroll
  for (int l = 0; l <= J; ++l) {
    const T sl = B.S[G_S + l];
    c[l] = mk<T>(B.S[G_H + 2 * (l * 3 + J)] * sl, B.S[G_H + 2 * (l * 3 + J) + 1] * sl);
  }
  constexpr int NE = J == 0 ? 4 : J == 1 ? 8 : 1;   // 1 + 2 (J + 1) values used
  T et[NE];
#pragma unroll
  for (int l = 0; l < NE; ++l) et[l] = T(0);
  CL_NODES(s) {
    cx<T> a = w[q];
    cx<T> uu[J + 1];
#pragma unroll
    for (int l = 0; l <= J; ++l) {
      uu[l] = u[l][q];
      a = sub_mul<T>(a, c[l], uu[l]);
    }
    add_abs2<T>(et[0], a);
    if constexpr (J < 2) {
      u[J + 1][q] = a;
#pragma unroll
      for (int l = 0; l <= J; ++l) {
        add_cmul<T>(et[1 + 2 * l], et[2 + 2 * l], a, uu[l]);
      }
    }
  }
  cl_push_sum<NE, NT>(B, et);   // synchronises the block: u_{J+1} is complete
  if constexpr (J < 2) start_apply<KT, NT>(B, s, u[J + 1]);
  cl_sync();
  cl_totals<NE, NT>(B);
  if (B.tid == 0) fin_b<J, T, T, T>(B.S, B.tot);
  __syncthreads();
  return true;
}

// nu GMRES(3) steps; z: x is zero on entry, so that the first step's u0 is b;
// left (complex64): leave b - A x in u0.  complex64 steps after the first take
// the residual that the previous update formed by linearity (sstep.cuh): ten
// applications per V(2,2) cycle and level instead of sixteen.
template <class KT, int NT, class T>
__device__ __forceinline__ void gmres(Blk<T>& B, const Slab<T>& s, int nu, bool z, bool left) {
  cx<T>* x = B.m + s.L->ox;
  const cx<T>* b = B.m + s.L->ob;
  cx<T>* const u[3] = {B.m + B.a->ou, B.m + B.a->ou + B.a->nu, B.m + B.a->ou + 2 * B.a->nu};
  for (int step = 0; step < nu; ++step) {
    if (z && step == 0) {
      CL_NODES(s) u[0][q] = b[q];
    } else if (sizeof(T) == 8 || !ss_carried(step)) {
      residual<KT, NT>(B, s, u[0]);
    }
    if constexpr (sizeof(T) == 8) {
      cx<T>* w = B.m + B.a->ou + 3 * B.a->nu;
      T a0[1] = {T(0)};
      CL_NODES(s) add_abs2<T>(a0[0], u[0][q]);
      cl_push_sum<1, NT>(B, a0);
      start_apply<KT, NT>(B, s, u[0]);
      cl_sync();
      cl_totals<1, NT>(B);
      if (B.tid == 0) fin_init<T, T, T>(B.S, B.tot);
      __syncthreads();
      if (arnoldi<0, KT, NT>(B, s, u, w) && arnoldi<1, KT, NT>(B, s, u, w)) arnoldi<2, KT, NT>(B, s, u, w);
      const int m = (int)B.S[G_M];
      if (m > 0) {
        cx<T> c[3];
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          const T sl = B.S[G_S + l];
          c[l] = mk<T>(B.S[G_Y + 2 * l] * sl, B.S[G_Y + 2 * l + 1] * sl);
        }
        CL_NODES(s) {
          cx<T> a = x[q];
#pragma unroll
          for (int l = 0; l < 3; ++l)
            if (l < m) a = fma_c<T>(c[l], u[l][q], a);
          x[q] = a;
        }
      }
      __syncthreads();
    } else {
      const T sc = s.L->scale, sg = s.L->sigma;
      cx<T>* v3s = B.m + B.a->ou + 3 * B.a->nu;
      const bool nr = step + 1 < nu ? ss_carried(step + 1) : left;   // the next residual is wanted
      T gm[SS_NV];
#pragma unroll
      for (int k = 0; k < SS_NV; ++k) gm[k] = T(0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {   // v_{k+1} = (scale A - sigma) v_k
        __syncthreads();
        start_apply<KT, NT>(B, s, u[k]);
        cl_sync();
        if (k < 2) {
          CL_NODES(s) {
            const cx<T> a = combine<KT>(B, s, jl, i), vk = u[k][q];
            u[k + 1][q] = mk<T>(fma(sc, a.x, -sg * vk.x), fma(sc, a.y, -sg * vk.y));
          }
        } else {
          CL_NODES(s) {
            const cx<T> a = combine<KT>(B, s, jl, i), v2 = u[2][q];
            const cx<T> v3 = mk<T>(fma(sc, a.x, -sg * v2.x), fma(sc, a.y, -sg * v2.y));
            ss_gram_add(gm, u[0][q], u[1][q], v2, v3);
            if (nr) v3s[q] = v3;
          }
        }
      }
      cl_push_sum<SS_NV, NT>(B, gm);
      cl_sync();
      cl_totals<SS_NV, NT>(B);
      if (B.tid == 0) ss_solve(B.tot, sc, sg, B.S);
      __syncthreads();
      cx<T> y[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) y[k] = mk<T>(B.S[2 * k], B.S[2 * k + 1]);
      cx<T> c[4];
      ss_residual_coef(y, T(1) / sc, sg, c);
      CL_NODES(s) {
        cx<T> e = z && step == 0 ? mk<T>(0, 0) : x[q];
        const cx<T> v[3] = {u[0][q], u[1][q], u[2][q]};
#pragma unroll
        for (int k = 0; k < 3; ++k) e = fma_c<T>(y[k], v[k], e);
        x[q] = e;
        if (nr) {
          cx<T> r = mul<T>(c[0], v[0]);
          r = fma_c<T>(c[1], v[1], r);
          r = fma_c<T>(c[2], v[2], r);
          u[0][q] = fma_c<T>(c[3], v3s[q], r);
        }
      }
      __syncthreads();
    }
  }
}

// --------------------------------------------------------------- transfers

// b_{l+1} = R (b - A x) and x_{l+1} = 0; left: b - A x is in u0
template <class KT, int NT, class T>
__device__ __forceinline__ void restrict_to(Blk<T>& B, const Slab<T>& s, int l, bool left) {
  const ClLev<T>& L = *s.L;
  cx<T>* r = B.m + B.a->ou;
  cx<T>* t = B.m + B.a->ou + B.a->nu;   // rows restricted along x
  if (!left) residual<KT, NT>(B, s, r);
  __syncthreads();
  const int n1c = (L.nx >> 1) + 1;
  const T w0 = L.w0, w1 = L.w1, w2 = L.w2;
  for (int q = B.tid; q < s.nr * n1c; q += NT) {
    const int jl = __umulhi(q, B.lev[l + 1].magic), I = q - jl * n1c;
    const cx<T>* row = r + jl * s.n1 + 2 * I;
    cx<T> v = scl<T>(w0, row[0]);
    if (I > 0) v = add<T>(v, add<T>(scl<T>(w1, row[-1]), scl<T>(w2, row[-2])));
    if (2 * I < L.nx) v = add<T>(v, add<T>(scl<T>(w1, row[1]), scl<T>(w2, row[2])));
    t[q] = v;
  }
  cl_sync();
  const Slab<T> c(B, l + 1);
  cx<T>* bc = B.m + c.L->ob;
  cx<T>* xc = B.m + c.L->ox;
  CL_NODES(c) {
    cx<T> v[5];   // rows off the grid: zero
#pragma unroll
    for (int d = -2; d <= 2; ++d) {
      const int j = 2 * (c.r0 + jl) + d, jc = min(max(j, 0), L.ny), o = __umulhi(jc, L.mrp);
      v[d + 2] = cl_ld_if(cl_map(t + (jc - o * L.rp) * n1c + i, o), j == jc, cx<T>());
    }
    cx<T> acc = mk<T>(0, 0);
#pragma unroll
    for (int d = -2; d <= 2; ++d) acc = add<T>(acc, scl<T>(d == 0 ? w0 : (d == 1 || d == -1) ? w1 : w2, v[d + 2]));
    bc[q] = scl<T>(T(0.25), acc);
    xc[q] = mk<T>(0, 0);
  }
  __syncthreads();
}

// x_l += P x_{l+1}
template <int NT, class T> __device__ __forceinline__ void prolong(Blk<T>& B, const Slab<T>& s, int l) {
  const ClLev<T>& L = *s.L;
  const ClLev<T>& C = B.lev[l + 1];
  cx<T>* x = B.m + L.ox;
  const cx<T>* e = B.m + C.ox;
  const T w0 = L.w0, w1 = L.w1, w2 = L.w2;
  cl_sync();
  CL_NODES(s) {
    // coarse rows J - 1 .. J + 1 (even j; J, J + 1 for odd j), columns alike:
    // the needed ones of the nine loads, all in flight before the first sum
    const int I = i >> 1, j = s.r0 + jl, J = j >> 1;
    const bool oi = i & 1, oj = j & 1;
    cx<T> m[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int JJ = J - 1 + a, jc = min(max(JJ, 0), C.ny), o = __umulhi(jc, C.mrp);
      const bool row = JJ == jc && !(a == 0 && oj);
      const unsigned p = cl_map(e + (jc - o * C.rp) * C.n1 + I, o);
      m[a][0] = cl_ld_if(p - (unsigned)sizeof(cx<T>), row && !oi && I > 0, cx<T>());
      m[a][1] = cl_ld_if(p, row, cx<T>());
      m[a][2] = cl_ld_if(p + (unsigned)sizeof(cx<T>), row && I < C.nx, cx<T>());
    }
    cx<T> r[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      r[a] = oi ? scl<T>(w1, add<T>(m[a][1], m[a][2]))
                : add<T>(add<T>(scl<T>(w0, m[a][1]), scl<T>(w2, m[a][0])), scl<T>(w2, m[a][2]));
    }
    const cx<T> v = oj ? scl<T>(w1, add<T>(r[1], r[2])) : add<T>(scl<T>(w2, add<T>(r[0], r[2])), scl<T>(w0, r[1]));
    x[q] = add<T>(x[q], v);
  }
  __syncthreads();
}

// x = A_c^{-1} b on the coarsest level, FP64: the right-hand side gathered
// in every block, one warp per row of the inverse.
template <int NT, class T> __device__ __forceinline__ void coarse(Blk<T>& B, const Slab<T>& s) {
  const ClLev<T>& L = *s.L;
  const int N = B.a->N, lane = B.tid & 31;
  double2* rs = reinterpret_cast<double2*>(B.m + B.a->oX);
  const int per = L.rp * s.n1;   // nodes of a full slab
  cl_sync();
  for (int q = B.tid; q < N; q += NT) {
    const int o = q / per;
    rs[q] = cvt<double, T>(cl_ld(cl_map(B.m + L.ob + (q - o * per), o), cx<T>()));
  }
  __syncthreads();
  for (int q = B.rank + B.C * (B.tid >> 5); q < N; q += B.C * (NT / 32)) {
    const double2* row = B.a->inv + (long long)q * N;
    double2 acc = make_double2(0, 0);
    for (int k = lane; k < N; k += 32) acc = fma_c<double>(row[k], rs[k], acc);
    double v[2] = {acc.x, acc.y};
    const double t = lane_sum<2, double>(v, lane);   // lanes 0..15 the real part, 16..31 the imaginary part
    const double ti = __shfl_down_sync(0xffffffffu, t, 16);
    const int o = q / per;
    if (lane == 0) cl_st(cl_map(B.m + L.ox + (q - o * per), o), mk<T>((T)t, (T)ti));
  }
  cl_sync();
}

// ------------------------------------------------------------------ kernel

template <class KT, int NT, class T>
__device__ __forceinline__ void level_step(Blk<T>& B, const ClStep& st) {
  const Slab<T> s(B, st.level);
  if (st.op == CL_JACOBI) jacobi<KT, NT>(B, s, st.arg, st.zero != 0);
  else if (st.op == CL_GMRES) gmres<KT, NT>(B, s, st.arg, st.zero != 0, st.left != 0);
  else restrict_to<KT, NT>(B, s, st.level, st.left != 0);
}

template <class T, int NT> __device__ __forceinline__ void cluster_cycle(const ClArgs<T>& a, int rhs, cx<T>* smem) {
  Blk<T> B;
  B.a = &a;
  B.m = smem;
  B.rank = (int)cl_rank();
  B.C = (int)cl_size();
  B.tid = threadIdx.x;
  B.par = B.rpar = 0;
  ClLev<T>* lt = reinterpret_cast<ClLev<T>*>(smem + a.olev);
  B.lev = lt;
  B.red = reinterpret_cast<T*>(smem + a.ored);
  B.tot = B.red + 2 * B.C * CL_NV;
  B.wsum = B.tot + CL_NV;
  B.S = B.wsum + CL_NV * (NT / 32);
  if (a.active && !a.active[rhs]) return;   // the whole cluster
  {
    const int nw = (int)(sizeof(ClLev<T>) / 4) * a.nlev;
    for (int k = B.tid; k < nw; k += NT) reinterpret_cast<int*>(lt)[k] = reinterpret_cast<const int*>(a.lev)[k];
  }
  __syncthreads();
  // operator factors and inverse diagonals of the slabs
  for (int l = 0; l < a.nlev; ++l) {
    const Slab<T> s(B, l);
    const ClLev<T>& L = *s.L;
    if (L.od >= 0) {
      cx<T>* d = smem + L.od;
      if (L.kind == 1) {
        CL_NODES(s) d[q] = L.c0.abc2 ? Op0<T, true>{L.c0, L.kf, L.nx, L.ny}.diag_inv(i, s.r0 + jl)
                                     : Op0<T>{L.c0, L.kf, L.nx, L.ny}.diag_inv(i, s.r0 + jl);
      } else {
        CL_NODES(s) d[q] = L.dinv[(long long)s.r0 * s.n1 + q];
      }
    }
    if (L.ost >= 0) {   // a warp per coefficient plane, all copies in flight at once
      const int K = 2 * (L.kind == 2 ? 2 : 3) + 1, np = L.rp * s.n1;
      for (int e = B.tid >> 5; e < K * K; e += NT / 32) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(smem + L.ost + e * np);
        const cx<T>* g = L.st + e * L.plane + (long long)s.r0 * s.n1;
        for (int q = B.tid & 31; q < s.nodes; q += 32)
          asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d + q * (unsigned)sizeof(cx<T>)), "l"(g + q),
                       "n"(sizeof(cx<T>))
                       : "memory");
      }
    }
    if (L.kind >= 4 && L.ogx >= 0) {
      const int K = L.kind == 4 ? 5 : 7;
      cx<T>* gx = smem + L.ogx;
      T* wx = reinterpret_cast<T*>(smem + L.owx);
      for (int e = B.tid; e < K * s.n1; e += NT) {   // [K][n1]: lanes of one row read consecutive columns
        const int i = e / K, k = e - i * K;
        gx[k * s.n1 + i] = L.gx[e];
        wx[k * s.n1 + i] = L.wx[e];
      }
      cx<T>* hy = smem + L.ohy;
      T* wy = reinterpret_cast<T*>(smem + L.owy);
      for (int e = B.tid; e < K * s.nr; e += NT) {
        hy[e] = L.hy[s.r0 * K + e];
        wy[e] = L.wy[s.r0 * K + e];
      }
    }
  }
  {   // the first level's right-hand side and iterate
    const Slab<T> s(B, 0);
    const cx<T>* gb = a.b + (long long)rhs * a.g.vstride;
    const cx<T>* gx = a.x + (long long)rhs * a.g.vstride;
    CL_NODES(s) {
      const int p = a.g.at(i, s.r0 + jl);
      smem[s.L->ob + q] = gb[p];
      smem[s.L->ox + q] = a.x_zero ? mk<T>(0, 0) : gx[p];
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  cl_sync();   // every block of the cluster runs; the slabs are loaded
  for (int k = 0; k < a.nsteps; ++k) {
    const ClStep st = a.steps[k];
    if (st.op == CL_COARSE) {
      coarse<NT>(B, Slab<T>(B, st.level));
    } else if (st.op == CL_PROLONG) {
      prolong<NT>(B, Slab<T>(B, st.level), st.level);
    } else {
      switch (lt[st.level].kind) {
        case 1: level_step<KindOf<1>, NT>(B, st); break;
        case 2:
          if (lt[st.level].ost >= 0) level_step<KindOf<2, true>, NT>(B, st);
          else level_step<KindOf<2>, NT>(B, st);
          break;
        case 3:
          if (lt[st.level].ost >= 0) level_step<KindOf<3, true>, NT>(B, st);
          else level_step<KindOf<3>, NT>(B, st);
          break;
        case 4: level_step<KindOf<4>, NT>(B, st); break;
        default: level_step<KindOf<5>, NT>(B, st); break;
      }
    }
  }
  const Slab<T> s(B, 0);
  cx<T>* gx = a.x + (long long)rhs * a.g.vstride;
  CL_NODES(s) gx[a.g.at(i, s.r0 + jl)] = smem[s.L->ox + q];
  cl_sync();   // no block leaves while another may still read its shared memory
}

template <class T, int NT>
__global__ void __launch_bounds__(NT, 1) k_cluster_cycle(const __grid_constant__ ClArgs<T> a) {
  extern __shared__ double2 cl_smem[];
  cluster_cycle<T, NT>(a, blockIdx.x / cl_size(), reinterpret_cast<cx<T>*>(cl_smem));
}

// One cluster per problem of a ragged batch (one right-hand side each).
template <class T, int NT>
__global__ void __launch_bounds__(NT, 1) k_cluster_cycle_rag(const __grid_constant__ ClRag<T> L) {
  extern __shared__ double2 cl_smem[];
  cluster_cycle<T, NT>(L.a[blockIdx.x / cl_size()], 0, reinterpret_cast<cx<T>*>(cl_smem));
}

// complex64 phases are latency-bound and want one node per thread; complex128
// ones are bound by the SM's FP64 pipe, which 8 warps fill.
template <class T> constexpr int cl_threads() { return sizeof(T) == 4 ? 512 : 256; }

constexpr int CL_SMEM = 225 * 1024;   // dynamic shared memory of a block (227 KB less the static part)

template <class T> const void* kern(bool rag) {
  return rag ? (const void*)k_cluster_cycle_rag<T, cl_threads<T>()> : (const void*)k_cluster_cycle<T, cl_threads<T>()>;
}

template <class T> cudaError_t configure(bool rag) {
  cudaError_t e = cudaFuncSetAttribute(kern<T>(rag), cudaFuncAttributeMaxDynamicSharedMemorySize, CL_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern<T>(rag), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

template <class T> cudaError_t launch(bool rag, void* arg, int C, int n, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(C * n));
  cfg.blockDim = dim3(cl_threads<T>());
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  void* args[1] = {arg};
  return cudaLaunchKernelExC(&cfg, kern<T>(rag), args);
}

}  // namespace

// Clusters of 2, 4, .. CL_MAXC blocks that the current device runs at once,
// and the kernels' attributes on it: a property of the device, asked for once
// (the queries take about half a millisecond, a tenth of a setup).
template <class T> static const int* cluster_counts() {
  constexpr int MAXDEV = 64, NC = 5;
  static_assert(1 << (NC - 1) == CL_MAXC, "cluster sizes");
  static std::mutex mu;
  static int table[MAXDEV][NC];   // [k]: clusters of 2^k blocks
  static bool known[MAXDEV];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAXDEV) return nullptr;
  std::lock_guard<std::mutex> lk(mu);
  if (!known[dev]) {
    if (configure<T>(false) != cudaSuccess || configure<T>(true) != cudaSuccess) return nullptr;
    for (int k = 1; k < NC; ++k) {
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(1u << k);
      cfg.blockDim = dim3(cl_threads<T>());
      cfg.dynamicSmemBytes = CL_SMEM;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = 1u << k;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kern<T>(false), &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
      }
      table[dev][k] = n;
    }
    known[dev] = true;
  }
  return table[dev];
}

template <class T> int cluster_size(int B) {
  const int* n = cluster_counts<T>();
  if (!n) return 0;
  for (int k = 4; k >= 1; --k)
    if (n[k] >= B) return 1 << k;
  return 1;
}

template <class T> bool cluster_layout(std::vector<ClLev<T>>& lv, int C, bool gmres, int N, ClArgs<T>& a) {
  // offsets in elements of cx<T>; every piece starts on a 16-byte boundary
  const int al = 16 / (int)sizeof(cx<T>);
  long long at = 0;
  auto take = [&](long long n) {
    const long long o = at;
    at += (n + al - 1) / al * al;
    return (int)o;
  };
  auto reals = [&](long long n) { return (n + 1) / 2; };
  long long nu = 0, nX = 0;
  const int nl = (int)lv.size();
  for (int l = 0; l < nl; ++l) {
    ClLev<T>& L = lv[l];
    const int R = op_radius(L.kind);
    L.n1 = L.nx + 1;
    L.rp = std::max(CL_MINROWS, cdiv(L.ny + 1, C));
    L.magic = (unsigned)(((1ull << 32) + L.n1 - 1) / L.n1);
    L.mrp = (unsigned)(((1ull << 32) + L.rp - 1) / L.rp);
    const long long nodes = (long long)L.rp * L.n1;
    if (nodes > (1 << 16)) return false;   // also keeps nodes * n1 in 32 bits (magic)
    const bool last = l == nl - 1;
    L.ox = take(nodes);
    L.ob = take(nodes);
    L.od = last || gmres ? -1 : take(nodes);
    L.ost = L.ogx = L.owx = L.ohy = L.owy = -1;
    if (last) continue;   // the coarsest level is solved, not smoothed
    if (L.kind >= 4) {
      const int K = 2 * R + 1;
      L.ogx = take((long long)K * L.n1);
      L.owx = take(reals((long long)K * L.n1));
      L.ohy = take((long long)K * L.rp);
      L.owy = take(reals((long long)K * L.rp));
    }
    nu = std::max(nu, nodes);
    nX = std::max(nX, (long long)(L.rp + 2 * R) * L.n1 * (L.kind >= 4 ? 2 : 1));
  }
  nu = (nu + al - 1) / al * al;
  nX = std::max((nX + al - 1) / al * al, (long long)(((size_t)N * sizeof(double2) / 2 + sizeof(cx<T>)) / sizeof(cx<T>) + al) / al * al);
  a.nu = (int)nu;
  a.nX = (int)nX;
  a.ou = take(nu * (gmres ? 4 : 2));
  a.oX = take(2 * nX);
  a.ored = take(reals((long long)CL_NV * (2 * C + 1 + cl_threads<T>() / 32) + GS));
  a.olev = take((long long)(sizeof(ClLev<T>) * nl + sizeof(cx<T>) - 1) / (long long)sizeof(cx<T>));
  if (at * (long long)sizeof(cx<T>) > CL_SMEM) return false;
  // what is left to the stored stencils, the coarsest level's first
  for (int l = nl - 2; l >= 0; --l) {
    const int K = 2 * op_radius(lv[l].kind) + 1;
    const long long n = (long long)K * K * lv[l].rp * lv[l].n1;
    if (lv[l].kind != 2 && lv[l].kind != 3) continue;
    if ((at + n + al) * (long long)sizeof(cx<T>) > CL_SMEM) break;
    lv[l].ost = take(n);
  }
  const long long bytes = at * (long long)sizeof(cx<T>);
  a.smem = (int)bytes;
  a.nlev = nl;
  a.C = C;
  a.N = N;
  return true;
}

template <class T> cudaError_t launch_cluster_cycle(const ClArgs<T>& a, int B, cudaStream_t s) {
  ClArgs<T> c = a;
  return launch<T>(false, &c, a.C, B, (size_t)a.smem, s);
}

template <class T> void launch_cluster_cycle_rag(const std::vector<ClArgs<T>>& v, cudaStream_t s) {
  static thread_local ClRag<T> L;
  for (size_t q0 = 0; q0 < v.size(); q0 += RMAXP) {
    const int n = (int)std::min<size_t>(RMAXP, v.size() - q0);
    int smem = 0;
    for (int q = 0; q < n; ++q) {
      L.a[q] = v[q0 + q];
      smem = std::max(smem, v[q0 + q].smem);
    }
    launch<T>(true, &L, v[q0].C, n, (size_t)smem, s);
  }
}

}  // namespace hmg
