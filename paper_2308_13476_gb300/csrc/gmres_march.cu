// GMRES(3) smoothing step (Sec. 5.3 of the paper) on the fine level in four
// row-marching passes plus the update.
//
// The node-parallel version (kernels_gmres.cu) stores w = A v_j and needs
// eight grid passes, about 28 vector reads and writes per step.  Here each
// warp owns a strip of columns and walks down a chunk of rows, keeping the
// rows it needs of every field in registers (horizontal neighbours come from
// the adjacent lanes by shuffles).  Row m of the next Arnoldi vector is
// formed as soon as rows m-1..m+1 of its input are in registers (w = A v_j is
// recomputed, never stored), and A is applied to the new vector one row
// behind, so the dots of Arnoldi step j+1 come out of the pass that creates
// u_{j+1}:
//   M0: u0 = b - A x                      |u0|^2, <u0, A u0>
//   M1: u1 = s0 A u0 - c00 u0             |u1|^2, <u1, u0>, <u_l, A u1>
//   M2: u2 = s1 A u1 - sum c_l1 u_l       |u2|^2, <u2, u_l>, <u_l, A u2>
//   M3: u3 = s2 A u2 - sum c_l2 u_l       |u3|^2 (not stored)
//   then x += sum y_l s_l u_l (g_update).
// That is 16 vector passes per step (complex128; the complex64 cycles take
// the s-step marches of sstep_march.cu).  The scalar steps between passes are
// the same FP64 Gram-matrix updates and Givens solve (gmres.cuh) in the same order
// as the node-parallel version; only the dots of A u_{j+1} are taken before
// the scale s_{j+1} is known, and scaled afterwards.
//
// Geometry: a lane holds NP adjacent nodes (two for complex64, one 16-byte
// load; one for complex128).  A warp loads 32 NP columns starting two left of
// its strip; after the two stencil applications of a pass the outer two
// columns on each side are invalid, so a strip is 32 NP - 4 columns wide and
// neighbouring strips overlap by four loaded columns.  Rows: a warp covers a
// chunk of rows (see MGeo) and reads two rows above and below it.  Nodes outside the
// grid are zero in every produced vector (they are not unknowns).
//
// Rows arrive through a per-lane ring of NS 16-byte shared-memory slots per
// field, filled by cp.async NS - 1 rows ahead of use (each lane reads back
// only what it copied, so no barrier is needed).  A pass with fewer input
// fields keeps more rows in flight (NS = 8, 6, 4 for one, two, three fields),
// so that every pass has about the same bytes in flight per SM: with one warp
// per block and at most 32 blocks per SM, a one-field pass staging three rows
// ahead ran at half the bandwidth of the three-field pass.  Every field keeps
// the rows it uses in a ring of four registers; row r sits in register slot
// (r - j0 + 2) mod 4, and the march is unrolled by four so that these slots
// are compile-time names (no copies as the ring advances).  The block's
// reduction scratch reuses the staging ring once the march has ended.  A warp whose loaded
// columns and computed rows hold no boundary node takes the interior path:
// the stencil without boundary tests (the same arithmetic as Op0::apply5's
// interior case).
#include <algorithm>

#include "gmres.cuh"
#include "internal.h"
#include "march.cuh"
#include "ragged.cuh"
#include "ragged_api.h"

namespace hmg {

namespace {

// M0 at iteration t: x and b rows t arrive; u0 row t-1 = b - A x formed from
// x rows t-2..t; A u0 on row t-2.
template <class T, int MD> struct P0 {
  static constexpr int NP = MNP<T>::NP;
  MIn<T, MD, 2> m;   // 0: x, 1: b
  cx<T>* us;
  Row<T> U[4];
  T acc[3];
  template <int S> __device__ __forceinline__ void step(int t) {
    m.template fetch<S>(t);
    const MCtx<T, MD>& c = m.c;
    if (t < c.j0) return;
    const Row<T> ax = c.apply(m.F[0][Sl<S, -2>::v], m.F[0][Sl<S, -1>::v], m.F[0][Sl<S, 0>::v], t - 1);
    Row<T> u;
#pragma unroll
    for (int n = 0; n < NP; ++n) u.v[n] = psub<T>(m.F[1][Sl<S, -1>::v].v[n], ax.v[n]);   // both zero outside the grid
    U[Sl<S, -1>::v] = u;
    if (c.own_row(t - 1)) mstore(us, c.g, c.i, t - 1, u);
#pragma unroll
    for (int n = 0; n < NP; ++n)
      if (c.cnt(n, t - 1)) add_abs2<T>(acc[0], u.v[n]);
    if (t - 2 >= c.j0) {
      const Row<T> au = c.apply(U[Sl<S, -3>::v], U[Sl<S, -2>::v], U[Sl<S, -1>::v], t - 2);
#pragma unroll
      for (int n = 0; n < NP; ++n)
        if (c.cnt(n, t - 2)) {
          add_cmul<T>(acc[1], acc[2], U[Sl<S, -2>::v].v[n], au.v[n]);
        }
    }
  }
};

// M0 on a zero x (u0 = b, not stored): b row t arrives; |u0|^2 on row t-1
// and A u0 on row t-2, in P0's order (the same sums as P0 with x = 0).
template <class T, int MD> struct P0Z {
  static constexpr int NP = MNP<T>::NP;
  MIn<T, MD, 1> m;   // 0: b
  T acc[3];
  template <int S> __device__ __forceinline__ void step(int t) {
    m.template fetch<S>(t);
    const MCtx<T, MD>& c = m.c;
    if (t < c.j0) return;
    const Row<T>(&U)[4] = m.F[0];
#pragma unroll
    for (int n = 0; n < NP; ++n)
      if (c.cnt(n, t - 1)) add_abs2<T>(acc[0], U[Sl<S, -1>::v].v[n]);
    if (t - 2 >= c.j0) {
      const Row<T> au = c.apply(U[Sl<S, -3>::v], U[Sl<S, -2>::v], U[Sl<S, -1>::v], t - 2);
#pragma unroll
      for (int n = 0; n < NP; ++n)
        if (c.cnt(n, t - 2)) {
          add_cmul<T>(acc[1], acc[2], U[Sl<S, -2>::v].v[n], au.v[n]);
        }
    }
  }
};

// M1 at iteration t: u0 row t arrives; u1 row t-1 formed; A u1 on row t-2.
template <class T, int MD> struct P1 {
  static constexpr int NP = MNP<T>::NP;
  MIn<T, MD, 1> m;   // 0: u0
  cx<T>* ws;
  T s0;
  cx<T> c0;
  Row<T> U[4];
  T acc[7];
  template <int S> __device__ __forceinline__ void step(int t) {
    m.template fetch<S>(t);
    const MCtx<T, MD>& c = m.c;
    if (t < c.j0) return;
    const Row<T>(&V)[4] = m.F[0];
    const Row<T> av = c.apply(V[Sl<S, -2>::v], V[Sl<S, -1>::v], V[Sl<S, 0>::v], t - 1);
    Row<T> u;
#pragma unroll
    for (int n = 0; n < NP; ++n) {
      const cx<T> c[1] = {c0};
      const cx<T> v[1] = {V[Sl<S, -1>::v].v[n]};
      u.v[n] = scl_minus<T, 1>(s0, av.v[n], c, v);
    }
    U[Sl<S, -1>::v] = u;
    if (c.own_row(t - 1)) mstore(ws, c.g, c.i, t - 1, u);
#pragma unroll
    for (int n = 0; n < NP; ++n)
      if (c.cnt(n, t - 1)) {
        add_abs2<T>(acc[0], u.v[n]);
        add_cmul<T>(acc[1], acc[2], u.v[n], V[Sl<S, -1>::v].v[n]);
      }
    if (t - 2 >= c.j0) {
      const Row<T> au = c.apply(U[Sl<S, -3>::v], U[Sl<S, -2>::v], U[Sl<S, -1>::v], t - 2);
#pragma unroll
      for (int n = 0; n < NP; ++n)
        if (c.cnt(n, t - 2)) {
          add_cmul<T>(acc[3], acc[4], V[Sl<S, -2>::v].v[n], au.v[n]);
          add_cmul<T>(acc[5], acc[6], U[Sl<S, -2>::v].v[n], au.v[n]);
        }
    }
  }
};

// M2 at iteration t: u1 and u0 rows t arrive; u2 row t-1 formed; A u2 on
// row t-2.
template <class T, int MD> struct P2 {
  static constexpr int NP = MNP<T>::NP;
  MIn<T, MD, 2> m;   // 0: u1, 1: u0
  cx<T>* ws;
  T s1;
  cx<T> c0, c1;
  Row<T> U[4];
  T acc[11];
  template <int S> __device__ __forceinline__ void step(int t) {
    m.template fetch<S>(t);
    const MCtx<T, MD>& c = m.c;
    if (t < c.j0) return;
    const Row<T>(&V)[4] = m.F[0];
    const Row<T>(&Z)[4] = m.F[1];
    const Row<T> av = c.apply(V[Sl<S, -2>::v], V[Sl<S, -1>::v], V[Sl<S, 0>::v], t - 1);
    Row<T> u;
#pragma unroll
    for (int n = 0; n < NP; ++n) {
      const cx<T> c[2] = {c0, c1};
      const cx<T> v[2] = {Z[Sl<S, -1>::v].v[n], V[Sl<S, -1>::v].v[n]};
      u.v[n] = scl_minus<T, 2>(s1, av.v[n], c, v);
    }
    U[Sl<S, -1>::v] = u;
    if (c.own_row(t - 1)) mstore(ws, c.g, c.i, t - 1, u);
#pragma unroll
    for (int n = 0; n < NP; ++n)
      if (c.cnt(n, t - 1)) {
        add_abs2<T>(acc[0], u.v[n]);
        add_cmul<T>(acc[1], acc[2], u.v[n], Z[Sl<S, -1>::v].v[n]);
        add_cmul<T>(acc[3], acc[4], u.v[n], V[Sl<S, -1>::v].v[n]);
      }
    if (t - 2 >= c.j0) {
      const Row<T> au = c.apply(U[Sl<S, -3>::v], U[Sl<S, -2>::v], U[Sl<S, -1>::v], t - 2);
#pragma unroll
      for (int n = 0; n < NP; ++n)
        if (c.cnt(n, t - 2)) {
          add_cmul<T>(acc[5], acc[6], Z[Sl<S, -2>::v].v[n], au.v[n]);
          add_cmul<T>(acc[7], acc[8], V[Sl<S, -2>::v].v[n], au.v[n]);
          add_cmul<T>(acc[9], acc[10], U[Sl<S, -2>::v].v[n], au.v[n]);
        }
    }
  }
};

// M3 at iteration t: u2, u0 and u1 rows t arrive; u3 on row t-1.
template <class T, int MD> struct P3 {
  static constexpr int NP = MNP<T>::NP;
  MIn<T, MD, 3> m;   // 0: u2, 1: u0, 2: u1
  T s2;
  cx<T> cl[3];
  T acc[1];
  template <int S> __device__ __forceinline__ void step(int t) {
    m.template fetch<S>(t);
    const MCtx<T, MD>& c = m.c;
    if (t < c.j0 + 1) return;
    const Row<T>(&V)[4] = m.F[0];
    const Row<T> av = c.apply(V[Sl<S, -2>::v], V[Sl<S, -1>::v], V[Sl<S, 0>::v], t - 1);
#pragma unroll
    for (int n = 0; n < NP; ++n)
      if (c.cnt(n, t - 1)) {
        const cx<T> v[3] = {m.F[1][Sl<S, -1>::v].v[n], m.F[2][Sl<S, -1>::v].v[n], V[Sl<S, -1>::v].v[n]};
        const cx<T> u = scl_minus<T, 3>(s2, av.v[n], cl, v);
        add_abs2<T>(acc[0], u);
      }
  }
};

template <class T> __host__ __device__ constexpr int strip_w() { return 32 * MNP<T>::NP - 4; }

// Arguments of the march kernels for one problem (the flattened launches of a
// ragged batch carry one per problem).
template <class T> struct GmA {
  Grid g;
  MGeo mg;
  Op0<T> op;
  const cx<T>* x;
  const cx<T>* b;
  cx<T>* u0;
  cx<T>* u1;
  cx<T>* u2;
  double* st;
  double* partial;
  unsigned* tickets;
  const int* active;
};

// Common prologue (one warp per block).  i: first node of this lane; outl:
// the lane's nodes are in the strip's output columns.
#define MPRO                                                                  \
  constexpr int NP = MNP<T>::NP;                                              \
  const int rhs = blockIdx.z;                                                 \
  if (active && !active[rhs]) return;                                         \
  const long long off = (long long)rhs * g.vstride;                           \
  const int lane = threadIdx.x & 31;                                          \
  int strip, j0, j1;                                                          \
  mg.template map<MM<MD>>(blockIdx.x, strip, j0, j1);                         \
  const int cs = strip * strip_w<T>() - 2;                                    \
  const int i = cs + NP * lane;                                               \
  const bool outl = NP * lane >= 2 && NP * lane + NP <= 32 * NP - 2;          \
  T* S = gstate<T>(st, rhs);                                                  \
  const MCtx<T, MD> ctx{op, g, i, j0, j1, outl};

// Runs pass P on the warp's strip and chunk (rows j0-2 .. t1 read) and
// returns its sums in acc.  stg: the warp's staging area, [NF][NS slots][32
// lanes] of 16 bytes, free again (every copy landed, the warp converged) on
// return.
template <template <class, int> class P, class T, int MD, int NV, class Init>
__device__ __forceinline__ void run_pass(const MCtx<T, MD>& c, int t1, const void* stg, T (&acc)[NV], Init&& init) {
  P<T, MD> p;
  p.m.c = c;
  p.m.sbase = (uint32_t)__cvta_generic_to_shared(stg) + (threadIdx.x & 31) * 16;
  p.m.t1 = t1;
  init(p);
#pragma unroll
  for (int k = 0; k < NV; ++k) p.acc[k] = T(0);
  p.m.prime(c.j0 - 2);
  march(p, c.j0 - 2, t1);
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncwarp();
#pragma unroll
  for (int k = 0; k < NV; ++k) acc[k] = p.acc[k];
}

// The interior and boundary launches of a pass may run one after the other
// or side by side: every block publishes its sums (interior blocks in
// records 0 .. ni-1, boundary blocks after them) and takes a ticket counted
// over both launches; the block holding the last ticket sums all records in
// record order and runs the scalar step F.
// blk: the block's index inside its own launch (the body's blockIdx.x).
template <int MD, int NV, class T, class F>
__device__ __forceinline__ void finish(const T (&acc)[NV], double* sh, double* partial, unsigned* tickets, int rhs,
                                       int blk, const MGeo& mg, T* S, F f) {
  double v[NV];
  const int nrec = mg.nrec();
  if (reduce_last_at<NV, T>(acc, v, sh, partial, tickets, rhs, nrec, blk, mg.template rec0<MM<MD>>(), nrec))
    staged<T>(S, v, f);
}

// M0: u0 = b - A x; |u0|^2 and <u0, A u0>.
template <class T, int MD>
__device__ __forceinline__ void gm_init_body(uint3 vblk, Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ x,
                                              const cx<T>* __restrict__ b, cx<T>* __restrict__ u0, double* st,
                                              double* partial, unsigned* tickets, const int* __restrict__ active) {
  const uint3 blockIdx = vblk;   // the block index inside this problem's launch
  MPRO
  T acc[3];
  __shared__ __align__(16) unsigned char stg[ring_bytes<2>()];
  double* sh = reinterpret_cast<double*>(stg);
  run_pass<P0>(ctx, j1 + 1, stg, acc, [&](auto& p) {
    p.m.src[0] = x + off;
    p.m.src[1] = b + off;
    p.us = u0 + off;
  });
  finish<MD>(acc, sh, partial, tickets, rhs, (int)blockIdx.x, mg, S, [](auto* s, const double* q) {
    fin_init<T>(s, q);
    if (s[G_BRK] == 0) {   // <u0, w> with w = s0 A u0
      const double d[2] = {q[1] * s[G_S], q[2] * s[G_S]};
      fin_a<0, T>(s, d);
    }
  });
}

template <class T, int MD>
__global__ void __launch_bounds__(32) gm_init(Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ x,
                                              const cx<T>* __restrict__ b, cx<T>* __restrict__ u0, double* st,
                                              double* partial, unsigned* tickets, const int* __restrict__ active) {
  gm_init_body<T, MD>(blockIdx, g, mg, op, x, b, u0, st, partial, tickets, active);
}

template <class T, int MD>
__global__ void __launch_bounds__(32) gm_init_rag(const __grid_constant__ RagLaunch<GmA<T>> L) {
  uint3 vb;
  dim3 vg;
  const GmA<T>& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  gm_init_body<T, MD>(vb, a.g, a.mg, a.op, a.x, a.b, a.u0, a.st, a.partial, a.tickets, a.active);
}

// M0 on a zero x: u0 = b (the caller passes b as u0 to the later passes).
template <class T, int MD>
__global__ void __launch_bounds__(32) gm_init_zero(Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ b,
                                                   double* st, double* partial, unsigned* tickets,
                                                   const int* __restrict__ active) {
  MPRO
  T acc[3];
  __shared__ __align__(16) unsigned char stg[ring_bytes<1>()];
  double* sh = reinterpret_cast<double*>(stg);
  run_pass<P0Z>(ctx, j1 + 1, stg, acc, [&](auto& p) { p.m.src[0] = b + off; });
  finish<MD>(acc, sh, partial, tickets, rhs, (int)blockIdx.x, mg, S, [](auto* s, const double* q) {
    fin_init<T>(s, q);
    if (s[G_BRK] == 0) {
      const double d[2] = {q[1] * s[G_S], q[2] * s[G_S]};
      fin_a<0, T>(s, d);
    }
  });
}

// M1: u1 = s0 A u0 - c00 u0; |u1|^2, <u1, u0>, then <u0, A u1>, <u1, A u1>.
template <class T, int MD>
__device__ __forceinline__ void gm_step1_body(uint3 vblk, Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ u0,
                                               cx<T>* __restrict__ u1, double* st, double* partial,
                                               unsigned* tickets, const int* __restrict__ active) {
  const uint3 blockIdx = vblk;   // the block index inside this problem's launch
  MPRO
  if (S[G_BRK] != 0) return;   // uniform per RHS
  const T s0 = (T)S[G_S];
  const cx<T> c0 = mk<T>((T)(S[G_H] * S[G_S]), (T)(S[G_H + 1] * S[G_S]));
  T acc[7];
  __shared__ __align__(16) unsigned char stg[ring_bytes<1>()];
  double* sh = reinterpret_cast<double*>(stg);
  run_pass<P1>(ctx, j1 + 1, stg, acc, [&](auto& p) {
    p.m.src[0] = u0 + off;
    p.ws = u1 + off;
    p.s0 = s0;
    p.c0 = c0;
  });
  finish<MD>(acc, sh, partial, tickets, rhs, (int)blockIdx.x, mg, S, [](auto* s, const double* q) {
    fin_b<0, T>(s, q);
    if (s[G_BRK] == 0) {
      const double s1 = s[G_S + 1];
      const double d[4] = {q[3] * s1, q[4] * s1, q[5] * s1, q[6] * s1};
      fin_a<1, T>(s, d);
    }
  });
}

template <class T, int MD>
__global__ void __launch_bounds__(32) gm_step1(Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ u0,
                                               cx<T>* __restrict__ u1, double* st, double* partial,
                                               unsigned* tickets, const int* __restrict__ active) {
  gm_step1_body<T, MD>(blockIdx, g, mg, op, u0, u1, st, partial, tickets, active);
}

template <class T, int MD>
__global__ void __launch_bounds__(32) gm_step1_rag(const __grid_constant__ RagLaunch<GmA<T>> L) {
  uint3 vb;
  dim3 vg;
  const GmA<T>& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  gm_step1_body<T, MD>(vb, a.g, a.mg, a.op, a.u0, a.u1, a.st, a.partial, a.tickets, a.active);
}

// M2: u2 = s1 A u1 - c01 u0 - c11 u1; |u2|^2, <u2, u0>, <u2, u1>, then
// <u_l, A u2> for l = 0, 1, 2.
template <class T, int MD>
__device__ __forceinline__ void gm_step2_body(uint3 vblk, Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ u0,
                                               const cx<T>* __restrict__ u1, cx<T>* __restrict__ u2, double* st,
                                               double* partial, unsigned* tickets, const int* __restrict__ active) {
  const uint3 blockIdx = vblk;   // the block index inside this problem's launch
  MPRO
  if (S[G_BRK] != 0 || S[G_M] < 1) return;
  const T s1 = (T)S[G_S + 1];
  const cx<T> c0 = mk<T>((T)(S[G_H + 2 * 1] * S[G_S]), (T)(S[G_H + 2 * 1 + 1] * S[G_S]));
  const cx<T> c1 = mk<T>((T)(S[G_H + 2 * 4] * S[G_S + 1]), (T)(S[G_H + 2 * 4 + 1] * S[G_S + 1]));
  T acc[11];
  __shared__ __align__(16) unsigned char stg[ring_bytes<2>()];
  double* sh = reinterpret_cast<double*>(stg);
  run_pass<P2>(ctx, j1 + 1, stg, acc, [&](auto& p) {
    p.m.src[0] = u1 + off;
    p.m.src[1] = u0 + off;
    p.ws = u2 + off;
    p.s1 = s1;
    p.c0 = c0;
    p.c1 = c1;
  });
  finish<MD>(acc, sh, partial, tickets, rhs, (int)blockIdx.x, mg, S, [](auto* s, const double* q) {
    fin_b<1, T>(s, q);
    if (s[G_BRK] == 0) {
      const double s2 = s[G_S + 2];
      const double d[6] = {q[5] * s2, q[6] * s2, q[7] * s2, q[8] * s2, q[9] * s2, q[10] * s2};
      fin_a<2, T>(s, d);
    }
  });
}

template <class T, int MD>
__global__ void __launch_bounds__(32) gm_step2(Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ u0,
                                               const cx<T>* __restrict__ u1, cx<T>* __restrict__ u2, double* st,
                                               double* partial, unsigned* tickets, const int* __restrict__ active) {
  gm_step2_body<T, MD>(blockIdx, g, mg, op, u0, u1, u2, st, partial, tickets, active);
}

template <class T, int MD>
__global__ void __launch_bounds__(32) gm_step2_rag(const __grid_constant__ RagLaunch<GmA<T>> L) {
  uint3 vb;
  dim3 vg;
  const GmA<T>& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  gm_step2_body<T, MD>(vb, a.g, a.mg, a.op, a.u0, a.u1, a.u2, a.st, a.partial, a.tickets, a.active);
}

// M3: |u3|^2 with u3 = s2 A u2 - sum_l c_l2 u_l; then the least-squares
// solve (fin_b<2>).
template <class T, int MD>
__device__ __forceinline__ void gm_step3_body(uint3 vblk, Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ u0,
                                               const cx<T>* __restrict__ u1, const cx<T>* __restrict__ u2,
                                               double* st, double* partial, unsigned* tickets,
                                               const int* __restrict__ active) {
  const uint3 blockIdx = vblk;   // the block index inside this problem's launch
  MPRO
  if (S[G_BRK] != 0 || S[G_M] < 2) return;
  const T s2 = (T)S[G_S + 2];
  cx<T> cl[3];
#pragma unroll
  for (int l = 0; l < 3; ++l)
    cl[l] = mk<T>((T)(S[G_H + 2 * (l * 3 + 2)] * S[G_S + l]), (T)(S[G_H + 2 * (l * 3 + 2) + 1] * S[G_S + l]));
  T acc[1];
  __shared__ __align__(16) unsigned char stg[ring_bytes<3>()];
  double* sh = reinterpret_cast<double*>(stg);
  run_pass<P3>(ctx, j1, stg, acc, [&](auto& p) {
    p.m.src[0] = u2 + off;
    p.m.src[1] = u0 + off;
    p.m.src[2] = u1 + off;
    p.s2 = s2;
    p.cl[0] = cl[0];
    p.cl[1] = cl[1];
    p.cl[2] = cl[2];
  });
  finish<MD>(acc, sh, partial, tickets, rhs, (int)blockIdx.x, mg, S, [](auto* s, const double* q) { fin_b<2, T>(s, q); });
}

template <class T, int MD>
__global__ void __launch_bounds__(32) gm_step3(Grid g, MGeo mg, Op0<T, MA2<MD>> op, const cx<T>* __restrict__ u0,
                                               const cx<T>* __restrict__ u1, const cx<T>* __restrict__ u2,
                                               double* st, double* partial, unsigned* tickets,
                                               const int* __restrict__ active) {
  gm_step3_body<T, MD>(blockIdx, g, mg, op, u0, u1, u2, st, partial, tickets, active);
}

template <class T, int MD>
__global__ void __launch_bounds__(32) gm_step3_rag(const __grid_constant__ RagLaunch<GmA<T>> L) {
  uint3 vb;
  dim3 vg;
  const GmA<T>& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  gm_step3_body<T, MD>(vb, a.g, a.mg, a.op, a.u0, a.u1, a.u2, a.st, a.partial, a.tickets, a.active);
}

// Interior chunks are tall (few halo rows) unless the grid has too few
// strips to give every SM several warps.  Interior strips: loaded columns in
// 1..nx-1.
template <class T> MGeo march_geo(const Grid& g, int B) {
  constexpr int NP = MNP<T>::NP, SW = strip_w<T>();
  MGeo m;
  m.fill(g.nx, g.ny, SW, 32 * NP, 2, 3);
  const int inner_rows = g.ny - 5;
  const long long want = (long long)device_sms() * 48;   // warps to fill the GPU a few times over
  int ch = 64;
  while (ch > 8 && (long long)m.nstrips * cdiv(inner_rows, ch) * B < want) ch /= 2;
  m.chunks(ch);
  return m;
}

}  // namespace

// The x update of the node-parallel smoother (kernels_gmres.cu).
template <class T> void launch_gmres_update(const Grid& g, cx<T>* x, const GmresBufs& gb, int B, const int* active,
                                            cudaStream_t s);

long long gmres_march_blocks(const Grid& g, int B) {
  return march_geo<double>(g, B).nrec();
}

template <class T>
void gmres_smooth_march(const Grid& g, const OpView<T>& opv, cx<T>* x, const cx<T>* b, int nu, int B,
                        const int* active, const GmresBufs& gb, cudaStream_t s) {
  cx<T>* u0 = (cx<T>*)gb.u[0];
  cx<T>* u1 = (cx<T>*)gb.u[1];
  cx<T>* u2 = (cx<T>*)gb.u[2];
  double* P = gb.partial;
  unsigned* tk = gb.tickets;
  double* st = gb.st;
  const Op0<T> op{opv.c0, opv.kf, g.nx, g.ny};
  const MGeo mg = march_geo<T>(g, B);
  const dim3 gi(mg.ni, 1, B), ge(mg.ne(), 1, B), gbd(mg.nb, 1, B);
  // the edge-strip and band launches of each pass on the side stream, beside
  // the interior one (their few warps then overlap the interior launch)
  const bool fork = gb.side && mg.ni;
  cudaStream_t sb = fork ? gb.side : s;
  auto pass = [&](auto interior, auto edge, auto bands) {
    if (fork) {
      cudaEventRecord(gb.ev_fork, s);
      cudaStreamWaitEvent(gb.side, gb.ev_fork, 0);
    }
    if (mg.ne()) edge();
    bands();
    if (mg.ni) interior();
    if (fork) {
      cudaEventRecord(gb.ev_join, gb.side);
      cudaStreamWaitEvent(s, gb.ev_join, 0);
    }
  };
  // the edge-strip and band launches take the boundary operator: with the
  // second-order absorbing rows its compile-time variant (modes 6 and 4)
  auto body = [&](auto opb, auto a2) {
    constexpr int ME = decltype(a2)::value ? 6 : 2, MB = decltype(a2)::value ? 4 : 0;
    for (int step = 0; step < nu; ++step) {
      // a zero x: u0 = b itself (read-only in every later pass)
      const bool z = step == 0 && gb.x_zero;
      if (z) {
        pass([&] { gm_init_zero<T, 1><<<gi, 32, 0, s>>>(g, mg, op, b, st, P, tk, active); },
             [&] { gm_init_zero<T, ME><<<ge, 32, 0, sb>>>(g, mg, opb, b, st, P, tk, active); },
             [&] { gm_init_zero<T, MB><<<gbd, 32, 0, sb>>>(g, mg, opb, b, st, P, tk, active); });
      } else {
        pass([&] { gm_init<T, 1><<<gi, 32, 0, s>>>(g, mg, op, x, b, u0, st, P, tk, active); },
             [&] { gm_init<T, ME><<<ge, 32, 0, sb>>>(g, mg, opb, x, b, u0, st, P, tk, active); },
             [&] { gm_init<T, MB><<<gbd, 32, 0, sb>>>(g, mg, opb, x, b, u0, st, P, tk, active); });
      }
      const cx<T>* v0 = z ? b : u0;
      GmresBufs gs = gb;
      gs.u[0] = (void*)v0;
      pass([&] { gm_step1<T, 1><<<gi, 32, 0, s>>>(g, mg, op, v0, u1, st, P, tk, active); },
           [&] { gm_step1<T, ME><<<ge, 32, 0, sb>>>(g, mg, opb, v0, u1, st, P, tk, active); },
           [&] { gm_step1<T, MB><<<gbd, 32, 0, sb>>>(g, mg, opb, v0, u1, st, P, tk, active); });
      pass([&] { gm_step2<T, 1><<<gi, 32, 0, s>>>(g, mg, op, v0, u1, u2, st, P, tk, active); },
           [&] { gm_step2<T, ME><<<ge, 32, 0, sb>>>(g, mg, opb, v0, u1, u2, st, P, tk, active); },
           [&] { gm_step2<T, MB><<<gbd, 32, 0, sb>>>(g, mg, opb, v0, u1, u2, st, P, tk, active); });
      pass([&] { gm_step3<T, 1><<<gi, 32, 0, s>>>(g, mg, op, v0, u1, u2, st, P, tk, active); },
           [&] { gm_step3<T, ME><<<ge, 32, 0, sb>>>(g, mg, opb, v0, u1, u2, st, P, tk, active); },
           [&] { gm_step3<T, MB><<<gbd, 32, 0, sb>>>(g, mg, opb, v0, u1, u2, st, P, tk, active); });
      launch_gmres_update<T>(g, x, gs, B, active, s);
    }
  };
  if (opv.c0.abc2) body(Op0<T, true>{opv.c0, opv.kf, g.nx, g.ny}, std::true_type{});
  else body(op, std::false_type{});
}

// The same smoothing steps on every problem of a ragged batch: each pass is
// one flattened launch per kind of warp (interior strips; edge strips and
// bands on the side stream), over the problems' own geometries.
template <class T>
void gmres_smooth_march_rag(const std::vector<RagLevel<T>>& v, int nu, cudaStream_t s, cudaStream_t side,
                            cudaEvent_t fork, cudaEvent_t join) {
  const int n = (int)v.size();
  std::vector<GmA<T>> A(n);
  bool any_interior = false;
  for (int q = 0; q < n; ++q) {
    const RagLevel<T>& L = v[q];
    const MGeo mg = march_geo<T>(L.g, 1);
    any_interior |= mg.ni > 0;
    A[q] = GmA<T>{L.g, mg, Op0<T>{L.op.c0, L.op.kf, L.g.nx, L.g.ny}, L.x, L.b, (cx<T>*)L.gb.u[0],
                  (cx<T>*)L.gb.u[1], (cx<T>*)L.gb.u[2], L.gb.st, L.gb.partial, L.gb.tickets, L.active};
  }
  const bool fk = side && any_interior;
  cudaStream_t sb = fk ? side : s;
  auto launch = [&](auto kern, int md, cudaStream_t st) {
    rag_launch<GmA<T>>(n, kern, dim3(32), 0, st, [&](int q, GmA<T>& a, int& gx, int&) {
      a = A[q];
      gx = md == 1 ? a.mg.ni : (md == 2 ? a.mg.ne() : a.mg.nb);
      return true;
    });
  };
  auto pass = [&](auto ki, auto ke, auto kb) {
    if (fk) {
      cudaEventRecord(fork, s);
      cudaStreamWaitEvent(side, fork, 0);
    }
    launch(ke, 2, sb);
    launch(kb, 0, sb);
    launch(ki, 1, s);
    if (fk) {
      cudaEventRecord(join, side);
      cudaStreamWaitEvent(s, join, 0);
    }
  };
  for (int step = 0; step < nu; ++step) {
    pass(gm_init_rag<T, 1>, gm_init_rag<T, 2>, gm_init_rag<T, 0>);
    pass(gm_step1_rag<T, 1>, gm_step1_rag<T, 2>, gm_step1_rag<T, 0>);
    pass(gm_step2_rag<T, 1>, gm_step2_rag<T, 2>, gm_step2_rag<T, 0>);
    pass(gm_step3_rag<T, 1>, gm_step3_rag<T, 2>, gm_step3_rag<T, 0>);
    launch_gmres_update_rag<T>(v, s);
  }
}

template void gmres_smooth_march_rag<double>(const std::vector<RagLevel<double>>&, int, cudaStream_t, cudaStream_t,
                                             cudaEvent_t, cudaEvent_t);
template void gmres_smooth_march<double>(const Grid&, const OpView<double>&, double2*, const double2*, int, int,
                                         const int*, const GmresBufs&, cudaStream_t);

}  // namespace hmg
