// GMRES(3) kernels that apply A on the constant-k coarse levels (Kronecker
// form A = W_y (x) G_x + H_y (x) W_x, radius R = 2 or 3), as column marches.
//
// OpK::apply evaluates, for every output node, the 2R+1 row sums
// s1 = G_x v and s2 = W_x v of the rows around it and then combines them
// along y: about 6 (2R+1)^2 FMAs per node, which makes these levels
// arithmetic-bound.  Here a thread owns one column and walks down a chunk of
// rows: each row's two sums are formed once, kept in a ring of 2R+1 rows in
// registers, and combined for the output row R behind.  The sums and the
// combination run in the same order as OpK::apply, so A v is the same value;
// the work drops to about 12 (2R+1) FMAs per node and the kernels become
// bandwidth-bound.  Outputs, reductions and scalar steps are those of
// g_init and g_arn_a (kernels_gmres.cu); g_arn_b and g_update, which do not
// apply A, are shared.
#include <algorithm>
#include <type_traits>

#include "gmres.cuh"
#include "internal.h"
#include "kron.cuh"
#include "ragged.cuh"
#include "ragged_api.h"

namespace hmg {

namespace {

// Arguments of the column marches for one problem (the flattened launches of a
// ragged batch carry one per problem); each kernel reads the fields it takes.
template <class T, int R> struct KmA {
  Grid g;
  KGeo kg;
  OpK<T, R> op;
  const cx<T>* x;
  const cx<T>* b;
  cx<T>* u0;
  cx<T>* u1;
  cx<T>* u2;
  cx<T>* w;
  double* st;
  double* partial;
  unsigned* tickets;
  const int* active;
};

// What km_init leaves: u0 = b - A x and partial |u0|^2 (as g_init), only u0
// (the residual before the restriction; no norm, no state), or a weighted
// Jacobi sweep u0 = x + (omega diag A)^{-1} (b - A x)
enum { KM_NORM = 0, KM_RES = 1, KM_JACOBI = 2 };
template <class T, int R, int OUT = KM_NORM>
__device__ __forceinline__ void km_init_body(uint3 vblk, dim3 vgrid, Grid g, KGeo kg, OpK<T, R> op, const cx<T>* __restrict__ x, const cx<T>* __restrict__ b, cx<T>* __restrict__ u0, double* st, double* partial, unsigned* tickets, const int* __restrict__ active) {
  const uint3 blockIdx = vblk;   // the block and grid inside this problem's launch
  const dim3 gridDim = vgrid;
  (void)blockIdx;
  (void)gridDim;
  KPRO
  T a0[1] = {T(0)};
  __shared__ __align__(16) cx<T> kbsm[KW][KSL][32];   // b, staged with x
  if (has) {
    KRing<T, R> ring;
    ring.init(op, i, col);
    ring.vs = x + off;
    ring.g = g;
    ring.cw0 = cw0;
    ring.lane = lane;
    ring.sm = &ksm[wib][0][0];
    ring.r0 = j0 - R;
    ring.os = b + off;
    ring.osm = &kbsm[wib][0][0];
    const int last = j1 + R - 1;
    ring.prime(last);
    kmarch<KU<T, R>>(j0 - R, last, [&](auto ph, int r) {
      constexpr int P = decltype(ph)::value;
      ring.template advance<P>(r, last);
      const int m = r - R;
      if (m >= j0 && col) {
        const int p = g.at(i, m);
        cx<T> res = sub<T>(ring.own_at(m), ring.template combine<P>(op, m));
        if constexpr (OUT == KM_JACOBI) res = fma_c<T>(op.diag_inv(i, m), res, ring.staged_at(m));
        u0[off + p] = res;
        if constexpr (OUT == KM_NORM) add_abs2<T>(a0[0], res);
      }
    });
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  }
  if constexpr (OUT == KM_NORM) {
    double v[1];
    if (reduce_last<1, T>(a0, v, sh, partial, tickets, rhs, nblk, blk) && threadIdx.x == 0)
      fin_init<T>(gstate<T>(st, rhs), v);
  }
}

// km_init on a zero x: u0 = b (the caller passes b as u0 to the later
// passes); each lane sums |b|^2 down its column of the chunk, in km_init's
// order and over its blocks, so the state equals km_init's on a zero x.
template <class T>
__global__ void __launch_bounds__(KW * 32) km_init_zero(Grid g, KGeo kg, const cx<T>* __restrict__ b, double* st,
                                                        double* partial, unsigned* tickets,
                                                        const int* __restrict__ active) {
  __shared__ double sh[NVMAX * 32];
  const int rhs = blockIdx.z;
  if (active && !active[rhs]) return;
  const long long off = (long long)rhs * g.vstride;
  const int lane = threadIdx.x & 31;
  const int gw = blockIdx.x * KW + (threadIdx.x >> 5);
  const bool has = gw < kg.ncw * kg.nchunks;
  const int i = (has ? gw % kg.ncw : 0) * 32 + lane;
  const int j0 = (has ? gw / kg.ncw : 0) * kg.ch, j1 = min(j0 + kg.ch, g.ny + 1);
  T a0[1] = {T(0)};
  if (has && i <= g.nx) {
    const cx<T>* bs = b + off;
#pragma unroll 4
    for (int m = j0; m < j1; ++m) add_abs2<T>(a0[0], bs[g.at(i, m)]);
  }
  double v[1];
  if (reduce_last<1, T>(a0, v, sh, partial, tickets, rhs, gridDim.x, blockIdx.x) && threadIdx.x == 0)
    fin_init<T>(gstate<T>(st, rhs), v);
}

template <class T, int R, int OUT = KM_NORM>
__global__ void __launch_bounds__(KW * 32) km_init(Grid g, KGeo kg, OpK<T, R> op, const cx<T>* __restrict__ x, const cx<T>* __restrict__ b, cx<T>* __restrict__ u0, double* st, double* partial, unsigned* tickets, const int* __restrict__ active) {
  km_init_body<T, R, OUT>(blockIdx, gridDim, g, kg, op, x, b, u0, st, partial, tickets, active);
}

template <class T, int R>
__global__ void __launch_bounds__(KW * 32) km_init_rag(const __grid_constant__ RagLaunch<KmA<T, R>> L) {
  uint3 vb;
  dim3 vg;
  const KmA<T, R>& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  km_init_body<T, R>(vb, vg, a.g, a.kg, a.op, a.x, a.b, a.u0, a.st, a.partial, a.tickets, a.active);
}

// w = s_J A u_J; partial dots <u_l, w>, l <= J (as g_arn_a)
template <class T, int R, int J>
__device__ __forceinline__ void km_arn_a_body(uint3 vblk, dim3 vgrid, Grid g, KGeo kg, OpK<T, R> op, const cx<T>* __restrict__ u0, const cx<T>* __restrict__ u1, const cx<T>* __restrict__ u2, cx<T>* __restrict__ w, double* __restrict__ st, double* partial, unsigned* tickets, const int* __restrict__ active) {
  const uint3 blockIdx = vblk;   // the block and grid inside this problem's launch
  const dim3 gridDim = vgrid;
  (void)blockIdx;
  (void)gridDim;
  KPRO
  T* S = gstate<T>(st, rhs);
  if (S[G_BRK] != 0 || S[G_M] < J) return;   // uniform per RHS
  const cx<T>* uJ = J == 0 ? u0 : (J == 1 ? u1 : u2);
  T acc[2 * (J + 1)];
#pragma unroll
  for (int k = 0; k < 2 * (J + 1); ++k) acc[k] = T(0);
  if (has) {
    const T sJ = (T)S[G_S + J];
    const cx<T>* us[3] = {u0 + off, u1 + off, u2 + off};
    KMARCH_SETUP(uJ + off)
    kmarch<KU<T, R>>(j0 - R, last, [&](auto ph, int r) {
      constexpr int P = decltype(ph)::value;
      ring.template advance<P>(r, last);
      const int m = r - R;
      if (m >= j0 && col) {
        const int p = g.at(i, m);
        const cx<T> a = scl<T>(sJ, ring.template combine<P>(op, m));
        w[off + p] = a;
#pragma unroll
        for (int l = 0; l <= J; ++l)   // u_J is the staged vector
          add_cmul<T>(acc[2 * l], acc[2 * l + 1], l == J ? ring.staged_at(m) : us[l][p], a);
      }
    });
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  }
  double v[2 * (J + 1)];
  if (reduce_last<2 * (J + 1), T>(acc, v, sh, partial, tickets, rhs, nblk, blk))
    staged<T>(S, v, [](auto* s, const double* q) { fin_a<J, T>(s, q); });
}

template <class T, int R, int J>
__global__ void __launch_bounds__(KW * 32) km_arn_a(Grid g, KGeo kg, OpK<T, R> op, const cx<T>* __restrict__ u0, const cx<T>* __restrict__ u1, const cx<T>* __restrict__ u2, cx<T>* __restrict__ w, double* __restrict__ st, double* partial, unsigned* tickets, const int* __restrict__ active) {
  km_arn_a_body<T, R, J>(blockIdx, gridDim, g, kg, op, u0, u1, u2, w, st, partial, tickets, active);
}

template <class T, int R, int J>
__global__ void __launch_bounds__(KW * 32) km_arn_a_rag(const __grid_constant__ RagLaunch<KmA<T, R>> L) {
  uint3 vb;
  dim3 vg;
  const KmA<T, R>& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  km_arn_a_body<T, R, J>(vb, vg, a.g, a.kg, a.op, a.u0, a.u1, a.u2, a.w, a.st, a.partial, a.tickets, a.active);
}

// Blocks that share the device's time in the choice of the chunk height
// (kron_geo).  complex64: the blocks of the launched march (residual or Jacobi
// sweep) resident at once.  complex128: one per SM, because one warp per
// scheduler already fills the FP64 pipe, so a second block on an SM doubles its
// time (8 x 129^2, radius 3: 86 -> 56 us with one block of 9 rows per SM).
template <class T, int R, int OUT> long long kron_capacity() {
  static const long long cap = [] {
    int per = 1;
    if constexpr (sizeof(T) == 4) {
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, km_init<T, R, OUT>, KW * 32, 0);
      cudaGetLastError();
    }
    return (long long)std::max(per, 1) * device_sms();
  }();
  return cap;
}

}  // namespace

template <class T> void launch_gmres_update(const Grid& g, cx<T>* x, const GmresBufs& gb, int B, const int* active,
                                            cudaStream_t s);
template <class T, int J> void launch_arn_b(const Grid& g, const GmresBufs& gb, cx<T>* un, int B, const int* active,
                                            cudaStream_t s);

long long kron_march_blocks(const Grid& g, int B) {   // the most for any chunk height: the shortest
  (void)B;
  return cdiv((long long)cdiv(g.nx + 1, 32) * cdiv(g.ny + 1, KCH_MIN), KW);
}

template <class T>
void gmres_smooth_kron(const Grid& g, const OpView<T>& opv, cx<T>* x, const cx<T>* b, int nu, int B,
                       const int* active, const GmresBufs& gb, cudaStream_t s) {
  cx<T>* u0 = (cx<T>*)gb.u[0];
  cx<T>* u1 = (cx<T>*)gb.u[1];
  cx<T>* u2 = (cx<T>*)gb.u[2];
  cx<T>* w = (cx<T>*)gb.w;
  double* P = gb.partial;
  unsigned* tk = gb.tickets;
  double* st = gb.st;
  auto run = [&](auto op, auto rad) {
    constexpr int R = decltype(rad)::value;
    const KGeo kg = kron_geo(g, B, R, kron_capacity<T, R, KM_NORM>(), gb.kron_ch);
    const dim3 grd(cdiv((long long)kg.ncw * kg.nchunks, KW), 1, B);
    for (int step = 0; step < nu; ++step) {
      // a zero x: u0 = b itself (read-only in every later pass)
      const bool z = step == 0 && gb.x_zero;
      const cx<T>* v0 = z ? b : u0;
      GmresBufs gs = gb;
      gs.u[0] = (void*)v0;
      if (z) km_init_zero<T><<<grd, KW * 32, 0, s>>>(g, kg, b, st, P, tk, active);
      else km_init<T, R><<<grd, KW * 32, 0, s>>>(g, kg, op, x, b, u0, st, P, tk, active);
      km_arn_a<T, R, 0><<<grd, KW * 32, 0, s>>>(g, kg, op, v0, u1, u2, w, st, P, tk, active);
      launch_arn_b<T, 0>(g, gs, u1, B, active, s);
      km_arn_a<T, R, 1><<<grd, KW * 32, 0, s>>>(g, kg, op, v0, u1, u2, w, st, P, tk, active);
      launch_arn_b<T, 1>(g, gs, u2, B, active, s);
      km_arn_a<T, R, 2><<<grd, KW * 32, 0, s>>>(g, kg, op, v0, u1, u2, w, st, P, tk, active);
      launch_arn_b<T, 2>(g, gs, nullptr, B, active, s);
      launch_gmres_update<T>(g, x, gs, B, active, s);
    }
  };
  if (opv.kind == 4) run(kron_op<T, 2>(opv, g.nx, g.ny), std::integral_constant<int, 2>{});
  else run(kron_op<T, 3>(opv, g.nx, g.ny), std::integral_constant<int, 3>{});
}

namespace {
template <int OUT, class T>
void kron_pass(const Grid& g, const OpView<T>& opv, const cx<T>* x, const cx<T>* b, cx<T>* r, int B, const int* active,
               int kron_ch, cudaStream_t s) {
  auto run = [&](auto op, auto rad) {
    constexpr int R = decltype(rad)::value;
    const KGeo kg = kron_geo(g, B, R, kron_capacity<T, R, OUT>(), kron_ch);
    const dim3 grd(cdiv((long long)kg.ncw * kg.nchunks, KW), 1, B);
    km_init<T, R, OUT><<<grd, KW * 32, 0, s>>>(g, kg, op, x, b, r, nullptr, nullptr, nullptr, active);
  };
  if (opv.kind == 4) run(kron_op<T, 2>(opv, g.nx, g.ny), std::integral_constant<int, 2>{});
  else run(kron_op<T, 3>(opv, g.nx, g.ny), std::integral_constant<int, 3>{});
}
}  // namespace

template <class T>
void launch_kron_residual(const Grid& g, const OpView<T>& opv, const cx<T>* x, const cx<T>* b, cx<T>* r, int B,
                          const int* active, int kron_ch, cudaStream_t s) {
  kron_pass<KM_RES, T>(g, opv, x, b, r, B, active, kron_ch, s);
}
template <class T>
void launch_kron_jacobi(const Grid& g, const OpView<T>& opv, const cx<T>* x, const cx<T>* b, cx<T>* xo, int B,
                        const int* active, int kron_ch, cudaStream_t s) {
  kron_pass<KM_JACOBI, T>(g, opv, x, b, xo, B, active, kron_ch, s);
}

// The same smoothing steps on every problem of a ragged batch (the problems'
// levels at the same depth share the radius): each kernel of a step is one
// flattened launch over the problems' own chunk geometries.
template <class T>
void gmres_smooth_kron_rag(const std::vector<RagLevel<T>>& v, int nu, cudaStream_t s) {
  if (v.empty()) return;
  const int n = (int)v.size();
  auto run = [&](auto rad) {
    constexpr int R = decltype(rad)::value;
    std::vector<KmA<T, R>> A(n);
    for (int q = 0; q < n; ++q) {
      const RagLevel<T>& L = v[q];
      const OpView<T>& o = L.op;
      const OpK<T, R> op = kron_op<T, R>(o, L.g.nx, L.g.ny);
      const KGeo kg = kron_geo(L.g, 1, R, kron_capacity<T, R, KM_NORM>(), L.gb.kron_ch);
      A[q] = KmA<T, R>{L.g, kg, op, L.x, L.b, (cx<T>*)L.gb.u[0], (cx<T>*)L.gb.u[1], (cx<T>*)L.gb.u[2],
                       (cx<T>*)L.gb.w, L.gb.st, L.gb.partial, L.gb.tickets, L.active};
    }
    auto launch = [&](auto kern, auto set) {
      rag_launch<KmA<T, R>>(n, kern, dim3(KW * 32), 0, s, [&](int q, KmA<T, R>& a, int& gx, int&) {
        a = A[q];
        set(a, v[q]);
        gx = cdiv((long long)a.kg.ncw * a.kg.nchunks, KW);
        return true;
      });
    };
    auto none = [](KmA<T, R>&, const RagLevel<T>&) {};
    for (int step = 0; step < nu; ++step) {
      launch(km_init_rag<T, R>, none);
      launch(km_arn_a_rag<T, R, 0>, none);
      launch_arn_b_rag<T, 0>(v, true, s);
      launch(km_arn_a_rag<T, R, 1>, none);
      launch_arn_b_rag<T, 1>(v, true, s);
      launch(km_arn_a_rag<T, R, 2>, none);
      launch_arn_b_rag<T, 2>(v, false, s);
      launch_gmres_update_rag<T>(v, s);
    }
  };
  if (v[0].op.kind == 4) run(std::integral_constant<int, 2>{});
  else run(std::integral_constant<int, 3>{});
}

template void gmres_smooth_kron_rag<double>(const std::vector<RagLevel<double>>&, int, cudaStream_t);
template void launch_kron_residual<double>(const Grid&, const OpView<double>&, const double2*, const double2*,
                                           double2*, int, const int*, int, cudaStream_t);
template void launch_kron_residual<float>(const Grid&, const OpView<float>&, const float2*, const float2*, float2*,
                                          int, const int*, int, cudaStream_t);
template void launch_kron_jacobi<double>(const Grid&, const OpView<double>&, const double2*, const double2*, double2*,
                                         int, const int*, int, cudaStream_t);
template void launch_kron_jacobi<float>(const Grid&, const OpView<float>&, const float2*, const float2*, float2*, int,
                                        const int*, int, cudaStream_t);
template void gmres_smooth_kron<double>(const Grid&, const OpView<double>&, double2*, const double2*, int, int,
                                        const int*, const GmresBufs&, cudaStream_t);

}  // namespace hmg
