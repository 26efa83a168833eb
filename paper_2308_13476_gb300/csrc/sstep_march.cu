// GMRES(3) smoothing step of the complex64 cycles on the fine level: two row
// marches and no stored Krylov vector.
//
// The s-step form (sstep.cuh) needs no global sum between the operator
// applications of a step, so all of them run in one march: rows of x and b
// arrive, and behind the row t being read the warp forms
//   r = b - A x on row t-1,  v1 = B r on row t-2,  v2 = B v1 on row t-3,
//   v3 = B v2 on row t-4,    B = scale A - sigma,
// and adds the Gram matrix of (r, v1, v2, v3) on row t-4 (ss_gram).  The last
// block solves the normal equations.  The second march forms r, v1 and v2
// again and writes x' = x + y0 r + y1 v1 + y2 v2 to another vector, since
// the neighbouring strips still read x (ss_update; in the refinement loop it
// adds x' to the FP64 iterate instead).  That is 2 + 3 vector passes per
// step (1 + 2 on a zero x, where r = b) against the Arnoldi form's 13, with
// about twice the arithmetic.
//
// What bounds it: the issue slots (about 200 instructions per row of 56 nodes
// and pass, half of them FP32) with the vector passes close behind: at 64 x
// 1025^2 the Gram march takes 323 us (1.08 GB of vectors, 49 % of measured HBM
// bandwidth) and the update 264 us (1.6 GB, 90 %), together 587 us against the
// 1210 us of the Arnoldi form's passes; one 1025^2 right-hand side 31 against
// 85 us.
//
// A lane holds two adjacent nodes; a warp loads 64 columns starting four left
// of its strip and writes 56.  Rows: four above and below the chunk (three
// for the update).
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "march.cuh"
#include "pack.cuh"
#include "ragged.cuh"
#include "ragged_api.h"
#include "sstep.cuh"

namespace hmg {
namespace {

constexpr int SHW = 4, SSW = 64 - 2 * SHW, SBR = 4;

// Arguments of the marches for one problem.
struct SmA {
  Grid g;
  MGeo mg;
  Op0<float> op;
  float scale, sigma;
  const float2* x;
  const float2* b;
  float2* xo;          // update: x'
  double2* outer;      // update: the FP64 iterate x' is added to (null: x' stored)
  double* st;
  double* partial;
  unsigned* tickets;
  const int* active;
  int nblk;            // blocks per right-hand side
  const float* rscale; // update into outer: x' is divided by rscale[2 rhs]
};

// Warp modes: 0 interior strips (branch-free five-point stencil), 1 strips
// and rows with boundary nodes (first-order absorbing rows: the stencil with
// lane-constant column weights and row weights, which are zero off the grid),
// 2 the same with the second-order absorbing rows (Op0<float, true>).
//
// The input rows arrive through a per-lane ring of 8 shared-memory slots per
// field, four rows ahead: row r sits in half ((r - t0) / 4) mod 2, slot (r -
// t0) mod 4, so that the march, unrolled by four, names its slots at compile
// time and only swaps halves.
constexpr int RING = 8 * 512;   // bytes of one field's ring

template <int MODE, int NF, bool VK> struct SIn {
  Op0<float, MODE == 2> op;
  int i, ny, j0, n, pitch, ok;  // n: output rows
  float sc, sg;
  float d, e, q, ih2;           // interior coefficients (constant k): A x = d x - ih2 sum; B v = e v + q sum
  float wx[2];                  // column weights (mode 1): 1, 1/2 on columns 0 and nx, 0 off the grid
  const float2* src[NF];        // this lane's nodes of row t + 4 of the input fields
  uint32_t sh, half;            // shared address of this lane's slot 0 of field 0, offset of row t's half
  int left;                     // rows still to issue
  Row<float> F[NF][4];          // register ring: row r in slot (r - t0) mod 4

  // the next row in flight, into the slot at `slot`, with what extra(slot) adds to it
  template <class E> __device__ __forceinline__ void issue(uint32_t slot, E&& extra) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      if (left > 0)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(slot + f * RING), "l"(src[f]), "r"(ok)
                     : "memory");
      src[f] += pitch;
    }
    --left;
    extra(slot);
    stage_commit();
  }
  template <class E> __device__ __forceinline__ void prime(E&& extra) {
#pragma unroll
    for (int k = 0; k < 4; ++k) issue(sh + k * 512, extra);   // half 0
  }
  // row t + 4 in flight, row t into the register ring
  template <int S, class E> __device__ __forceinline__ void fetch(E&& extra) {
    issue(sh + (half ^ (4 * 512)) + S * 512, extra);
    stage_wait<4>();
#pragma unroll
    for (int f = 0; f < NF; ++f)
      F[f][S] = stage_read(reinterpret_cast<const float4*>(__cvta_shared_to_generic(sh + half + f * RING + S * 512)));
  }

  // row weight: 1, 1/2 on rows 0 and ny, 0 off the grid
  __device__ __forceinline__ float wrow(int m) const {
    return (unsigned)m > (unsigned)ny ? 0.f : (m == 0 || m == ny) ? 0.5f : 1.f;
  }
  __device__ __forceinline__ float kat(int in, int m) const {
    if (!VK || !op.kf) return op.c.k;
    if constexpr (MODE != 0) in = min(max(in, 0), op.nx);
    return op.kf[min(max(m, 0), ny) * (op.nx + 1) + in];   // rows the march warms up on may be off the grid
  }
  // RES: bb - A v, else B v, on row m from rows m-1..m+1 of v
  template <bool RES>
  __device__ __forceinline__ Row<float> apply(const Row<float>& dn, const Row<float>& c, const Row<float>& up, int m,
                                              const Row<float>& bb) const {
    const float2 west = shfl_up1<float>(c.v[1]), east = shfl_dn1<float>(c.v[0]);
    Row<float> r;
#pragma unroll
    for (int n_ = 0; n_ < 2; ++n_) {
      const float2 xe = n_ == 0 ? c.v[1] : east, xw = n_ == 1 ? c.v[0] : west, v = c.v[n_];
      const int in = i + n_;
      if constexpr (MODE == 0) {
        const float2 sn = add2(add2(xe, xw), add2(up.v[n_], dn.v[n_]));
        float dd = d, ee = e;
        if constexpr (VK) {
          const float k = kat(in, m);
          dd = fmaf(-k, k, 4.f * ih2);
          ee = -sc * k * k;
        }
        if constexpr (RES) r.v[n_] = fma2(bc2(-dd), v, fma2(bc2(ih2), sn, bb.v[n_]));
        else r.v[n_] = fma2(bc2(ee), v, mul2(bc2(q), sn));
      } else if constexpr (MODE == 1) {
        const float wy = wrow(m), w = wx[n_] * wy, k = kat(in, m);
        const float bt = k * op.c.inv_h * ((wx[n_] == 0.5f ? wy : 0.f) + (wy == 0.5f ? wx[n_] : 0.f));
        const float2 sn = fma2(bc2(wy), add2(xe, xw), mul2(bc2(wx[n_]), add2(up.v[n_], dn.v[n_])));
        const float in_grid = w > 0.f ? 1.f : 0.f;
        if constexpr (RES) {
          const float ar = w * fmaf(-k, k, 4.f * ih2);
          const float2 t = fma2(bc2(-ar), v, fma2(bc2(in_grid * ih2), sn, bb.v[n_]));
          r.v[n_] = make_float2(fmaf(-bt, v.y, t.x), fmaf(bt, v.x, t.y));
        } else {
          const float er = fmaf(-w * sc, k * k, w - sg), ei = sc * bt;
          const float2 t = fma2(bc2(er), v, mul2(bc2(in_grid * q), sn));
          r.v[n_] = make_float2(fmaf(ei, v.y, t.x), fmaf(-ei, v.x, t.y));
        }
      } else {
        r.v[n_] = zc<float>();
        if (m >= 0 && m <= ny && in >= 0 && in <= op.nx) {
          const float2 a = op.apply5(v, xe, xw, up.v[n_], dn.v[n_], in, m);
          r.v[n_] = RES ? sub2(bb.v[n_], a) : make_float2(fmaf(sc, a.x, -sg * v.x), fmaf(sc, a.y, -sg * v.y));
        }
      }
    }
    return r;
  }
};

// P::step<S>(t) for t = t0, t0 + 1, ..: full groups of four rows up to at
// least t1 (the rows past t1 repeat old data and are not output).
template <class P> __device__ __forceinline__ void smarch(P& p, int t0, int t1) {
#pragma unroll 1
  for (int t = t0; t <= t1; t += 4) {
    p.template step<0>(t);
    p.template step<1>(t + 1);
    p.template step<2>(t + 2);
    p.template step<3>(t + 3);
    p.m.half ^= 4 * 512;
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// The Gram sums in packed form: norms and real parts as sums of component
// products, imaginary parts as scalars.
struct GramAcc {
  float2 n[4], re[6];
  float im[6];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < 4; ++k) n[k] = zc<float>();
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      re[k] = zc<float>();
      im[k] = 0.f;
    }
  }
  __device__ __forceinline__ void add(float2 a, float2 b, float2 c, float2 d) {
    const float2 v[4] = {a, b, c, d};
    int k = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      n[i] = fma2(v[i], v[i], n[i]);
#pragma unroll
      for (int j = i + 1; j < 4; ++j, ++k) {
        re[k] = fma2(v[i], v[j], re[k]);
        im[k] = fmaf(v[i].x, v[j].y, fmaf(-v[i].y, v[j].x, im[k]));
      }
    }
  }
  __device__ __forceinline__ void out(float (&g)[SS_NV], bool mine) const {
#pragma unroll
    for (int k = 0; k < 4; ++k) g[k] = mine ? n[k].x + n[k].y : 0.f;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      g[4 + 2 * k] = mine ? re[k].x + re[k].y : 0.f;
      g[5 + 2 * k] = mine ? im[k] : 0.f;
    }
  }
};

// Krylov rows behind the row t being read: r on row t - D, v1 on t - D - 1
// and v2 on t - D - 2.  Z: x = 0, so r = b and the rows of r arrive themselves
// (D = 0).  The first rows a march forms are of no use (their inputs were not
// read); nothing output depends on them.
template <int MODE, bool Z, bool VK> struct SMarch {
  static constexpr int NF = Z ? 1 : 2, D = Z ? 0 : 1;
  SIn<MODE, NF, VK> m;   // x, b (Z: b)
  Row<float> R[4], V1[4], V2[4];
  template <int S, int K> __device__ __forceinline__ const Row<float>& r() const {   // r on row t - K
    if constexpr (Z) return m.F[0][Sl<S, -K>::v];
    else return R[Sl<S, -K>::v];
  }
  template <int S, class E> __device__ __forceinline__ void rows(int t, E&& extra) {
    m.template fetch<S>(extra);
    if constexpr (!Z)
      R[Sl<S, -1>::v] = m.template apply<true>(m.F[0][Sl<S, -2>::v], m.F[0][Sl<S, -1>::v], m.F[0][Sl<S, 0>::v], t - 1,
                                               m.F[NF - 1][Sl<S, -1>::v]);
    V1[Sl<S, -D - 1>::v] = m.template apply<false>(r<S, D + 2>(), r<S, D + 1>(), r<S, D>(), t - D - 1, r<S, D>());
    V2[Sl<S, -D - 2>::v] = m.template apply<false>(V1[Sl<S, -D - 3>::v], V1[Sl<S, -D - 2>::v], V1[Sl<S, -D - 1>::v],
                                                   t - D - 2, V1[Sl<S, -D - 1>::v]);
  }
};

template <int MODE, bool Z, bool VK> struct SGram : SMarch<MODE, Z, VK> {
  using M = SMarch<MODE, Z, VK>;
  GramAcc acc;
  template <int S> __device__ __forceinline__ void step(int t) {
    constexpr int D = M::D;
    this->template rows<S>(t, [](uint32_t) {});
    if ((unsigned)(t - D - 3 - this->m.j0) >= (unsigned)this->m.n) return;
    const Row<float> v3 = this->m.template apply<false>(this->V2[Sl<S, -D - 4>::v], this->V2[Sl<S, -D - 3>::v],
                                                        this->V2[Sl<S, -D - 2>::v], t - D - 3, this->V2[0]);
#pragma unroll
    for (int n = 0; n < 2; ++n)
      acc.add(this->template r<S, D + 3>().v[n], this->V1[Sl<S, -D - 3>::v].v[n], this->V2[Sl<S, -D - 3>::v].v[n],
              v3.v[n]);
  }
};

template <int MODE, bool Z, bool VK, bool OUT> struct SUpd : SMarch<MODE, Z, VK> {
  using M = SMarch<MODE, Z, VK>;
  float2* xo;        // this lane's nodes of the output row of step t (moves with t)
  double2* x64;      // OUT: the same of the FP64 iterate,
  const double2* xs; // and of the row 4 steps ahead, staged with the input rows (fields NF, NF + 1 of the ring)
  int rs;            // that row, counted from j0
  int nv;            // nodes of this lane to write (0: none)
  double ig;         // OUT: 1 / rscale
  float2 y[3];
  __device__ __forceinline__ void stage64(uint32_t slot) {
#pragma unroll
    for (int n = 0; n < 2; ++n)
      if ((unsigned)rs < (unsigned)this->m.n && n < nv)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(slot + (M::NF + n) * RING), "l"(xs + n)
                     : "memory");
    ++rs;
    xs += this->m.pitch;
  }
  template <int S> __device__ __forceinline__ void step(int t) {
    constexpr int D = M::D;
    const bool mine = (unsigned)(t - D - 2 - this->m.j0) < (unsigned)this->m.n;
    this->template rows<S>(t, [&](uint32_t slot) {
      if constexpr (OUT) stage64(slot);
    });
    if (mine) {
      float2 u[2];
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const float2 v[3] = {this->template r<S, D + 2>().v[n], this->V1[Sl<S, -D - 2>::v].v[n],
                             this->V2[Sl<S, -D - 2>::v].v[n]};
        float2 a, w = mul2(bc2(y[0].y), v[0]);
        if constexpr (Z) a = mul2(bc2(y[0].x), v[0]);
        else a = fma2(bc2(y[0].x), v[0], this->m.F[0][Sl<S, -D - 2>::v].v[n]);
#pragma unroll
        for (int l = 1; l < 3; ++l) {
          a = fma2(bc2(y[l].x), v[l], a);
          w = fma2(bc2(y[l].y), v[l], w);
        }
        u[n] = make_float2(a.x - w.y, a.y + w.x);
      }
      if constexpr (OUT) {
#pragma unroll
        for (int n = 0; n < 2; ++n)
          if (n < nv) {
            const double2 o = *reinterpret_cast<const double2*>(
                __cvta_shared_to_generic(this->m.sh + this->m.half + (M::NF + n) * RING + S * 512));
            x64[n] = make_double2(fma(ig, f64_from_f32(u[n].x), o.x), fma(ig, f64_from_f32(u[n].y), o.y));
          }
      } else {
        if (nv == 2) *reinterpret_cast<float4*>(xo) = make_float4(u[0].x, u[0].y, u[1].x, u[1].y);
        else if (nv == 1) *xo = u[0];
      }
    }
    if constexpr (OUT) x64 += this->m.pitch;
    else xo += this->m.pitch;
  }
};

constexpr int SWB = 4;   // warps per block
constexpr int SWO = 2;   // of the update that stages the FP64 iterate too (16 KB per warp)

// Strip and rows [j0, j1) of warp w of a problem's launch and its mode: edge
// strips first, then the bands, then the interior strips (the slower warps
// start first).  -1: no work.
__device__ __forceinline__ int sm_map(const MGeo& mg, int w, int& strip, int& j0, int& j1) {
  const int ne = mg.ne();
  if (w < ne) mg.template map<2>(w, strip, j0, j1);
  else if (w < ne + mg.nb) mg.template map<0>(w - ne, strip, j0, j1);
  else if (w < ne + mg.nb + mg.ni) mg.template map<1>(w - ne - mg.nb, strip, j0, j1);
  else return -1;
  return w < ne + mg.nb ? 1 : 0;
}

template <bool Z, int MODE, int NF, bool VK>
__device__ __forceinline__ void sm_setup(SIn<MODE, NF, VK>& m, const SmA& a, int strip, int j0, int j1, long long off,
                                         const void* stg) {
  const int lane = threadIdx.x & 31;
  m.op = Op0<float, MODE == 2>{a.op.c, a.op.kf, a.g.nx, a.g.ny};
  m.i = strip * SSW - SHW + 2 * lane;
  m.ny = a.g.ny;
  m.j0 = j0;
  m.n = j1 - j0;
  m.pitch = a.g.pitch;
  m.ok = m.i <= a.g.nx ? 16 : 0;
  m.sc = a.scale;
  m.sg = a.sigma;
  m.ih2 = a.op.c.inv_h2;
  m.d = fmaf(-a.op.c.k, a.op.c.k, 4.f * m.ih2);
  m.e = -a.scale * a.op.c.k * a.op.c.k;
  m.q = -a.scale * m.ih2;
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    const int in = m.i + n;
    m.wx[n] = in < 0 || in > a.g.nx ? 0.f : (in == 0 || in == a.g.nx) ? 0.5f : 1.f;
  }
  m.sh = (uint32_t)__cvta_generic_to_shared(stg) + lane * 16;
  m.half = 0;
  const long long at = off + a.g.at(m.ok ? m.i : 0, j0 - SHW);
  m.src[0] = (Z ? a.b : a.x) + at;
  if constexpr (NF == 2) m.src[1] = a.b + at;
  m.left = m.n + 2 * SHW;   // rows j0 - 4 .. j1 + 3
}

template <int MODE, bool Z, bool VK>
__device__ __forceinline__ void gram_run(const SmA& a, int strip, int j0, int j1, long long off, const void* stg,
                                         float (&g)[SS_NV]) {
  SGram<MODE, Z, VK> p;
  sm_setup<Z>(p.m, a, strip, j0, j1, off, stg);
  p.acc.clear();
  p.m.prime([](uint32_t) {});
  smarch(p, j0 - SHW, j1 + SHW - 1);
  const int lane = threadIdx.x & 31;
  p.acc.out(g, lane >= SHW / 2 && lane < 32 - SHW / 2);
}

template <int MODE, bool Z, bool VK, bool OUT>
__device__ __forceinline__ void upd_run(const SmA& a, int strip, int j0, int j1, int rhs, long long off,
                                        const void* stg) {
  SUpd<MODE, Z, VK, OUT> p;
  sm_setup<Z>(p.m, a, strip, j0, j1, off, stg);
  const float* S = gstate<float>(a.st, rhs);
#pragma unroll
  for (int l = 0; l < 3; ++l) p.y[l] = make_float2(S[2 * l], S[2 * l + 1]);
  const int lane = threadIdx.x & 31;
  p.nv = lane >= SHW / 2 && lane < 32 - SHW / 2 ? min(max(a.g.nx + 1 - p.m.i, 0), 2) : 0;
  const long long at = off + a.g.at(p.m.i, j0 - SHW - 2 - SMarch<MODE, Z, VK>::D);
  p.xo = a.xo + at;
  p.x64 = a.outer + at;
  p.xs = p.x64;
  if constexpr (OUT) p.ig = f64_from_f32(rcp_pow2(a.rscale[2 * rhs]));
  p.rs = -SHW - 2 - SMarch<MODE, Z, VK>::D;
  p.m.prime([&](uint32_t slot) {
    if constexpr (OUT) p.stage64(slot);
  });
  smarch(p, j0 - SHW, j1 + SHW - 1);
}

// Runs F with the warp's mode (boundary mode GM) as an integral constant.
template <int GM, class F> __device__ __forceinline__ void sm_mode(int mode, F&& f) {
  if (mode == 1) f(std::integral_constant<int, GM>{});
  else if (mode == 0) f(std::integral_constant<int, 0>{});
}

template <bool Z, bool VK, bool A2> __device__ __forceinline__ void ss_gram_body(const SmA& a, int blk, int rhs) {
  if (a.active && !a.active[rhs]) return;
  __shared__ __align__(16) unsigned char stg[SWB][(Z ? 1 : 2) * RING];
  const long long off = (long long)rhs * a.g.vstride;
  const int warp = threadIdx.x >> 5;
  int strip, j0, j1;
  const int mode = sm_map(a.mg, blk * SWB + warp, strip, j0, j1);
  float g[SS_NV];
#pragma unroll
  for (int k = 0; k < SS_NV; ++k) g[k] = 0.f;
  sm_mode<A2 ? 2 : 1>(mode, [&](auto md) {
    constexpr int MD = decltype(md)::value;
    gram_run<MD, Z, (VK || MD != 0)>(a, strip, j0, j1, off, stg[warp], g);
  });
  __syncthreads();   // the staging rings are free: the sums reuse them
  ss_finish<SWB * 32>(g, reinterpret_cast<double*>(&stg[0][0]), a.partial, a.tickets, rhs, a.nblk, blk, threadIdx.x,
                      a.scale, a.sigma, a.st);
}
template <bool Z, bool VK, bool A2, bool OUT>
__device__ __forceinline__ void ss_update_body(const SmA& a, int blk, int rhs) {
  if (a.active && !a.active[rhs]) return;
  constexpr int W = OUT ? SWO : SWB;
  __shared__ __align__(16) unsigned char stg[W][((Z ? 1 : 2) + (OUT ? 2 : 0)) * RING];
  const long long off = (long long)rhs * a.g.vstride;
  const int warp = threadIdx.x >> 5;
  int strip, j0, j1;
  const int mode = sm_map(a.mg, blk * W + warp, strip, j0, j1);
  sm_mode<A2 ? 2 : 1>(mode, [&](auto md) {
    constexpr int MD = decltype(md)::value;
    upd_run<MD, Z, (VK || MD != 0), OUT>(a, strip, j0, j1, rhs, off, stg[warp]);
  });
}

template <bool Z, bool VK, bool A2>
__global__ void __launch_bounds__(SWB * 32, 4) ss_gram(const __grid_constant__ SmA a) {
  ss_gram_body<Z, VK, A2>(a, blockIdx.x, blockIdx.z);
}
template <bool Z, bool VK, bool A2, bool OUT>
__global__ void __launch_bounds__((OUT ? SWO : SWB) * 32, OUT ? 6 : 4) ss_update(const __grid_constant__ SmA a) {
  ss_update_body<Z, VK, A2, OUT>(a, blockIdx.x, blockIdx.z);
}
// Flattened over a ragged batch (constant k, first-order absorbing rows).
__global__ void __launch_bounds__(SWB * 32, 4) ss_gram_rag(const __grid_constant__ RagLaunch<SmA> L) {
  uint3 vb;
  dim3 vg;
  const SmA& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  ss_gram_body<false, false, false>(a, vb.x, 0);
}
__global__ void __launch_bounds__(SWB * 32, 4) ss_update_rag(const __grid_constant__ RagLaunch<SmA> L) {
  uint3 vb;
  dim3 vg;
  const SmA& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  ss_update_body<false, false, false, false>(a, vb.x, 0);
}

// Chunk height: the launch runs in ceil(blocks / resident) rounds of warps
// that march ch + 8 rows each; the height that minimises the product.
// Resident: 4 blocks of 4 warps per SM (the register bound above).
MGeo ss_geo(const Grid& g, int B) {
  MGeo m{};
  m.fill(g.nx, g.ny, SSW, 64, SHW, SBR);
  const long long resident = 4LL * device_sms();
  long long best = -1;
  int bch = 8;
  for (int ch = 4; ch <= 256; ch += 4) {
    m.chunks(ch);
    const long long blocks = (long long)cdiv(m.nrec(), SWB) * B;
    const long long cost = ((blocks + resident - 1) / resident) * (ch + 2 * SHW);
    if (best < 0 || cost <= best) {   // the tallest of equal cost
      best = cost;
      bch = ch;
    }
  }
  m.chunks(bch);
  return m;
}

}  // namespace

long long ss_march_blocks(const Grid& g, int B) { return cdiv(ss_geo(g, B).nrec(), SWB); }

float2* gmres_smooth_ss_march(const Grid& g, const OpView<float>& opv, float2* x, float2* xt, const float2* b, int nu,
                              int B, const int* active, const GmresBufs& gb, cudaStream_t s) {
  SmA a{g, ss_geo(g, B), Op0<float>{opv.c0, opv.kf, g.nx, g.ny}, gb.scale, gb.sigma, x, b, xt, gb.outer,
        gb.st, gb.partial, gb.tickets, active, 0, gb.rscale};
  a.nblk = cdiv(a.mg.nrec(), SWB);
  const dim3 grid(a.nblk, 1, B);
  auto steps = [&](auto vk, auto a2) {
    constexpr bool VK = decltype(vk)::value, A2 = decltype(a2)::value;
    for (int step = 0; step < nu; ++step) {
      const bool z = step == 0 && gb.x_zero, out = step == nu - 1 && gb.outer;
      if (z) ss_gram<true, VK, A2><<<grid, SWB * 32, 0, s>>>(a);
      else ss_gram<false, VK, A2><<<grid, SWB * 32, 0, s>>>(a);
      const dim3 go(cdiv(a.mg.nrec(), SWO), 1, B);
      if (z && out) ss_update<true, VK, A2, true><<<go, SWO * 32, 0, s>>>(a);
      else if (z) ss_update<true, VK, A2, false><<<grid, SWB * 32, 0, s>>>(a);
      else if (out) ss_update<false, VK, A2, true><<<go, SWO * 32, 0, s>>>(a);
      else ss_update<false, VK, A2, false><<<grid, SWB * 32, 0, s>>>(a);
      if (out) break;   // x' went to the FP64 iterate
      std::swap(x, xt);
      a.x = x;
      a.xo = xt;
    }
  };
  if (opv.c0.abc2) steps(std::true_type{}, std::true_type{});
  else if (opv.kf) steps(std::true_type{}, std::false_type{});
  else steps(std::false_type{}, std::false_type{});
  return x;
}

// The same steps on every problem of a ragged batch, in place: an odd number
// of steps leaves the result in xt, which the caller swaps in (v[q].x).
void gmres_smooth_ss_march_rag(std::vector<RagLevel<float>>& v, int nu, cudaStream_t s) {
  const int n = (int)v.size();
  std::vector<SmA> A(n);
  for (int q = 0; q < n; ++q) {
    RagLevel<float>& L = v[q];
    A[q] = SmA{L.g, ss_geo(L.g, 1), Op0<float>{L.op.c0, L.op.kf, L.g.nx, L.g.ny}, L.gb.scale, L.gb.sigma, L.x, L.b,
               L.xt, nullptr, L.gb.st, L.gb.partial, L.gb.tickets, L.active, 0, nullptr};
    A[q].nblk = cdiv(A[q].mg.nrec(), SWB);
  }
  auto launch = [&](auto kern) {
    rag_launch<SmA>(n, kern, dim3(SWB * 32), 0, s, [&](int q, SmA& a, int& gx, int&) {
      a = A[q];
      gx = a.nblk;
      return true;
    });
  };
  for (int step = 0; step < nu; ++step) {   // constant k (a ragged batch has no k fields)
    launch(ss_gram_rag);
    launch(ss_update_rag);
    for (int q = 0; q < n; ++q) {
      std::swap(v[q].x, v[q].xt);
      A[q].x = v[q].x;
      A[q].xo = v[q].xt;
    }
  }
}

}  // namespace hmg
