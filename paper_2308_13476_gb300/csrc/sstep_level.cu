// GMRES(3) smoothing of the complex64 cycles on the levels that store their
// Krylov vectors: Kronecker-form levels as column marches, stored stencils
// (and every level without marches) with node-parallel kernels.
//
// A step in s-step form (sstep.cuh) is three applications v1 = B r, v2 = B v1
// and v3 = B v2, the last one with the Gram sums of (r, v1, v2, v3) and the
// solve, and one update of x and, by linearity, of the residual:
//   x' = x + scale sum_k z_k v_k,   r' = r - sum_k z_k (v_{k+1} + sigma v_k),
// so that the next step (and the restriction after the pre-smoothing) needs
// no application for its residual: a V(2,2) cycle applies A ten times per
// level instead of sixteen, in four launches per step of which one carries a
// global sum.  The residual is formed afresh at the start of a smoothing call
// and after SS_REFRESH updates.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "kron.cuh"
#include "pack.cuh"
#include "ragged.cuh"
#include "ragged_api.h"
#include "sstep.cuh"

namespace hmg {
namespace {

// What one application forms: RES b - A v, NEXT B v, GRAM v3 = B v2 with the
// Gram sums and the solve.
enum { RES = 0, NEXT = 1, GRAM = 2 };

// Arguments of one launch (one problem of a ragged batch).
struct SlA {
  Grid g;
  const float2* v;     // applied vector (x, r, v1, v2)
  const float2* b;     // RES: right-hand side
  const float2* r;     // GRAM: r
  const float2* v1;    // GRAM: v1
  float2* out;         // result (GRAM: null if v3 is not needed)
  float scale, sigma;
  double* st;
  double* partial;
  unsigned* tickets;
  const int* active;
  int B;
};

// ------------------------------------------------------- node-parallel form

// A v at the thread's node pair (i0, j) for RB right-hand sides vs apart.
template <class Op, int RB> struct RbApply {
  __device__ __forceinline__ static void run(const Op& op, const float2* x, long long vs, int nrb, int p, int pitch,
                                             int i0, int j, Pack<float> (&y)[RB]) {
#pragma unroll
    for (int q = 0; q < RB; ++q)
      if (q < nrb) y[q] = apply_pack<float>(op, x + q * vs, p, pitch, i0, j);
  }
};
// Stored stencils: each coefficient is read once for the RB right-hand sides
// and both nodes, and a row of v once for the 2R + 1 coefficients (16-byte
// loads): the kernel is bound by L1 and L2 bandwidth, not by arithmetic.
template <int R, int RB> struct RbApply<OpS<float, R>, RB> {
  __device__ __forceinline__ static void run(const OpS<float, R>& op, const float2* x, long long vs, int nrb, int p,
                                             int pitch, int i0, int j, Pack<float> (&y)[RB]) {
    constexpr int K = 2 * R + 1;
    const bool two = i0 + 1 <= op.nx;
    const float2* st = op.st + (long long)j * (op.nx + 1) + i0;
#pragma unroll
    for (int q = 0; q < RB; ++q) y[q].v[0] = y[q].v[1] = make_float2(0.f, 0.f);
#pragma unroll
    for (int dy = -R; dy <= R; ++dy) {
      float2 w[RB][2 * R + 2];   // v at columns i0 - R .. i0 + R + 1 of row j + dy
      const int pr = p + dy * pitch;
#pragma unroll
      for (int q = 0; q < RB; ++q) {
        const float2* row = x + q * vs + pr;
        if (q < nrb) {
          if constexpr (R & 1) {
            w[q][0] = row[-R];
            w[q][2 * R + 1] = row[R + 1];
          }
#pragma unroll
          for (int c = R & 1; c + 1 < 2 * R + 2 - (R & 1); c += 2) {
            const float4 t = *reinterpret_cast<const float4*>(row + c - R);
            w[q][c] = make_float2(t.x, t.y);
            w[q][c + 1] = make_float2(t.z, t.w);
          }
        } else {
#pragma unroll
          for (int c = 0; c < 2 * R + 2; ++c) w[q][c] = make_float2(0.f, 0.f);
        }
      }
#pragma unroll
      for (int dx = 0; dx < K; ++dx) {
        const float2* c = st + ((dy + R) * K + dx) * op.plane;
        const float2 c0 = c[0], c1 = two ? c[1] : make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < RB; ++q) {
          y[q].v[0] = fma_c<float>(c0, w[q][dx], y[q].v[0]);
          y[q].v[1] = fma_c<float>(c1, w[q][dx + 1], y[q].v[1]);
        }
      }
    }
  }
};

template <class Op, int MODE, int RB>
__global__ void __launch_bounds__(BX * BY) sl_apply(const __grid_constant__ SlA a, const __grid_constant__ Op op) {
  const Grid& g = a.g;
  const int r0 = blockIdx.z * RB, nrb = min(RB, a.B - r0);
  bool any = a.active == nullptr;
  for (int q = 0; q < nrb && !any; ++q) any = a.active[r0 + q] != 0;
  if (!any) return;
  const int i0 = (blockIdx.x * BX + threadIdx.x) * 2, j = blockIdx.y * BY + threadIdx.y;
  const int nv = j <= g.ny ? min(2, g.nx + 1 - i0) : 0;
  const long long vs = g.vstride, off = r0 * vs;
  const int p = g.at(i0, j), tid = threadIdx.x + threadIdx.y * BX;
  constexpr int NT = BX * BY;
  Pack<float> y[RB];
  if (nv > 0) RbApply<Op, RB>::run(op, a.v + off, vs, nrb, p, g.pitch, i0, j, y);
  __shared__ double sh[MODE != GRAM ? 1 : RB == 1 ? NT : RB * SS_NV * (NT / 32)];
  unsigned act = 0;   // block-uniform
#pragma unroll
  for (int q = 0; q < RB; ++q) {
    if (q >= nrb || (a.active && !a.active[r0 + q])) continue;
    act |= 1u << q;
    const long long o = off + q * vs;
    float gm[SS_NV];
    if constexpr (MODE == GRAM) {
#pragma unroll
      for (int k = 0; k < SS_NV; ++k) gm[k] = 0.f;
    }
    if (nv > 0) {
      Pack<float> w;
      if constexpr (MODE == RES) {
        w = load_pack(a.b + o, p);
#pragma unroll
        for (int n = 0; n < 2; ++n) w.v[n] = sub2(w.v[n], y[q].v[n]);
      } else {
        const Pack<float> v = load_pack(a.v + o, p);
#pragma unroll
        for (int n = 0; n < 2; ++n) w.v[n] = fma2(bc2(a.scale), y[q].v[n], mul2(bc2(-a.sigma), v.v[n]));
        if constexpr (MODE == GRAM) {
          const Pack<float> r = load_pack(a.r + o, p), v1 = load_pack(a.v1 + o, p);
#pragma unroll
          for (int n = 0; n < 2; ++n)
            if (n < nv) ss_gram_add(gm, r.v[n], v1.v[n], v.v[n], w.v[n]);
        }
      }
      if (MODE != GRAM || a.out) store_pack(a.out + o, p, w, nv);
    }
    if constexpr (MODE == GRAM) ss_warp_sums<NT>(gm, sh + q * SS_NV * (NT / 32), tid);
  }
  if constexpr (MODE == GRAM)
    ss_finish_rb<NT, RB>(sh, a.partial, a.tickets, r0, act, gridDim.x * gridDim.y, blockIdx.y * gridDim.x + blockIdx.x,
                         tid, a.scale, a.sigma, a.st);
}

// One node per thread and one right-hand side per block, stored stencils: the
// launch of a level that the blocks above would leave under-filled.  A
// thread's (2R+1)^2 coefficients come from L2 once and nothing is reused, so
// what bounds it is how many of those loads are in flight: they are issued in
// groups of stencil rows (all five rows of radius 2, three of radius 3 at a
// time), coefficients and v together, before the first multiply-add, and a
// thread has half the loads and the launch twice the threads of the pair form.
// Layered model 1281 x 449, one right-hand side, with the grouped loads of the
// cluster launch (cluster.cuh): 237 -> 162 ms.
template <int R>
__device__ __forceinline__ float2 stencil_node(const float2* st, long long plane, const float2* v, int pitch) {
  constexpr int K = 2 * R + 1, G = R == 2 ? 5 : 3;
  float2 acc = make_float2(0.f, 0.f);
#pragma unroll
  for (int d0 = 0; d0 < K; d0 += G) {
    float2 c[G * K], x[G * K];
#pragma unroll
    for (int e = 0; e < G * K; ++e) {
      if (d0 * K + e >= K * K) break;
      c[e] = __ldg(st + (long long)(d0 * K + e) * plane);
      x[e] = v[(d0 + e / K - R) * pitch + e % K - R];
    }
#pragma unroll
    for (int e = 0; e < G * K; ++e) {
      if (d0 * K + e >= K * K) break;
      acc = fma_c<float>(c[e], x[e], acc);
    }
  }
  return acc;
}

template <int R, int MODE, int NY>
__global__ void __launch_bounds__(BX * NY, 512 / (BX * NY)) sl_one(const __grid_constant__ SlA a,
                                                                   const __grid_constant__ OpS<float, R> op) {
  const Grid& g = a.g;
  const int rhs = blockIdx.z;
  if (a.active && !a.active[rhs]) return;
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * NY + threadIdx.y;
  const long long off = (long long)rhs * g.vstride;
  float gm[SS_NV];
  if constexpr (MODE == GRAM) {
#pragma unroll
    for (int k = 0; k < SS_NV; ++k) gm[k] = 0.f;
  }
  if (i <= g.nx && j <= g.ny) {
    const long long p = off + g.at(i, j);
    const float2 y = stencil_node<R>(op.st + (long long)j * (op.nx + 1) + i, op.plane, a.v + p, g.pitch);
    float2 w;
    if constexpr (MODE == RES) {
      w = sub2(a.b[p], y);
    } else {
      const float2 v = a.v[p];
      w = fma2(bc2(a.scale), y, mul2(bc2(-a.sigma), v));
      if constexpr (MODE == GRAM) ss_gram_add(gm, a.r[p], a.v1[p], v, w);
    }
    if (MODE != GRAM || a.out) a.out[p] = w;
  }
  if constexpr (MODE == GRAM) {
    __shared__ double sh[BX * NY];
    ss_finish<BX * NY>(gm, sh, a.partial, a.tickets, rhs, gridDim.x * gridDim.y, blockIdx.y * gridDim.x + blockIdx.x,
                       threadIdx.x + threadIdx.y * BX, a.scale, a.sigma, a.st);
  }
}

// ------------------------------------------------------------ column marches

template <int R> struct KlA {
  SlA a;
  KGeo kg;
  OpK<float, R> op;
};

template <int R, int MODE> __device__ __forceinline__ void kl_apply_body(const KlA<R>& L, int blk, int nblk, int rhs) {
  using T = float;
  const SlA& a = L.a;
  const Grid& g = a.g;
  const KGeo& kg = L.kg;
  constexpr int NO = MODE == RES ? 1 : MODE == GRAM ? 2 : 0;   // vectors read at the lane's own nodes
  __shared__ __align__(16) float2 ksm[KW][KSL][KRing<T, R>::WD];
  __shared__ __align__(16) float2 osm[NO > 0 ? KW : 1][NO > 0 ? NO : 1][KSL][32];
  __shared__ double sh[MODE == GRAM ? KW * 32 : 1];
  if (a.active && !a.active[rhs]) return;
  const long long off = (long long)rhs * g.vstride;
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = blk * KW + wib;
  const bool has = gw < kg.ncw * kg.nchunks;
  float gm[SS_NV];
#pragma unroll
  for (int k = 0; k < SS_NV; ++k) gm[k] = 0.f;
  if (has) {
    const int cw0 = (gw % kg.ncw) * 32, i = cw0 + lane;
    const int j0 = (gw / kg.ncw) * kg.ch, j1 = min(j0 + kg.ch, g.ny + 1);
    const bool col = i <= g.nx;
    KRing<T, R> ring;
    ring.init(L.op, i, col);
    ring.vs = a.v + off;
    ring.g = g;
    ring.cw0 = cw0;
    ring.lane = lane;
    ring.sm = &ksm[wib][0][0];
    ring.r0 = j0 - R;
    if constexpr (NO > 0) {
      ring.os = (MODE == RES ? a.b : a.r) + off;
      ring.osm = &osm[wib][0][0][0];
    }
    if constexpr (NO > 1) {
      ring.os2 = a.v1 + off;
      ring.osm2 = &osm[wib][1][0][0];
    }
    const int last = j1 + R - 1;
    ring.prime(last);
    float2* out = a.out + off;
    kmarch<KU<T, R>>(j0 - R, last, [&](auto ph, int r) {
      constexpr int P = decltype(ph)::value;
      ring.template advance<P>(r, last);
      const int m = r - R;
      if (m >= j0 && col) {
        const float2 y = ring.template combine<P>(L.op, m);
        if constexpr (MODE == RES) {
          out[g.at(i, m)] = sub2(ring.own_at(m), y);
        } else {   // sigma = 0 on these levels
          const float2 w = mul2(bc2(a.scale), y);
          if constexpr (MODE == GRAM) ss_gram_add(gm, ring.own_at(m), ring.own2_at(m), ring.staged_at(m), w);
          if (MODE != GRAM || a.out) out[g.at(i, m)] = w;
        }
      }
    });
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  }
  if constexpr (MODE == GRAM)
    ss_finish<KW * 32>(gm, sh, a.partial, a.tickets, rhs, nblk, blk, threadIdx.x, a.scale, a.sigma,
                       a.st);
}

template <int R, int MODE> __global__ void __launch_bounds__(KW * 32) kl_apply(const __grid_constant__ KlA<R> L) {
  kl_apply_body<R, MODE>(L, blockIdx.x, gridDim.x, blockIdx.z);
}
template <int R, int MODE>
__global__ void __launch_bounds__(KW * 32) kl_apply_rag(const __grid_constant__ RagLaunch<KlA<R>> L) {
  uint3 vb;
  dim3 vg;
  const KlA<R>& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  kl_apply_body<R, MODE>(a, vb.x, vg.x, 0);
}

// Blocks of a march resident on the device at once: each mode has its own
// chunk height, since the Gram march takes twice the registers of the others.
template <int R, int MODE> long long kl_capacity() {
  static const long long cap = [] {
    int per = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kl_apply<R, MODE>, KW * 32, 0);
    cudaGetLastError();
    return (long long)std::max(per, 1) * device_sms();
  }();
  return cap;
}

// -------------------------------------------------------------------- update

struct SuA {
  Grid g;
  float2* x;
  const float2* r;     // r (b on a zero x)
  const float2* v1;
  const float2* v2;
  const float2* v3;    // NR
  float2* rn;          // NR: the new residual
  double2* outer;      // OUT: the FP64 iterate to which x' is added (x' is not stored)
  float iscale, sigma;
  const double* st;
  const int* active;
  const float* rscale; // OUT: x' is divided by rscale[2 rhs]
};

// Z: x is zero (not read).  NR: the residual too.
template <bool Z, bool NR, bool OUT>
__device__ __forceinline__ void sl_update_body(const SuA& a, uint3 blk, int rhs) {
  if (a.active && !a.active[rhs]) return;
  const Grid& g = a.g;
  const int i0 = (blk.x * BX + threadIdx.x) * 2, nv = min(2, g.nx + 1 - i0);
  if (nv <= 0) return;
  const long long off = (long long)rhs * g.vstride;
  const float* S = gstate<float>(a.st, rhs);
  float2 y[3], c[4];
#pragma unroll
  for (int k = 0; k < 3; ++k) y[k] = make_float2(S[2 * k], S[2 * k + 1]);
  if constexpr (NR) ss_residual_coef(y, a.iscale, a.sigma, c);
  [[maybe_unused]] double ig = 1.0;
  if constexpr (OUT) ig = f64_from_f32(rcp_pow2(a.rscale[2 * rhs]));
  for (int q = 0, j = blk.y * BY * g.ry + threadIdx.y; q < g.ry; ++q, j += BY) {
    if (j > g.ny) break;
    const long long p = off + g.at(i0, j);
    const Pack<float> r = load_pack(a.r + p, 0), v1 = load_pack(a.v1 + p, 0), v2 = load_pack(a.v2 + p, 0);
    Pack<float> x, v3;
    if constexpr (!Z) x = load_pack(a.x + p, 0);
    if constexpr (NR) v3 = load_pack(a.v3 + p, 0);
    Pack<float> rn;
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      float2 e = Z ? make_float2(0.f, 0.f) : x.v[n];
      e = fma_c<float>(y[0], r.v[n], e);
      e = fma_c<float>(y[1], v1.v[n], e);
      x.v[n] = fma_c<float>(y[2], v2.v[n], e);
      if constexpr (NR) {
        float2 t = mul<float>(c[0], r.v[n]);
        t = fma_c<float>(c[1], v1.v[n], t);
        t = fma_c<float>(c[2], v2.v[n], t);
        rn.v[n] = fma_c<float>(c[3], v3.v[n], t);
      }
    }
    if constexpr (OUT) {
#pragma unroll
      for (int n = 0; n < 2; ++n)
        if (n < nv) {
          double2 o = a.outer[p + n];
          o.x = fma(ig, f64_from_f32(x.v[n].x), o.x);
          o.y = fma(ig, f64_from_f32(x.v[n].y), o.y);
          a.outer[p + n] = o;
        }
    } else {
      store_pack(a.x + p, 0, x, nv);
    }
    if constexpr (NR) store_pack(a.rn + p, 0, rn, nv);
  }
}

template <bool Z, bool NR, bool OUT> __global__ void __launch_bounds__(BX * BY) sl_update(const __grid_constant__ SuA a) {
  sl_update_body<Z, NR, OUT>(a, blockIdx, blockIdx.z);
}
template <bool NR> __global__ void __launch_bounds__(BX * BY) sl_update_rag(const __grid_constant__ RagLaunch<SuA> L) {
  uint3 vb;
  dim3 vg;
  const SuA& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  sl_update_body<false, NR, false>(a, vb, 0);
}

dim3 pack_blocks(const Grid& g, int B) { return dim3(cdiv(g.nx + 1, BX * 2), cdiv(g.ny + 1, BY * g.ry), B); }

void launch_update(const SuA& a, int B, bool z, bool nr, bool out, cudaStream_t s) {
  const dim3 grd = pack_blocks(a.g, B), blk(BX, BY);
  if (out) {
    if (z) sl_update<true, false, true><<<grd, blk, 0, s>>>(a);
    else sl_update<false, false, true><<<grd, blk, 0, s>>>(a);
  } else if (z) {
    if (nr) sl_update<true, true, false><<<grd, blk, 0, s>>>(a);
    else sl_update<true, false, false><<<grd, blk, 0, s>>>(a);
  } else {
    if (nr) sl_update<false, true, false><<<grd, blk, 0, s>>>(a);
    else sl_update<false, false, false><<<grd, blk, 0, s>>>(a);
  }
}

}  // namespace

long long sl_blocks(const Grid& g) { return (long long)cdiv(g.nx + 1, BX) * cdiv(g.ny + 1, BY); }

void gmres_smooth_ss(const Grid& g, const OpView<float>& opv, bool march, float2* x, const float2* b, int nu,
                     bool want_r, int B, const int* active, const GmresBufs& gb, cudaStream_t s) {
  float2* const u0 = (float2*)gb.u[0];
  float2* const u1 = (float2*)gb.u[1];
  float2* const u2 = (float2*)gb.u[2];
  float2* const w = (float2*)gb.w;
  SlA a{g, nullptr, b, nullptr, u1, nullptr, gb.scale, gb.sigma, gb.st, gb.partial, gb.tickets, active, B};
  SuA u{g, x, nullptr, u1, u2, w, u0, gb.outer, 1.f / gb.scale, gb.sigma, gb.st, active, gb.rscale};
  // apply(mode, v, out): one application of this level's kernels
  auto steps = [&](auto apply) {
    const float2* r = u0;
    for (int step = 0; step < nu; ++step) {
      const bool z = step == 0 && gb.x_zero, last = step == nu - 1;
      const bool nr = last ? want_r : ss_carried(step + 1), out = last && gb.outer;
      if (z) {
        r = b;
      } else if (!ss_carried(step)) {
        apply(std::integral_constant<int, RES>{}, x, u0);
        r = u0;
      }
      a.r = u.r = r;
      apply(std::integral_constant<int, NEXT>{}, r, u1);
      apply(std::integral_constant<int, NEXT>{}, u1, u2);
      apply(std::integral_constant<int, GRAM>{}, u2, nr ? w : nullptr);
      launch_update(u, B, z, nr, out, s);
      r = u0;
    }
  };
  if (march && opv.kind >= 4) {
    auto run = [&](auto rad) {
      constexpr int R = decltype(rad)::value;
      const OpK<float, R> op = kron_op<float, R>(opv, g.nx, g.ny);
      steps([&](auto mode, const float2* v, float2* o) {
        constexpr int MODE = decltype(mode)::value;
        const KGeo kg = kron_geo(g, B, R, kl_capacity<R, MODE>(), gb.kron_ch);
        const dim3 grd(cdiv((long long)kg.ncw * kg.nchunks, KW), 1, B);
        a.v = v;
        a.out = o;
        kl_apply<R, MODE><<<grd, KW * 32, 0, s>>>(KlA<R>{a, kg, op});
      });
    };
    if (opv.kind == 4) run(std::integral_constant<int, 2>{});
    else run(std::integral_constant<int, 3>{});
    return;
  }
  // Node-parallel.  Stored stencils: node pairs of up to four right-hand sides
  // per block (a coefficient is then read once for them) as long as the launch
  // keeps two blocks per SM, else one node of one right-hand side per thread,
  // in blocks of 512 threads once blocks of 256 would be more than two per SM
  // (half as many records for the last block to add).  The other operators
  // have nothing to share.
  const long long nb = (long long)cdiv(g.nx + 1, BX * 2) * cdiv(g.ny + 1, BY), fill = 2LL * device_sms();
  with_op<float>(opv, g.nx, g.ny, [&](auto op) {
    using Op = decltype(op);
    auto go = [&](auto rb) {
      constexpr int N = decltype(rb)::value;
      const dim3 grd(cdiv(g.nx + 1, BX * 2), cdiv(g.ny + 1, BY), cdiv(B, N)), blk(BX, BY);
      steps([&](auto mode, const float2* v, float2* o) {
        constexpr int MODE = decltype(mode)::value;
        a.v = v;
        a.out = o;
        sl_apply<Op, MODE, N><<<grd, blk, 0, s>>>(a, op);
      });
    };
    if constexpr (std::is_same_v<Op, OpS<float, 2>> || std::is_same_v<Op, OpS<float, 3>>) {
      constexpr int R = std::is_same_v<Op, OpS<float, 2>> ? 2 : 3;
      auto one = [&](auto ny) {
        constexpr int NY = decltype(ny)::value;
        const dim3 grd(cdiv(g.nx + 1, BX), cdiv(g.ny + 1, NY), B), blk(BX, NY);
        steps([&](auto mode, const float2* v, float2* o) {
          constexpr int MODE = decltype(mode)::value;
          a.v = v;
          a.out = o;
          sl_one<R, MODE, NY><<<grd, blk, 0, s>>>(a, op);
        });
      };
      if (B >= 4 && nb * cdiv(B, 4) >= fill) go(std::integral_constant<int, 4>{});
      else if (B >= 2 && nb * cdiv(B, 2) >= fill) go(std::integral_constant<int, 2>{});
      else if (sl_blocks(g) * B > fill) one(std::integral_constant<int, 16>{});
      else one(std::integral_constant<int, 8>{});
    } else {
      go(std::integral_constant<int, 1>{});
    }
  });
}

// The same steps on a Kronecker-form level of every problem of a ragged batch.
void gmres_smooth_ss_rag(const std::vector<RagLevel<float>>& v, int nu, bool want_r, cudaStream_t s) {
  if (v.empty()) return;
  const int n = (int)v.size();
  auto run = [&](auto rad) {
    constexpr int R = decltype(rad)::value;
    std::vector<KlA<R>> A(n);
    for (int q = 0; q < n; ++q) {
      const RagLevel<float>& L = v[q];
      A[q].a = SlA{L.g, nullptr, L.b, (float2*)L.gb.u[0], (float2*)L.gb.u[1], nullptr, L.gb.scale, L.gb.sigma,
                   L.gb.st, L.gb.partial, L.gb.tickets, L.active, 1};
      A[q].op = kron_op<float, R>(L.op, L.g.nx, L.g.ny);
    }
    auto apply = [&](auto mode, auto vec, auto out) {
      constexpr int MODE = decltype(mode)::value;
      rag_launch<KlA<R>>(n, kl_apply_rag<R, MODE>, dim3(KW * 32), 0, s, [&](int q, KlA<R>& a, int& gx, int&) {
        a = A[q];
        a.kg = kron_geo(a.a.g, 1, R, kl_capacity<R, MODE>(), v[q].gb.kron_ch);
        a.a.v = vec(v[q]);
        a.a.out = out(v[q]);
        gx = cdiv((long long)a.kg.ncw * a.kg.nchunks, KW);
        return true;
      });
    };
    auto buf = [](int k) { return [k](const RagLevel<float>& L) { return (float2*)(k < 3 ? L.gb.u[k] : L.gb.w); }; };
    for (int step = 0; step < nu; ++step) {
      const bool nr = step == nu - 1 ? want_r : ss_carried(step + 1);
      if (!ss_carried(step)) apply(std::integral_constant<int, RES>{}, [](const RagLevel<float>& L) { return L.x; }, buf(0));
      apply(std::integral_constant<int, NEXT>{}, buf(0), buf(1));
      apply(std::integral_constant<int, NEXT>{}, buf(1), buf(2));
      apply(std::integral_constant<int, GRAM>{}, buf(2), [&](const RagLevel<float>& L) { return nr ? (float2*)L.gb.w : nullptr; });
      auto update = [&](auto kern) {
        rag_launch<SuA>(n, kern, dim3(BX, BY), 0, s, [&](int q, SuA& a, int& gx, int& gy) {
          const RagLevel<float>& L = v[q];
          a = SuA{L.g, L.x, (float2*)L.gb.u[0], (float2*)L.gb.u[1], (float2*)L.gb.u[2], (float2*)L.gb.w,
                  (float2*)L.gb.u[0], nullptr, 1.f / L.gb.scale, L.gb.sigma, L.gb.st, L.active, nullptr};
          const dim3 d = pack_blocks(L.g, 1);
          gx = d.x;
          gy = d.y;
          return true;
        });
      };
      if (nr) update(sl_update_rag<true>);
      else update(sl_update_rag<false>);
    }
  };
  if (v[0].op.kind == 4) run(std::integral_constant<int, 2>{});
  else run(std::integral_constant<int, 3>{});
}

}  // namespace hmg
