// FP64 residual of the refinement loop: r = b - A x in FP64, written in float
// for the next complex64 cycle, with the stopping test fused.
//
// What bounds it is the FP64 pipe (two multiply-adds per clock and SM, 1/64 of
// the FP32 rate): 40 bytes per node take 396 us at 64 x 1025^2, ten FP64
// instructions per node 1070 us.  So the interior is a row march that spends
// eight: with the diagonal pair sums
//   u(i, j) = x(i + 1, j) + x(i, j + 1)
// the four neighbours of a node are u(i, j) + u(i - 1, j - 1), two adds per
// component instead of three, and b - d x + (1/h^2) (..) two multiply-adds.
// Everything else stays off that pipe: the casts to float are integer
// arithmetic (f32_from_f64_rn, the hardware's rounding) and the norm is
// summed from the float residual, compensated within a lane, in FP32 within
// a warp and in FP64 across warps and blocks, which resolves the stopping
// test's relative residual to about 1e-7 of itself.
//
// A warp walks down a strip of 64 columns, two nodes per lane, and writes the
// inner 62 of them (a node needs its left neighbour's u and its right
// neighbour's x: shuffles); the rows of x and b two steps ahead are in flight
// in registers, so that a few warps per SM keep the pipe busy.  Against the
// node-parallel form with ten FP64 instructions per node: 64 x 1025^2 1740 ->
// 1212 us (87 % of the pipe's measured rate), 16 x 513^2 with a k field 143 ->
// 104 us, one 1025^2 46 -> 32 us; 64 right-hand sides on 1025^2 623 -> 576 ms.  The nodes
// of the boundary ring take Op0::apply5 in warps of their own: their rows
// cost three times as much and would hold up every edge strip.
#include "internal.h"
#include "ragged.cuh"
#include "ragged_api.h"

namespace hmg {
namespace {

constexpr int RMW = 4;          // warps per block
constexpr int RMB = 5;          // blocks per SM (register bound of the launch)
constexpr int RMS = 62;         // columns written per strip
constexpr int RMN = 4;          // boundary nodes per lane

// Interior strips and chunks of rows, and boundary warps, of one right-hand side.
struct RmGeo {
  int ns, ch, nch, nring, nw;   // strips, rows per chunk, chunks, boundary nodes, warps
  __host__ __device__ int blocks() const { return (nw + RMW - 1) / RMW; }
};

// One warp per scheduler nearly fills the FP64 pipe, so the chunk height is the
// one of the least work per SM: ceil(blocks / SMs) blocks of ch rows and about
// 1.5 more for their start, plus one block's time that nothing overlaps.
RmGeo rm_geo(const Grid& g, int B) {
  RmGeo m{};
  m.ns = cdiv(g.nx - 1, RMS);
  m.nring = 2 * (g.nx + 1) + 2 * (g.ny - 1);
  long long best = -1;
  for (int ch = 4; ch <= 128; ch += 2) {
    RmGeo t = m;
    t.ch = ch;
    t.nch = cdiv(g.ny - 1, ch);
    t.nw = t.ns * t.nch + cdiv(m.nring, 32 * RMN);
    const long long cost = cdiv((long long)t.blocks() * B, (long long)device_sms()) * (2LL * ch + 3) + (2 * ch + 3);
    if (best < 0 || cost <= best) {
      best = cost;
      m = t;
    }
  }
  return m;
}

struct RmA {
  Grid g;
  RmGeo m;
  Op0<double> op;
  const double2* x;
  const double2* b;
  float2* r32;
  Ctl c;
  int count;
};

__device__ __forceinline__ double2 dadd2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 shfl_down2(double2 v) {
  return make_double2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ double2 shfl_up2(double2 v) {
  return make_double2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ float2 cast2(double2 v) { return make_float2(f32_from_f64_rn(v.x), f32_from_f64_rn(v.y)); }

// Compensated sum of the squares.
struct CSum {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float t) {
    const float s = hi + t, z = s - hi;
    lo += (hi - (s - z)) + (t - z);
    hi = s;
  }
  // past the largest float lo is inf - inf: the sum is then hi, inf
  __device__ __forceinline__ float total() const { return lo == lo ? hi + lo : hi; }
};

template <bool VK> struct RmMarch {
  const double2 *x, *b;   // this lane's first node of row j + 3 and j + 2 (the next to load)
  const double* k;        // VK: this lane's first node of row j + 2
  float2* r;              // this lane's first node of row j
  int pitch, n1;
  bool ok0, ok1, out0, out1;
  float gs;                   // factor of the stored residual (Ctl::rscale)
  double ih2, dc;
  double2 X[2][2], Q[2][2];   // rows in flight: x of rows j + 1, j + 2 and b of rows j, j + 1
  double D[2][2];             // VK: k of rows j, j + 1
  double2 xc[2], u[2];        // x of row j, u of row j - 1
  CSum sum;

  __device__ __forceinline__ void load(double2 (&v)[2], const double2* p) const {
    v[0] = ok0 ? p[0] : make_double2(0.0, 0.0);
    v[1] = ok1 ? p[1] : make_double2(0.0, 0.0);
  }
  __device__ __forceinline__ void loadk(double (&v)[2]) const {
    v[0] = ok0 ? k[0] : 0.0;
    v[1] = ok1 ? k[1] : 0.0;
  }
  // row j of the march; more: rows whose loads are still to be issued
  template <int S> __device__ __forceinline__ void step(bool morex, bool moreb) {
    const double2 xn[2] = {X[S][0], X[S][1]}, q[2] = {Q[S][0], Q[S][1]};
    double d[2] = {dc, dc};
    if constexpr (VK) {
#pragma unroll
      for (int n = 0; n < 2; ++n) d[n] = fma(-D[S][n], D[S][n], dc);
    }
    if (morex) load(X[S], x);
    if (moreb) {
      load(Q[S], b);
      if constexpr (VK) loadk(D[S]);
    }
    x += pitch;
    b += pitch;
    if constexpr (VK) k += n1;
    const double2 east = shfl_down2(xc[0]), uw = shfl_up2(u[1]);
    const double2 un[2] = {dadd2(xc[1], xn[0]), dadd2(east, xn[1])};
    const double2 s[2] = {dadd2(un[0], uw), dadd2(un[1], u[0])};
    float2 f[2];
#pragma unroll
    for (int n = 0; n < 2; ++n)
      f[n] = cast2(make_double2(fma(ih2, s[n].x, fma(-d[n], xc[n].x, q[n].x)),
                                fma(ih2, s[n].y, fma(-d[n], xc[n].y, q[n].y))));
    const float2 o[2] = {mul2(bc2(gs), f[0]), mul2(bc2(gs), f[1])};
    if (out0 && out1) *reinterpret_cast<float4*>(r) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
    else if (out0) r[0] = o[0];
    else if (out1) r[1] = o[1];
    r += pitch;
    const float t0 = fmaf(f[0].x, f[0].x, f[0].y * f[0].y), t1 = fmaf(f[1].x, f[1].x, f[1].y * f[1].y);
    sum.add((out0 ? t0 : 0.f) + (out1 ? t1 : 0.f));
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      xc[n] = xn[n];
      u[n] = un[n];
    }
  }
};

template <bool A2, bool VK> __device__ __forceinline__ void rm_body(const RmA& a, int blk, int rhs) {
  if (!a.c.active[rhs]) return;   // block-uniform
  __shared__ double sh[32];
  const Grid& g = a.g;
  const int lane = threadIdx.x & 31, w = blk * RMW + (threadIdx.x >> 5);
  const long long off = (long long)rhs * g.vstride;
  const double2* xs = a.x + off;
  const double2* bs = a.b + off;
  float2* rs = a.r32 + off;
  const float gs = a.c.rscale[2 * rhs + 1];
  CSum sum;
  if (w < a.m.ns * a.m.nch) {
    const int strip = w % a.m.ns, i = strip * RMS + 2 * lane;
    const int j0 = 1 + (w / a.m.ns) * a.m.ch, j1 = min(j0 + a.m.ch, g.ny);
    RmMarch<VK> p;
    p.ok0 = i <= g.nx;
    p.ok1 = i + 1 <= g.nx;
    p.out0 = lane > 0 && i < g.nx;
    p.out1 = lane < 31 && i + 1 < g.nx;
    p.gs = gs;
    p.pitch = g.pitch;
    p.n1 = g.nx + 1;
    p.ih2 = a.op.c.inv_h2;
    p.dc = VK ? 4.0 * p.ih2 : fma(-a.op.c.k, a.op.c.k, 4.0 * p.ih2);
    const int at = g.at(p.ok0 ? i : 0, j0);
    const double2* x0 = xs + at;
    double2 xm[2];
    p.load(xm, x0 - p.pitch);
    p.load(p.xc, x0);
    p.load(p.X[0], x0 + p.pitch);
    p.b = bs + at;
    p.load(p.Q[0], p.b);
    if constexpr (VK) {
      p.k = a.op.kf + (long long)j0 * p.n1 + (p.ok0 ? i : 0);
      p.loadk(p.D[0]);
      p.k += p.n1;
    }
    if (j0 + 1 < j1) {
      p.load(p.X[1], x0 + 2 * p.pitch);
      p.load(p.Q[1], p.b + p.pitch);
      if constexpr (VK) {
        p.loadk(p.D[1]);
        p.k += p.n1;
      }
    }
    p.x = x0 + 3 * p.pitch;
    p.b += 2 * p.pitch;
    p.r = rs + at;
    const double2 east = shfl_down2(xm[0]);
    p.u[0] = dadd2(xm[1], p.xc[0]);
    p.u[1] = dadd2(east, p.xc[1]);
#pragma unroll 1
    for (int j = j0; j < j1; j += 2) {   // x is read up to row j1 <= ny, b up to row j1 - 1
      p.template step<0>(j + 2 < j1, j + 2 < j1);
      if (j + 1 < j1) p.template step<1>(j + 3 < j1, j + 3 < j1);
    }
    sum = p.sum;
  } else if (w < a.m.nw) {
    const Op0<double, A2> op{a.op.c, a.op.kf, g.nx, g.ny};
#pragma unroll 1
    for (int n = 0; n < RMN; ++n) {
      int q = ((w - a.m.ns * a.m.nch) * RMN + n) * 32 + lane, i, j;
      if (q >= a.m.nring) break;
      if (q < 2 * (g.nx + 1)) {   // first and last row, then the ends of the rows between
        j = q <= g.nx ? 0 : g.ny;
        i = q <= g.nx ? q : q - (g.nx + 1);
      } else {
        q -= 2 * (g.nx + 1);
        i = q < g.ny - 1 ? 0 : g.nx;
        j = 1 + (q < g.ny - 1 ? q : q - (g.ny - 1));
      }
      const int at = g.at(i, j);
      const float2 f = cast2(sub<double>(bs[at], op.apply(xs, at, g.pitch, i, j)));
      rs[at] = mul2(bc2(gs), f);
      sum.add(fmaf(f.x, f.x, f.y * f.y));
    }
  }
  const float a0[1] = {sum.total()};
  double v[1];
  __syncwarp();
  if (reduce_last<1, float>(a0, v, sh, a.c.partial, a.c.tickets, rhs, a.m.blocks(), blk) && threadIdx.x == 0)
    stop_update(a.c, rhs, v[0], a.count, gs);
}

template <bool A2, bool VK>   // the k field's rows in flight take the registers of one block
__global__ void __launch_bounds__(RMW * 32, VK ? RMB - 1 : RMB) k_resid_cast_stop(const __grid_constant__ RmA a) {
  rm_body<A2, VK>(a, blockIdx.x, blockIdx.z);
}
// Flattened over a ragged batch (constant k, first-order absorbing rows).
__global__ void __launch_bounds__(RMW * 32, RMB - 1) k_resid_cast_stop_rag(const __grid_constant__ RagLaunch<RmA> L) {
  uint3 vb;
  dim3 vg;
  const RmA& a = L.a[rag_problem(L, blockIdx.x, vb, vg)];
  rm_body<false, false>(a, vb.x, 0);
}

}  // namespace

long long resid_blocks(const Grid& g, int B) { return rm_geo(g, B).blocks(); }

void launch_resid_cast_stop(const Grid& g, const OpView<double>& v, const double2* x, const double2* b, float2* r32,
                            int B, const Ctl& c, int count, cudaStream_t s) {
  const RmA a{g, rm_geo(g, B), Op0<double>{v.c0, v.kf, g.nx, g.ny}, x, b, r32, c, count};
  const dim3 grd(a.m.blocks(), 1, B);
  auto go = [&](auto kern) { kern<<<grd, RMW * 32, 0, s>>>(a); };
  if (v.c0.abc2) go(v.kf ? k_resid_cast_stop<true, true> : k_resid_cast_stop<true, false>);
  else go(v.kf ? k_resid_cast_stop<false, true> : k_resid_cast_stop<false, false>);
}

void launch_resid_cast_stop_rag(const std::vector<RagOuter>& v, int count, cudaStream_t s) {
  rag_launch<RmA>((int)v.size(), k_resid_cast_stop_rag, dim3(RMW * 32), 0, s, [&](int q, RmA& a, int& gx, int&) {
    const RagOuter& O = v[q];
    a = RmA{O.g, rm_geo(O.g, 1), O.op, O.x, O.b, O.r32, O.c, count};
    gx = a.m.blocks();
    return true;
  });
}

}  // namespace hmg
