// Building blocks of the fine level's row marches (gmres_march.cu, complex128;
// sstep_march.cu, complex64, which has its own stencil and staging): a warp walks a strip of columns down a chunk of rows, with
// the rows it needs in registers, horizontal neighbours by shuffles and input
// rows staged ahead through a per-lane cp.async ring.
#pragma once
#include "gmres.cuh"
#include "internal.h"

namespace hmg {
namespace {

// staging slots per field of a pass with NF input fields
template <int NF> struct Ring { static constexpr int NS = NF == 1 ? 8 : NF == 2 ? 6 : 4; };
// shared memory of a pass: the staging ring, and afterwards the [NVMAX][32]
// doubles of the block reduction
template <int NF> constexpr int ring_bytes() {
  return NF * Ring<NF>::NS * 32 * 16 > NVMAX * 32 * 8 ? NF * Ring<NF>::NS * 32 * 16 : NVMAX * 32 * 8;
}

template <class T> struct MNP { static constexpr int NP = 1; };
template <> struct MNP<float> { static constexpr int NP = 2; };

template <class T> struct Row { cx<T> v[MNP<T>::NP]; };

template <class T> __device__ __forceinline__ cx<T> zc() { return mk<T>(T(0), T(0)); }
template <class T> __device__ __forceinline__ Row<T> zrow() {
  Row<T> r;
#pragma unroll
  for (int n = 0; n < MNP<T>::NP; ++n) r.v[n] = zc<T>();
  return r;
}

// Asynchronous copy of this lane's 16 bytes of row j (nodes i..) into a
// shared-memory slot; columns right of the grid are zero-filled (the padded
// layout makes the two columns left of the grid and the rows -2..ny+2
// readable zeros).
template <class T>
__device__ __forceinline__ void stage_row(uint32_t dst, const cx<T>* __restrict__ s, const Grid& g, int i, int j) {
  const bool ok = i <= g.nx;
  const cx<T>* src = s + g.at(ok ? i : 0, j);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ Row<float> stage_read(const float4* p) {
  const float4 q = *p;
  Row<float> r;
  r.v[0] = make_float2(q.x, q.y);
  r.v[1] = make_float2(q.z, q.w);
  return r;
}
__device__ __forceinline__ Row<double> stage_read(const double2* p) {
  Row<double> r;
  r.v[0] = *p;
  return r;
}
template <class T> struct SlotT { using type = double2; };
template <> struct SlotT<float> { using type = float4; };

__device__ __forceinline__ void mstore(double2* __restrict__ d, const Grid& g, int i, int j, const Row<double>& r) {
  if (i <= g.nx) d[g.at(i, j)] = r.v[0];
}

template <class T> __device__ __forceinline__ cx<T> shfl_up1(cx<T> a) {
  return mk<T>(__shfl_up_sync(0xffffffffu, a.x, 1), __shfl_up_sync(0xffffffffu, a.y, 1));
}
template <class T> __device__ __forceinline__ cx<T> shfl_dn1(cx<T> a) {
  return mk<T>(__shfl_down_sync(0xffffffffu, a.x, 1), __shfl_down_sync(0xffffffffu, a.y, 1));
}

// March modes: MD = 1 interior strips (branch-free stencil), MD = 2 edge
// strips over interior rows (the same stencil, with the boundary row of
// Op0::apply5 on columns 0 and nx and zero off the grid), MD = 0 everything
// else (the 3-row bands; every warp on grids of fewer than 7 rows).  MD + 4
// (modes 0 and 2 only): the same with the second-order absorbing rows of
// Op0<T, true> on the boundary nodes (interior strips touch none).
template <int MD> constexpr int MM = MD & 3;
template <int MD> constexpr bool MA2 = (MD & 4) != 0;
// Per-warp march context.
template <class T, int MD> struct MCtx {
  static constexpr int NP = MNP<T>::NP;
  Op0<T, MA2<MD>> op;
  Grid g;
  int i;       // first node of this lane
  int j0, j1;  // chunk rows [j0, j1)
  bool outl;   // the lane's nodes are in the strip's output columns

  // (A v) on row m from rows m-1, m, m+1 of v; zero for nodes outside the
  // grid.  All lanes must call it (shuffles).
  __device__ __forceinline__ Row<T> apply(const Row<T>& dn, const Row<T>& c, const Row<T>& up, int m) const {
    const cx<T> west = shfl_up1<T>(c.v[NP - 1]);
    const cx<T> east = shfl_dn1<T>(c.v[0]);
    Row<T> r;
#pragma unroll
    for (int n = 0; n < NP; ++n) {
      const cx<T> xe = n + 1 < NP ? c.v[n + 1 < NP ? n + 1 : 0] : east;
      const cx<T> xw = n > 0 ? c.v[n > 0 ? n - 1 : 0] : west;
      const int in = i + n;
      if (MM<MD> != 0) {   // Op0::apply5, interior case
        const cx<T> xn = up.v[n], xs = dn.v[n], xp = c.v[n];
        const int ik = MM<MD> == 2 ? min(max(in, 0), op.nx) : in;   // edge strips: k of an in-grid node
        const T k = op.kf ? op.kf[m * (op.nx + 1) + ik] : op.c.k;
        const T d = fma(-k, k, T(4) * op.c.inv_h2);
        const T sr = (xe.x + xw.x) + (xn.x + xs.x), si = (xe.y + xw.y) + (xn.y + xs.y);
        r.v[n] = mk<T>(fma(d, xp.x, -op.c.inv_h2 * sr), fma(d, xp.y, -op.c.inv_h2 * si));
        if (MM<MD> == 2) {   // rows are interior here; columns 0 and nx take the
                         // boundary row of Op0::apply5, columns off the grid zero
          const bool bcol = in == 0 || in == op.nx, inside = in >= 0 && in <= op.nx;
          if (bcol) r.v[n] = op.apply5(xp, xe, xw, xn, xs, in, m);
          if (!inside) r.v[n] = zc<T>();
        }
      } else {
        r.v[n] = (m >= 0 && m <= op.ny && in >= 0 && in <= op.nx)
                     ? op.apply5(c.v[n], xe, xw, up.v[n], dn.v[n], in, m)
                     : zc<T>();
      }
    }
    return r;
  }
  // node n of the lane counts in the dots of row m
  __device__ __forceinline__ bool cnt(int n, int m) const {
    return outl && (MM<MD> == 1 || i + n <= g.nx) && m >= j0 && m < j1;
  }
  __device__ __forceinline__ bool own_row(int m) const { return outl && m >= j0 && m < j1; }
};

// Register slot of row t + d at unroll phase S (the march starts at t0 = j0 -
// 2 with phase 0, so row r sits in slot (r - j0 + 2) mod 4).
template <int S, int D> struct Sl { static constexpr int v = (S + D + 8) & 3; };

// The NF input fields of a pass: shared-memory staging and register rings.
// Staging slot (f, k) of a lane is at sbase + (f NS + k) 512 bytes.
template <class T, int MD, int NF> struct MIn {
  static constexpr int NS = Ring<NF>::NS, AH = NS - 1;   // AH: rows in flight ahead of use
  MCtx<T, MD> c;
  const cx<T>* src[NF];
  uint32_t sbase;   // shared address of this lane's slot 0 of field 0
  Row<T> F[NF][4];  // register ring: row r in slot (r - j0 + 2) mod 4
  int t1;           // last row the march reads
  int sw, sr;       // staging slots of the next row to issue and to read

  __device__ __forceinline__ void issue(int r, int slot) {
#pragma unroll
    for (int f = 0; f < NF; ++f) stage_row<T>(sbase + (f * NS + slot) * 32 * 16, src[f], c.g, c.i, r);
  }
  // rows t0 .. t0 + AH - 1 in flight, in slots 0 .. AH - 1
  __device__ __forceinline__ void prime(int t0) {
#pragma unroll
    for (int d = 0; d < AH; ++d) {
      if (t0 + d <= t1) issue(t0 + d, d);
      stage_commit();
    }
    sw = AH;
    sr = 0;
  }
  // row t + AH in flight (into the slot row t - 1 left), row t into the
  // register ring
  template <int S> __device__ __forceinline__ void fetch(int t) {
    if (t + AH <= t1) issue(t + AH, sw);
    sw = sw + 1 == NS ? 0 : sw + 1;
    stage_commit();
    stage_wait<AH>();
#pragma unroll
    for (int f = 0; f < NF; ++f)
      F[f][Sl<S, 0>::v] = stage_read(reinterpret_cast<const typename SlotT<T>::type*>(
          __cvta_shared_to_generic(sbase + (f * NS + sr) * 32 * 16)));
    sr = sr + 1 == NS ? 0 : sr + 1;
  }
};

// Runs p.step<S>(t) for t = t0..t1, S = (t - t0) mod 4.
template <class P> __device__ __forceinline__ void march(P& p, int t0, int t1) {
#pragma unroll 1
  for (int t = t0; t <= t1; t += 4) {
    p.template step<0>(t);
    if (t + 1 > t1) break;
    p.template step<1>(t + 1);
    if (t + 2 > t1) break;
    p.template step<2>(t + 2);
    if (t + 3 > t1) break;
    p.template step<3>(t + 3);
  }
}

// Per-warp geometry inside one right-hand side.  With band = 1 the interior
// set is every strip over rows [br, ny+1-br) in chunks of ch rows: strips
// [e_lo, e_hi), whose loaded columns hold no boundary column, take the
// branch-free stencil; the others (the edge strips) take it too and replace
// it by the boundary row of Op0::apply5 on columns 0 and nx and by zero off
// the grid (lane-constant choices: their rows are interior).  br is the
// number of boundary-row bands such that no row a chunk computes is a
// boundary row: one more than the rows computed above a chunk (3 for two
// stencil applications, 4 for the three past the residual).  The boundary set
// is the br-row bands at the top and bottom of every strip.  With band = 0
// every warp is a boundary warp, in chunks of chb rows from row 0.
struct MGeo {
  int nstrips, ny, band, ch, chb, br;
  int e_lo, e_hi;   // strips of the interior set without a boundary column
  int nci;          // chunks per strip over rows [br, ny+1-br)
  int ni, nb;       // warps of the interior strips and of the bands (or of the whole grid)
  // strip and rows [j0, j1) of warp w of the set
  // interior strips [e_lo, e_hi), the edge strips outside that range, each
  // over rows [br, ny+1-br) in chunks of ch rows
  __host__ __device__ __forceinline__ int ne() const { return (nstrips - (e_hi - e_lo)) * nci; }
  template <int MD> __host__ __device__ __forceinline__ void map(int w, int& strip, int& j0, int& j1) const {
    if (MD != 0) {
      const int nse = nstrips - (e_hi - e_lo), nsm = MD == 1 ? e_hi - e_lo : nse;
      const int sidx = w % nsm;
      strip = MD == 1 ? e_lo + sidx : (sidx < e_lo ? sidx : e_hi + (sidx - e_lo));
      j0 = br + (w / nsm) * ch;
      j1 = j0 + ch < ny + 1 - br ? j0 + ch : ny + 1 - br;
      return;
    }
    if (!band) {
      strip = w % nstrips;
      j0 = (w / nstrips) * chb;
      j1 = j0 + chb < ny + 1 ? j0 + chb : ny + 1;
      return;
    }
    strip = w % nstrips;
    j0 = w < nstrips ? 0 : ny + 1 - br;
    j1 = j0 + br;
  }
  // first reduction record of a mode's warps: interior, then edge, then the rest
  template <int MD> __host__ __device__ __forceinline__ int rec0() const {
    return MD == 1 ? 0 : (MD == 2 ? ni : ni + ne());
  }
  __host__ __device__ __forceinline__ int nrec() const { return ni + ne() + nb; }
  // The sets of a grid with strips of sw output columns that load lw columns
  // from hw left of the strip (strip columns), for the chunk height ch.
  __host__ void fill(int nx, int ny_, int sw, int lw, int hw, int br_) {
    nstrips = (nx + sw) / sw;
    ny = ny_;
    br = br_;
    band = ny >= 2 * br;
    chb = 16;
    e_lo = e_hi = 0;
    if (!band) return;
    for (int s = 0; s < nstrips; ++s) {
      const int cs = s * sw - hw;
      if (cs >= 1 && cs + lw - 1 <= nx - 1) {
        if (e_hi == 0) e_lo = s;
        e_hi = s + 1;
      }
    }
  }
  __host__ void chunks(int rows) {
    ch = rows;
    if (band) {
      nci = (ny + 1 - 2 * br + ch - 1) / ch;
      ni = (e_hi - e_lo) * nci;
      nb = 2 * nstrips;
    } else {
      nci = ni = 0;
      nb = nstrips * ((ny + chb) / chb);
    }
  }
};

}  // namespace
}  // namespace hmg
