// Column marches over a Kronecker-form level (A = W_y (x) G_x + H_y (x) W_x,
// radius R): the row staging, the row-sum ring and the combination along y
// shared by kron_march.cu (complex128 GMRES(3), residuals) and sstep_level.cu
// (complex64 s-step GMRES(3)).
#pragma once
#include <algorithm>
#include <type_traits>

#include "gmres.cuh"
#include "internal.h"

namespace hmg {
namespace {

constexpr int KW = 4;   // warps per block; a warp covers 32 columns of one chunk of rows

struct KGeo {
  int ncw;      // 32-column groups
  int ch;       // rows per chunk
  int nchunks;
};

template <int P, int K, class F> __device__ __forceinline__ void kmarch_phases(int r, int last, F& f) {
  if constexpr (P < K) {
    if (r + P > last) return;
    f(std::integral_constant<int, P>{}, r + P);
    kmarch_phases<P + 1, K>(r, last, f);
  }
}
// Runs f(phase, r) for r = r0 .. last, phase = (r - r0) mod K as an
// std::integral_constant.
template <int K, class F> __device__ __forceinline__ void kmarch(int r0, int last, F&& f) {
#pragma unroll 1
  for (int r = r0; r <= last; r += K) kmarch_phases<0, K>(r, last, f);
}

// Whether the march over a radius-R level is unrolled so that its register
// ring never moves (KU = 2R+1 phases), or keeps one phase and shifts the ring
// by a row per step (KU = 1).  complex64 unrolls both radii (with the y
// coefficients of the interior rows in the parameter bank the radius-3
// passes stay within their launch bounds); the complex128 radius-3 marches
// would spill unrolled and keep the shifting ring.
template <class T, int R> constexpr int KU = (R == 2 || sizeof(T) == 4) ? 2 * R + 1 : 1;

// A v down column i: the input rows arrive in order through a per-warp
// shared-memory ring (each row's 32 + 2RA columns around the warp's columns,
// RA >= R, copied by cp.async KD rows ahead of use, so the 2R+1 neighbours of a lane
// are read from shared memory instead of being loaded from L2 2R+1 times);
// advance<P>() forms the two row sums of the lane's column and puts them in
// slot P of the register ring of the last 2R+1 rows, and combine<P>() returns
// (A v)(i, m) once that ring holds rows m-R..m+R.  With R = 2 the march over
// rows is unrolled by 2R+1 (kmarch, KU), so that row r sits in the
// compile-time slot P = (r - r0) mod (2R+1) and the ring never moves; with
// R = 3 the ring shifts by one row per step.
constexpr int KD = 4;    // rows in flight ahead of use
constexpr int KSL = 8;   // ring slots (a power of two > KD)

// Staged columns left (and right) of a warp's 32: R, rounded up to even for
// complex64 so that a staged row starts on a 16-byte boundary (the warp's
// first column is a multiple of 32, the row pitch a multiple of 4).
template <class T, int R> constexpr int kron_ra() { return sizeof(T) == 4 ? (R + 1) & ~1 : R; }

// Copy row r's staged columns cw0 - RA .. cw0 + 31 + RA of vs into dst.
// complex64: one 16-byte copy of a column pair per lane, for the first
// 16 + RA lanes; a pair that starts at column nx takes the zero halo column
// nx + 1 with it, a pair right of it is zero-filled.  complex128: one
// 16-byte element per copy.  The padded layout covers the columns left of
// the grid and the rows past either edge.
template <class T, int RA>
__device__ __forceinline__ void stage_kron_row(cx<T>* dst, const cx<T>* vs, const Grid& g, int cw0, int lane,
                                               int r) {
  constexpr int WD = 32 + 2 * RA;
  if constexpr (sizeof(cx<T>) == 8) {
    if (lane < WD / 2) {
      const int col = cw0 - RA + 2 * lane;
      const bool ok = col <= g.nx;
      const cx<T>* src = vs + g.at(ok ? col : 0, r);
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + 2 * lane);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
    }
  } else {
#pragma unroll
    for (int e = lane; e < WD; e += 32) {
      const int col = cw0 - RA + e;
      const bool ok = col <= g.nx;
      const cx<T>* src = vs + g.at(ok ? col : 0, r);
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + e);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
    }
  }
}

// Copy row r's own 32 columns cw0 .. cw0 + 31 of vs into dst (no halo): a
// vector read only at the lane's own node, staged with the applied one so
// that its loads are in flight KD rows ahead too.
template <class T>
__device__ __forceinline__ void stage_own_row(cx<T>* dst, const cx<T>* vs, const Grid& g, int cw0, int lane, int r) {
  if constexpr (sizeof(cx<T>) == 8) {
    if (lane < 16) {
      const int col = cw0 + 2 * lane;
      const bool ok = col <= g.nx;
      const cx<T>* src = vs + g.at(ok ? col : 0, r);
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + 2 * lane);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
    }
  } else {
    const int col = cw0 + lane;
    const bool ok = col <= g.nx;
    const cx<T>* src = vs + g.at(ok ? col : 0, r);
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + lane);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
  }
}

// combination along y for output row m = r - R, r the row just taken in
// slot P of a ring of the last K = 2R+1 row sums: row m + dy sits in slot
// (P + 1 + R + dy) mod K, or in slot dy + R of a shifting ring (KU = 1).
// Rows whose y-factors are the translation-invariant interior ones take the
// coefficients from the operator's parameter-bank copy (the same values);
// the others load their row's coefficients.
template <class T, int R, int K, int KUR, int P>
__device__ __forceinline__ cx<T> kcombine(const OpK<T, R>& op, int m, const cx<T> (&s1)[K], const cx<T> (&s2)[K]) {
  cx<T> acc = mk<T>(T(0), T(0));
  if (m >= op.ty0 && m < op.ty1) {
    if constexpr (sizeof(T) == 4 && R == 2) {   // packed: Re h and w_y with s, Im h apart, joined once
      float2 pr = make_float2(0.f, 0.f), pi = make_float2(0.f, 0.f);
#pragma unroll
      for (int dy = -R; dy <= R; ++dy) {
        const int q = KUR == 1 ? dy + R : (P + 1 + R + dy) % K;
        pr = fma2(op.pk.wyb[dy + R], s1[q], pr);
        pr = fma2(op.pk.hyr[dy + R], s2[q], pr);
        pi = fma2(op.pk.hyi[dy + R], s2[q], pi);
      }
      return make_float2(pr.x - pi.y, pr.y + pi.x);
    }
#pragma unroll
    for (int dy = -R; dy <= R; ++dy) {
      const int q = KUR == 1 ? dy + R : (P + 1 + R + dy) % K;
      const T wy = op.wyc[dy + R];
      acc = mk<T>(fma(wy, s1[q].x, acc.x), fma(wy, s1[q].y, acc.y));
      acc = fma_c<T>(op.hyc[dy + R], s2[q], acc);
    }
    return acc;
  }
  const cx<T>* H = op.hy + m * K;
  const T* Wy = op.wy + m * K;
#pragma unroll
  for (int dy = -R; dy <= R; ++dy) {
    const int q = KUR == 1 ? dy + R : (P + 1 + R + dy) % K;
    const T wy = __ldg(Wy + dy + R);
    acc = mk<T>(fma(wy, s1[q].x, acc.x), fma(wy, s1[q].y, acc.y));
    acc = fma_c<T>(__ldg(H + dy + R), s2[q], acc);
  }
  return acc;
}

template <class T, int R> struct KRing {
  static constexpr int K = 2 * R + 1;
  static constexpr int RA = kron_ra<T, R>();
  static constexpr int WD = 32 + 2 * RA;   // staged row width
  cx<T> G[K];
  T Wx[K];
  cx<T> s1[K], s2[K];
  const cx<T>* vs;   // slice of the applied vector
  Grid g;
  int cw0, lane;     // the warp's first column, the lane
  cx<T>* sm;         // the warp's ring, [KSL][WD]
  int r0;            // first row of the march (slot 0)
  const cx<T>* os = nullptr;   // optional vectors read at the lane's own nodes (no halo)
  cx<T>* osm = nullptr;        // their rings, [KSL][32]
  const cx<T>* os2 = nullptr;
  cx<T>* osm2 = nullptr;

  __device__ __forceinline__ void init(const OpK<T, R>& op, int i, bool col) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      G[k] = col ? op.gx[i * K + k] : mk<T>(T(0), T(0));
      Wx[k] = col ? op.wx[i * K + k] : T(0);
      s1[k] = mk<T>(T(0), T(0));
      s2[k] = mk<T>(T(0), T(0));
    }
  }
  // copy row r's staged columns into its slot
  __device__ __forceinline__ void issue(int r) {
    stage_kron_row<T, RA>(sm + ((r - r0) & (KSL - 1)) * WD, vs, g, cw0, lane, r);
    if (os) stage_own_row<T>(osm + ((r - r0) & (KSL - 1)) * 32, os, g, cw0, lane, r);
    if (os2) stage_own_row<T>(osm2 + ((r - r0) & (KSL - 1)) * 32, os2, g, cw0, lane, r);
  }
  // the applied vector and the own-node vector at row m (m >= r - KSL + KD,
  // r the row last taken: the slot is not yet reused), the lane's column
  __device__ __forceinline__ cx<T> staged_at(int m) const { return sm[((m - r0) & (KSL - 1)) * WD + lane + RA]; }
  __device__ __forceinline__ cx<T> own_at(int m) const { return osm[((m - r0) & (KSL - 1)) * 32 + lane]; }
  __device__ __forceinline__ cx<T> own2_at(int m) const { return osm2[((m - r0) & (KSL - 1)) * 32 + lane]; }
  __device__ __forceinline__ static void commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
  // rows r0 .. r0 + KD - 1 in flight
  __device__ __forceinline__ void prime(int last) {
#pragma unroll
    for (int d = 0; d < KD; ++d) {
      if (r0 + d <= last) issue(r0 + d);
      commit();
    }
  }
  // take input row r (rows up to `last` exist): row r + KD in flight, row r's
  // sums into the register ring.  All lanes of the warp call it.
  template <int P> __device__ __forceinline__ void advance(int r, int last) {
    __syncwarp();   // every lane is done with the slot row r + KD reuses
    if (r + KD <= last) issue(r + KD);
    commit();
    asm volatile("cp.async.wait_group %0;\n" ::"n"(KD) : "memory");
    __syncwarp();   // row r, copied by all lanes, is visible to all
    const cx<T>* row = sm + ((r - r0) & (KSL - 1)) * WD + lane + RA;
    cx<T> a = mk<T>(T(0), T(0)), c = mk<T>(T(0), T(0));
#pragma unroll
    for (int dx = -R; dx <= R; ++dx) {
      const cx<T> xv = row[dx];
      a = fma_c<T>(G[dx + R], xv, a);
      c = mk<T>(fma(Wx[dx + R], xv.x, c.x), fma(Wx[dx + R], xv.y, c.y));
    }
    if constexpr (KU<T, R> == 1) {
#pragma unroll
      for (int k = 0; k < K - 1; ++k) {
        s1[k] = s1[k + 1];
        s2[k] = s2[k + 1];
      }
    }
    s1[KU<T, R> == 1 ? K - 1 : P] = a;
    s2[KU<T, R> == 1 ? K - 1 : P] = c;
  }
  // combination along y for output row m = r - R, r the row just taken in
  // slot P: row m + dy sits in slot (P + 1 + R + dy) mod K, or in slot dy + R
  // of the shifting ring (KU = 1)
  template <int P> __device__ __forceinline__ cx<T> combine(const OpK<T, R>& op, int m) const {
    return kcombine<T, R, K, KU<T, R>, P>(op, m, s1, s2);
  }
};

// Common prologue.  A warp owns 32 columns of one chunk of rows; `has`: the
// warp has work; `col`: the lane's column is inside the grid.
#define KPRO                                                                  \
  __shared__ double sh[NVMAX * 32];                                           \
  __shared__ __align__(16) cx<T> ksm[KW][KSL][KRing<T, R>::WD];              \
  const int rhs = blockIdx.z;                                                 \
  if (active && !active[rhs]) return;                                         \
  const long long off = (long long)rhs * g.vstride;                           \
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;                  \
  const int gw = blockIdx.x * KW + wib;                                       \
  const bool has = gw < kg.ncw * kg.nchunks;                                  \
  const int cw0 = (has ? gw % kg.ncw : 0) * 32, i = cw0 + lane;               \
  const int j0 = (has ? gw / kg.ncw : 0) * kg.ch, j1 = min(j0 + kg.ch, g.ny + 1); \
  const bool col = has && i <= g.nx;                                          \
  const int nblk = gridDim.x, blk = blockIdx.x;

#define KMARCH_SETUP(vsrc)                                                    \
  KRing<T, R> ring;                                                           \
  ring.init(op, i, col);                                                      \
  ring.vs = (vsrc);                                                           \
  ring.g = g;                                                                 \
  ring.cw0 = cw0;                                                             \
  ring.lane = lane;                                                           \
  ring.sm = &ksm[wib][0][0];                                                  \
  ring.r0 = j0 - R;                                                           \
  const int last = j1 + R - 1;                                                \
  ring.prime(last);

constexpr int KCH_MIN = 8, KCH_MAX = 64;   // rows per chunk

// Rows per chunk for a level: each warp marches ch + 2R rows, and the
// launch runs in ceil(blocks / cap) rounds of the cap blocks the GPU holds
// at once, so the chunk height minimising rounds x (ch + 2R) is taken (the
// tallest on ties).  A fixed height can leave a last round of a few blocks:
// 64-row chunks of a 513^2 level with 64 right-hand sides give 2.05 rounds.
KGeo kron_geo(const Grid& g, int B, int R, long long cap, int forced = 0) {
  KGeo k;
  k.ncw = cdiv(g.nx + 1, 32);
  if (forced > 0) {   // a fixed height (the autotuner's axis), at least the shortest
    k.ch = std::max(forced, KCH_MIN);
    k.nchunks = cdiv(g.ny + 1, k.ch);
    return k;
  }
  long long best = -1;
  for (int ch = KCH_MAX; ch >= KCH_MIN; --ch) {
    const long long blocks = (long long)cdiv((long long)k.ncw * cdiv(g.ny + 1, ch), KW) * B;
    const long long cost = (long long)cdiv(blocks, cap) * (ch + 2 * R);
    if (best < 0 || cost < best) {
      best = cost;
      k.ch = ch;
    }
  }
  k.nchunks = cdiv(g.ny + 1, k.ch);
  return k;
}

}  // namespace
}  // namespace hmg
