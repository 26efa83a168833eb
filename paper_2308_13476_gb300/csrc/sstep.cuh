// GMRES(3) of the complex64 cycles in s-step form.
//
// One smoothing step minimises ||b - A (x + c)|| over c in span{r, A r,
// A^2 r}.  The Arnoldi form needs a global sum after every operator
// application (and again after every orthogonalisation).  Here the basis is
//   v_0 = r,  v_{k+1} = (scale A - sigma) v_k,  k = 0..2,
// which no sum interrupts, and one sum gives its Gram matrix <v_i, v_j>.
// With w_j = scale A v_j = v_{j+1} + sigma v_j the minimiser is x + scale
// sum_j z_j v_j, z the solution of the 3 x 3 normal equations
//   <w_i, w_j> z_j = <w_i, r>.
// scale (about the inverse of the level's diagonal) keeps the powers in
// range; sigma = 1 on the fine level, where scale A has its spectrum around
// 1, keeps the basis well conditioned (median condition of the scaled normal
// matrix over a solve 9 to 24, against 600 to 1100 with sigma = 0), and sigma = 0
// the coarse levels' (17 to 45 on the first of them, against 2e4 to 7e4 with
// sigma = 1; 30 to 2400 below).  The least-squares minimum is flat, so an error e
// in z raises the residual only by e^2: with FP32 scalars the cycle counts of
// constant-k, variable-k, W-cycle and linear-transfer solves to 1e-6 and to 1e-11
// stay within 10 % (at least two) of the complex128 path's, which keeps the
// Arnoldi form, whose iterates follow modified Gram-Schmidt to rounding.  The
// cycle runs on its residual times a power of two near the inverse of its norm
// (Ctl::rscale), so that the squares summed here stay in the float range.
#pragma once
#include "common.cuh"
#include "gmres.cuh"

namespace hmg {

// scale and sigma of level l of a hierarchy with fine cell size h, for an
// operator of the given kind (OpView::kind): h_l^2 / 4, about the inverse of
// the diagonal of the Galerkin operators as of the five-point one.
inline double ss_scale(double h, int l) { return 0.25 * h * h * (double)(1ll << (2 * l)); }
inline double ss_sigma(int kind) { return kind == 1 ? 1.0 : 0.0; }

// Steps between two fresh residuals on the levels whose update forms the next
// residual by linearity, and whether step `step` of a smoothing call starts
// from one that the previous update left.
constexpr int SS_REFRESH = 4;
__host__ __device__ inline bool ss_carried(int step) { return step % SS_REFRESH != 0; }

// Coefficients of r, v_1, v_2, v_3 in the next residual,
//   r' = (1 - sigma z_0) r - (z_0 + sigma z_1) v_1 - (z_1 + sigma z_2) v_2 - z_2 v_3,
// from y = scale z.
__device__ __forceinline__ void ss_residual_coef(const float2 (&y)[3], float iscale, float sigma, float2 (&c)[4]) {
  float2 z[4];
#pragma unroll
  for (int k = 0; k < 3; ++k) z[k] = make_float2(y[k].x * iscale, y[k].y * iscale);
  z[3] = make_float2(0.f, 0.f);
  c[0] = make_float2(1.f - sigma * z[0].x, -sigma * z[0].y);
#pragma unroll
  for (int k = 1; k < 4; ++k)
    c[k] = make_float2(-fmaf(sigma, z[k].x, z[k - 1].x), -fmaf(sigma, z[k].y, z[k - 1].y));
}

// Values of one Gram sum: |v_0|^2 .. |v_3|^2, then <v_i, v_j> (re, im) for
// (i, j) = (0,1), (0,2), (0,3), (1,2), (1,3), (2,3).
constexpr int SS_NV = 16;

template <class T>
__device__ __forceinline__ void ss_gram_add(T (&g)[SS_NV], cx<T> v0, cx<T> v1, cx<T> v2, cx<T> v3) {
  const cx<T> v[4] = {v0, v1, v2, v3};
  int k = 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    g[i] = fma(v[i].x, v[i].x, fma(v[i].y, v[i].y, g[i]));
#pragma unroll
    for (int j = i + 1; j < 4; ++j, k += 2) {
      g[k] = fma(v[i].x, v[j].x, fma(v[i].y, v[j].y, g[k]));
      g[k + 1] = fma(v[i].x, v[j].y, fma(-v[i].y, v[j].x, g[k + 1]));
    }
  }
}

// y[0..6) = scale z (re, im): the coefficients of v_0..v_2.  LDL^H of the
// normal matrix scaled to a unit diagonal; a pivot at rounding level ends
// the basis there (the remaining coefficients are 0), as a breakdown of the
// Arnoldi process would.
template <class V, class St> __device__ __forceinline__ void ss_solve(const V* g, float scale, float sigma, St* y) {
  // the sums relative to |r|^2: z does not depend on their common factor, and
  // near convergence |r|^2 alone is too small for products of its inverses
  float d[4], er[4][4], ei[4][4];   // <v_i, v_j> for i < j
  const V f = V(1) / (g[0] > V(1e-36f) ? g[0] : V(1e-36f));
#pragma unroll
  for (int i = 0, k = 4; i < 4; ++i) {
    d[i] = (float)(g[i] * f);
#pragma unroll
    for (int j = i + 1; j < 4; ++j, k += 2) {
      er[i][j] = (float)(g[k] * f);
      ei[i][j] = (float)(g[k + 1] * f);
    }
  }
  // M_ij = <w_i, w_j> (lower triangle, i >= j) and f_i = <w_i, r>
  float m[3], l10r, l10i, l20r, l20i, l21r, l21i, fr[3], fi[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) m[j] = fmaf(sigma, fmaf(sigma, d[j], 2.f * er[j][j + 1]), d[j + 1]);
  // <w_1, w_0> = <v_2, v_1> + s <v_2, v_0> + s <v_1, v_1> + s^2 <v_1, v_0>
  l10r = fmaf(sigma, er[0][2] + fmaf(sigma, er[0][1], d[1]), er[1][2]);
  l10i = -fmaf(sigma, fmaf(sigma, ei[0][1], ei[0][2]), ei[1][2]);
  // <w_2, w_0> = <v_3, v_1> + s <v_3, v_0> + s <v_2, v_1> + s^2 <v_2, v_0>
  l20r = fmaf(sigma, er[0][3] + fmaf(sigma, er[0][2], er[1][2]), er[1][3]);
  l20i = -fmaf(sigma, ei[0][3] + fmaf(sigma, ei[0][2], ei[1][2]), ei[1][3]);
  // <w_2, w_1> = <v_3, v_2> + s <v_3, v_1> + s <v_2, v_2> + s^2 <v_2, v_1>
  l21r = fmaf(sigma, er[1][3] + fmaf(sigma, er[1][2], d[2]), er[2][3]);
  l21i = -fmaf(sigma, fmaf(sigma, ei[1][2], ei[1][3]), ei[2][3]);
  fr[0] = fmaf(sigma, d[0], er[0][1]);
  fi[0] = -ei[0][1];
  fr[1] = fmaf(sigma, er[0][1], er[0][2]);
  fi[1] = -fmaf(sigma, ei[0][1], ei[0][2]);
  fr[2] = fmaf(sigma, er[0][2], er[0][3]);
  fi[2] = -fmaf(sigma, ei[0][2], ei[0][3]);
  float s[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    s[j] = m[j] > 0.f ? rsqrtf(m[j]) : 0.f;
    fr[j] *= s[j];
    fi[j] *= s[j];
  }
  const float s10 = s[1] * s[0], s20 = s[2] * s[0], s21 = s[2] * s[1];
  l10r *= s10; l10i *= s10;
  l20r *= s20; l20i *= s20;
  l21r *= s21; l21i *= s21;
  constexpr float tiny = 2e-7f;
  const float d1 = 1.f - fmaf(l10r, l10r, l10i * l10i);
  const bool k1 = d1 > tiny;
  const float i1 = k1 ? 1.f / d1 : 0.f;
  // c = <w_2, w_1> - l20 conj(l10): the unnormalised L_21 d1
  const float cr = l21r - fmaf(l20r, l10r, l20i * l10i), ci = l21i - fmaf(l20i, l10r, -(l20r * l10i));
  const float er21 = cr * i1, ei21 = ci * i1;
  const float d2 = 1.f - fmaf(l20r, l20r, l20i * l20i) - fmaf(cr, er21, ci * ei21);
  const bool k2 = k1 && d2 > tiny;
  const float i2 = k2 ? 1.f / d2 : 0.f;
  // forward: t = L^{-1} f
  const float t1r = fr[1] - fmaf(l10r, fr[0], -(l10i * fi[0])), t1i = fi[1] - fmaf(l10r, fi[0], l10i * fr[0]);
  const float t2r = fr[2] - fmaf(l20r, fr[0], -(l20i * fi[0])) - fmaf(er21, t1r, -(ei21 * t1i));
  const float t2i = fi[2] - fmaf(l20r, fi[0], l20i * fr[0]) - fmaf(er21, t1i, ei21 * t1r);
  // back: z = L^{-H} D^{-1} t
  const float z2r = t2r * i2, z2i = t2i * i2;
  const float z1r = t1r * i1 - fmaf(er21, z2r, ei21 * z2i), z1i = t1i * i1 - fmaf(er21, z2i, -(ei21 * z2r));
  const float z0r = fr[0] - fmaf(l10r, z1r, l10i * z1i) - fmaf(l20r, z2r, l20i * z2i);
  const float z0i = fi[0] - fmaf(l10r, z1i, -(l10i * z1r)) - fmaf(l20r, z2i, -(l20i * z2r));
  y[0] = (St)(scale * s[0] * z0r);
  y[1] = (St)(scale * s[0] * z0i);
  y[2] = (St)(scale * s[1] * z1r);
  y[3] = (St)(scale * s[1] * z1i);
  y[4] = (St)(scale * s[2] * z2r);
  y[5] = (St)(scale * s[2] * z2i);
}

// The block's Gram sums of one right-hand side by warp, sh[value * warps +
// warp]: float within the warps, FP64 from there on.
template <int NT> __device__ __forceinline__ void ss_warp_sums(float (&g)[SS_NV], double* sh /* [SS_NV * NT / 32] */, int tid) {
  const int lane = tid & 31;
  const float t = lane_sum<SS_NV, float>(g, lane);
  if ((lane & 1) == 0) sh[lane_value<SS_NV>(lane) * (NT / 32) + (tid >> 5)] = (double)t;
}

// Grid-wide Gram sums of RB right-hand sides from rhs0 on inside the kernel
// that forms v_3, and the solves: every block publishes its sums (sh:
// ss_warp_sums of each right-hand side, one after the other), the block with
// the last ticket adds the nrec records of each and solves for y in the state
// at S.  The RB right-hand sides share the ticket, the fences and the wait for
// the records: NT / RB threads take one of them, 16 values side by side,
// every thread one value of every NT / RB / 16-th record, in record order.
// act: bit q set if right-hand side rhs0 + q takes part.  Reproducible: the
// order does not depend on which block is last.  Must be reached by every
// thread of every block of these right-hand sides; the records of tickets[rhs0]
// are complete at the last ticket.
template <int NT, int RB>
__device__ __forceinline__ void ss_finish_rb(double* sh /* [RB * SS_NV * max(NT / 32, NT / RB / 16)] */, double* partial,
                                             unsigned* tickets, int rhs0, unsigned act, int nrec, int blk, int tid,
                                             float scale, float sigma, double* st) {
  constexpr int W = NT / 32, N = NT / RB, G = N / SS_NV;   // threads and records per pass of one right-hand side
  static_assert(NT % 32 == 0 && SS_NV * RB <= NT && N % SS_NV == 0 && N % 32 == 0 && SS_NV == 16, "block shape");
  __shared__ int s_last;
  __syncthreads();
  if (tid < SS_NV * RB && (act >> (tid / SS_NV) & 1)) {
    double v = sh[tid * W];
#pragma unroll
    for (int w = 1; w < W; ++w) v += sh[tid * W + w];
    partial[((long long)(rhs0 + tid / SS_NV) * nrec + blk) * SS_NV + tid % SS_NV] = v;
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&tickets[rhs0], 1u) == (unsigned)(nrec - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int q = tid / N, t = tid - q * N;
  const bool on = act >> q & 1;
  if (on) {
    const double* rec = partial + (long long)(rhs0 + q) * nrec * SS_NV + t;   // record t / 16, value t % 16
    double v = 0.0;
    int b = t / SS_NV;
    for (; b + 7 * G < nrec; b += 8 * G, rec += 8 * N) {
      double a[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) a[k] = __ldcg(rec + k * N);
      v += ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
    }
    for (; b < nrec; b += G, rec += N) v += __ldcg(rec);
    sh[tid] = v;
  }
  __syncthreads();
  if (on && t < SS_NV) {
    double v = sh[tid];
#pragma unroll
    for (int k = 1; k < G; ++k) v += sh[tid + k * SS_NV];
    sh[tid] = v;
  }
  __syncthreads();
  if (tid == 0) tickets[rhs0] = 0u;
  if (on && t == 0) ss_solve(sh + q * N, scale, sigma, gstate<float>(st, rhs0 + q));
}

// The same for one right-hand side (sh: [NT]).
template <int NT>
__device__ __forceinline__ void ss_finish(float (&g)[SS_NV], double* sh, double* partial, unsigned* tickets, int rhs,
                                          int nrec, int blk, int tid, float scale, float sigma, double* st) {
  ss_warp_sums<NT>(g, sh, tid);
  ss_finish_rb<NT, 1>(sh, partial, tickets, rhs, 1u, nrec, blk, tid, scale, sigma, st);
}

}  // namespace hmg
