// Scalar part of the GMRES(3) smoother (Sec. 5.3 of the paper), shared by
// the grid-wide kernels, the coarse-cycle cluster and the cooperative interpreter: the
// per-RHS state layout, the Hessenberg updates of one Arnoldi step (modified
// Gram-Schmidt written with the Gram matrix of the basis) and the FP64 Givens
// least-squares solve.  Each function runs in one thread.
#pragma once
#include "common.cuh"

namespace hmg {

// Per-RHS scalar state, GS doubles each.
constexpr int GS = 96;
constexpr int G_BETA = 0;
constexpr int G_S = 1;      // s_0..s_3
constexpr int G_H = 8;      // Hbar[i][j] complex, i < 4, j < 3: 8 + 2*(i*3+j)
constexpr int G_G = 32;     // Gram <v_i, v_l> complex 4x4: 32 + 2*(i*4+l)
constexpr int G_Y = 64;     // y complex, 3
constexpr int G_M = 70;     // number of Arnoldi columns
constexpr int G_BRK = 71;   // 1 = stop (breakdown or beta == 0)


// min || beta e1 - Hbar y || by Givens rotations; Hbar is (m+1) x m.  The
// arithmetic runs in Ts (FP64 for the complex128 path, FP32 for the
// complex64 cycles of the mixed path); the state S is stored in St: FP64 in
// global memory, or Ts where one thread block owns the state (every stored
// value is a Ts value, so both storages give the same results).  The summed
// inputs v of the fin_* steps come in V: FP64 from the grid-wide sums, Ts
// from the block sums of the coarse-cycle launches.
//
// The scalars sit on the serial path of every smoothing step (one thread,
// every launch of the Arnoldi process waits for them), so their cost is the
// length of the dependent chain: square roots and divides above all, which on
// the FP64 pipe are sequences of a dozen dependent instructions each.  The
// subdiagonal of Hbar is real (a norm), so the rotation
//   G = t [[conj(a), b], [-b, a]],  t = (|a|^2 + b^2)^(-1/2)
// zeroes it with one reciprocal square root per column, leaves the real
// diagonal (|a|^2 + b^2) t and makes t its reciprocal: the back substitution
// needs no divide (three rsqrt where the |a|, |b|, r form took nine square
// roots and twelve to eighteen divides).  Measured on whole solves: FP64
// W(2,2) on 161^2 325.8 -> 297.7 ms, FP64 8 x 513^2 538.7 -> 521.2 ms,
// complex64 V(2,2) on 81^2 9.12 -> 8.43 ms.
template <class Ts, class St = double> __device__ __forceinline__ void lsq(St* S) {
  const int m = (int)S[G_M];
  if (m <= 0) return;
  Ts Hr[3][3], Hi[3][3], t[3], gr[3], gi[3];   // rows 0..2 of Hbar's upper triangle, the rotated right-hand side
  Ts yr[3] = {0, 0, 0}, yi[3] = {0, 0, 0};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    t[c] = gr[c] = gi[c] = Ts(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Hr[a][c] = (Ts)S[G_H + 2 * (a * 3 + c)];
      Hi[a][c] = (Ts)S[G_H + 2 * (a * 3 + c) + 1];
    }
  }
  gr[0] = (Ts)S[G_BETA];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (c >= m) break;
    const Ts ar = Hr[c][c], ai = Hi[c][c], b = (Ts)S[G_H + 2 * ((c + 1) * 3 + c)];
    const Ts n2 = fma(ar, ar, fma(ai, ai, b * b));
    if (n2 == Ts(0)) continue;   // a zero column: y_c = 0
    t[c] = rsqrt(n2);
    const Ts pr = ar * t[c], pi = ai * t[c], q = b * t[c];
#pragma unroll
    for (int col = c + 1; col < 3; ++col) {
      const Ts xr = Hr[c][col], xi = Hi[c][col], zr = Hr[c + 1][col], zi = Hi[c + 1][col];
      Hr[c][col] = fma(pr, xr, fma(pi, xi, q * zr));
      Hi[c][col] = fma(pr, xi, fma(-pi, xr, q * zi));
      Hr[c + 1][col] = fma(-q, xr, fma(pr, zr, -(pi * zi)));
      Hi[c + 1][col] = fma(-q, xi, fma(pr, zi, pi * zr));
    }
    const Ts xr = gr[c], xi = gi[c];
    gr[c] = fma(pr, xr, pi * xi);
    gi[c] = fma(pr, xi, -(pi * xr));
    if (c < 2) {
      gr[c + 1] = -q * xr;
      gi[c + 1] = -q * xi;
    }
  }
#pragma unroll
  for (int c = 2; c >= 0; --c) {
    if (c >= m) continue;
    Ts vr = gr[c], vi = gi[c];
#pragma unroll
    for (int q = c + 1; q < 3; ++q) {   // y_q = 0 for q >= m
      vr = fma(-Hr[c][q], yr[q], fma(Hi[c][q], yi[q], vr));
      vi = fma(-Hr[c][q], yi[q], fma(-Hi[c][q], yr[q], vi));
    }
    yr[c] = vr * t[c];
    yi[c] = vi * t[c];
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    S[G_Y + 2 * c] = (St)yr[c];
    S[G_Y + 2 * c + 1] = (St)yi[c];
  }
}

// ---- scalar steps of one Arnoldi pass, run by one thread ----

// sqrt(n2) given s = rsqrt(n2) (0 for n2 = 0): one product instead of a
// second iterated square root; a NaN or infinite n2 keeps its sqrt.
template <class Ts> __device__ __forceinline__ Ts norm_of(Ts n2, Ts s) { return s > Ts(0) ? n2 * s : sqrt(n2); }

template <class Ts, class St = double, class V = double> __device__ __forceinline__ void fin_init(St* S, const V* v) {
  for (int k = 0; k < GS; ++k) S[k] = St(0);
  const Ts n2 = (Ts)v[0], s0 = n2 > Ts(0) ? rsqrt(n2) : Ts(0);
  S[G_BETA] = (St)norm_of(n2, s0);
  S[G_M] = St(0);
  if (n2 == Ts(0)) S[G_BRK] = St(1);
  else S[G_S + 0] = (St)s0;
}

// h_lJ = <v_l, w> - sum_{q<l} h_qJ <v_l, v_q>, with <v_l, w> = s_l <u_l, w>
template <int J, class Ts, class St = double, class V = double> __device__ __forceinline__ void fin_a(St* S, const V* v) {
  Ts hr[J + 1], hi[J + 1];
  for (int l = 0; l <= J; ++l) {
    const Ts sl = (Ts)S[G_S + l];
    Ts dr = sl * (Ts)v[2 * l], di = sl * (Ts)v[2 * l + 1];
    for (int q = 0; q < l; ++q) {
      const Ts gr = (Ts)S[G_G + 2 * (l * 4 + q)], gi = (Ts)S[G_G + 2 * (l * 4 + q) + 1];
      dr -= hr[q] * gr - hi[q] * gi;
      di -= hr[q] * gi + hi[q] * gr;
    }
    hr[l] = dr;
    hi[l] = di;
    S[G_H + 2 * (l * 3 + J)] = (St)dr;
    S[G_H + 2 * (l * 3 + J) + 1] = (St)di;
  }
}

// h_{J+1,J} = ||u_{J+1}||, breakdown test, Gram entries of v_{J+1}; the least
// squares problem is solved once the Arnoldi process stops.
template <int J, class Ts, class St = double, class V = double> __device__ __forceinline__ void fin_b(St* S, const V* v) {
  const Ts n2 = (Ts)v[0], sn = n2 > Ts(0) ? rsqrt(n2) : Ts(0), hn = norm_of(n2, sn);
  S[G_H + 2 * ((J + 1) * 3 + J)] = (St)hn;
  S[G_H + 2 * ((J + 1) * 3 + J) + 1] = St(0);
  S[G_M] = St(J + 1);
  if (hn <= Ts(1e-14) * (Ts)S[G_BETA]) {
    S[G_BRK] = St(1);
  } else {
    S[G_S + J + 1] = (St)sn;
    if (J < 2) {
      for (int l = 0; l <= J; ++l) {   // <v_{J+1}, v_l> = s_{J+1} s_l <u_{J+1}, u_l>
        const Ts f = sn * (Ts)S[G_S + l];
        S[G_G + 2 * ((J + 1) * 4 + l)] = (St)(f * (Ts)v[1 + 2 * l]);
        S[G_G + 2 * ((J + 1) * 4 + l) + 1] = (St)(f * (Ts)v[2 + 2 * l]);
      }
    }
  }
  if (J == 2 || S[G_BRK] != St(0)) lsq<Ts, St>(S);
}

// The per-RHS state in global memory: GS values of the cycle's working
// precision T per right-hand side (the scalar steps compute in T and store T
// values, so FP32 storage gives what FP64 storage would; kernels of a
// complex64 cycle then read their coefficients without FP64 instructions).
template <class T> __device__ __forceinline__ T* gstate(double* st, int rhs) {
  return reinterpret_cast<T*>(st) + (long long)rhs * GS;
}
template <class T> __device__ __forceinline__ const T* gstate(const double* st, int rhs) {
  return reinterpret_cast<const T*>(st) + (long long)rhs * GS;
}

// Runs a scalar step on the RHS state in shared memory (all threads of the
// block copy it in and out; thread 0 computes), so its many dependent reads
// and writes stay on chip.
template <class T, class St, class F>
__device__ __forceinline__ void staged(St* S, const double* v, F f) {
  __shared__ St Ssh[GS];
  const int tid = threadIdx.x + threadIdx.y * blockDim.x, nt = blockDim.x * blockDim.y;
  for (int k = tid; k < GS; k += nt) Ssh[k] = S[k];
  __syncthreads();
  if (tid == 0) f(Ssh, v);
  __syncthreads();
  for (int k = tid; k < GS; k += nt) S[k] = Ssh[k];
}

}  // namespace hmg
