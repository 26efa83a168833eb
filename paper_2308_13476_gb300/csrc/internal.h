// Host-side declarations shared by the helmmg translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "common.cuh"

namespace hmg {

// Operator of one level in precision T, as handed to the launch wrappers.
// kind 1: matrix-free fine-level operator (c0, kf); kind 2 / 3: stored
// Galerkin stencil of that radius (st, dinv, plane); kind 4 / 5: constant-k
// Kronecker form of radius 2 / 3 (gx, wx, hy, wy, dinv).
template <class T> struct OpView {
  int kind;
  Op0Consts<T> c0;
  const T* kf;
  const cx<T>* st;
  const cx<T>* dinv;
  long long plane;
  const cx<T>* gx;
  const T* wx;
  const cx<T>* hy;
  const T* wy;
  // constant-k levels: rows [ty0, ty1) whose y-factor rows are hyc / wyc
  int ty0, ty1;
  cx<T> hyc[7];
  T wyc[7];
};
__host__ __device__ inline int op_radius(int kind) { return kind == 1 ? 1 : (kind == 2 || kind == 4) ? 2 : 3; }

// Dispatch a generic lambda on the operator functor of a view.
// The Kronecker-form operator of a view, with its translation-invariant
// y-factor rows (parameter-bank copies) when it has them.
template <class T, int R> inline OpK<T, R> kron_op(const OpView<T>& v, int nx, int ny) {
  OpK<T, R> o{v.gx, v.wx, v.hy, v.wy, v.dinv, nx, ny};
  o.ty0 = v.ty0;
  o.ty1 = v.ty1;
  for (int k = 0; k < 2 * R + 1; ++k) {
    o.hyc[k] = v.hyc[k];
    o.wyc[k] = v.wyc[k];
    if constexpr (sizeof(T) == 4) {
      o.pk.hyr[k] = make_float2(v.hyc[k].x, v.hyc[k].x);
      o.pk.hyi[k] = make_float2(v.hyc[k].y, v.hyc[k].y);
      o.pk.wyb[k] = make_float2(v.wyc[k], v.wyc[k]);
    }
  }
  return o;
}

template <class T, class F> inline void with_op(const OpView<T>& v, int nx, int ny, F&& f) {
  switch (v.kind) {
    case 1:   // the second-order absorbing rows are a separate instantiation
      if (v.c0.abc2) f(Op0<T, true>{v.c0, v.kf, nx, ny});
      else f(Op0<T>{v.c0, v.kf, nx, ny});
      break;
    case 2: f(OpS<T, 2>{v.st, v.dinv, v.plane, nx, ny}); break;
    case 3: f(OpS<T, 3>{v.st, v.dinv, v.plane, nx, ny}); break;
    case 4: f(kron_op<T, 2>(v, nx, ny)); break;
    default: f(kron_op<T, 3>(v, nx, ny)); break;
  }
}

// Node-parallel kernels (kernels_level.cu).  `active[b]` == 0 skips RHS b.
// B = number of right-hand sides.
template <class T> void launch_residual(const Grid& g, const OpView<T>& op, const cx<T>* x, const cx<T>* b,
                                        cx<T>* r, int B, const int* active, cudaStream_t s);
template <class T> void launch_apply(const Grid& g, const OpView<T>& op, const cx<T>* x, cx<T>* y, int B,
                                     const int* active, cudaStream_t s);
// x = null: x is zero (the sweep is xout = (omega diag A)^{-1} b).
template <class T> void launch_jacobi(const Grid& g, const OpView<T>& op, const cx<T>* x, const cx<T>* b,
                                      cx<T>* xout, int B, const int* active, cudaStream_t s);
// Streaming multiprocessors of the device, for the launches' geometry: asked for
// once, so that a buffer sized by a geometry and the launches that fill it
// always go by one number.
inline int device_sms() {
  static const int n = [] {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      cudaGetLastError();
    return sms > 0 ? sms : 1;
  }();
  return n;
}
// Per-solve control block of the stopping test (device arrays, one entry per
// RHS unless noted).  tolp = {tol, divergence threshold}; partial/tickets are
// the scratch of the fused reductions (reduce_last).
struct Ctl {
  const double* bnorm;
  const double* tolp;
  int* active;
  int* state;
  int* cycles;
  double* relres;
  double* hist;
  int hist_len;
  int* n_active;        // one int
  double* partial;
  unsigned* tickets;
  float* rscale;        // complex64 cycles, [B][2] (null: complex128): see inv_pow2
};
// The power of two next to 1 / v, of a v that may be 0 or not finite.  A
// complex64 cycle runs on its right-hand side times such a power of the
// residual's norm and its result is divided by it again: every step of a cycle
// is homogeneous, so no digit of the iterates depends on it, and the Gram sums
// of the s-step smoother (squares of unnormalised vectors) stay in the float
// range for residuals of any size (with the residual itself, solves that pass
// below 1e-19 per node took 30 to 60 % more cycles).  rscale[2 rhs] is the
// factor of the right-hand side at hand, rscale[2 rhs + 1] that of the next one,
// from the norm before it.
__device__ __forceinline__ float inv_pow2(double v) {
  const int e = (int)((unsigned long long)__double_as_longlong(v) >> 52 & 0x7ff) - 1023;
  return __uint_as_float((unsigned)(127 - max(-126, min(126, e))) << 23);
}
// 1 / s of such a power of two: its exponent mirrored
__device__ __forceinline__ float rcp_pow2(float s) { return __uint_as_float((254u << 23) - __float_as_uint(s)); }
// Stopping test for one right-hand side, run by the last block of a norm
// reduction: relres = sqrt(sumsq) / ||b||; count != 0 means a cycle has just
// finished.  A RHS that meets tol (state 1) or diverges (state 2: not finite
// or above the threshold) is deactivated.
// gs: the factor that the residual was written with (Ctl::rscale).
__device__ __forceinline__ void stop_update(const Ctl& c, int rhs, double sumsq, int count, float gs = 1.f) {
  const double tol = c.tolp[0], diverge = c.tolp[1];
  const double nrm = sqrt(sumsq), rr = nrm / c.bnorm[rhs];
  c.relres[rhs] = rr;
  if (c.rscale) {
    c.rscale[2 * rhs] = gs;
    c.rscale[2 * rhs + 1] = inv_pow2(nrm);
  }
  if (count) {
    const int cy = ++c.cycles[rhs];
    if (cy <= c.hist_len) c.hist[(long long)rhs * c.hist_len + cy - 1] = rr;
  }
  int st = 0;
  if (!(rr == rr) || rr > diverge) st = 2;
  else if (rr <= tol) st = 1;
  if (st) {
    c.state[rhs] = st;
    c.active[rhs] = 0;
    atomicSub(c.n_active, 1);
  }
}

// ||b - A x|| per RHS with the stopping test fused (count != 0: a cycle just finished).
template <class T> void launch_resnorm_stop(const Grid& g, const OpView<T>& op, const cx<T>* x, const cx<T>* b,
                                            int B, const Ctl& c, int count, cudaStream_t s);
// Mixed path, FP64 outer loop: r = b - A x in FP64, written as float into r32
// (same Grid) times rscale[2 rhs + 1], stopping test fused (resid_march.cu;
// resid_blocks() records per RHS in the partial buffer); and x += e / rscale[2
// rhs] (FP64 += float), masked.
long long resid_blocks(const Grid& g, int B);
void launch_resid_cast_stop(const Grid& g, const OpView<double>& op, const double2* x, const double2* b,
                            float2* r32, int B, const Ctl& c, int count, cudaStream_t s);
void launch_update_mixed(const Grid& g, double2* x, const float2* e, int B, const int* active, const float* rscale,
                         cudaStream_t s);
// out[b] = ||v_b|| (one kernel); rscale: the factors of Ctl::rscale from it.
template <class T> void launch_vecnorm_fin(const Grid& g, const cx<T>* v, int B, double* out, double* partial,
                                           unsigned* tickets, cudaStream_t s, float* rscale = nullptr);
// Transfers (weights xw, Eq. (xex) or linear): r_c = R r_f and x_f += P e_c.
template <class T> void launch_restrict(const Grid& gf, const Grid& gc, const cx<T>* rf, cx<T>* rc, int B,
                                        const int* active, const Xfer& xw, cudaStream_t s);
template <class T> void launch_prolong_add(const Grid& gf, const Grid& gc, const cx<T>* ec, cx<T>* xf, int B,
                                           const int* active, const Xfer& xw, cudaStream_t s);
template <class T> void launch_copy_masked(const Grid& g, const cx<T>* src, cx<T>* dst, int B, const int* active,
                                           cudaStream_t s);
// Dense user array [B][ny+1][nx+1] complex128 <-> padded vector; conj != 0 conjugates.
template <class T> void launch_pack(const Grid& g, const double2* user, cx<T>* v, int B, int conj, cudaStream_t s);
template <class T> void launch_unpack(const Grid& g, const cx<T>* v, double2* user, int B, int conj, cudaStream_t s);
// Coarsest-grid solve with the stored FP64 inverse (setup.cu).
template <class T> void launch_coarse_solve(const Grid& g, const double2* inv, int N, const cx<T>* r, cx<T>* e,
                                            int B, const int* active, cudaStream_t s);

// Setup kernels (setup.cu).  All FP64.
void launch_op0consts(Op0Consts<double>* c64, Op0Consts<float>* c32, double h, double k, double omega,
                      double beta2, int abc, cudaStream_t s);
// Galerkin coarse stencil (radius rc) from the fine operator: fine kind 1 uses
// the matrix-free definition with the CSL shift beta2; kind 2/3 a stored stencil.
void launch_galerkin(const OpView<double>& fine, int fnx, int fny, double2* coarse_st, int cnx, int cny, int rc,
                     double beta2, const Xfer& xw, cudaStream_t s);
void launch_diaginv(const double2* st, int rc, long long plane, double omega, double2* dinv, cudaStream_t s);
void launch_to_float(const double2* src, float2* dst, long long n, cudaStream_t s);
void launch_to_float_real(const double* src, float* dst, long long n, cudaStream_t s);
// 1D factors of the constant-k fine operator (radius 1, rows [n+1][3]):
// g = L1/h^2 - (1 + i beta2) k^2 W1 - i (k/h) B1 (the x factor) when shifted,
// h = L1/h^2 - i (k/h) B1 (the y factor), w = W1.
void launch_factors0(int n, double h, double k, double beta2, double2* g, double2* hf, double2* w, cudaStream_t s);
// 1D Galerkin coarsening X_c = (P1^T / 2) X P1 of a banded [nf+1][2rf+1] row
// array into [nc+1][2rc+1] (nc = nf / 2).
void launch_galerkin_1d(const double2* X, int nf, int rf, double2* Xc, int rc, const Xfer& xw, cudaStream_t s);
// Real parts of a complex row array (the W factors are real).
void launch_real_part(const double2* a, double* b, long long n, cudaStream_t s);
// Per-node 1/(omega * diagonal) of a level operator (any kind).
void launch_diaginv_op(const OpView<double>& op, int nx, int ny, double omega, double2* dinv, cudaStream_t s);
// Dense matrix of a level operator (N = (nx+1)(ny+1) <= 4096) and its inverse.
void launch_dense(const OpView<double>& op, int nx, int ny, double2* M, cudaStream_t s);
void launch_gauss_jordan(double2* M, double2* inv, int N, int* status, cudaStream_t s);
// Per-node stencil export [ny+1][nx+1][2r+1][2r+1] complex128 of a level operator.
void launch_export_stencil(const OpView<double>& op, int nx, int ny, int r, double2* out, cudaStream_t s);

// GMRES(3) smoother (kernels_gmres.cu).  State layout per RHS in `gs`.
struct GmresBufs {
  void* u[3];          // Arnoldi vectors (unnormalised), precision T
  void* w;             // A v_j
  double* partial;     // block partials of the fused reductions
  unsigned* tickets;   // one per RHS, 0 at rest
  double* st;          // per-RHS scalars, see kernels_gmres.cu
  cudaStream_t side;   // optional second stream (with the two events) on
  cudaEvent_t ev_fork; // which the fine level's boundary launches run beside
  cudaEvent_t ev_join; // the interior ones; null: one stream
  double2* outer;      // complex64 level 0 inside the FP64 refinement: the FP64
                       // iterate to which the last smoothing step's result is
                       // added by the fused update (null: none)
  int kron_ch;         // rows per chunk of the Kronecker-level column marches
                       // (0: chosen from the kernel's occupancy)
  int x_zero;          // x is zero on entry: the first step takes b itself as
                       // u0 = b - A x (no apply, no u0 write; b is read-only
                       // in every pass) and only sums |b|^2 for its norm
  float scale, sigma;  // complex64 s-step basis of the level (sstep.cuh)
  const float* rscale; // complex64: Ctl::rscale (the update of outer divides by it)
};
template <class T> void gmres_smooth(const Grid& g, const OpView<T>& op, cx<T>* x, const cx<T>* b, int nu, int B,
                                     const int* active, const GmresBufs& gb, cudaStream_t s);

// The same smoother on the fine level (kind 1), complex128, in four row-marching passes
// plus the update (gmres_march.cu); the partial buffer must hold
// gmres_march_blocks() records per RHS.
long long gmres_march_blocks(const Grid& g, int B);
template <class T> void gmres_smooth_march(const Grid& g, const OpView<T>& op, cx<T>* x, const cx<T>* b, int nu,
                                           int B, const int* active, const GmresBufs& gb, cudaStream_t s);

// The same smoother on the fine level in complex64: two row marches per step
// in s-step form (sstep_march.cu).  x' alternates between x and xt; returns
// the one that holds the result (with gb.outer the last step's result went to
// the FP64 iterate instead).  The partial buffer must hold ss_march_blocks()
// records per RHS.
long long ss_march_blocks(const Grid& g, int B);
float2* gmres_smooth_ss_march(const Grid& g, const OpView<float>& op, float2* x, float2* xt, const float2* b, int nu,
                              int B, const int* active, const GmresBufs& gb, cudaStream_t s);

// The same smoother in complex64 on a level that stores its Krylov vectors, in
// s-step form (sstep_level.cu): Kronecker-form levels as column marches when
// march, all others node-parallel.  want_r: leave r = b - A x in gb.u[0] (not
// with gb.outer).  The partial buffer must hold sl_blocks() and
// kron_march_blocks() records per RHS.
long long sl_blocks(const Grid& g);
void gmres_smooth_ss(const Grid& g, const OpView<float>& op, bool march, float2* x, const float2* b, int nu,
                     bool want_r, int B, const int* active, const GmresBufs& gb, cudaStream_t s);

// The same smoother on a Kronecker-form level (kinds 4, 5), complex128, with
// the kernels that apply A written as column marches (kron_march.cu); the partial buffer
// must hold kron_march_blocks() records per RHS.
long long kron_march_blocks(const Grid& g, int B);
template <class T> void gmres_smooth_kron(const Grid& g, const OpView<T>& op, cx<T>* x, const cx<T>* b, int nu, int B,
                                          const int* active, const GmresBufs& gb, cudaStream_t s);
// r = b - A x on a Kronecker-form level as a column march (the residual that
// the restriction then reads; kron_ch as in GmresBufs).
template <class T> void launch_kron_residual(const Grid& g, const OpView<T>& op, const cx<T>* x, const cx<T>* b,
                                             cx<T>* r, int B, const int* active, int kron_ch, cudaStream_t s);
// A weighted-Jacobi sweep on a Kronecker-form level as a column march.
template <class T> void launch_kron_jacobi(const Grid& g, const OpView<T>& op, const cx<T>* x, const cx<T>* b,
                                           cx<T>* xout, int B, const int* active, int kron_ch, cudaStream_t s);

// Steps of the small levels' part of a cycle, walked by the cooperative
// interpreter (coop.cu).
enum { C_JACOBI = 0, C_GMRES = 1, C_RESTRICT = 2, C_ZERO = 3, C_COARSE = 4, C_PROLONG = 5, C_COPY = 6 };
template <class T> struct CLevel {
  Grid g;
  Xfer xw;                  // transfers between this level and the next
  int kind;                 // as OpView::kind
  Op0Consts<T> c0;
  const T* kf;
  const cx<T>* st;
  const cx<T>* dinv;
  long long plane;
  const cx<T>* gx;
  const T* wx;
  const cx<T>* hy;
  const T* wy;
  cx<T>* b;                 // right-hand side of the level
  cx<T>* r;                 // residual scratch
  cx<T>* u[3];              // GMRES(3) basis (null without GMRES)
  cx<T>* w;
};
struct CStep {
  int op, level, arg, pad;  // arg: GMRES steps
  void* p0;                 // iterate of `level` (in place), or source
  void* p1;                 // destination (Jacobi, copy) or coarse correction (prolong)
};

// Coarse-cycle launch (cluster.cuh): the levels lc..L-1 of one right-hand side
// in the shared memory of a cluster of C blocks, which walks a host-recorded
// list of steps.
constexpr int CL_MAXC = 16;      // blocks per cluster
constexpr int CL_MINROWS = 3;    // rows per block at least (the largest operator radius)
constexpr int CL_NV = 16;        // values of a cluster-wide sum
enum { CL_JACOBI = 0, CL_GMRES = 1, CL_RESTRICT = 2, CL_COARSE = 3, CL_PROLONG = 4 };
struct ClStep {
  int op, level, arg, zero;   // level: counted from lc; arg: sweeps or steps; zero: x is zero on entry
  int left;                   // complex64 GMRES: leave the residual in u0; restriction: it is there
};
template <class T> struct ClLev {
  int nx, ny, n1, rp;         // intervals, nodes per row, rows per block
  int kind;                   // as OpView::kind
  unsigned magic, mrp;        // q / n1 = umulhi(q, magic) for the slab's nodes, j / rp = umulhi(j, mrp) for the rows
  int ox, ob, od;             // shared memory (elements): iterate, right-hand side, inverse diagonal (-1: none)
  int ost;                    // stored stencil of the slab, [(2R+1)^2][rp n1] (-1: read from L2)
  int ogx, owx, ohy, owy;     // Kronecker factors: x rows transposed to [2R+1][n1], the slab's y rows
  T scale, sigma;             // s-step basis (sstep.cuh)
  T w0, w1, w2;               // transfers between this level and the next (Xfer)
  Op0Consts<T> c0;
  const T* kf;
  const cx<T>* st;
  const cx<T>* dinv;
  long long plane;
  const cx<T>* gx;
  const T* wx;
  const cx<T>* hy;
  const T* wy;
};
template <class T> struct ClArgs {
  const ClLev<T>* lev;        // nlev levels, device
  const ClStep* steps;        // device
  int nlev, nsteps, C;
  int x_zero;                 // x is zero on entry (not read)
  int N;                      // coarsest nodes, and the FP64 inverse
  const double2* inv;
  const int* active;
  Grid g;                     // of the first level
  const cx<T>* b;             // its right-hand side and iterate
  cx<T>* x;
  int ou, nu, oX, nX, ored, olev, smem;   // shared memory layout (elements; smem in bytes)
};
// Largest cluster (a power of two, at most CL_MAXC) of which B run at once, so
// that no right-hand side of the handle waits for another's visit to end; 0: none.
// The handles of a ragged batch ask for their own B only: their clusters together
// can be more than the device holds, and then take turns.
template <class T> int cluster_size(int B);
// Fills the layout of levels (nx, ny, kind set) into lv and a; false if a
// slab does not fit in a block's shared memory.
template <class T> bool cluster_layout(std::vector<ClLev<T>>& lv, int C, bool gmres, int N, ClArgs<T>& a);
template <class T> cudaError_t launch_cluster_cycle(const ClArgs<T>& a, int B, cudaStream_t s);

// Cooperative multi-CTA interpreter (coop.cu): the same steps, all blocks of
// the GPU, grid-wide barriers between phases.
constexpr int COOP_THREADS = 256;
constexpr int COOP_MAXLEV = 16;
struct CoopCtl {
  unsigned* bar;          // {arrival count, generation}, zero at rest
  int* err;               // set to 1 when a barrier wait gave up
  long long spin_limit;   // polls per barrier wait
  double* partial;        // [B * bpr][NVMAX] block sums
};
template <class T> int coop_max_blocks(int N);
template <class T> cudaError_t launch_cycle_coop(const CLevel<T>* levels, int nlev, const CStep* steps, int nsteps,
                                                 const double2* inv, int N, const int* active, int B, int grid,
                                                 const CoopCtl& c, cudaStream_t s);

// Fused halo-tile kernels (fused.cu): r_c = R (b - A x) in one pass (any
// level), and up to jacobi_fused_max_nu() fine-level Jacobi sweeps in one pass.
template <class T> void launch_resid_restrict(const Grid& gf, const Grid& gc, const OpView<T>& op, const cx<T>* x,
                                              const cx<T>* b, cx<T>* rc, int B, const int* active, const Xfer& xw,
                                              cudaStream_t s);
template <class T> void launch_jacobi_fused(const Grid& g, const OpView<T>& op, const cx<T>* x, const cx<T>* b,
                                            cx<T>* xo, int nu, int B, const int* active, cudaStream_t s);
int jacobi_fused_max_nu();
cudaError_t configure_fused_kernels();

// Outer iterate of the mixed path in float-float arithmetic (mixed_ff.cu):
// level-0 vectors hold each node as the float4 {re.hi, im.hi, re.lo, im.lo}
// in the space of a complex128 vector.
struct FF {
  float h, l;
};
struct FFConsts {
  FF d, ih2, sb;   // 4/h^2 - k^2, 1/h^2, k/h (constant k)
};
// Constants, and for variable k the per-node diagonal w (4/h^2 - k^2) into dP.
void launch_ff_setup(double h, double k, const double* kf, int nx, int ny, FFConsts* consts, float2* dP,
                     cudaStream_t s);
// r = b - A x in float-float, written as float into r32, stopping test fused.
void launch_ff_resid_cast_stop(const Grid& g, const FFConsts& K, const double* kf, double h, const float2* dP,
                               const void* x, const void* b, float2* r32, int B, const Ctl& c, int count,
                               cudaStream_t s);
// x += e (float-float += float), masked.
void launch_ff_update(const Grid& g, void* x, const float2* e, int B, const int* active, const float* rscale,
                      cudaStream_t s);
void launch_ff_pack(const Grid& g, const double2* user, void* v, int B, int conj, cudaStream_t s);
void launch_ff_unpack(const Grid& g, const void* v, double2* user, int B, int conj, cudaStream_t s);
void launch_ff_norm(const Grid& g, const void* v, int B, double* out, double* partial, unsigned* tickets,
                    float* rscale, cudaStream_t s);

// Flexible GMRES(m) outer loop with one cycle as the right preconditioner
// (fgmres.cu).  V: m+1 basis vectors and Z: m preconditioned vectors, both
// in the cycle's precision; vector q of RHS b at base + q * vlen + b * vstride.
constexpr int FG_MAXM = 32;
// Per-RHS FP64 scalars of the restart cycle: the rotated Hessenberg columns
// (column j, row i), the Gram matrix of V (row a, column b: <v_a, v_b>), the
// rotations (cs real, sn complex), g, y, beta and the scales s_j of the
// unnormalised basis (v_j = s_j u_j); complex values as (re, im).
struct FgLayout {
  int m;
  __host__ __device__ int h(int j, int i) const { return 2 * (j * (m + 1) + i); }
  __host__ __device__ int gram(int a, int b) const { return 2 * m * (m + 1) + 2 * (a * (m + 1) + b); }
  __host__ __device__ int cs(int i) const { return 2 * m * (m + 1) + 2 * (m + 1) * (m + 1) + i; }
  __host__ __device__ int sn(int i) const { return cs(m) + 2 * i; }
  __host__ __device__ int g(int i) const { return sn(m) + 2 * i; }
  __host__ __device__ int y(int i) const { return g(m + 1) + 2 * i; }
  __host__ __device__ int beta() const { return y(m); }
  __host__ __device__ int s(int j) const { return beta() + 1 + j; }
  __host__ __device__ int size() const { return s(m + 1); }
};
struct FgArgs {
  Grid g;                  // fine level
  Op0Consts<double> c0;    // fine operator (FP64: restart residual)
  const double* kf;
  Op0Consts<float> c0f;    // and in FP32 (Arnoldi passes of the mixed path)
  const float* kf32;
  int B, m;
  int nbr, ncx, ns, nvp;   // blocks per RHS, strip columns, strips, values per partial record
  long long vlen;          // g.vstride * B
  void* V;
  void* Z;
  double2* X;
  const double2* b;
  double* S;               // [B][sd] scalars (FgLayout)
  int sd;
  int* kst;                // [B][2]: steps of the current restart cycle, steps allowed in it
  int* active;             // 1 while the RHS is inside a restart cycle
  int* state;              // 0 running, 1 converged, 2 not finite
  int* cycles;             // preconditioner applications
  double* relres;          // true relative residual at the last restart
  double* hist;            // residual estimate after every application
  int hist_len;
  int* n_active;
  const double* bnorm;
  double tol;
  int max_cycles;
  double* partial;         // [B][nvp][nbr]
  unsigned* tickets;       // [B], 0 at rest
  float* rscale;           // complex64 cycles: as Ctl::rscale, of the cycle's right-hand side
};
// Strip geometry and blocks per RHS (nbr, ncx, ns, nvp) for a fine grid.
void fg_geometry(const Grid& g, int B, bool fp64z, FgArgs& a);
// cb, cxv: the cycle's level-0 right-hand side and iterate (the restart and
// orth passes write the next basis vector into cb and zero cxv).
template <class T> void launch_fg_restart(const FgArgs& a, cx<T>* cb, cx<T>* cxv, cudaStream_t s);
template <class T> void launch_fg_dots(const FgArgs& a, int j, const cx<T>* z, cudaStream_t s);
template <class T> void launch_fg_orth(const FgArgs& a, int j, cx<T>* cb, cx<T>* cxv, cudaStream_t s);
template <class T> void launch_fg_update(const FgArgs& a, cudaStream_t s);

// Dense two-grid analysis of the two finest levels (analysis.cu).  out[0] =
// ||T0||_2, out[1] = 1 if Gamma~ is Hermitian positive definite, out[2] =
// ||Gamma~||_1 / kappa_1(Gamma~), out[3] = power iterations, out[4] = 1 if
// the power method met its stopping test, out[5] = 1 if A_1 was singular.
cudaError_t two_grid_analysis(const OpView<double>& fine, const OpView<double>& coarse, int fnx, int fny, int cnx,
                              int cny, double omega, const Xfer& xw, int nu, int max_iter, double* out,
                              cudaStream_t s);

// Gradient of the receiver misfit (kernels_level.cu).
void launch_gradient(int nx, int ny, double h, const double* m, double omega_f, const double2* u,
                     const double2* lam, int nsrc, double* g, cudaStream_t s);

inline int cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

// Sets the message mg_last_error() returns on this host thread (capi.cu).
void hmg_set_error(const char* msg);

}  // namespace hmg
