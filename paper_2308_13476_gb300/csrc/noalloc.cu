// mg_residual_norm_static: the fine-level residual norm without any device
// allocation.
//
// Every other entry point of this library works through a handle whose
// mg_setup allocates device memory, and the norm reductions inside them
// keep their block partials in that memory.  Some callers cannot allocate
// device memory at the point where they need a residual: code that runs
// while another framework's memory pool owns the device (its caching
// allocator has reserved what it needs and raw allocations would fight it or
// fail), code on a latency-critical loop where an allocation's implicit
// device-wide synchronisation is not acceptable, or code in a context where
// allocation is simply not permitted.  This entry point keeps its scratch (the
// per-block partial sums and the completion ticket) in one file-scope device
// array instead, sized for a fixed maximum number of thread blocks.
//
// Set-up: the first call on each device looks up the array's device address
// with cudaGetSymbolAddress (the array's name in host code is only a host-side
// stand-in, not a device address) and caches it; make that first call on a
// device before any stream capture.  Calls share the array and it keeps the
// last call's contents, so each call clears its ticket first; calls whose
// kernels overlap on the GPU (different streams, or different host threads
// on the same device) race on the array and must be serialised by the caller.
#include <mutex>

#include "../../include/helmmg.h"
#include "internal.h"

namespace hmg {

namespace {
constexpr int NA_TILE = 32;                           // grids are accepted by their count of 32 x 32 tiles
constexpr int NA_MAX_BLOCKS = 16384;                  // -> at most 16.7 M nodes
constexpr int NA_NT = 256;                            // threads per block
constexpr int NA_RESIDENT = 6;                        // blocks of the one-node form that run at once on an SM
constexpr int NA_MAX_DEVICES = 64;
}  // namespace

// [blk][2] partial sums (|r|^2, |b|^2) followed by the ticket; 256 KiB + 256 B.
static __device__ __align__(256) double g_noalloc_scratch[2 * NA_MAX_BLOCKS + 32];

// The norms on the caller's dense [ny+1][nx+1] layout, RY nodes per thread: a
// block takes RY * 256 consecutive nodes, so that no thread is left without
// one at the grid's right edge.
//
// What bounds it is the FP64 pipe (two multiply-adds per clock and SM), so an
// interior node costs 14 FP64 instructions: b - d x + (1/h^2) (E + W + N + S)
// with d = 4/h^2 - k^2, five per component, and two for each norm.  Edge rows
// and columns take the operator of the solver (Op0::apply5) on zero off the
// grid.  One node per thread while all blocks run at once: the pipe is then
// evenly loaded and every load is in flight; above that four, for fewer
// records in the last block.  Per call, 32 x 32-node tiles with 35 FP64
// instructions per node -> this form: 257^2 18.7 -> 12.4 us (most of it the
// launches of the clear and the kernel), 513^2 29 -> 20.6 us, 1001^2 82 -> 43
// us, 2001^2 287 -> 136 us.
template <int RY, bool VK>
__global__ void __launch_bounds__(NA_NT) k_resnorm_dense(const __grid_constant__ Op0<double> op, int nodes, double dc,
                                                         const double2* __restrict__ x, const double2* __restrict__ b,
                                                         double* scratch, double* __restrict__ out) {
  __shared__ double sh[2 * NA_NT / 32];
  __shared__ int s_last;
  const int nx = op.nx, ny = op.ny, n1 = nx + 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nblk = gridDim.x, blk = blockIdx.x;
  const double ih2 = op.c.inv_h2;
  double v[2] = {0.0, 0.0};
#pragma unroll
  for (int r = 0; r < RY; ++r) {
    const int q = (blk * RY + r) * NA_NT + tid;
    if (q >= nodes) break;
    const int j = q / n1, i = q - j * n1;
    const double2 xp = x[q], bq = b[q], z = make_double2(0.0, 0.0);
    const double2 xe = i < nx ? x[q + 1] : z, xw = i > 0 ? x[q - 1] : z;
    const double2 xn = j < ny ? x[q + n1] : z, xs = j > 0 ? x[q - n1] : z;
    double2 t;
    if (i > 0 && i < nx && j > 0 && j < ny) {
      double d = dc;
      if constexpr (VK) {
        const double k = op.kf[q];
        d = fma(-k, k, 4.0 * ih2);
      }
      t.x = fma(ih2, (xe.x + xw.x) + (xn.x + xs.x), fma(-d, xp.x, bq.x));
      t.y = fma(ih2, (xe.y + xw.y) + (xn.y + xs.y), fma(-d, xp.y, bq.y));
    } else {
      t = sub<double>(bq, op.apply5(xp, xe, xw, xn, xs, i, j));
    }
    v[0] = fma(t.x, t.x, fma(t.y, t.y, v[0]));
    v[1] = fma(bq.x, bq.x, fma(bq.y, bq.y, v[1]));
  }
  // both sums of the block in threads 0 and 16 (FP64 adds: 6 per warp, then one per warp)
  auto block_sums = [&](double (&a)[2]) {
    const double t = lane_sum<2, double>(a, lane);
    if ((lane & 15) == 0) sh[lane_value<2>(lane) * (NA_NT / 32) + warp] = t;
    __syncthreads();
    double s = 0.0;
    if (warp == 0 && (lane & 15) == 0) {
#pragma unroll
      for (int w = 0; w < NA_NT / 32; ++w) s += sh[lane_value<2>(lane) * (NA_NT / 32) + w];
    }
    return s;
  };
  const bool own = warp == 0 && (lane & 15) == 0;
  const double s = block_sums(v);
  unsigned* ticket = reinterpret_cast<unsigned*>(scratch + 2 * NA_MAX_BLOCKS);
  if (own) {
    scratch[2 * blk + lane_value<2>(lane)] = s;
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(ticket, 1u) == (unsigned)(nblk - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a[2] = {0.0, 0.0};
  for (int q = tid; q < nblk; q += NA_NT) {
    const double2 p = __ldcg(reinterpret_cast<const double2*>(scratch) + q);
    a[0] += p.x;
    a[1] += p.y;
  }
  const double total = block_sums(a);
  if (own) out[lane_value<2>(lane)] = sqrt(total);
  if (tid == 0) *ticket = 0u;
}

}  // namespace hmg

using namespace hmg;

static std::mutex g_noalloc_mu;
static double* g_noalloc_ptr[NA_MAX_DEVICES] = {};

extern "C" mg_status mg_residual_norm_static(int nx, int ny, double h, const double* k_field, double k_const,
                                             const void* x, const void* b, double* out, void* stream) {
  if (nx < 2 || ny < 2 || !(h > 0) || !x || !b || !out || (!k_field && !(k_const >= 0))) {
    hmg_set_error("mg_residual_norm_static: need nx, ny >= 2, h > 0, k >= 0 and non-NULL x, b, out");
    return MG_EINVAL;
  }
  const long long nbx = cdiv(nx + 1LL, NA_TILE), nby = cdiv(ny + 1LL, NA_TILE);
  if (nbx * nby > NA_MAX_BLOCKS) {
    hmg_set_error("mg_residual_norm_static: grid too large for the static scratch (at most 16384 blocks of 32 x 32 "
                  "nodes, about 16.7 M nodes)");
    return MG_EINVAL;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) {
    hmg_set_error("mg_residual_norm_static: no usable current device");
    return MG_ECUDA;
  }
  double* scratch;
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {   // once per device: the array's device address
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p) {
        hmg_set_error("mg_residual_norm_static: cudaGetSymbolAddress failed");
        return MG_ECUDA;
      }
      g_noalloc_ptr[dev] = (double*)p;
    }
    scratch = g_noalloc_ptr[dev];
  }
  cudaStream_t s = (cudaStream_t)stream;
  e = cudaMemsetAsync(scratch + 2 * NA_MAX_BLOCKS, 0, sizeof(unsigned), s);   // ticket starts at zero
  if (e != cudaSuccess) {
    hmg_set_error("mg_residual_norm_static: clearing the ticket failed");
    return MG_ECUDA;
  }
  const int nodes = (nx + 1) * (ny + 1);   // at most 2^24 here
  Op0<double> op{};
  op.c.inv_h2 = 1.0 / (h * h);
  op.c.inv_h = 1.0 / h;
  op.c.k = k_field ? 0.0 : k_const;
  op.kf = k_field;
  op.nx = nx;
  op.ny = ny;
  const double dc = 4.0 * op.c.inv_h2 - op.c.k * op.c.k;
  const double2 *xv = (const double2*)x, *bv = (const double2*)b;
  auto launch = [&](auto kern, int ry) { kern<<<cdiv(nodes, NA_NT * ry), NA_NT, 0, s>>>(op, nodes, dc, xv, bv, scratch, out); };
  if (cdiv(nodes, NA_NT) <= NA_RESIDENT * device_sms()) launch(k_field ? k_resnorm_dense<1, true> : k_resnorm_dense<1, false>, 1);
  else launch(k_field ? k_resnorm_dense<4, true> : k_resnorm_dense<4, false>, 4);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    hmg_set_error("mg_residual_norm_static: kernel launch failed");
    return MG_ECUDA;
  }
  return MG_OK;
}
