// Device helpers shared by the libmrcm kernels.
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace mrcm {

// Raises kernel K's dynamic shared-memory limit to the device maximum, once per kernel and
// process (thread-safe).  Launches then pass their own size: the limit only gates launches and
// does not change occupancy, and a limit that never moves cannot be lowered by another thread
// between its own set and launch (request workers launch the same kernels with different sizes).
template <auto K>
cudaError_t raise_smem_limit() {
  static const cudaError_t err = [] {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, K);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    return e;
  }();
  return err;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over a block (blockDim.x multiple of 32, <= 1024).  Every thread receives the total.
// Deterministic: fixed order for a fixed block size.
__device__ __forceinline__ double block_sum(double v, double* smem32) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) smem32[wid] = v;
  __syncthreads();
  const int nw = blockDim.x >> 5;
  double t = lane < nw ? smem32[lane] : 0.0;
  t = warp_sum(t);
  return t;
}

// Grid-wide deterministic reduction of NV values per thread.  Each block writes its partial sums
// to partials[v * gridDim.x + blockIdx.x]; the last block to finish (atomic ticket) adds the
// partials in block order and writes *outs[v] (the square root for entries with the sqrt bit set
// in sqrt_mask); the ticket counter is reset for the next launch.
template <int NV>
__device__ __forceinline__ void grid_reduce(double (&v)[NV], double* partials, unsigned* counter,
                                            double* const (&outs)[NV], double* smem32, int sqrt_mask = 0) {
  __shared__ bool last;
  for (int k = 0; k < NV; ++k) {
    double t = block_sum(v[k], smem32);
    if (threadIdx.x == 0) partials[k * gridDim.x + blockIdx.x] = t;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned ticket = atomicAdd(counter, 1u);
    last = (ticket == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int k = 0; k < NV; ++k) {
    double acc = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
      acc += *((volatile double*)&partials[k * gridDim.x + b]);
    double t = block_sum(acc, smem32);
    if (threadIdx.x == 0) *outs[k] = ((sqrt_mask >> k) & 1) ? sqrt(t) : t;
  }
  if (threadIdx.x == 0) *counter = 0u;
}

// Two-point-flux pieces (Sec. 3): half transmissibility tau = 2 K |f| / h_a.
__device__ __forceinline__ double half_trans(double k, double area, double ha) { return 2.0 * k * area / ha; }

// Robin face coefficient t_R = (1/tau_in + beta/|f|)^-1, beta = alpha H / K_H (Eq. 5-6).
__device__ __forceinline__ double robin_tr(double k_in, double k_out, double area, double ha, double Hs,
                                           double alpha, double* beta_out, double* tau_out) {
  const double tau = half_trans(k_in, area, ha);
  const double kh = 2.0 * k_in * k_out / (k_in + k_out);
  const double beta = alpha * Hs / kh;
  if (beta_out) *beta_out = beta;
  if (tau_out) *tau_out = tau;
  return 1.0 / (1.0 / tau + beta / area);
}

// The five-point operator (A v)_c = sum over the four faces of T_f (v_c - v_c') (no flow into cells outside
// the grid, whose v is 0: a boundary face contributes T_f v_c), applied by a march down columns: a warp
// takes 31 columns (its first lane holds the column to their left) and the rows [j0, j1), and each face
// difference is formed once, for the cell on either side of it: the x difference goes to the next lane
// by a shuffle, the y difference is kept for the next row.  emit(cell, base, s) gets, for each cell, the
// face sum folded into base(cell) as base + sign * A v, in the order east, west, north, south.
//
// Bound by the FP64 pipe (1.6 operations a clock and SM), so what counts is FP64 instructions per cell:
// two subtractions and four FMAs here, against four and five with every cell forming its own four
// differences.  2048^2 cells: 73.8 -> 57.4 us (51 at the pipe's rate, 20 of HBM traffic).
// Rows come in groups of STENCIL_ROWS whose loads are all in flight together.
constexpr int STENCIL_ROWS = 4;
constexpr int STENCIL_COLS = 31;

template <int SIGN, class Base, class Emit>
__device__ __forceinline__ void stencil_march(const Geo& g, const double* __restrict__ v, int col0, int j0, int j1,
                                              Base base, Emit emit) {
  const int lane = threadIdx.x & 31, i = col0 + lane - 1;
  const bool in = i >= 0 && i < g.nx, own = in && lane > 0;
  auto at = [&](int j) { return in && j >= 0 && j < g.ny ? v[(size_t)j * g.nx + i] : 0.0; };
  double vc = at(j0), ds = at(j0 - 1) - vc, Ts = own ? g.Ty[(size_t)j0 * g.nx + i] : 0.0;
  for (int j = j0; j < j1; j += STENCIL_ROWS) {
    double vn[STENCIL_ROWS], vr[STENCIL_ROWS], Tw[STENCIL_ROWS], Te[STENCIL_ROWS], Tn[STENCIL_ROWS], b[STENCIL_ROWS];
#pragma unroll
    for (int q = 0; q < STENCIL_ROWS; ++q) {
      const bool on = own && j + q < j1;
      vn[q] = j + q < j1 ? at(j + q + 1) : 0.0;
      vr[q] = on && lane == 31 && i + 1 < g.nx ? v[(size_t)(j + q) * g.nx + i + 1] : 0.0;
      const double* Tx = g.Tx + (size_t)(j + q) * (g.nx + 1) + i;
      Tw[q] = on ? Tx[0] : 0.0;
      Te[q] = on ? Tx[1] : 0.0;
      Tn[q] = on ? g.Ty[(size_t)(j + q + 1) * g.nx + i] : 0.0;
      b[q] = on ? base((size_t)(j + q) * g.nx + i) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < STENCIL_ROWS; ++q) {
      const double right = __shfl_down_sync(0xffffffffu, vc, 1);
      const double de = vc - (lane == 31 ? vr[q] : right);
      const double dw = __shfl_up_sync(0xffffffffu, de, 1);   // v_west - v_c
      const double dn = vc - vn[q];
      double s = fma(SIGN * Te[q], de, b[q]);
      s = fma(-SIGN * Tw[q], dw, s);
      s = fma(SIGN * Tn[q], dn, s);
      s = fma(-SIGN * Ts, ds, s);
      if (own && j + q < j1) emit((size_t)(j + q) * g.nx + i, s);
      ds = dn;
      vc = vn[q];
      Ts = Tn[q];
    }
  }
}
// The same for one cell alone, base + SIGN A v in the same order (bit for bit the march's)
template <int SIGN>
__device__ __forceinline__ double face_sum(const Geo& g, const double* __restrict__ v, int i, int j, double base) {
  const size_t c = (size_t)j * g.nx + i;
  const double vc = v[c];
  const double vw = i > 0 ? v[c - 1] : 0.0;
  const double ve = i < g.nx - 1 ? v[c + 1] : 0.0;
  const double vs = j > 0 ? v[c - g.nx] : 0.0;
  const double vn = j < g.ny - 1 ? v[c + g.nx] : 0.0;
  const double* Tx = g.Tx + (size_t)j * (g.nx + 1) + i;
  const double* Ty = g.Ty + c;
  double s = fma(SIGN * Tx[1], vc - ve, base);
  s = fma(SIGN * Tx[0], vc - vw, s);
  s = fma(SIGN * Ty[g.nx], vc - vn, s);
  return fma(SIGN * Ty[0], vc - vs, s);
}
__device__ __forceinline__ double apply_A(const Geo& g, const double* __restrict__ v, int i, int j) {
  return face_sum<1>(g, v, i, j, 0.0);
}

// Launch shape of a kernel of 128-thread blocks that march `rows` rows per warp (blockIdx.y).  Long marches
// where they still give every SM a dozen warps (2 M cells), short ones below, and none (one thread per
// cell, apply_A) below half a million cells, where a launch is bound by latency: there a march of 16 or
// 4 rows took 2 to 4 us more than a thread per cell (two launches at 512^2: 21.3 against 17.3 us).
inline bool stencil_marches(int nx, int ny) { return (size_t)nx * ny >= (size_t)1 << 19; }
inline int stencil_rows(int nx, int ny) { return (size_t)nx * ny >= (size_t)1 << 21 ? 16 : STENCIL_ROWS; }
inline dim3 stencil_grid(int nx, int ny) {
  const int cols = 4 * STENCIL_COLS, rows = stencil_rows(nx, ny);
  return dim3((nx + cols - 1) / cols, (ny + rows - 1) / rows);
}
__device__ __forceinline__ int stencil_col0() { return (blockIdx.x * 4 + (threadIdx.x >> 5)) * STENCIL_COLS; }

// Grid-wide barrier for cooperative launches (every block co-resident).  bar[0] counts arrivals
// (zero between barriers), bar[1] is the generation.  A block that polls more than
// BARRIER_SPIN_LIMIT times sets FLAG_TIMEOUT in *flags and returns false instead of waiting on.

// Returns false if the wait gave up (the flag is set; the caller returns).
__device__ __forceinline__ bool grid_barrier(unsigned* bar, int* flags) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = bar + 1;
    const unsigned my = *gen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u);
    s_ok = 1;
    if (arrived == gridDim.x - 1) {
      bar[0] = 0u;
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      long long spins = 0;
      while (*gen == my) {
        if (++spins > BARRIER_SPIN_LIMIT) {
          atomicOr(flags, FLAG_TIMEOUT);
          s_ok = 0;
          break;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
  return s_ok != 0;
}

}  // namespace mrcm
