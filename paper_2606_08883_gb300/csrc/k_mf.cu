// Coupling system of MRCM-O (Eq. 13-14) by a multifrontal LU over a nested dissection of the
// subdomain grid, without row interchanges.
//
// Each interface carries 2 nq unknowns and the 2 nq rows homed at them (flux and pressure rows),
// and a row couples the unknowns of the one or two subdomains it joins, so a rectangle of
// subdomains whose interior interfaces are eliminated leaves couplings only among the interfaces of
// its boundary.  The host plan (plan.cpp) cuts the grid recursively; a front eliminates the
// separator of its rectangle (or every interior interface of a leaf rectangle).  With the front
// F = [F11 F12; F21 F22] (pivot unknowns P first, boundary unknowns U after),
//   F11^-1 (Gauss-Jordan without pivoting),  D = F11^-1 F12,  B = F21 F11^-1,
//   S = F22 - F21 D  (added into the parent front),
// and a solve of G x = g runs forward through the levels, v_P = g_P + children's w, w_U = v_U - B v_P,
// then backward, x_P = F11^-1 v_P - D x_U.  Every product has a fixed order, so the solution is
// deterministic.  A zero or non-finite pivot, or |S| above NOPIV_MAX_GROWTH max |G|, sets
// FLAG_NOPIV_REJECTED and the caller falls back to the pivoted band LU of k_coarse.cu.
#include <algorithm>

#include <cooperative_groups.h>

#include "common.cuh"

namespace mrcm {

constexpr int MF_THREADS = 256;
constexpr int MF_GJ_CL = 8;          // CTAs of the cluster that inverts a large pivot block
constexpr int MF_GJ_CLUSTER_NP = 64; // pivot blocks this large (and divisible by MF_GJ_CL) use it

// Magnitudes as bit patterns (those of non-negative doubles order like the values; anything not finite counts
// as +inf), compared as integers: FP64 compares, like FP64 negations, take the FP64 pipe.
__device__ __forceinline__ unsigned long long mag(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
  return b < 0x7ff0000000000000ULL ? b : 0x7ff0000000000000ULL;
}
__device__ __forceinline__ bool nonzero_finite(double d) {
  const unsigned long long b = mag(d);
  return b != 0 && b != 0x7ff0000000000000ULL;
}
// -v by its sign bit
__device__ __forceinline__ double flip_sign(double v) {
  return __hiloint2double(__double2hiint(v) ^ (int)0x80000000, __double2loint(v));
}
// the largest magnitude across the CTA into a maximum in global memory
__device__ __forceinline__ void cta_max_to(unsigned long long v, unsigned long long* dst) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
    v = u > v ? u : v;
  }
  if ((threadIdx.x & 31) == 0 && v) atomicMax(dst, v);
}

// One MF_TILE x MF_TILE tile of C (rows x cols of it) = (acc ? C : 0) + alpha A (rows x K) B (K x cols),
// row-major operands with leading dimensions in global memory, one output per thread of the CTA; both
// operands are staged in shared memory (sm: MF_TILE (2 K + 1) + K doubles).  Each output is one sum in
// increasing k.  Returns the magnitude of the entry written.
__device__ unsigned long long cta_tile(int rows, int cols, int K, const double* A, int lda, const double* B, int ldb, double* C, int ldc,
                           double alpha, bool acc, double* sm) {
  double* As = sm;                            // [MF_TILE][K + 1]
  double* Bs = sm + MF_TILE * (K + 1);        // [K][MF_TILE]
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int r = wid; r < MF_TILE; r += MF_THREADS / 32)
    for (int k = lane; k < K; k += 32) As[r * (K + 1) + k] = r < rows ? A[(size_t)r * lda + k] : 0.0;
  for (int t = tid; t < K * MF_TILE; t += MF_THREADS) {
    const int k = t / MF_TILE, c = t % MF_TILE;
    Bs[t] = c < cols ? B[(size_t)k * ldb + c] : 0.0;
  }
  const int r = tid / MF_TILE, c = tid % MF_TILE;
  const bool on = r < rows && c < cols;
  const double old = on && acc ? C[(size_t)r * ldc + c] : 0.0;
  __syncthreads();
  double s = 0.0;
  for (int k = 0; k < K; ++k) s = fma(As[r * (K + 1) + k], Bs[k * MF_TILE + c], s);
  const double v = fma(alpha, s, old);
  if (on) C[(size_t)r * ldc + c] = v;
  return on ? mag(v) : 0ULL;
}

__device__ __forceinline__ unsigned long long* mf_stats(const MfDev& m) {
  return reinterpret_cast<unsigned long long*>(m.scr + 2);
}

// Gauss-Jordan inversion in registers of np rows by nc columns [c0, c0 + nc) of the pivot block (entry
// t = thread + MF_THREADS r of the nc-wide rows; pivot k takes the scaled row r_j = a_kj / a_kk and the column
// c_i = a_ik, then a_ij -= c_i r_j off row and column k, row k = r_j, column k = -c_i / a_kk, a_kk = 1 / a_kk).  The
// column is published by the step before, over the whole block, the row by this CTA.  Bound by the FP64 pipe of its
// SM: an update is one FMA per entry with every lane busy, the division and the scaled row and column cost a handful
// per warp, and the column is published with its sign flipped by an integer operation because an FP64 negation per
// entry is an FP64 instruction too.
template <int R>
struct GjBlock {
  double a[R];
  int ij[R];   // row << 8 | column; unused entries: the spare slot (np, nc)
  int nr;      // rounds with entries
  __device__ __forceinline__ void load(const double* F, int f, int np, int nc) {
    const int di = MF_THREADS / nc, dj = MF_THREADS - di * nc;
    int i = threadIdx.x / nc, j = threadIdx.x - i * nc;
    nr = (np * nc + MF_THREADS - 1) / MF_THREADS;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool on = i < np;
      ij[r] = on ? i << 8 | j : np << 8 | nc;
      a[r] = on ? F[(size_t)i * f + j] : 0.0;
      i += di;
      j += dj;
      if (j >= nc) {
        j -= nc;
        ++i;
      }
    }
  }
  __device__ __forceinline__ void store(double* F, int f, int np) const {
#pragma unroll
    for (int r = 0; r < R; ++r)
      if ((ij[r] >> 8) < np) F[(size_t)(ij[r] >> 8) * f + (ij[r] & 255)] = a[r];
  }
  // row and column k, this one negated (own column kc, or none if outside), into the published arrays
  __device__ __forceinline__ void publish(int k, int kc, double* row, double* col) const {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = ij[r] >> 8, j = ij[r] & 255;
      if (i == k) row[j] = a[r];
      if (j == kc) col[i] = flip_sign(a[r]);
    }
  }
  // pivot k with nc (the column, negated), w (nc times rp), rowr (the row times rp) and rp (1 / pivot); publishes row
  // and column k + 1
  __device__ __forceinline__ void pivot(int k, int kc, const double* nc, const double* w, const double* rowr, double rp,
                                        double* next_row, double* next_col) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r >= nr) break;
      const int i = ij[r] >> 8, j = ij[r] & 255;
      double v = fma(nc[i], rowr[j], a[r]);
      if (i == k) v = j == kc ? rp : rowr[j];
      else if (j == kc) v = w[i];
      a[r] = v;
      if (i == k + 1) next_row[j] = v;
      if (j == kc + 1) next_col[i] = flip_sign(v);
    }
  }
};

// The children's Schur complements into the fronts of a level, a row of F per warp: entry (i, j) is the sum over
// the children that hold both unknowns (their message slots say which and where), 0 elsewhere.  With one CTA per
// front adding its children entry by entry, the upper levels' assembly alone took 25 to 45 us each.
__global__ void __launch_bounds__(MF_THREADS) k_mf_gather(MfDev m, int first) {
  const MfFront fr = m.fr[m.order[first + blockIdx.x]];
  const int f = fr.np + fr.nu, i = blockIdx.y * (MF_THREADS / 32) + (threadIdx.x >> 5);
  if (i >= f) return;
  const int2 si = m.inv[fr.io + i];
  const double* S[2] = {nullptr, nullptr};   // row of the child's S that belongs to row i
  int wo[2] = {0, 0};
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int slot = c == 0 ? si.x : si.y;
    if (c < fr.nch && slot >= 0) {
      const MfFront cf = m.fr[fr.ch[c]];
      const int fc = cf.np + cf.nu;
      wo[c] = cf.wo;
      S[c] = m.F + cf.fo + (size_t)(cf.np + slot - cf.wo) * fc + cf.np;
    }
  }
  double* row = m.F + fr.fo + (size_t)i * f;
#pragma unroll 4
  for (int j = threadIdx.x & 31; j < f; j += 32) {
    const int2 sj = m.inv[fr.io + j];
    double v = S[0] && sj.x >= 0 ? S[0][sj.x - wo[0]] : 0.0;
    if (S[1] && sj.y >= 0) v += S[1][sj.y - wo[1]];
    row[j] = v;
  }
}

// The entry of a child's S that belongs to its message slots (row, column)
__device__ __forceinline__ double schur_entry(const MfDev& m, const MfFront& ch, int row, int col) {
  const int fc = ch.np + ch.nu;
  return m.F[ch.fo + (size_t)(ch.np + row - ch.wo) * fc + ch.np + col - ch.wo];
}

// One CTA per front of a level: the original entries of the pivot rows and columns, and F11^-1 of the blocks that
// one CTA inverts.
template <int R>
__global__ void __launch_bounds__(MF_THREADS) k_mf_front(MfDev m, const double* __restrict__ ab, int first,
                                                         int* flags) {
  extern __shared__ __align__(16) double smd[];
  const int fid = m.order[first + blockIdx.x];
  const MfFront fr = m.fr[fid];
  const int np = fr.np, nu = fr.nu, f = np + nu;
  double* __restrict__ F = m.F + fr.fo;
  // the original entries with the children's (k_mf_gather), in batches of AB per thread, every load of a batch
  // issued before its stores (the positions are distinct).  An entry is (original + first child) + second child:
  // where both children have one, they are read again and added in that order.
  constexpr int AB = 8;
  MfFront ch[2] = {};
  for (int c = 0; c < 2; ++c)
    if (fr.nch == 2) ch[c] = m.fr[fr.ch[c]];
  unsigned long long amax = 0;
  for (int t0 = threadIdx.x; t0 < fr.na; t0 += AB * MF_THREADS) {
    int dst[AB];
    double v[AB], o[AB], o2[AB];
#pragma unroll
    for (int e = 0; e < AB; ++e) {
      const int t = t0 + e * MF_THREADS;
      dst[e] = -1;
      v[e] = o[e] = o2[e] = 0.0;
      if (t < fr.na) {
        const int2 p = m.asmv[fr.ao + t];
        dst[e] = p.x;
        v[e] = ab[p.y];
        bool both = false;
        if (fr.nch == 2) {
          const int2 si = m.inv[fr.io + p.x / f], sj = m.inv[fr.io + p.x % f];
          both = si.x >= 0 && sj.x >= 0 && si.y >= 0 && sj.y >= 0;
          if (both) {
            o[e] = schur_entry(m, ch[0], si.x, sj.x);
            o2[e] = schur_entry(m, ch[1], si.y, sj.y);
          }
        }
        if (!both) o[e] = F[p.x];
      }
    }
#pragma unroll
    for (int e = 0; e < AB; ++e)
      if (dst[e] >= 0) {
        F[dst[e]] = (v[e] + o[e]) + o2[e];
        const unsigned long long b = mag(v[e]);
        amax = b > amax ? b : amax;
      }
  }
  cta_max_to(amax, mf_stats(m));
  __syncthreads();
  // F12 aside: the tiles of D = F11^-1 F12 overwrite it while others still read it
  double* Fc = F + (size_t)f * f + (size_t)nu * np;
  for (int i = threadIdx.x >> 5; i < np; i += MF_THREADS / 32)
    for (int j = threadIdx.x & 31; j < nu; j += 32) Fc[(size_t)i * nu + j] = F[(size_t)i * f + np + j];
  if (np >= MF_GJ_CLUSTER_NP && np % MF_GJ_CL == 0) return;   // F11^-1 by k_mf_gj_cluster
  // F11^-1 (at most R MF_THREADS entries: the launcher picks R by the level's largest block)
  const int tid = threadIdx.x;
  double* row = smd;                      // [2][np + 1] row k, double-buffered
  double* col = row + 2 * (np + 1);       // [2][np + 1] column k, negated
  double* w = col + 2 * (np + 1);         // [np + 1] column k / pivot (both negated)
  double* rowr = w + np + 1;              // [np + 1] row k / pivot
  double* s_r = rowr + np + 1;            // 1 / pivot
  for (int t = tid; t < 6 * (np + 1); t += MF_THREADS) smd[t] = 0.0;
  GjBlock<R> blk;
  blk.load(F, f, np, np);
  __syncthreads();
  blk.publish(0, 0, row, col);
  __syncthreads();
  bool bad = false;
  for (int k = 0; k < np; ++k) {
    const int c = (k & 1) * (np + 1), n = np + 1 - c;
    if (tid < np) {
      double d = flip_sign(col[c + k]);
      if (!nonzero_finite(d)) {
        bad = true;
        d = 1.0;
      }
      const double r = 1.0 / d;
      w[tid] = col[c + tid] * r;
      rowr[tid] = row[c + tid] * r;
      if (tid == 0) *s_r = r;
    }
    __syncthreads();
    blk.pivot(k, k, col + c, w, rowr, *s_r, row + n, col + n);
    __syncthreads();
  }
  blk.store(F, f, np);
  if (bad) atomicOr(flags, FLAG_NOPIV_REJECTED);
}

// F11^-1 of a large pivot block by the same Gauss-Jordan steps, over a cluster of MF_GJ_CL CTAs:
// CTA q keeps columns [q cw, (q + 1) cw) of F11 in its registers (cw = np / MF_GJ_CL); per pivot the
// owner of column k has published it (double-buffered), one cluster barrier, every CTA reads it through
// distributed shared memory, scales it and updates its columns.  Entry by entry the arithmetic is that of
// the one-CTA form.  One cluster per front of the level; fronts too small for it return at once.
__global__ void __launch_bounds__(MF_THREADS, 1) k_mf_gj_cluster(MfDev m, int first, int* flags) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) double smd[];
  const int q = (int)cl.block_rank();
  const int fid = m.order[first + blockIdx.x / MF_GJ_CL];
  const MfFront fr = m.fr[fid];
  const int np = fr.np, f = fr.np + fr.nu;
  if (np < MF_GJ_CLUSTER_NP || np % MF_GJ_CL != 0) return;   // uniform over the cluster
  const int cw = np / MF_GJ_CL, c0 = q * cw;
  double* F = m.F + fr.fo;
  constexpr int R = MF_MAX_NP * MF_MAX_NP / MF_GJ_CL / MF_THREADS;
  double* pub = smd;                   // [2][np + 1] the pivot column, negated, published by its owner
  double* nc = pub + 2 * (np + 1);     // [np + 1] this CTA's copy of it
  double* w = nc + np + 1;             // [np + 1] the same divided by the pivot
  double* row = w + np + 1;            // [2][cw + 1] this CTA's part of the pivot row
  double* rowr = row + 2 * (cw + 1);   // [cw + 1] the same divided by the pivot
  double* s_r = rowr + cw + 1;         // 1 / pivot
  const int tid = threadIdx.x;
  for (int t = tid; t < 4 * (np + 1) + 3 * (cw + 1); t += MF_THREADS) smd[t] = 0.0;
  GjBlock<R> blk;
  blk.load(F + c0, f, np, cw);
  __syncthreads();
  blk.publish(0, q == 0 ? 0 : -1, row, pub);
  bool bad = false;
  for (int k = 0; k < np; ++k) {
    const int owner = k / cw, kc = k - c0;   // this CTA's column of pivot k, in [0, cw) at its owner only
    const int c = k & 1, n = c ^ 1;
    cl.sync();
    const double* rp = cl.map_shared_rank(pub + c * (np + 1), owner);
    if (tid < np) {   // np <= MF_MAX_NP < MF_THREADS
      double d = flip_sign(rp[k]);
      const double ci = rp[tid];
      if (!nonzero_finite(d)) {
        bad = true;
        d = 1.0;
      }
      const double r = 1.0 / d;
      nc[tid] = ci;
      w[tid] = ci * r;
      if (tid < cw) rowr[tid] = row[c * (cw + 1) + tid] * r;
      if (tid == 0) *s_r = r;
    }
    __syncthreads();
    blk.pivot(k, kc, nc, w, rowr, *s_r, row + n * (cw + 1), pub + n * (np + 1));
  }
  cl.sync();   // no CTA leaves while another may still read its published column
  blk.store(F + c0, f, np);
  if (bad) atomicOr(flags, FLAG_NOPIV_REJECTED);
}

// Tile tasks of a level, MF_TILE x MF_TILE outputs at (r0, c0) each: kind 0, of D = F11^-1 F12 (in place of
// F12, from its copy); kind 1, of B = F21 F11^-1; kind 2, of S = F22 - F21 D.  The fronts are few and small, so
// the tiles are too: a 32-wide slab of a leaf's D (48 pivots) kept one SM's FP64 pipe 42 us while most SMs had
// none; now 13 us for the level (16 leaves), 138 -> 71 us for 256.
__global__ void __launch_bounds__(MF_THREADS) k_mf_tiles(MfDev m, int first) {
  static_assert(MF_TILE * MF_TILE == MF_THREADS, "one output per thread");
  extern __shared__ __align__(16) double smd[];
  const int4 tk = m.task[first + blockIdx.x];
  const MfFront fr = m.fr[tk.x];
  const int np = fr.np, nu = fr.nu, f = np + nu, r0 = tk.z, c0 = tk.w;
  double* F = m.F + fr.fo;
  double* Bx = F + (size_t)f * f;
  const double* Fc = Bx + (size_t)nu * np;
  if (tk.y == 0) {
    cta_tile(min(MF_TILE, np - r0), min(MF_TILE, nu - c0), np, F + (size_t)r0 * f, f, Fc + c0, nu,
             F + (size_t)r0 * f + np + c0, f, 1.0, false, smd);
  } else if (tk.y == 1) {
    cta_tile(min(MF_TILE, nu - r0), min(MF_TILE, np - c0), np, F + (size_t)(np + r0) * f, f, F + c0, f,
             Bx + (size_t)r0 * np + c0, np, 1.0, false, smd);
  } else {
    const unsigned long long s = cta_tile(min(MF_TILE, nu - r0), min(MF_TILE, nu - c0), np, F + (size_t)(np + r0) * f, f, F + np + c0, f,
                              F + (size_t)(np + r0) * f + np + c0, f, -1.0, true, smd);
    cta_max_to(s, mf_stats(m) + 1);
  }
}

__global__ void k_mf_check(MfDev m, int* flags) {
  const unsigned long long* st = mf_stats(m);
  const double gmax = __longlong_as_double((long long)st[0]), smax = __longlong_as_double((long long)st[1]);
  if (!(smax <= NOPIV_MAX_GROWTH * gmax) || !isfinite(gmax)) atomicOr(flags, FLAG_NOPIV_REJECTED);
}

cudaError_t launch_mf_factor(const MfDev& m, const Plan& P, const double* ab, int* flags, cudaStream_t st) {
  // the limits go to the device maximum once (raise_smem_limit): request workers launch these kernels
  // from several host threads with different sizes, and a per-launch limit could be lowered by
  // another thread between its set and its launch
  cudaError_t e = raise_smem_limit<k_mf_tiles>();
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(m.scr + 2, 0, 16, st);   // the statistics; the solve epoch runs on
  if (e != cudaSuccess) return e;
  for (int L = 0; L + 1 < (int)P.mf_level.size(); ++L) {
    const int nf = P.mf_level[L + 1] - P.mf_level[L];
    // shared memory by the level's own pivot blocks, so that several small fronts share an SM
    bool big = false;                   // a pivot block for the cluster form
    size_t np_one = 1, np_max = 1;      // the largest block of the one-CTA form, and of all
    int f_max = 1;
    for (int i = P.mf_level[L]; i < P.mf_level[L + 1]; ++i) {
      const MfFront& fr = P.mf_front[P.mf_order[i]];
      const bool cl = fr.np >= MF_GJ_CLUSTER_NP && fr.np % MF_GJ_CL == 0;
      big = big || cl;
      if (!cl) np_one = std::max(np_one, (size_t)fr.np);
      np_max = std::max(np_max, (size_t)fr.np);
      f_max = std::max(f_max, fr.np + fr.nu);
    }
    const size_t sm_tiles = 8 * (MF_TILE * (2 * np_max + 1) + np_max);
    if (nf > 0) {
      k_mf_gather<<<dim3(nf, (f_max + MF_THREADS / 32 - 1) / (MF_THREADS / 32)), MF_THREADS, 0, st>>>(m, P.mf_level[L]);
      count_launch(1);
      const int rounds = (int)((np_one * np_one + MF_THREADS - 1) / MF_THREADS);
      const size_t sm = 8 * (6 * (np_one + 1) + 1);
      // R rounds of MF_THREADS entries: 36 and 64 (blocks of 81 to 128 unknowns that no cluster takes) fill the
      // 255 registers of a thread and spill 912 and 480 bytes of them around the assembly and the division; still
      // ahead of the block in shared memory (set-up with blocks of 90 unknowns 1.40 -> 1.12 ms, of 126 2.48 -> 1.92)
#define MRCM_MF_FRONT(R) k_mf_front<R><<<nf, MF_THREADS, sm, st>>>(m, ab, P.mf_level[L], flags)
      if (rounds <= 2) MRCM_MF_FRONT(2);
      else if (rounds <= 4) MRCM_MF_FRONT(4);
      else if (rounds <= 9) MRCM_MF_FRONT(9);
      else if (rounds <= 16) MRCM_MF_FRONT(16);
      else if (rounds <= 25) MRCM_MF_FRONT(25);
      else if (rounds <= 36) MRCM_MF_FRONT(36);
      else MRCM_MF_FRONT(64);
#undef MRCM_MF_FRONT
      count_launch(1);
      if (big) {
        const size_t sm_gj = 8 * (4 * (np_max + 1) + 3 * (np_max / MF_GJ_CL + 1) + 1);
        cudaError_t e2 = raise_smem_limit<k_mf_gj_cluster>();
        if (e2 != cudaSuccess) return e2;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = MF_GJ_CL;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(nf * MF_GJ_CL);
        cfg.blockDim = dim3(MF_THREADS);
        cfg.dynamicSmemBytes = sm_gj;
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e2 = cudaLaunchKernelEx(&cfg, k_mf_gj_cluster, m, P.mf_level[L], flags);
        if (e2 != cudaSuccess) return e2;
        count_launch(1);
      }
    }
    const int nb = P.mf_task_c[L] - P.mf_task_b[L];
    if (nb > 0) {
      k_mf_tiles<<<nb, MF_THREADS, sm_tiles, st>>>(m, P.mf_task_b[L]);
      count_launch(1);
    }
    const int nc = P.mf_task_b[L + 1] - P.mf_task_c[L];
    if (nc > 0) {
      k_mf_tiles<<<nc, MF_THREADS, sm_tiles, st>>>(m, P.mf_task_c[L]);
      count_launch(1);
    }
  }
  k_mf_check<<<1, 1, 0, st>>>(m, flags);
  count_launch(1);
  return cudaGetLastError();
}

// y_r = sum_k A[r][k] x[k] for r < rows (A row-major with leading dimension lda, in shared or global memory), for
// some rows of a front's block of `all` rows.  Every row is 4 d sums (d, a power of two up to 8, as many as the CTA
// would have threads for all rows): chain (q, c) takes the columns q + (c + 4 i) d of the whole groups of four, and
// (q, 0) the up to three left over; then c in pairs, then q in the order of a butterfly.  One chain per thread.  d
// depends on the front alone, so a front cut into parts gives the bits of the whole one.  emit(r, y) by the first
// thread of the row.
template <class Emit>
__device__ __forceinline__ void mf_rows(const double* A, int lda, int rows, int all, int cols, const double* x, Emit emit) {
  int d = 1;
  while (d < 8 && d * 2 * all <= MF_THREADS) d *= 2;
  const int tpr = 4 * d, c = threadIdx.x & 3, q = (threadIdx.x >> 2) & (d - 1), per = MF_THREADS / tpr;
  for (int r0 = 0; r0 < rows; r0 += per) {
    const int r = r0 + threadIdx.x / tpr;
    double s = 0.0;
    if (r < rows) {
      const double* a = A + (size_t)r * lda;
      int k = q;
      for (; k + 3 * d < cols; k += 4 * d) s = fma(a[k + c * d], x[k + c * d], s);
      if (c == 0)
        for (; k < cols; k += d) s = fma(a[k], x[k], s);
    }
    for (int o = 1; o < tpr; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (r < rows && c == 0 && q == 0) emit(r, s);
  }
}

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// Messages: a double in a 16-byte slot as two 64-bit words, each a half of it below the solve's epoch (the slots of
// NCCL's LL protocol).  Each word is one access of the memory model, also in a vector of two (of four 32-bit
// elements, as the slots were written before, every one is an access of its own, and a reader could take a new epoch
// beside an old half).  So two words with the solve's epoch hold the solve's value whatever order they arrive in,
// and no fence or separate flag is needed.
__device__ __forceinline__ void msg_put(ulonglong2* slot, double v, unsigned E) {
  const unsigned long long e = (unsigned long long)E << 32;
  asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};\n" ::"l"(slot), "l"(e | (unsigned)__double2loint(v)),
               "l"(e | (unsigned)__double2hiint(v))
               : "memory");
}
// Polls a slot.  The wait is bounded: when it gives up, here or in any other CTA (FLAG_TIMEOUT is set),
// it returns 0, and the other waits of the launch give up at their 1,024th poll.  The CTA goes on with what it has
// (every front's messages are written, with the current epoch), and the status word tells the host.
__device__ __forceinline__ double msg_get(const ulonglong2* slot, unsigned E, int* flags, long long polls) {
  for (long long spins = 0; spins < polls; ++spins) {
    unsigned long long lo, hi;
    asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];\n" : "=l"(lo), "=l"(hi) : "l"(slot) : "memory");
    if ((unsigned)(lo >> 32) == E && (unsigned)(hi >> 32) == E) return __hiloint2double((int)hi, (int)lo);
    if ((spins & 1023) == 1023 && (*(volatile int*)flags & FLAG_TIMEOUT)) return 0.0;
  }
  atomicOr(flags, FLAG_TIMEOUT);
  return 0.0;
}

// Solve, one cooperative launch.  A part of a front takes its rows forward (w_U = v_U - B v_P, with
// v_P = g_P + the children's w, v_U their part mapped into U) and backward (x_P = F11^-1 v_P - D x_U);
// it polls the entries that it needs from the children's parts, or of x from the ancestors', each entry
// carrying the solve's epoch.  The epoch lives in device memory: every CTA reads it at the start, the
// last CTA to finish advances it, so repeated launches (also from a captured graph) never take an old
// entry for a current one.  All CTAs are resident, and each takes its parts in increasing level
// (decreasing, backward), so every wait ends; the waits are bounded all the same.  What a part reads
// besides (its rows of B or [F11^-1 D], copied into shared memory, its slots) is requested before it
// waits.  Rows are dotted by up to a warp each, in an order that does not depend on the parts.
//
// The dependence chain bounds it: 2 x levels hand-overs, each a write, a poll and a short product.  With
// the whole front on one CTA the upper levels' products alone took 2.4 to 4.7 us there (128 x 128 FMA at
// 1.6 a clock), and a completion flag per front cost a fence, a poll by one thread and a second read:
// 134 us on 64 x 64 subdomains (9 levels), 76 us on 32 x 32, 49 us on 16 x 16, with the right-hand side
// formed by a launch of its own; now 60, 34 and 23 us.
__global__ void __launch_bounds__(MF_THREADS, 2) k_mf_solve(MfDev m, const double* __restrict__ mom0,
                                                         double* __restrict__ g, int* flags, int mcap) {
  extern __shared__ __align__(16) double smd[];
  double* v = smd;           // [max_f]
  double* M = v + m.max_f;   // [mcap] rows of B or of [F11^-1 D], with an odd stride
  volatile unsigned* vep = m.scr + 8;
  const unsigned E = *vep + 1u;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  auto stage = [&](const double* A, int rows, int cols) -> bool {   // rows x cols, contiguous rows of A
    if (rows * (cols + 1) > mcap) return false;
    for (int r = wid; r < rows; r += MF_THREADS / 32)
      for (int k = lane; k < cols; k += 32) cp_async8(M + (size_t)r * (cols + 1) + k, A + (size_t)r * cols + k);
    return true;
  };
  const int last = m.nitem - 1 - (m.nitem - 1 - (int)blockIdx.x) % (int)gridDim.x;
  for (int it = blockIdx.x; it < m.nitem; it += gridDim.x) {
    const MfItem w = m.item[it];
    const MfFront fr = m.fr[w.front];
    const int np = fr.np, f = fr.np + fr.nu, rows = w.u1 - w.u0;
    const double* Bx = m.F + fr.fo + (size_t)f * f + (size_t)w.u0 * np;
    const bool staged = stage(Bx, rows, np);
    for (int t = tid; t < np + rows; t += MF_THREADS) {
      const int pos = fr.io + (t < np ? t : t + w.u0);
      const int2 slot = m.inv[pos];
      double val = 0.0;
      if (t < np) {
        const int2 o = m.rhs[m.idx[pos]];
        val = o.y >= 0 ? -(mom0[o.x] + mom0[o.y]) : -(mom0[o.x] - mom0[~o.y]);
      }
      if (slot.x >= 0) val += msg_get(m.W + slot.x, E, flags, m.polls);
      if (slot.y >= 0) val += msg_get(m.W + slot.y, E, flags, m.polls);
      v[t] = val;
      if (t < np) m.V[w.vo + t] = val;
    }
    cp_async_wait_all();
    __syncthreads();
    mf_rows(staged ? M : Bx, staged ? np + 1 : np, rows, fr.nu, np, v,
            [&](int r, double t) { msg_put(m.W + fr.wo + w.u0 + r, v[np + r] - t, E); });
    __syncthreads();
  }
  for (int it = last; it >= 0; it -= gridDim.x) {
    const MfItem w = m.item[it];
    const MfFront fr = m.fr[w.front];
    const int np = fr.np, f = fr.np + fr.nu, rows = w.p1 - w.p0;
    const double* F = m.F + fr.fo + (size_t)w.p0 * f;
    const bool staged = stage(F, rows, f);
    for (int t = tid; t < f; t += MF_THREADS)
      v[t] = t < np ? m.V[w.vo + t] : -msg_get(m.X + m.idx[fr.io + t], E, flags, m.polls);
    cp_async_wait_all();
    __syncthreads();
    mf_rows(staged ? M : F, staged ? f + 1 : f, rows, np, f, v, [&](int r, double t) {
      const int u = m.idx[fr.io + w.p0 + r];
      msg_put(m.X + u, t, E);
      g[u] = t;
    });
    __syncthreads();
  }
  // the last CTA to finish advances the epoch (a CTA that gave up still counts itself)
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(m.scr + 9, 1u) == gridDim.x - 1) {
      m.scr[9] = 0u;
      __threadfence();
      *vep = E;
    }
  }
}

cudaError_t launch_mf_solve(const MfDev& m, const double* mom0, double* g, int* flags, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = raise_smem_limit<k_mf_solve>();
  if (e != cudaSuccess) return e;
  // v and the staged rows: about 50 KB, so two CTAs fit an SM (one if the largest front is very wide)
  const size_t sm = 8 * ((size_t)m.max_f + (size_t)m.mcap);
  const int per_sm = sm <= 112 * 1024 ? 2 : 1;
  MfDev mm = m;
  int mcap = m.mcap;
  void* args[] = {(void*)&mm, (void*)&mom0, (void*)&g, (void*)&flags, (void*)&mcap};
  const int grid = m.nitem < per_sm * sms ? m.nitem : per_sm * sms;
  e = cudaLaunchCooperativeKernel((const void*)k_mf_solve, dim3(grid), dim3(MF_THREADS), args, sm, st);
  count_launch(1);
  return e;
}

}  // namespace mrcm
