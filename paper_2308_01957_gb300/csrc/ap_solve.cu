// Damped float64 solve of the Levenberg-Marquardt step and the on-device
// accept / reject (Sec. "Optimization methods": Marquardt 1963, Transtrum &
// Sethna 2012, Gavin 2022; the step never meets a singular matrix).
//
// Per group g with parameters gp[0..n):
//   M = (J^T W J)_gg + lambda_g diag(D),  D = diag(J^T W J)_gg floored at
//   1e-12 max(D); solve M delta = (J^T W r)_g.
// A failed factorisation (or a non-positive curvature p^T M p in CG) raises
// lambda_g x10 and retries, at most 8 times; then the status word gets
// AP_ERR_NOT_SPD and delta_g = 0.
#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>

#include "ap_internal.cuh"

namespace cg = cooperative_groups;

namespace ap {

constexpr int CHOL_THREADS = 128;
constexpr int PCG_THREADS = 1024;
constexpr int LM_RETRIES = 8;
constexpr double DIAG_FLOOR = 1e-12;
constexpr int PCG_MAX_IT = 4000;
// stop when the preconditioned residual r^T M^-1 r has fallen by PCG_RTOL^2:
// invariant to the scaling of the parameters (fluxes vs positions)
constexpr double PCG_RTOL = 1e-11;

// Block reductions: warp shuffles, then warp 0 combines the warp partials
// with a fixed shuffle tree and broadcasts through shared memory (one warp
// does the float64 adds, not every thread).  red[] holds 33 doubles.
__device__ __forceinline__ double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double s = lane < nw ? red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[32] = s;
  }
  __syncthreads();
  return red[32];
}

__device__ __forceinline__ double block_max(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double s = lane < nw ? red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
    if (lane == 0) red[32] = s;
  }
  __syncthreads();
  return red[32];
}

// ---------------------------------------------------------------------------
// dense factorisation of a small group (up to 64 parameters), one CTA each; the
// matrix in shared memory.
//
// Cholesky in the form L diag(d) L^T (the same pivots, no square roots), right
// looking, one barrier per column: a thread owns a row (two threads share its
// columns) and updates it with the column's unscaled entries; the scaled ones go to
// the upper triangle; the thread that completes the next pivot also divides one by
// it (in every thread, the divisions would take as long as the updates).
// The right-hand side rides along as row n, which makes the forward substitution
// part of the factorisation; one warp does the back substitution by columns.
// Bound by the float64 pipe (a warp's FMA holds it for some 17 clocks, n^3 / 170
// of them) and the column's latency chain.  64 groups of up to 57 parameters
// 240 -> 90 us, one of 8 parameters 21 -> 9 us (divisions per element, an index
// division per update and a one-thread substitution took the time).
// ---------------------------------------------------------------------------
__host__ __device__ inline int chol_pitch(int n) { return n | 1; }   // odd: rows on different banks

__global__ void __launch_bounds__(CHOL_THREADS) chol_kernel(
    const GroupDev* __restrict__ groups, const int* __restrict__ gparams, const int64_t* __restrict__ row_ptr,
    const int32_t* __restrict__ lcol, const int64_t* __restrict__ dpos, const double* __restrict__ vals,
    const double* __restrict__ jtwr, double* lambda, double* delta, int max_n, int* status) {
  extern __shared__ double sm[];
  __shared__ double red[33];
  const int g = blockIdx.x;
  const GroupDev G = groups[g];
  if (G.dense != 1) return;
  const int n = G.n, P = chol_pitch(n);
  const int* gp = gparams + G.p0;
  double* A = sm;                                        // rows 0..n - 1, and the right-hand side as row n
  double* D = A + (max_n + 1) * chol_pitch(max_n);       // damping diagonal
  double* z = D + max_n;                                 // D^-1 L^-1 b
  double* inv = z + max_n;                               // reciprocal pivots
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double d0 = 0.0;
  if (tid < n) {
    const int64_t e = dpos[gp[tid]];
    d0 = e >= 0 ? vals[e] : 0.0;
  }
  const double dmax = block_max(fmax(d0, 0.0), red);
  if (tid < n) D[tid] = fmax(d0, dmax > 0.0 ? DIAG_FLOOR * dmax : 1.0);
  double lam = lambda[g];
  bool ok = false;
  for (int attempt = 0; attempt <= LM_RETRIES && !ok; ++attempt) {
    __syncthreads();
    for (int idx = tid; idx < n * P; idx += CHOL_THREADS) A[idx] = 0.0;
    if (tid < n) A[n * P + tid] = jtwr[gp[tid]];
    __syncthreads();
    for (int r = warp; r < n; r += CHOL_THREADS / 32) {
      const int pr = gp[r];
      for (int64_t e = row_ptr[pr] + lane; e < row_ptr[pr + 1]; e += 32) {
        const int c = lcol[e];
        if (c >= 0 && c <= r) A[r * P + c] = vals[e];
      }
    }
    __syncthreads();
    if (tid < n) A[tid * P + tid] += lam * D[tid];
    if (tid == 0 && n > 0) inv[0] = 1.0 / A[0];
    __syncthreads();
    ok = true;
    for (int k = 0; k < n; ++k) {
      const double d = A[k * P + k], iv = inv[k];
      // 2^-1022 <= d < 2^1022 (one integer comparison, the same for every thread):
      // 1 / d is a normal number; other positive pivots divide
      const bool normal = (unsigned)(__double2hiint(d) - 0x00100000) < 0x7fd00000u - 0x00100000u;
      if (!normal && (!(d > 0.0) || !isfinite(d))) {
        ok = false;
        break;
      }
      const int r = k + 1 + (tid & 63), q = tid >> 6;
      if (r <= n) {
        const double l = normal ? A[r * P + k] * iv : A[r * P + k] / d;
        double* row = A + r * P;
        const int c1 = r < n ? r : n - 1;
#pragma unroll 4
        for (int c = k + 1 + q; c <= c1; c += 2) row[c] -= l * A[c * P + k];
        if (q == 0) {
          if (r < n) A[k * P + r] = l;
          else z[k] = l;
        }
        if (tid == 0 && r < n) inv[r] = 1.0 / row[r];
      }
      __syncthreads();
    }
    if (!ok) lam *= 10.0;
  }
  if (!ok) {
    if (tid < n) delta[gp[tid]] = 0.0;
    if (tid == 0) { atomicCAS(status, 0, AP_ERR_NOT_SPD); lambda[g] = lam; }
    return;
  }
  // L^T x = z: x_k is final once the columns past k have been taken out
  if (warp == 0) {
    double xa = lane < n ? z[lane] : 0.0, xb = lane + 32 < n ? z[lane + 32] : 0.0;
    for (int k = n - 1; k > 0; --k) {
      const double xk = __shfl_sync(0xffffffffu, k < 32 ? xa : xb, k & 31);
      if (lane < k) xa -= A[lane * P + k] * xk;
      if (lane + 32 < k) xb -= A[(lane + 32) * P + k] * xk;
    }
    if (lane < n) delta[gp[lane]] = xa;
    if (lane + 32 < n) delta[gp[lane + 32]] = xb;
    if (lane == 0) lambda[g] = lam;
  }
}

// ---------------------------------------------------------------------------
// block-Jacobi preconditioned conjugate gradients, one CTA per group of up to
// PCG_SMEM_N parameters, vectors in shared memory.  Plans precomputed on the
// host: lcol[e] (group-local column of CSR entry e), dpos[p] (CSR position of
// row p's diagonal), bpos[PCG_BLK2 b + PCG_BLK a + c] (position of entry
// (a, c) of preconditioner block b, -1 if structurally zero).
// ---------------------------------------------------------------------------
constexpr int PCG_SMEM_N = 2048;

// The damped block (m x m, m <= PCG_BLK) into A (row stride PCG_BLK) and
// its explicit inverse in place, by Gauss-Jordan elimination without
// pivoting (the block is symmetric positive definite, else a pivot fails):
// applying the preconditioner is then one small matrix-vector product with
// no float64 division.
__device__ bool factor_block(const int64_t* bq, const double* vals, const double* D, int s0, int m, double lam,
                             double* A) {
  for (int a = 0; a < m; ++a)
    for (int c = 0; c < m; ++c) {
      const int64_t e = bq[a * PCG_BLK + c];
      double v = e >= 0 ? vals[e] : 0.0;
      if (a == c) v += lam * D[s0 + a];
      A[a * PCG_BLK + c] = v;
    }
  for (int k = 0; k < m; ++k) {
    const double piv = A[k * PCG_BLK + k];
    if (!(piv > 0.0) || !isfinite(piv)) return false;
    const double ip = 1.0 / piv;
    A[k * PCG_BLK + k] = 1.0;
    for (int c = 0; c < m; ++c) A[k * PCG_BLK + c] *= ip;
    for (int a = 0; a < m; ++a) {
      if (a == k) continue;
      const double f = A[a * PCG_BLK + k];
      A[a * PCG_BLK + k] = 0.0;
      for (int c = 0; c < m; ++c) A[a * PCG_BLK + c] -= f * A[k * PCG_BLK + c];
    }
  }
  return true;
}

__device__ __forceinline__ void apply_block(const double* Minv, const double* in, double* out, int s0, int m) {
  double x[PCG_BLK];
  for (int a = 0; a < m; ++a) x[a] = in[s0 + a];
  for (int a = 0; a < m; ++a) {
    double v = 0.0;
    for (int c = 0; c < m; ++c) v += Minv[a * PCG_BLK + c] * x[c];
    out[s0 + a] = v;
  }
}

__global__ void __launch_bounds__(PCG_THREADS) pcg_kernel(const GroupDev* __restrict__ groups, int n_groups,
                                                          const int* __restrict__ gparams,
                                                          const int* __restrict__ blk_ptr,
                                                          const int64_t* __restrict__ row_ptr,
                                                          const int32_t* __restrict__ lcol,
                                                          const int64_t* __restrict__ dpos,
                                                          const int64_t* __restrict__ bpos,
                                                          const double* __restrict__ vals,
                                                          const double* __restrict__ jtwr, double* lambda,
                                                          double* delta, double* blk_work, int* iters,
                                                          const int64_t* __restrict__ ch_e0,
                                                          const int64_t* __restrict__ ch_e1,
                                                          const int* __restrict__ ch_row, double* ch_part,
                                                          int* status) {
  extern __shared__ double vec[];
  __shared__ double red[33];
  __shared__ int fail;
  const int g = blockIdx.x;
  const GroupDev G = groups[g];
  if (G.dense != 0) return;
  const int n = G.n;
  const int* gp = gparams + G.p0;
  const int* bp = blk_ptr + G.b0;
  double* D = vec;
  double* x = D + n;
  double* r = x + n;
  double* z = r + n;
  double* p = z + n;
  double* q = p + n;
  double* Linv = blk_work + (int64_t)PCG_BLK2 * G.b0;
  const int tid = threadIdx.x;
  double dmax = 0.0, bn2 = 0.0;
  for (int i = tid; i < n; i += blockDim.x) {
    const int pr = gp[i];
    const int64_t e = dpos[pr];
    const double d = e >= 0 ? vals[e] : 0.0;
    D[i] = d;
    dmax = fmax(dmax, d);
    const double b = jtwr[pr];
    bn2 += b * b;
  }
  dmax = block_max(dmax, red);
  bn2 = block_sum(bn2, red);
  const double floor_v = dmax > 0.0 ? DIAG_FLOOR * dmax : 1.0;
  for (int i = tid; i < n; i += blockDim.x) D[i] = fmax(D[i], floor_v);
  double lam = lambda[g];
  bool ok = false;
  int it = 0;
  for (int attempt = 0; attempt <= LM_RETRIES && !ok; ++attempt) {
    __syncthreads();
    if (tid == 0) fail = 0;
    __syncthreads();
    for (int b = tid; b < G.nblk; b += blockDim.x)
      if (!factor_block(bpos + (int64_t)PCG_BLK2 * (G.b0 + b), vals, D, bp[b], bp[b + 1] - bp[b], lam,
                        Linv + (int64_t)PCG_BLK2 * b))
        fail = 1;
    for (int i = tid; i < n; i += blockDim.x) { x[i] = 0.0; r[i] = jtwr[gp[i]]; }
    __syncthreads();
    if (fail) { lam *= 10.0; continue; }
    for (int b = tid; b < G.nblk; b += blockDim.x)
      apply_block(Linv + (int64_t)PCG_BLK2 * b, r, z, bp[b], bp[b + 1] - bp[b]);
    __syncthreads();
    double rz = 0.0;
    for (int i = tid; i < n; i += blockDim.x) { p[i] = z[i]; rz += r[i] * z[i]; }
    rz = block_sum(rz, red);
    const double rz0 = rz;
    bool conv = bn2 == 0.0 || rz0 == 0.0;
    bool bad = false;
    const int cbeg = ch_row[G.p0], cend = ch_row[G.p0 + n];
    for (it = 0; it < PCG_MAX_IT && !conv; ++it) {
      __syncthreads();
      // SpMV: chunk partial sums, then each row sums its chunks in order
      for (int ch = cbeg + tid; ch < cend; ch += blockDim.x) {
        double sv = 0.0;
        for (int64_t e = ch_e0[ch]; e < ch_e1[ch]; ++e) sv += vals[e] * p[lcol[e]];
        ch_part[ch] = sv;
      }
      __syncthreads();
      double pq = 0.0;
      for (int i = tid; i < n; i += blockDim.x) {
        double sv = lam * D[i] * p[i];
        for (int ch = ch_row[G.p0 + i]; ch < ch_row[G.p0 + i + 1]; ++ch) sv += ch_part[ch];
        q[i] = sv;
        pq += p[i] * sv;
      }
      pq = block_sum(pq, red);
      if (!(pq > 0.0)) { bad = true; break; }
      const double alpha = rz / pq;
      for (int i = tid; i < n; i += blockDim.x) {
        x[i] += alpha * p[i];
        r[i] -= alpha * q[i];
      }
      __syncthreads();
      for (int b = tid; b < G.nblk; b += blockDim.x)
        apply_block(Linv + (int64_t)PCG_BLK2 * b, r, z, bp[b], bp[b + 1] - bp[b]);
      __syncthreads();
      double rz2 = 0.0;
      for (int i = tid; i < n; i += blockDim.x) rz2 += r[i] * z[i];
      rz2 = block_sum(rz2, red);
      if (rz2 <= PCG_RTOL * PCG_RTOL * rz0) { conv = true; ++it; break; }
      const double beta = rz2 / rz;
      rz = rz2;
      for (int i = tid; i < n; i += blockDim.x) p[i] = z[i] + beta * p[i];
    }
    __syncthreads();
    if (bad) { lam *= 10.0; continue; }
    if (!conv && tid == 0) atomicCAS(status, 0, AP_ERR_TIMEOUT);
    ok = true;
  }
  __syncthreads();
  if (!ok) {
    for (int i = tid; i < n; i += blockDim.x) delta[gp[i]] = 0.0;
    if (tid == 0) atomicCAS(status, 0, AP_ERR_NOT_SPD);
  } else {
    for (int i = tid; i < n; i += blockDim.x) delta[gp[i]] = x[i];
  }
  if (tid == 0) {
    lambda[g] = lam;
    if (iters) iters[g] = it;
  }
}

// ---------------------------------------------------------------------------
// Distributed block-Jacobi PCG: one group's system spread over several CTAs,
// either the CTAs of one thread-block cluster (one group per cluster, many
// clusters per launch) or every CTA of a cooperative launch (one large group
// per launch).
//
// The iteration is the Chronopoulos-Gear arrangement of preconditioned CG
// (Chronopoulos & Gear 1989), in which both inner products of an iteration
// are reduced together:
//   u = M^-1 r,  w = A u,  gamma = r.u,  delta = u.w
//   beta = gamma / gamma_old,  alpha = gamma / (delta - beta gamma / alpha_old)
//   p = u + beta p,  s = w + beta s,  x += alpha p,  r -= alpha s
// (first iteration: beta = 0, alpha = gamma / delta).  In exact arithmetic it
// produces the iterates of the textbook PCG in pcg_kernel.  Two barriers per
// iteration: one after the SpMV chunk partials of A u (with delta), one after
// the owners of the rows publish the next u (with gamma).
//
// Ownership: CTA k owns a contiguous run of preconditioner blocks (and so of
// rows), planned on the host; its x, r, p, s, D and block inverses live in
// its shared memory.  The SpMV is cut into chunks that any CTA may compute:
// rows of up to DIST_WARP_ROW entries into thread chunks of DIST_CHUNK
// entries, longer rows (the sky parameters couple to everything) into warp
// chunks of DIST_WCHUNK entries, so that no row has more than a few tens of
// partials to add.  What an iteration waits for is the count of float64 warp
// instructions (profiled on a 112-parameter fit: the float64 pipe 55 % busy,
// 600 of them per SM and iteration): a thread chunk costs 16 for 512 entries
// where a warp chunk costs 10 for 128.  The first chunk of every thread stays in
// registers over the iterations.  21 iterations of the 953-parameter field 298 ->
// 211 us, 43 of 16 overlapping galaxies 413 -> 299 us, 82 grid-wide ones of the
// 1536^2 crowded field 2.10 -> 1.84 ms.  In a cluster, u is broadcast into every CTA's shared memory and
// each chunk partial is stored straight into its row owner's shared memory
// (distributed shared memory); grid-wide, both go through global memory.
// Reductions: every CTA publishes its totals to its rank's slots; after the
// barrier every CTA adds the slots in rank order, so all CTAs hold the same
// bits and take the same branches.
// ---------------------------------------------------------------------------
constexpr int DIST_THREADS = 256;

struct GridBarrier {
  static constexpr bool kCluster = false;
  __device__ void sync() const { cg::this_grid().sync(); }
  __device__ int rank() const { return blockIdx.x; }
  __device__ int size() const { return gridDim.x; }
  __device__ int unit() const { return 0; }
  template <typename T>
  __device__ T* at(T* p, int) const { return p; }
};

struct ClusterBarrier {
  static constexpr bool kCluster = true;
  __device__ void sync() const { cg::this_cluster().sync(); }
  __device__ int rank() const { return (int)cg::this_cluster().block_rank(); }
  __device__ int size() const { return (int)cg::this_cluster().num_blocks(); }
  __device__ int unit() const { return blockIdx.x / size(); }
  // the same shared-memory object in CTA q of the cluster
  template <typename T>
  __device__ T* at(T* p, int q) const { return cg::this_cluster().map_shared_rank(p, q); }
};

// Totals over all CTAs of NV <= 3 values (value 0 is a max when max0).  A warp-wide
// float64 addition holds this part's one float64 pipe per SM for some 17 clocks
// whatever its lanes do, and they were what an iteration waited for, so the totals
// take as few of them as they can: every thread leaves its values in shared memory,
// warp k adds value k (8 terms per lane, then one tree) and publishes it to
// slot[par][k][rank] -- every CTA's copy in a cluster, the one global copy otherwise
// -- waits at the barrier and adds the slots in rank order (17 additions per value;
// a tree in every warp took 47).  Every thread returns the same NV values.
// red[] holds 3 DIST_THREADS + 3 doubles.
template <int NV, class Bar>
__device__ void dist_reduce(const Bar& bar, double v[3], bool max0, double* slots, int& par, double* red) {
  const int nct = bar.size(), rank = bar.rank();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) red[k * DIST_THREADS + threadIdx.x] = v[k];
  __syncthreads();
  const bool mx = warp == 0 && max0;
  auto join = [&](double x, double y) { return mx ? fmax(x, y) : x + y; };
  double* sp = slots + (size_t)(par * 3 + warp) * nct;
  if (warp < NV) {
    const double* r = red + warp * DIST_THREADS + lane;
    double x = join(r[0], r[32]), y = join(r[64], r[96]), z = join(r[128], r[160]), w = join(r[192], r[224]);
    x = join(join(x, y), join(z, w));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = join(x, __shfl_xor_sync(0xffffffffu, x, o));
    if (Bar::kCluster) {
      if (lane < nct) bar.at(sp, lane)[rank] = x;
    } else if (lane == 0) {
      sp[rank] = x;
    }
  }
  bar.sync();
  if (warp < NV) {
    double x = 0.0;   // (the max is over non-negative values)
    if constexpr (Bar::kCluster) {
      x = lane < nct ? sp[lane] : 0.0;
    } else {
      for (int q0 = lane; q0 < nct; q0 += 320) {   // ten slots per lane in flight
        double t[10];
#pragma unroll
        for (int j = 0; j < 10; ++j) t[j] = q0 + 32 * j < nct ? __ldcg(sp + q0 + 32 * j) : 0.0;
#pragma unroll
        for (int j = 0; j < 10; ++j) x = join(x, t[j]);
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      if (o >= nct) continue;   // uniform: the lanes past nct hold zeros
      x = join(x, __shfl_xor_sync(0xffffffffu, x, o));
    }
    if (lane == 0) red[3 * DIST_THREADS + warp] = x;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = red[3 * DIST_THREADS + k];
  par ^= 1;
}
static_assert(DIST_THREADS == 256, "eight terms per lane");

// read u: the CTA's own copy in a cluster, global memory (L2) otherwise
template <bool CL>
__device__ __forceinline__ double ld_u(const double* u, int i) {
  if (CL) return u[i];
  return __ldcg(u + i);
}

// thread chunk: at most DIST_CHUNK entries of one row, all loads issued first
template <bool CL>
__device__ __forceinline__ double dist_tchunk(const double* __restrict__ vals, const int32_t* __restrict__ lcol,
                                              const double* u, int64_t e0, int64_t e1) {
  double v[DIST_CHUNK];
  int c[DIST_CHUNK];
#pragma unroll
  for (int k = 0; k < DIST_CHUNK; ++k) {
    const bool in = e0 + k < e1;
    v[k] = in ? vals[e0 + k] : 0.0;
    c[k] = in ? lcol[e0 + k] : -1;
  }
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < DIST_CHUNK; ++k)
    if (c[k] >= 0) acc[k & 3] += v[k] * ld_u<CL>(u, c[k]);
  return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

// warp chunk: at most DIST_WCHUNK entries of one row, lane l takes entries
// l, l + 32, ...; every lane returns the (fixed-order) total
template <bool CL>
__device__ __forceinline__ double dist_wchunk(const double* __restrict__ vals, const int32_t* __restrict__ lcol,
                                              const double* u, int64_t e0, int64_t e1, int lane) {
  double a0 = 0.0, a1 = 0.0;
  int64_t e = e0 + lane;
  for (; e + 32 < e1; e += 64) {
    a0 += vals[e] * ld_u<CL>(u, lcol[e]);
    a1 += vals[e + 32] * ld_u<CL>(u, lcol[e + 32]);
  }
  if (e < e1) a0 += vals[e] * ld_u<CL>(u, lcol[e]);
  double s = a0 + a1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

template <class Bar>
__global__ void __launch_bounds__(DIST_THREADS, 2) pcg_dist_kernel(int g_fixed, const int* __restrict__ glist,
                                                                const GroupDev* __restrict__ groups,
                                                                const int* __restrict__ gparams,
                                                                const int* __restrict__ blk_ptr,
                                                                const int64_t* __restrict__ dpos,
                                                                const int64_t* __restrict__ bpos,
                                                                const double* __restrict__ vals,
                                                                const double* __restrict__ jtwr, double* lambda,
                                                                double* delta, double* work, double* gslots,
                                                                int* iters, DistPlan dp, DistSmem sz,
                                                                int* status) {
  constexpr bool CL = Bar::kCluster;
  const Bar bar;
  extern __shared__ double sm[];
  __shared__ double red[3 * DIST_THREADS + 3];
  const int nct = bar.size(), rank = bar.rank();
  const int tid = threadIdx.x, lane = tid & 31;
  const int g = CL ? glist[bar.unit()] : g_fixed;
  const GroupDev G = groups[g];
  const int* gp = gparams + G.p0;
  const int* bp = blk_ptr + G.b0;
  const int ob = dp.own_ptr[g];
  const int b0 = dp.own_blk[ob + rank], b1 = dp.own_blk[ob + rank + 1];
  const int R0 = bp[b0], R1 = bp[b1];
  const int P0 = dp.row[G.p0 + R0];   // first chunk partial of the owned rows
  // shared memory: [slots (cluster)] | x r p s D [nr] | block inverses [nb] | u [nu] | partials [np] (cluster)
  double* slots = CL ? sm : gslots;
  double* X = sm + (CL ? 6 * nct : 0);
  double* Rv = X + sz.nr;
  double* P = Rv + sz.nr;
  double* S = P + sz.nr;
  double* Dv = S + sz.nr;
  double* Lv = Dv + sz.nr;                    // packed block inverses of the owned blocks
  double* U = Lv + sz.nb;                     // cluster: u over the whole group; grid: u of the owned rows
  double* PART = U + sz.nu;                   // cluster: partials of the owned rows
  double* gu = work + (int64_t)6 * G.p0;      // grid: u over the whole group, in global memory
  const double* ug = CL ? U : gu;             // where the SpMV gathers u from
  // thread chunks go to the CTA's threads from the last one down, warp chunks to its
  // warps from the first one up: the warps with warp chunks get thread chunks last
  const int first = rank + nct * ((int)blockDim.x - 1 - tid), stride = nct * (int)blockDim.x;
  const int wfirst = rank + nct * (tid >> 5), wstride = nct * (int)(blockDim.x >> 5);
  int par = 0;
  if (CL) bar.sync();   // every CTA of the cluster is running before any remote store

  double v[3] = {0.0, 0.0, 0.0};
  for (int i = R0 + tid; i < R1; i += blockDim.x) {
    const int pr = gp[i];
    const int64_t e = dpos[pr];
    v[0] = fmax(v[0], e >= 0 ? vals[e] : 0.0);
    v[1] += jtwr[pr] * jtwr[pr];
  }
  dist_reduce<2>(bar, v, true, slots, par, red);
  const double floor_v = v[0] > 0.0 ? DIAG_FLOOR * v[0] : 1.0;
  const double bn2 = v[1];
  double lam = lambda[g];
  bool ok = false;
  int it = 0;
  const int tb = dp.tptr[g], te = dp.tptr[g + 1], wb = dp.wptr[g], we = dp.wptr[g + 1];

  // u of one row: publish to the SpMV (every CTA's copy, or global memory)
  auto publish_u = [&](int i, double val) {
    if (CL) {
      for (int q = 0; q < nct; ++q) bar.at(U, q)[i] = val;
    } else {
      gu[i] = val;
      U[i - R0] = val;
    }
  };
  auto own_u = [&](int i) -> double { return CL ? U[i] : U[i - R0]; };

  // block phases run in teams of PCG_BLK (16) lanes, one team per owned
  // block and one lane per row of it; the rounds are uniform over the CTA so
  // that the team shuffles and warp syncs always see the whole warp
  const int team = tid / PCG_BLK, tl = tid % PCG_BLK, tbase = lane & ~(PCG_BLK - 1);
  const int nteam = blockDim.x / PCG_BLK;
  const int nrounds = (b1 - b0 + nteam - 1) / nteam;
  // the chunks of the first round's row
  int pc0 = 0, pc1 = 0;
  if (b0 + team < b1 && tl < bp[b0 + team + 1] - bp[b0 + team]) {
    pc0 = dp.row[G.p0 + bp[b0 + team] + tl];
    pc1 = dp.row[G.p0 + bp[b0 + team] + tl + 1];
  }
  // the thread's first chunk stays in registers over all iterations
  double kv[DIST_CHUNK];
  int kc[DIST_CHUNK];
  const int kid = tb + first < te ? dp.tlist[tb + first] : -1;
  const int64_t ke0 = kid >= 0 ? dp.e0[kid] : 0, ke1 = kid >= 0 ? dp.e1[kid] : 0;
#pragma unroll
  for (int j = 0; j < DIST_CHUNK; ++j) {
    const bool in = ke0 + j < ke1;
    kv[j] = in ? vals[ke0 + j] : 0.0;
    kc[j] = in ? dp.lcol[ke0 + j] : -1;
  }

  for (int attempt = 0; attempt <= LM_RETRIES && !ok; ++attempt) {
    double fail = 0.0, gam = 0.0, dd = 0.0;
    for (int rd = 0; rd < nrounds; ++rd) {
      const int b = b0 + rd * nteam + team;
      const bool has = b < b1;
      const int s0 = has ? bp[b] : 0, m = has ? bp[b + 1] - s0 : 0, l0 = s0 - R0;
      const bool row = tl < m;
      double d = 0.0, rr = 0.0;
      if (row) {
        const int pr = gp[s0 + tl];
        const int64_t e = dpos[pr];
        d = fmax(e >= 0 ? vals[e] : 0.0, floor_v);
        rr = jtwr[pr];
        Dv[l0 + tl] = d;
        X[l0 + tl] = 0.0;
        Rv[l0 + tl] = rr;
        P[l0 + tl] = 0.0;
        S[l0 + tl] = 0.0;
      }
      // the damped block into its packed slot (lane tl: row tl), then its
      // inverse in place by Gauss-Jordan elimination without pivoting (M is
      // symmetric positive definite or the block fails), the lanes of the
      // team updating their rows step by step; steps past the warp's largest
      // block are skipped (mw is uniform over the warp)
      double* Li = Lv + (has ? dp.loff[G.b0 + b] : 0);
      if (row) {
        const int64_t* bq = bpos + (int64_t)PCG_BLK2 * (G.b0 + b) + tl * PCG_BLK;
        for (int c = 0; c < m; ++c) {
          const int64_t e = bq[c];
          Li[tl * m + c] = (e >= 0 ? vals[e] : 0.0) + (c == tl ? lam * d : 0.0);
        }
      }
      __syncwarp();
      bool good = true;
      const int mw = (int)__reduce_max_sync(0xffffffffu, (unsigned)m);
      for (int k = 0; k < mw; ++k) {
        const bool act = k < m;
        const double piv = act ? Li[k * m + k] : 1.0;
        __syncwarp();   // the pivot is read before row k changes
        good = good && (!act || (piv > 0.0 && isfinite(piv)));
        const double ip = 1.0 / piv;
        if (act && tl == k) {
          Li[k * m + k] = 1.0;
          for (int c = 0; c < m; ++c) Li[k * m + c] *= ip;
        }
        __syncwarp();   // row k is scaled
        if (act && row && tl != k) {
          const double f = Li[tl * m + k];
          Li[tl * m + k] = 0.0;
          for (int c = 0; c < m; ++c) Li[tl * m + c] -= f * Li[k * m + c];
        }
        __syncwarp();   // every row is updated before the next pivot is read
      }
      // every lane of the team saw the same pivots: lane 0 counts a failure
      if (has && tl == 0 && !good) fail += 1.0;
      // u = M^-1 r for the block
      double t = 0.0;
      for (int c = 0; c < mw; ++c) {
        const double rc = __shfl_sync(0xffffffffu, rr, tbase + c);
        if (row && c < m) t += Li[tl * m + c] * rc;
      }
      if (row) {
        gam += rr * t;
        dd += lam * d * t * t;
        publish_u(s0 + tl, t);
      }
    }
    v[0] = fail; v[1] = gam; v[2] = dd;
    dist_reduce<3>(bar, v, false, slots, par, red);
    if (v[0] > 0.0) { lam *= 10.0; continue; }
    gam = v[1];
    dd = v[2];
    const double gamma0 = gam;
    bool conv = bn2 == 0.0 || !(gamma0 > 0.0);
    bool bad = false;
    double gam_old = 1.0, alpha_old = 1.0;
    for (it = 0; it < PCG_MAX_IT && !conv;) {
      // w = A u as chunk partials; delta = u.(A u) + the damping part
      double del = 0.0;
      for (int k = wb + wfirst; k < we; k += wstride) {
        const int c = dp.wlist[k];
        const double sv = dist_wchunk<CL>(vals, dp.lcol, ug, dp.e0[c], dp.e1[c], lane);
        if (lane == 0) {
          if (CL) bar.at(PART, dp.owner[c])[dp.dst[c]] = sv;
          else dp.part[c] = sv;
          del += ld_u<CL>(ug, dp.lrow[c]) * sv;
        }
      }
      auto put = [&](int c, double sv) {   // a chunk's sum to its row's owner
        if (CL) bar.at(PART, dp.owner[c])[dp.dst[c]] = sv;
        else dp.part[c] = sv;
        del += ld_u<CL>(ug, dp.lrow[c]) * sv;
      };
      if (kid >= 0) {
        double a0 = 0.0, a1 = 0.0;
#pragma unroll
        for (int j = 0; j < DIST_CHUNK; j += 2) {
          if (kc[j] >= 0) a0 += kv[j] * ld_u<CL>(ug, kc[j]);
          if (kc[j + 1] >= 0) a1 += kv[j + 1] * ld_u<CL>(ug, kc[j + 1]);
        }
        put(kid, a0 + a1);
      }
      for (int k = tb + first + stride; k < te; k += stride) {
        const int c = dp.tlist[k];
        put(c, dist_tchunk<CL>(vals, dp.lcol, ug, dp.e0[c], dp.e1[c]));
      }
      v[0] = del;
      dist_reduce<1>(bar, v, false, slots, par, red);
      const double dlt = v[0] + dd;
      const double beta = it == 0 ? 0.0 : gam / gam_old;
      const double den = it == 0 ? dlt : dlt - beta * gam / alpha_old;
      if (!(den > 0.0) || !isfinite(den)) { bad = true; break; }
      const double alpha = gam / den;
      double gam2 = 0.0, dd2 = 0.0;
      for (int rd = 0; rd < nrounds; ++rd) {
        const int b = b0 + rd * nteam + team;
        const bool has = b < b1;
        const int s0 = has ? bp[b] : 0, m = has ? bp[b + 1] - s0 : 0, l = s0 - R0 + tl;
        const bool row = tl < m;
        double rr = 0.0;
        if (row) {
          const int i = s0 + tl;
          const int c0 = rd == 0 ? pc0 : dp.row[G.p0 + i], c1 = rd == 0 ? pc1 : dp.row[G.p0 + i + 1];
          const double ui = own_u(i);
          double w0 = lam * Dv[l] * ui, w1 = 0.0;
          constexpr int NP = CL ? 4 : 8;
          for (int ch = c0; ch < c1; ch += NP) {   // NP partials in flight
            double t[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) t[q] = ch + q < c1 ? (CL ? PART[ch + q - P0] : __ldcg(dp.part + ch + q)) : 0.0;
#pragma unroll
            for (int q = 0; q < NP; q += 2)
              if (ch + q < c1) {
                w0 += t[q];
                w1 += t[q + 1];
              }
          }
          const double pi = ui + beta * P[l];
          const double si = (w0 + w1) + beta * S[l];
          P[l] = pi;
          S[l] = si;
          X[l] += alpha * pi;
          rr = Rv[l] - alpha * si;
          Rv[l] = rr;
        }
        const double* Li = Lv + (has ? dp.loff[G.b0 + b] : 0) + tl * m;
        // two independent product chains (shorter dependency path), as wide
        // as the warp's largest block
        const int mw = (int)__reduce_max_sync(0xffffffffu, (unsigned)m);
        double t0 = 0.0, t1 = 0.0;
        for (int c = 0; c < mw; ++c) {
          const double rc = __shfl_sync(0xffffffffu, rr, tbase + c);
          if (row && c < m) {
            if (c & 1) t1 += Li[c] * rc;
            else t0 += Li[c] * rc;
          }
        }
        const double t = t0 + t1;
        if (row) {
          gam2 += rr * t;
          dd2 += lam * Dv[l] * t * t;
          // the SpMV of this iteration is complete in every CTA (barrier
          // above), so u may be overwritten
          publish_u(s0 + tl, t);
        }
      }
      v[0] = gam2; v[1] = dd2;
      dist_reduce<2>(bar, v, false, slots, par, red);
      gam_old = gam;
      alpha_old = alpha;
      gam = v[0];
      dd = v[1];
      ++it;
      conv = gam <= PCG_RTOL * PCG_RTOL * gamma0;
    }
    if (bad) { lam *= 10.0; continue; }
    if (!conv && rank == 0 && tid == 0) atomicCAS(status, 0, AP_ERR_TIMEOUT);
    ok = true;
  }
  for (int i = R0 + tid; i < R1; i += blockDim.x) delta[gp[i]] = ok ? X[i - R0] : 0.0;
  if (rank == 0 && tid == 0) {
    lambda[g] = lam;
    if (iters) iters[g] = it;
    if (!ok) atomicCAS(status, 0, AP_ERR_NOT_SPD);
  }
  if (CL) bar.sync();   // no CTA leaves while another may still address its shared memory
}

size_t dist_smem_bytes(const DistSmem& sz, int nct, bool cluster) {
  return sizeof(double) * ((cluster ? (size_t)6 * nct : 0) + 5 * (size_t)sz.nr + (size_t)sz.nb + sz.nu + sz.np);
}

int grid_pcg_blocks(int device, size_t smem) {
  int sms = 0, per = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  allow_max_dynamic_smem(pcg_dist_kernel<GridBarrier>);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, pcg_dist_kernel<GridBarrier>, DIST_THREADS, smem);
  return sms * std::min(per, 2);
}

int cluster_pcg_size(int device, size_t smem) {
  (void)device;
  allow_max_dynamic_smem(pcg_dist_kernel<ClusterBarrier>);
  cudaFuncSetAttribute(pcg_dist_kernel<ClusterBarrier>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  for (int cs : {16, 8, 4}) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(DIST_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, pcg_dist_kernel<ClusterBarrier>, &cfg) == cudaSuccess &&
        nclusters > 0)
      return cs;
    cudaGetLastError();
  }
  return 0;
}

// one cooperative launch per grid group (dense == 2), one cluster launch for
// all cluster groups (dense == 3)
int launch_pcg_dist(const GroupDev* groups_host, int n_groups, const SolvePlan& sp, const double* vals,
                    const double* jtwr, double* lambda, double* delta, const DistLaunch& dl, int* status,
                    cudaStream_t st) {
  const int* no_list = nullptr;
  for (int g = 0; g < n_groups; ++g) {
    if (groups_host[g].dense != 2) continue;
    void* args[] = {(void*)&g, (void*)&no_list, (void*)&sp.groups, (void*)&sp.gparams, (void*)&sp.blk_ptr,
                    (void*)&sp.dpos, (void*)&sp.bpos, (void*)&vals, (void*)&jtwr, (void*)&lambda, (void*)&delta,
                    (void*)&sp.work, (void*)&sp.part, (void*)&sp.iters, (void*)&sp.dist, (void*)&dl.grid_sz,
                    (void*)&status};
    const cudaError_t e = cudaLaunchCooperativeKernel((const void*)pcg_dist_kernel<GridBarrier>,
                                                      dim3(dl.grid_blocks), dim3(DIST_THREADS), args,
                                                      dist_smem_bytes(dl.grid_sz, dl.grid_blocks, false), st);
    if (e != cudaSuccess) return (int)e;
  }
  if (dl.n_cluster_groups > 0) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = dl.cluster_size;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(dl.n_cluster_groups * dl.cluster_size);
    cfg.blockDim = dim3(DIST_THREADS);
    cfg.dynamicSmemBytes = dist_smem_bytes(dl.cluster_sz, dl.cluster_size, true);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, pcg_dist_kernel<ClusterBarrier>, -1, sp.cluster_groups, sp.groups, sp.gparams,
                           sp.blk_ptr, sp.dpos, sp.bpos, vals, jtwr, lambda, delta, sp.work, sp.part, sp.iters,
                           sp.dist, dl.cluster_sz, status);
    if (e != cudaSuccess) return (int)e;
  }
  return 0;
}

void configure_solve() {
  allow_max_dynamic_smem(chol_kernel);
  allow_max_dynamic_smem(pcg_kernel);
}

void launch_lm_solve(int n_groups, const SolvePlan& sp, const double* vals, const double* jtwr, double* lambda,
                     double* delta, int* status, cudaStream_t st, int any_dense, int any_pcg, int max_dense,
                     int max_pcg) {
  if (n_groups <= 0) return;
  if (any_dense) {
    const size_t sm = (size_t)((max_dense + 1) * chol_pitch(max_dense) + 3 * max_dense) * sizeof(double);
    chol_kernel<<<n_groups, CHOL_THREADS, sm, st>>>(sp.groups, sp.gparams, sp.row_ptr, sp.lcol, sp.dpos, vals, jtwr,
                                                    lambda, delta, max_dense, status);
  }
  if (any_pcg)
    pcg_kernel<<<n_groups, PCG_THREADS, 6 * max_pcg * sizeof(double), st>>>(
        sp.groups, n_groups, sp.gparams, sp.blk_ptr, sp.row_ptr, sp.lcol, sp.dpos, sp.bpos, vals, jtwr, lambda,
        delta, sp.blk_work, sp.iters, sp.ch_e0, sp.ch_e1, sp.ch_row, sp.ch_part, status);
}

// ---------------------------------------------------------------------------
// trial point and accept / reject
// ---------------------------------------------------------------------------
__global__ void trial_kernel(const double* theta, const double* delta, const double* lo, const double* hi,
                             double* trial, int n) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) trial[p] = fmin(fmax(theta[p] + delta[p], lo[p]), hi[p]);
}

void launch_trial(const double* theta, const double* delta, const double* lo, const double* hi, double* trial, int n,
                  cudaStream_t st) {
  if (n > 0) trial_kernel<<<(n + 255) / 256, 256, 0, st>>>(theta, delta, lo, hi, trial, n);
}

constexpr double LAMBDA_DOWN = 9.0, LAMBDA_UP = 11.0, LAMBDA_MIN = 1e-12, LAMBDA_MAX = 1e12;

// Accept or reject, one launch: the first blocks update the groups and the
// parameters, the others copy an accepted group's trial state (source records,
// w r) over its current one, a chunk each (16-byte words where both ends are
// aligned).  Every block decides from the two chi^2 values itself, so nothing in
// the launch waits for the groups' flags; a chunk is 16 KB, four rounds of loads
// of its CTA (64 KB chunks in a launch of their own took 11 us on an image of one
// chunk).
// fwd_valid[g] = 1: after this launch the group's current source records and w r
// are in place (the trial's if it accepted, else those of the unchanged theta),
// and chi2_state holds its chi^2.
__device__ __forceinline__ bool lm_accepts(const double* chi2_now, const double* chi2_trial, int g) {
  const double c1 = chi2_trial[g];
  return isfinite(c1) && c1 < chi2_now[g];
}

__global__ void __launch_bounds__(256) accept_kernel(const double* __restrict__ chi2_now,
                                                     const double* __restrict__ chi2_trial, double* lambda,
                                                     double* chi2_state, double* log, int* fwd_valid, int n_groups,
                                                     const int* __restrict__ param_group, int n_params, double* theta,
                                                     const double* __restrict__ trial, int n_head,
                                                     const StateChunk* __restrict__ chunks) {
  if ((int)blockIdx.x >= n_head) {
    const StateChunk ch = chunks[blockIdx.x - n_head];
    if (!lm_accepts(chi2_now, chi2_trial, ch.group)) return;
    int done = 0;
    if ((((uintptr_t)ch.src | (uintptr_t)ch.dst) & 15) == 0) {
      const int nq = ch.n_words >> 2;
      const uint4* s4 = reinterpret_cast<const uint4*>(ch.src);
      uint4* d4 = reinterpret_cast<uint4*>(ch.dst);
#pragma unroll 4
      for (int i = threadIdx.x; i < nq; i += 256) d4[i] = __ldg(s4 + i);
      done = nq << 2;
    }
    for (int i = done + threadIdx.x; i < ch.n_words; i += 256) ch.dst[i] = ch.src[i];
    return;
  }
  const int t = blockIdx.x * 256 + threadIdx.x;
  if (t < n_params) {
    const int g = param_group[t];
    if (g >= 0 && lm_accepts(chi2_now, chi2_trial, g)) theta[t] = trial[t];
  }
  if (t < n_groups) {
    const double c0 = chi2_now[t], c1 = chi2_trial[t];
    const bool acc = lm_accepts(chi2_now, chi2_trial, t);
    double lam = lambda[t];
    lam = acc ? fmax(lam / LAMBDA_DOWN, LAMBDA_MIN) : fmin(lam * LAMBDA_UP, LAMBDA_MAX);
    lambda[t] = lam;
    chi2_state[t] = acc ? c1 : c0;
    fwd_valid[t] = 1;
    log[4 * t + 0] = c0;
    log[4 * t + 1] = c1;
    log[4 * t + 2] = lam;
    log[4 * t + 3] = acc;
  }
}

void launch_accept(const double* chi2_now, const double* chi2_trial, double* lambda, double* chi2_state, double* log,
                   int* fwd_valid, int n_groups, const int* param_group, int n_params, double* theta,
                   const double* trial, const StateChunk* chunks, int n_chunks, cudaStream_t st) {
  const int n_head = (std::max(n_groups, n_params) + 255) / 256;
  if (n_head + n_chunks > 0)
    accept_kernel<<<n_head + n_chunks, 256, 0, st>>>(chi2_now, chi2_trial, lambda, chi2_state, log, fwd_valid,
                                                     n_groups, param_group, n_params, theta, trial, n_head, chunks);
}

// Pointers carried by value in the kernel's arguments: the launch copies them,
// so the caller's host array need not outlive the call (no host sync).
struct PtrRun {
  void* p[PTR_RUN];
  int n;
};

__global__ void store_ptrs_kernel(PtrRun run, void** dst) {
  if ((int)threadIdx.x < run.n) dst[threadIdx.x] = run.p[threadIdx.x];
}

void launch_store_ptrs(void* const* src_host, int n, void** dst_dev, cudaStream_t st) {
  for (int k0 = 0; k0 < n; k0 += PTR_RUN) {
    PtrRun run;
    run.n = n - k0 < PTR_RUN ? n - k0 : PTR_RUN;
    for (int k = 0; k < run.n; ++k) run.p[k] = src_host[k0 + k];
    store_ptrs_kernel<<<1, PTR_RUN, 0, st>>>(run, dst_dev + k0);
  }
}

}  // namespace ap
