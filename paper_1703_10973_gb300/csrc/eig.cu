// FP64 symmetric eigensolver for Algorithm 1 step 1 (eig(W)), the NT scaling
// (eig(L^T S L)) and the step-length test (lambda_min).
//
//  1. Householder tridiagonalisation A = Q T Q^T: one CTA (n <= 64), a 16-CTA cluster
//     (its shared memory up to n ~ 880, through L2 up to 1024), the whole GPU with the
//     matrix in registers and shared memory (up to 2048) or in HBM; bounded barriers.
//  2. Eigenvalues of T by multisection on Sturm counts (one warp per eigenvalue).
//  3. Eigenvectors of T by inverse iteration with a pivoted tridiagonal LU (one vector
//     per CTA in shared memory, eight in global memory).
//  4. Re-orthogonalisation of the eigenvector block by up to two Cholesky-QR
//     passes (Gram matrix GEMM, Cholesky, triangular solve), which repair the
//     loss of orthogonality of inverse iteration inside eigenvalue clusters; a
//     pass whose Gram matrix is already the identity to 1e-12 stops there.
//  5. Back-transformation by the stored reflectors (no inter-CTA communication).
#include <cstring>
#include "internal.cuh"

#include <cooperative_groups.h>

#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include <algorithm>

namespace cg = cooperative_groups;

namespace sdpgb {

static inline unsigned cdiv(size_t a, size_t b) { return (unsigned)((a + b - 1) / b); }

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double bsum(double v, double* sh) {
  v = wsum(v);
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = (l < (int)(blockDim.x / 32)) ? sh[l] : 0.0;
    s = wsum(s);
  }
  __syncthreads();
  return s;  // valid in thread 0 (lane 0 of warp 0)
}

// Grid-wide barrier for a cooperative launch.  Every wait is bounded: after
// `spin` cycles of the SM clock (default about two seconds) the waiting CTA sets
// *flag and returns false; all CTAs then leave the kernel at their next barrier.
constexpr long long SPIN_CYCLES = 4000000000LL;

__device__ bool grid_barrier(unsigned int* bar, int* flag, long long spin) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    s_ok = 1;
    volatile unsigned int* vgen = bar + 1;
    const unsigned int gen = *vgen;
    __threadfence();
    const unsigned int arrived = atomicAdd(bar, 1u) + 1u;
    if (arrived == gridDim.x) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      const long long t0 = clock64();
      unsigned int spins = 0;
      while (*vgen == gen) {
        if (*(volatile int*)flag) { s_ok = 0; break; }
        if (clock64() - t0 > spin) { atomicExch(flag, 1); s_ok = 0; break; }
        if (++spins > 4096u) __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return s_ok != 0;
}

// ---------------------------------------------------------------------------
// 1. Tridiagonalisation (lower; A full symmetric storage, row-major)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_sytrd(int n, double* A, int lda, double* d, double* e,
                                               double* tauh, double* p, double* part,
                                               unsigned int* bar, int* flag, long long spin) {
  extern __shared__ double sm[];
  double* v = sm;       // n
  double* w = sm + n;   // n
  __shared__ double red[32];
  __shared__ double s_tau, s_beta, s_scale, s_K;
  const int wpb = blockDim.x / 32, wid = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int gwarp = blockIdx.x * wpb + wid, nwarps = gridDim.x * wpb;

  for (int j = 0; j < n - 2; ++j) {
    const int len = n - j - 1;
    const double* row = A + (size_t)j * lda + j + 1;
    // --- reflector H = I - tau v v^T with v[0] = 1 mapping row j onto beta e_1
    double s = 0.0;
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      const double x = __ldcg(row + i);
      v[i] = x;
      if (i > 0) s = fma(x, x, s);
    }
    s = bsum(s, red);
    if (threadIdx.x == 0) {
      const double x0 = v[0];
      double tau = 0.0, beta = x0, scale = 0.0;
      if (s > 0.0) {
        beta = -copysign(sqrt(fma(x0, x0, s)), x0);
        tau = (beta - x0) / beta;
        scale = 1.0 / (x0 - beta);
      }
      s_tau = tau; s_beta = beta; s_scale = scale;
    }
    __syncthreads();
    const double tau = s_tau, scale = s_scale;
    for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) v[i] *= scale;
    if (threadIdx.x == 0) v[0] = 1.0;
    __syncthreads();
    // --- p = tau A22 v for the rows this CTA owns; partial sums of p^T v
    double kp = 0.0;
    for (int i = j + 1 + gwarp; i < n; i += nwarps) {
      const double* ai = A + (size_t)i * lda + j + 1;
      double acc = 0.0;
      for (int l = lane; l < len; l += 32) acc = fma(__ldcg(ai + l), v[l], acc);
      acc = wsum(acc) * tau;
      if (lane == 0) {
        p[i] = acc;
        kp = fma(acc, v[i - j - 1], kp);
      }
    }
    kp = bsum(kp, red);
    if (threadIdx.x == 0) part[blockIdx.x] = kp;
    if (!grid_barrier(bar, flag, spin)) return;
    // --- w = p - (tau/2)(p^T v) v ; A22 -= v w^T + w v^T
    if (threadIdx.x < 32) {
      double K = 0.0;
      for (int b = lane; b < (int)gridDim.x; b += 32) K += __ldcg(part + b);
      K = wsum(K);
      if (lane == 0) s_K = 0.5 * tau * K;
    }
    __syncthreads();
    const double K = s_K;
    for (int l = threadIdx.x; l < len; l += blockDim.x) w[l] = __ldcg(p + j + 1 + l) - K * v[l];
    __syncthreads();
    for (int i = j + 1 + gwarp; i < n; i += nwarps) {
      double* ai = A + (size_t)i * lda + j + 1;
      const double vi = v[i - j - 1], wi = w[i - j - 1];
      for (int l = lane; l < len; l += 32) {
        const double x = __ldcg(ai + l);
        ai[l] = fma(-vi, w[l], fma(-wi, v[l], x));
      }
    }
    if (blockIdx.x == 0) {
      double* rj = A + (size_t)j * lda + j + 1;
      for (int l = threadIdx.x; l < len; l += blockDim.x) rj[l] = v[l];
      if (threadIdx.x == 0) {
        d[j] = __ldcg(A + (size_t)j * lda + j);
        e[j] = s_beta;
        tauh[j] = tau;
      }
    }
    if (!grid_barrier(bar, flag, spin)) return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (n >= 2) {
      d[n - 2] = __ldcg(A + (size_t)(n - 2) * lda + n - 2);
      e[n - 2] = __ldcg(A + (size_t)(n - 2) * lda + n - 1);
      tauh[n - 2] = 0.0;
    }
    d[n - 1] = __ldcg(A + (size_t)(n - 1) * lda + n - 1);
    e[n - 1] = 0.0;
    if (n >= 2) tauh[n - 1] = 0.0;
  }
}

// Resident form of k_sytrd for orders up to SYR_MAX_N: the matrix stays in the
// registers and shared memory of the whole GPU and a column costs one grid barrier.
// A warp owns one row for the whole reduction: lane q keeps the entries with index
// q mod 32, those below 1024 in registers, the rest in shared memory.  Per column j:
//   p_i = tau A[i, :] v for the owned row, published with the not yet updated row
//   j + 1; grid barrier; every CTA forms w and the updated row j + 1 itself, starts
//   the next reflector from it, and updates the owned rows.
// The sums are those of k_sytrd in the same order: a row's dot runs over the same
// residue classes (held by rotated lanes, turned back before the warp sum), p^T v
// over groups of eight rows as k_sytrd's blocks formed it (one row per warp there:
// its grid has at least n / 8 blocks), ||x||^2 over 256 threads.  Vectors are zero
// left of the active part, so no lane needs a predicate.
// Bound by the barrier, the reflector's square root and quotients, and the FP64
// pipe of 14 rows per SM; k_sytrd streams the trailing matrix twice per column and
// waits at two barriers.  n = 2000: 61.5 ms -> 40.3 ms.
constexpr int SYR_THREADS = 512, SYR_WARPS = SYR_THREADS / 32;
constexpr int SYR_REG = 32;                       // entries per lane in registers
constexpr int SYR_MAX_N = 2048;
static size_t sytrd_resident_smem(int n, int rows) {
  return ((size_t)std::max(0, n - 32 * SYR_REG) * rows + 5 * (size_t)n) * sizeof(double);
}
// Barrier number `target` / gridDim.x; false when a wait ran out somewhere.
__device__ bool syr_barrier(unsigned int* bar, int* flag, unsigned int target, long long spin) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    int ok = 1;
    const long long t0 = clock64();
    for (;;) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= target) break;
      if (*(volatile int*)flag) { ok = 0; break; }
      if (clock64() - t0 > spin) { atomicExch(flag, 1); ok = 0; break; }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}
__global__ void __launch_bounds__(SYR_THREADS, 1)
    k_sytrd_resident(int n, double* A, int lda, double* d, double* e, double* tauh, double* p0, double* p1, double* r0,
                     double* r1, int rpc, unsigned int* bar, int* flag, long long spin) {
  extern __shared__ double sm[];
  double* va = sm;                 // n each: the reflector, the next one, w, p, row j + 1
  double* vb = va + n;
  double* w = vb + n;
  double* p = w + n;
  double* rw = p + n;
  double* tail = rw + n;           // rpc rows x (n - 1024)
  __shared__ double red[32], part[(SYR_MAX_N + 7) / 8];
  __shared__ double s_tau, s_beta, s_scale, s_K;
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
  const int row = (int)blockIdx.x * rpc + wid;
  const bool own = wid < rpc && row < n;
  const int nt = max(0, n - 32 * SYR_REG);
  double* mytail = tail + (size_t)wid * nt;      // entry idx at [idx - 1024] (used only when own)
  double a[SYR_REG];
#pragma unroll
  for (int t = 0; t < SYR_REG; ++t) {
    const int idx = 32 * t + lane;
    a[t] = (own && idx < n) ? __ldcg(A + (size_t)row * lda + idx) : 0.0;
  }
  if (own)
    for (int x = lane; x < nt; x += 32) mytail[x] = __ldcg(A + (size_t)row * lda + 32 * SYR_REG + x);

  // Reflector of the row in rw (entries from c on): scalars in s_*, vector in v
  // (zeros left of c).  The sum runs over 256 threads as in k_sytrd.
  auto partial = [&](int c) {
    double s = 0.0;
    if (tid < 256)
      for (int l = tid; l < n - c; l += 256)
        if (l > 0) s = fma(rw[c + l], rw[c + l], s);
    if (wid < 8) {
      s = wsum(s);
      if (lane == 0) red[wid] = s;
    }
  };
  auto scalars = [&](int c) {      // warp 0
    double s = (lane < 8) ? red[lane] : 0.0;
    s = wsum(s);
    const double x0 = rw[c];
    double tau = 0.0, beta = x0, scale = 0.0;
    if (s > 0.0) {
      beta = -copysign(sqrt(fma(x0, x0, s)), x0);
      // two quotients in two lanes
      const double q = (lane == 1 ? 1.0 : beta - x0) / (lane == 1 ? x0 - beta : beta);
      tau = __shfl_sync(0xffffffffu, q, 0);
      scale = __shfl_sync(0xffffffffu, q, 1);
    }
    if (lane == 0) {
      s_tau = tau;
      s_beta = beta;
      s_scale = scale;
    }
  };
  auto finish = [&](int c, double* v) {
    const double scale = s_scale;
    for (int i = tid; i < n; i += SYR_THREADS) v[i] = (i < c) ? 0.0 : (i == c) ? 1.0 : rw[i] * scale;
  };

  for (int i = tid; i < n; i += SYR_THREADS) rw[i] = __ldcg(A + i);
  __syncthreads();
  double dnext = rw[0];
  partial(1);
  __syncthreads();
  if (wid == 0) scalars(1);
  __syncthreads();
  finish(1, va);
  __syncthreads();
  unsigned int target = 0;
  for (int j = 0; j < n - 2; ++j) {
    double* v = (j & 1) ? vb : va;
    double* vn = (j & 1) ? va : vb;
    double* pg = (j & 1) ? p1 : p0;
    double* rg = (j & 1) ? r1 : r0;
    const double tau = s_tau, beta = s_beta;
    const int t0 = (j + 1) >> 5;
    if (own && row > j) {
      double acc = 0.0;
#pragma unroll
      for (int t = 0; t < SYR_REG; ++t)
        if (t >= t0 && 32 * t < n) {
          const int idx = 32 * t + lane;
          acc = fma(a[t], (idx < n) ? v[idx] : 0.0, acc);
        }
#pragma unroll 4
      for (int x = max(0, 32 * t0 - 32 * SYR_REG) + lane; x < nt; x += 32) acc = fma(mytail[x], v[32 * SYR_REG + x], acc);
      acc = __shfl_sync(0xffffffffu, acc, (lane + j + 1) & 31);   // class of lane q in lane q
      acc = wsum(acc) * tau;
      if (lane == 0) __stcg(pg + row, acc);
      if (row == j + 1) {
#pragma unroll
        for (int t = 0; t < SYR_REG; ++t)
          if (32 * t + lane < n) __stcg(rg + 32 * t + lane, a[t]);
        for (int x = lane; x < nt; x += 32) __stcg(rg + 32 * SYR_REG + x, mytail[x]);
      }
    }
    target += gridDim.x;
    if (!syr_barrier(bar, flag, target, spin)) return;
    // p, the products p_i v_i in groups of eight rows, row j + 1
    const int len = n - j - 1;
    for (int l0 = 0; l0 < len; l0 += SYR_THREADS) {
      const int l = l0 + tid;
      double x = 0.0;
      if (l < len) {
        const double pi = __ldcg(pg + j + 1 + l);
        p[j + 1 + l] = pi;
        rw[j + 1 + l] = __ldcg(rg + j + 1 + l);
        x = fma(pi, v[j + 1 + l], 0.0);
      }
      x += __shfl_xor_sync(0xffffffffu, x, 4);
      x += __shfl_xor_sync(0xffffffffu, x, 2);
      x += __shfl_xor_sync(0xffffffffu, x, 1);
      if ((tid & 7) == 0 && l < len) part[l >> 3] = x;
    }
    __syncthreads();
    if (wid == 0) {
      double K = 0.0;
      for (int b = lane; b < ((len + 7) >> 3); b += 32) K += part[b];
      K = wsum(K);
      if (lane == 0) s_K = 0.5 * tau * K;
    } else if (blockIdx.x == 0) {
      // the reflector takes the place of row j
      for (int i = j + 1 + tid - 32; i < n; i += SYR_THREADS - 32) A[(size_t)j * lda + i] = v[i];
      if (tid == 32) {
        d[j] = dnext;
        e[j] = beta;
        tauh[j] = tau;
      }
    }
    __syncthreads();
    const double K = s_K;
    // w, then row j + 1 updated (v[j + 1] = 1)
    const double w1 = p[j + 1] - K * v[j + 1];
    for (int i = tid; i < n; i += SYR_THREADS) {
      if (i <= j) {
        w[i] = 0.0;
        continue;
      }
      const double wi = p[i] - K * v[i];
      w[i] = wi;
      rw[i] = fma(-1.0, wi, fma(-w1, v[i], rw[i]));
    }
    __syncthreads();
    dnext = rw[j + 1];
    if (j + 1 < n - 2) partial(j + 2);
    __syncthreads();
    if (wid == 0 && j + 1 < n - 2) scalars(j + 2);
    if (own && row > j) {
      const double vi = v[row], wi = w[row];
#pragma unroll
      for (int t = 0; t < SYR_REG; ++t)
        if (t >= t0 && 32 * t < n) {
          const int idx = 32 * t + lane;
          const double wl = (idx < n) ? w[idx] : 0.0, vl = (idx < n) ? v[idx] : 0.0;
          a[t] = fma(-vi, wl, fma(-wi, vl, a[t]));
        }
#pragma unroll 4
      for (int x = max(0, 32 * t0 - 32 * SYR_REG) + lane; x < nt; x += 32)
        mytail[x] = fma(-vi, w[32 * SYR_REG + x], fma(-wi, v[32 * SYR_REG + x], mytail[x]));
    }
    __syncthreads();
    if (j + 1 < n - 2) finish(j + 2, vn);
    __syncthreads();
  }
  // the last two rows: through shared memory, every entry at its index
  if (own && row >= n - 2) {
#pragma unroll
    for (int t = 0; t < SYR_REG; ++t) {
      const int idx = 32 * t + lane;
      if (idx >= n - 2 && idx < n) {
        if (idx == row) d[row] = a[t];
        else if (row == n - 2) e[n - 2] = a[t];
      }
    }
    for (int x = lane; x < nt; x += 32) {
      const int idx = 32 * SYR_REG + x;
      if (idx >= n - 2) {
        if (idx == row) d[row] = mytail[x];
        else if (row == n - 2) e[n - 2] = mytail[x];
      }
    }
    if (lane == 0) {
      tauh[row] = 0.0;
      if (row == n - 1) e[n - 1] = 0.0;
    }
  }
}

// Cluster form for small n: one thread-block cluster of SY_CS CTAs, so that
// the two barriers per column are hardware cluster barriers instead of grid
// barriers through global atomics, and the rest of the GPU stays free for
// other problems.  A stays in global memory (L2); warp g of the cluster owns
// rows i = g mod (number of warps) for the whole reduction.  Per column j:
//   every CTA rebuilds the reflector from row j (loaded through L2);
//   p_i = tau A22[i, :] v for the owned rows, each p_i broadcast into every
//   CTA's shared memory, and the CTA's share of p^T v likewise;
//   cluster barrier;  w = p - (tau / 2)(p^T v) v;  owned rows updated;
//   cluster barrier (row j + 1 is complete before anyone reads it).
// The shared arrays written remotely in column j + 1 are only read in steps of
// column j that precede its second barrier, so no buffer is overwritten early.
constexpr int SY_THREADS = 512;
__global__ void __launch_bounds__(SY_THREADS) k_sytrd_cluster(int n, double* A, int lda, double* d, double* e,
                                                               double* tauh) {
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  extern __shared__ double sm[];
  double* v = sm;            // n
  double* w = sm + n;        // n
  double* p = sm + 2 * n;    // n   (written by every CTA)
  __shared__ double kpart[32];  // one partial of p^T v per CTA of the cluster
  __shared__ double red[32];
  __shared__ double s_tau, s_beta, s_scale;
  const int wpb = blockDim.x / 32, wid = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int gwarp = rank * wpb + wid, nwarps = cs * wpb;

  for (int j = 0; j < n - 2; ++j) {
    const int len = n - j - 1;
    const double* row = A + (size_t)j * lda + j + 1;
    double s = 0.0;
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      const double x = __ldcg(row + i);
      v[i] = x;
      if (i > 0) s = fma(x, x, s);
    }
    s = bsum(s, red);
    if (threadIdx.x == 0) {
      const double x0 = v[0];
      double tau = 0.0, beta = x0, scale = 0.0;
      if (s > 0.0) {
        beta = -copysign(sqrt(fma(x0, x0, s)), x0);
        tau = (beta - x0) / beta;
        scale = 1.0 / (x0 - beta);
      }
      s_tau = tau; s_beta = beta; s_scale = scale;
    }
    __syncthreads();
    const double tau = s_tau, scale = s_scale;
    for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) v[i] *= scale;
    if (threadIdx.x == 0) v[0] = 1.0;
    __syncthreads();
    // owned rows: first owned row index >= j + 1
    double kp = 0.0;
    int i = gwarp + ((j + 1 - gwarp + nwarps - 1) / nwarps) * nwarps;
    if (gwarp >= j + 1) i = gwarp;
    for (; i < n; i += nwarps) {
      const double* ai = A + (size_t)i * lda + j + 1;
      // four independent accumulators keep four L2 loads in flight per lane
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
      int l = lane;
      for (; l + 96 < len; l += 128) {
        const double x0 = __ldcg(ai + l), x1 = __ldcg(ai + l + 32), x2 = __ldcg(ai + l + 64),
                     x3 = __ldcg(ai + l + 96);
        a0 = fma(x0, v[l], a0);
        a1 = fma(x1, v[l + 32], a1);
        a2 = fma(x2, v[l + 64], a2);
        a3 = fma(x3, v[l + 96], a3);
      }
      for (; l < len; l += 32) a0 = fma(__ldcg(ai + l), v[l], a0);
      double acc = wsum((a0 + a1) + (a2 + a3)) * tau;
      if (lane < cs) {
        double* dst = cluster.map_shared_rank(p, lane);
        dst[i - j - 1] = acc;
      }
      if (lane == 0) kp = fma(acc, v[i - j - 1], kp);
    }
    kp = bsum(kp, red);                                  // valid in thread 0
    const double kp0 = __shfl_sync(0xffffffffu, kp, 0);  // warp 0: every lane gets it
    if (threadIdx.x < cs) {
      double* dst = cluster.map_shared_rank(kpart, (int)threadIdx.x);
      dst[rank] = kp0;
    }
    cluster.sync();
    double K = 0.0;
    for (int c = 0; c < cs; ++c) K += kpart[c];
    K *= 0.5 * tau;
    for (int l = threadIdx.x; l < len; l += blockDim.x) w[l] = p[l] - K * v[l];
    __syncthreads();
    i = gwarp + ((j + 1 - gwarp + nwarps - 1) / nwarps) * nwarps;
    if (gwarp >= j + 1) i = gwarp;
    for (; i < n; i += nwarps) {
      double* ai = A + (size_t)i * lda + j + 1;
      const double vi = v[i - j - 1], wi = w[i - j - 1];
      int l = lane;
      for (; l + 96 < len; l += 128) {
        const double x0 = __ldcg(ai + l), x1 = __ldcg(ai + l + 32), x2 = __ldcg(ai + l + 64),
                     x3 = __ldcg(ai + l + 96);
        ai[l] = fma(-vi, w[l], fma(-wi, v[l], x0));
        ai[l + 32] = fma(-vi, w[l + 32], fma(-wi, v[l + 32], x1));
        ai[l + 64] = fma(-vi, w[l + 64], fma(-wi, v[l + 64], x2));
        ai[l + 96] = fma(-vi, w[l + 96], fma(-wi, v[l + 96], x3));
      }
      for (; l < len; l += 32) {
        const double x = __ldcg(ai + l);
        ai[l] = fma(-vi, w[l], fma(-wi, v[l], x));
      }
    }
    if (rank == 0) {
      double* rj = A + (size_t)j * lda + j + 1;
      for (int l = threadIdx.x; l < len; l += blockDim.x) rj[l] = v[l];
      if (threadIdx.x == 0) {
        d[j] = __ldcg(A + (size_t)j * lda + j);
        e[j] = s_beta;
        tauh[j] = tau;
      }
    }
    cluster.sync();
  }
  if (rank == 0 && threadIdx.x == 0) {
    if (n >= 2) {
      d[n - 2] = __ldcg(A + (size_t)(n - 2) * lda + n - 2);
      e[n - 2] = __ldcg(A + (size_t)(n - 2) * lda + n - 1);
      tauh[n - 2] = 0.0;
    }
    d[n - 1] = __ldcg(A + (size_t)(n - 1) * lda + n - 1);
    e[n - 1] = 0.0;
    if (n >= 2) tauh[n - 1] = 0.0;
  }
}

// Shared-memory-resident cluster form for orders whose matrix fits in the
// distributed shared memory of one cluster: row i lives in CTA i mod cs (slot
// i / cs) for the whole reduction, so the matrix-vector product and the rank-2
// update of every column read and write shared memory instead of streaming the
// trailing matrix through L2.  Per column j: every CTA copies row j from the CTA
// that owns it (a distributed-shared-memory read) and rebuilds the reflector;
// p_i = tau A22[i, :] v for the owned rows, broadcast into every CTA's p;
// cluster barrier; w = p - (tau / 2)(p^T v) v; owned rows updated; the owner of
// row j stores the reflector in it; cluster barrier.  Row j is read by the other
// CTAs before the first barrier and overwritten by its owner after it, and row
// j + 1 is complete at the second barrier, before anyone reads it.  The rows
// return to global memory at the end (the back-transformation reads them).
__global__ void __launch_bounds__(SY_THREADS) k_sytrd_cluster_smem(int n, double* A, int lda, double* d, double* e,
                                                                    double* tauh) {
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  extern __shared__ double sm[];
  const int slots = (n + cs - 1) / cs;
  double* rows = sm;                         // slots x n, row-major
  double* v = rows + (size_t)slots * n;      // n
  double* w = v + n;                         // n
  double* p = w + n;                         // n   (written by every CTA)
  __shared__ double kpart[32];
  __shared__ double red[32];
  __shared__ double s_tau, s_beta, s_scale;
  const int wpb = blockDim.x / 32, wid = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int sl = 0; sl < slots; ++sl) {
    const int i = sl * cs + rank;
    if (i >= n) break;
    for (int c = threadIdx.x; c < n; c += blockDim.x) rows[(size_t)sl * n + c] = __ldcg(A + (size_t)i * lda + c);
  }
  cluster.sync();
  for (int j = 0; j < n - 2; ++j) {
    const int len = n - j - 1;
    const double* rowj = cluster.map_shared_rank(rows, j % cs) + (size_t)(j / cs) * n + j + 1;
    double s = 0.0;
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      const double x = rowj[i];
      v[i] = x;
      if (i > 0) s = fma(x, x, s);
    }
    s = bsum(s, red);
    if (threadIdx.x == 0) {
      const double x0 = v[0];
      double tau = 0.0, beta = x0, scale = 0.0;
      if (s > 0.0) {
        beta = -copysign(sqrt(fma(x0, x0, s)), x0);
        tau = (beta - x0) / beta;
        scale = 1.0 / (x0 - beta);
      }
      s_tau = tau; s_beta = beta; s_scale = scale;
    }
    __syncthreads();
    const double tau = s_tau, scale = s_scale;
    for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) v[i] *= scale;
    if (threadIdx.x == 0) v[0] = 1.0;
    __syncthreads();
    // owned rows i = sl cs + rank > j
    const int sl0 = (j + 1 > rank) ? (j + 1 - rank + cs - 1) / cs : 0;
    double kp = 0.0;
    for (int sl = sl0 + wid; sl < slots; sl += wpb) {
      const int i = sl * cs + rank;
      if (i >= n) break;
      const double* ai = rows + (size_t)sl * n + j + 1;
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
      int l = lane;
      for (; l + 96 < len; l += 128) {
        a0 = fma(ai[l], v[l], a0);
        a1 = fma(ai[l + 32], v[l + 32], a1);
        a2 = fma(ai[l + 64], v[l + 64], a2);
        a3 = fma(ai[l + 96], v[l + 96], a3);
      }
      for (; l < len; l += 32) a0 = fma(ai[l], v[l], a0);
      const double acc = wsum((a0 + a1) + (a2 + a3)) * tau;
      if (lane < cs) {
        double* dst = cluster.map_shared_rank(p, lane);
        dst[i - j - 1] = acc;
      }
      if (lane == 0) kp = fma(acc, v[i - j - 1], kp);
    }
    kp = bsum(kp, red);
    const double kp0 = __shfl_sync(0xffffffffu, kp, 0);
    if (threadIdx.x < cs) {
      double* dst = cluster.map_shared_rank(kpart, (int)threadIdx.x);
      dst[rank] = kp0;
    }
    cluster.sync();
    double K = 0.0;
    for (int c = 0; c < cs; ++c) K += kpart[c];
    K *= 0.5 * tau;
    for (int l = threadIdx.x; l < len; l += blockDim.x) w[l] = p[l] - K * v[l];
    __syncthreads();
    for (int sl = sl0 + wid; sl < slots; sl += wpb) {
      const int i = sl * cs + rank;
      if (i >= n) break;
      double* ai = rows + (size_t)sl * n + j + 1;
      const double vi = v[i - j - 1], wi = w[i - j - 1];
      for (int l = lane; l < len; l += 32) ai[l] = fma(-vi, w[l], fma(-wi, v[l], ai[l]));
    }
    if (rank == j % cs) {
      double* rj = rows + (size_t)(j / cs) * n;
      for (int l = threadIdx.x; l < len; l += blockDim.x) rj[j + 1 + l] = v[l];
      if (threadIdx.x == 0) {
        d[j] = rj[j];
        e[j] = s_beta;
        tauh[j] = tau;
      }
    }
    cluster.sync();
  }
  if (threadIdx.x == 0) {
    if (n >= 2 && rank == (n - 2) % cs) {
      const double* r2 = rows + (size_t)((n - 2) / cs) * n;
      d[n - 2] = r2[n - 2];
      e[n - 2] = r2[n - 1];
      tauh[n - 2] = 0.0;
    }
    if (rank == (n - 1) % cs) {
      d[n - 1] = rows[(size_t)((n - 1) / cs) * n + n - 1];
      e[n - 1] = 0.0;
      if (n >= 2) tauh[n - 1] = 0.0;
    }
  }
  for (int sl = 0; sl < slots; ++sl) {
    const int i = sl * cs + rank;
    if (i >= n) break;
    for (int c = threadIdx.x; c < n; c += blockDim.x) A[(size_t)i * lda + c] = rows[(size_t)sl * n + c];
  }
}

// One-triangle shared-memory cluster form.  Row i keeps only its lower part
// A[i][0..i] (packed) in CTA i mod cs, so the matrix of order up to ~880 fits
// one 16-CTA cluster, and the symmetric rank-2 update touches one triangle:
// 2 len^2 FMAs per column instead of the 3 len^2 of the full-storage form.
// With lower storage, p = A22 v splits into a row part (the owner's dot of its
// lower row with v) and a column part (for column c, the sum over rows i > c
// of A[i][c] v_i, which every CTA forms over its own rows).  Per column j:
//   1: the CTA's column parts (thread per column) and row parts (warp per owned
//      row); cluster barrier;
//   2: the owner of row i adds its row part to the 16 CTAs' column parts for i
//      (fixed order), scales by tau and broadcasts p_i and its share of p^T v;
//      cluster barrier;
//   3: w = p - (tau / 2)(p^T v) v.  Every CTA has column j + 1 as it was before this
//      update (the owners broadcast it a column earlier) and updates it itself, so
//      the next reflector starts at once: one warp forms its scalars while the
//      warps of the other three schedulers update the owned rows on c in [j + 1, i],
//      store the reflector in column j and broadcast column j + 2.
// Three vectors rotate: b0 the reflector, b1 column j + 1, b2 first the column
// parts, then column j + 2.  Remote writes and the barriers that order them: b2 is
// written in step 3, after barrier 2 ended the reading of the column parts, and read
// in step 3 of the next column; p and kpart are written between barriers 1 and 2
// and read after barrier 2.  Every sum runs in a fixed order (those over the
// reflector in 512 threads' order, p^T v in that of 16 warps), so the result does not
// depend on timing.  An FP64 warp instruction holds its scheduler's pipe for 64
// cycles however many lanes it serves, so the trees of the sums share instructions:
// the first two levels in the warp that formed the sum, the others (and the 16 column
// parts of a row) four lanes per row.  At n = 565 the pipe bounds the first columns,
// latency the last ones.  With three barriers, 512 threads and the scalars on the way
// of the update a column took 15.4 us on average (n = 565: 8.7 ms), with whole warps
// for each sum 12.0 us (6.8 ms), now 10.9 us (6.1 ms).  At the end the rows are written back with
// the lower part mirrored into the upper one: row j then holds the reflector in
// A[j][j+1..], as the back-transformation expects.
constexpr int SYL_THREADS = 1024;
__device__ __forceinline__ size_t sy_off(int sl, int cs, int rank) {
  return (size_t)cs * sl * (sl - 1) / 2 + (size_t)sl * (rank + 1);
}
__global__ void __launch_bounds__(SYL_THREADS, 1) k_sytrd_cluster_lower(int n, double* A, int lda, double* d,
                                                                         double* e, double* tauh) {
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  extern __shared__ double sm[];
  const int slots = (n - rank + cs - 1) / cs;      // owned rows i = sl cs + rank < n
  // the vectors come first, at the same offset in every CTA (a remote access
  // maps the local offset); the packed rows, whose length depends on the
  // rank, follow them
  double* p = sm + 3 * (size_t)n;   // n (at least 8): tau A22 v (written remotely), then w
  double* rowp = p + max(n, 8);     // ceil(n / cs): row parts, then p_i, of the owned rows
  double* rows = rowp + (n + cs - 1) / cs;
  __shared__ double kpart[32];
  __shared__ double red[16][8];
  __shared__ double s_tau, s_beta, s_scale, s_K, s_w0;
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31, nw = SYL_THREADS / 32;
  for (int sl = 0; sl < slots; ++sl) {
    const int i = sl * cs + rank;
    double* ri = rows + sy_off(sl, cs, rank);
    for (int c = tid; c <= i; c += SYL_THREADS) ri[c] = __ldcg(A + (size_t)i * lda + c);
  }
  cluster.sync();
  // columns 0 and 1 to every CTA
  for (int sl = wid; sl < slots; sl += nw) {
    const int i = sl * cs + rank;
    const double* ri = rows + sy_off(sl, cs, rank);
    if (i >= 1 && lane < cs) cluster.map_shared_rank(sm, lane)[i - 1] = ri[0];
    if (i >= 2 && lane < cs) cluster.map_shared_rank(sm, lane)[n + i - 2] = ri[1];
  }
  cluster.sync();
  // sum of squares of x[1..len) in the order of 512 threads: warps 0 to 15, whose sums
  // (levels 4, 2, 1) end in scalars
  auto partial = [&](const double* x, int len) {
    if (tid < 512) {
      double s = 0.0;
      if (wid * 32 < len) {
        for (int l = tid; l < len; l += 512)
          if (l > 0) s = fma(x[l], x[l], s);
        s += __shfl_xor_sync(0xffffffffu, s, 16);
        s += __shfl_xor_sync(0xffffffffu, s, 8);
      }
      if (lane < 8) red[wid][lane] = s;
    }
  };
  auto scalars = [&](const double* x) {   // warp 0; the two quotients in two lanes
    // two lanes per warp of partial, four values each
    const double* rd = red[lane >> 1] + (lane & 1);
    double s = (rd[0] + rd[4]) + (rd[2] + rd[6]);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s = __shfl_sync(0xffffffffu, s, (2 * lane) & 31);
    s = wsum(lane < 16 ? s : 0.0);
    const double x0 = x[0];
    double tau = 0.0, beta = x0, scale = 0.0;
    if (s > 0.0) {
      beta = -copysign(sqrt(fma(x0, x0, s)), x0);
      const double q = (lane == 1 ? 1.0 : beta - x0) / (lane == 1 ? x0 - beta : beta);
      tau = __shfl_sync(0xffffffffu, q, 0);
      scale = __shfl_sync(0xffffffffu, q, 1);
    }
    if (lane == 0) {
      s_tau = tau;
      s_beta = beta;
      s_scale = scale;
    }
  };
  partial(sm, n - 1);
  __syncthreads();
  if (wid == 0) scalars(sm);
  __syncthreads();
  for (int l = tid; l < n - 1; l += SYL_THREADS) sm[l] = (l == 0) ? 1.0 : sm[l] * s_scale;
  __syncthreads();
  int rot = 0;                       // b0 = sm + rot n
  for (int j = 0; j < n - 2; ++j) {
    const int len = n - j - 1;
    const double* v = sm + (size_t)rot * n;
    const int r1 = (rot == 2) ? 0 : rot + 1, r2 = (r1 == 2) ? 0 : r1 + 1;
    double* xn = sm + (size_t)r1 * n;
    double* part = sm + (size_t)r2 * n;
    const double tau = s_tau, beta = s_beta;
    // ---- 1: column parts and row parts
    // (groups of four warps there and back: the first columns are the longest sums)
    for (int l = (wid & 4) ? tid + 32 * (3 - 2 * (wid & 3)) : tid; l < len; l += SYL_THREADS) {
      const int c = j + 1 + l;
      int sl = (c >= rank) ? (c - rank) / cs + 1 : 0;   // first owned row > c
      double acc = 0.0;
      size_t o = sy_off(sl, cs, rank);
#pragma unroll 4
      for (int i = sl * cs + rank; i < n; i += cs) {
        acc = fma(rows[o + c], v[i - j - 1], acc);
        o += (size_t)i + 1;                          // row i holds i + 1 entries
      }
      part[l] = acc;
    }
    const int sl0 = (j + 1 > rank) ? (j + 1 - rank + cs - 1) / cs : 0;   // first owned row > j
    for (int sl = sl0 + wid; sl < slots; sl += nw) {
      const int i = sl * cs + rank;
      const double* ri = rows + sy_off(sl, cs, rank) + j + 1;
      const int cnt = i - j;                         // c = j + 1 .. i
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
      int l = lane;
      for (; l + 96 < cnt; l += 128) {
        a0 = fma(ri[l], v[l], a0);
        a1 = fma(ri[l + 32], v[l + 32], a1);
        a2 = fma(ri[l + 64], v[l + 64], a2);
        a3 = fma(ri[l + 96], v[l + 96], a3);
      }
      for (; l < cnt; l += 32) a0 = fma(ri[l], v[l], a0);
      double s = (a0 + a1) + (a2 + a3);
      s += __shfl_xor_sync(0xffffffffu, s, 16);
      s += __shfl_xor_sync(0xffffffffu, s, 8);
      if (lane < 8) p[8 * (sl - sl0) + lane] = s;    // p is free until barrier 1
    }
    __syncthreads();
    // the sums' levels 4, 2, 1, four lanes per row
    for (int base = sl0 + 8 * wid; base < slots; base += 8 * nw) {
      const int sl = base + (lane >> 2);
      const double* x = p + 8 * (min(sl, slots - 1) - sl0) + (lane & 3);
      double s = x[0] + x[4];
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      if ((lane & 3) == 0 && sl < slots) rowp[sl] = s;
    }
    cluster.sync();
    // ---- 2: p_i for the owned rows, broadcast
    // four lanes per row, four of the 16 column parts and of the 16 copies each
    for (int base = sl0 + 8 * wid; base < slots; base += 8 * nw) {
      const int sl = base + (lane >> 2), q = lane & 3;
      const bool on = sl < slots;
      const int li = (on ? sl : slots - 1) * cs + rank - j - 1;
      double x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = cluster.map_shared_rank(part, q + 4 * u)[li];
      double s = (x[0] + x[2]) + (x[1] + x[3]);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      const double pi = (rowp[on ? sl : slots - 1] + (s + 0.0)) * tau;   // a sum of zeros is +0
      if (on) {
#pragma unroll
        for (int u = 0; u < 4; ++u) cluster.map_shared_rank(p, q + 4 * u)[li] = pi;
      }
      __syncwarp();
      if (on && q == 0) rowp[sl] = pi;
    }
    __syncthreads();
    if (wid == 0) {
      double kp = 0.0;
      if (lane < 16)
        for (int sl = sl0 + lane; sl < slots; sl += 16) kp = fma(rowp[sl], v[sl * cs + rank - j - 1], kp);
      kp = wsum(kp);
      if (lane < cs) cluster.map_shared_rank(kpart, lane)[rank] = kp;
    }
    cluster.sync();
    // ---- 3: w and the next column
    if (wid == 0) {
      double K = 0.0;
      for (int c = 0; c < cs; ++c) K += kpart[c];
      K *= 0.5 * tau;
      if (lane == 0) {
        s_K = K;
        s_w0 = p[0] - K * v[0];
      }
    }
    __syncthreads();
    const double K = s_K, w0 = s_w0;
    for (int l = tid; l < len; l += SYL_THREADS) {
      const double wl = (l == 0) ? w0 : p[l] - K * v[l];
      p[l] = wl;
      if (l > 0) xn[l - 1] = fma(-v[l], w0, fma(-wl, 1.0, xn[l - 1]));
    }
    __syncthreads();
    const bool more = j + 1 < n - 2;
    if (more) partial(xn, len - 1);
    __syncthreads();
    if (wid == 0 && more) scalars(xn);
    if ((wid & 3) != 0) {
      const double* w = p;
      for (int sl = sl0 + (wid >> 2) * 3 + (wid & 3) - 1; sl < slots; sl += nw / 4 * 3) {
        const int i = sl * cs + rank;
        const int li = i - j - 1;
        double* ri = rows + sy_off(sl, cs, rank);
        const double vi = v[li], wi = w[li];
        const int cnt = i - j;
        double* rr = ri + j + 1;
        for (int l = lane; l < cnt; l += 32) rr[l] = fma(-vi, w[l], fma(-wi, v[l], rr[l]));
        __syncwarp();
        if (lane == 0) ri[j] = vi;                       // reflector entry (row i, column j)
        if (i > j + 2 && lane < cs) cluster.map_shared_rank(part, lane)[i - j - 3] = ri[j + 2];
      }
      if (tid == 32) {
        if (rank == j % cs) d[j] = rows[sy_off(j / cs, cs, rank) + j];
        if (rank == 0) {
          e[j] = beta;
          tauh[j] = tau;
        }
      }
    }
    __syncthreads();
    if (more) {
      const double scale = s_scale;
      for (int l = tid; l < len - 1; l += SYL_THREADS) xn[l] = (l == 0) ? 1.0 : xn[l] * scale;
    }
    __syncthreads();
    rot = r1;
  }
  if (tid == 0) {
    if (rank == (n - 2) % cs) {
      d[n - 2] = rows[sy_off((n - 2) / cs, cs, rank) + n - 2];
      tauh[n - 2] = 0.0;
    }
    if (rank == (n - 1) % cs) {
      const double* rl = rows + sy_off((n - 1) / cs, cs, rank);
      d[n - 1] = rl[n - 1];
      e[n - 2] = rl[n - 2];
      e[n - 1] = 0.0;
      tauh[n - 1] = 0.0;
    }
  }
  for (int sl = 0; sl < slots; ++sl) {
    const int i = sl * cs + rank;
    const double* ri = rows + sy_off(sl, cs, rank);
    for (int c = tid; c <= i; c += SYL_THREADS) {
      const double x = ri[c];
      A[(size_t)i * lda + c] = x;
      A[(size_t)c * lda + i] = x;
    }
  }
  cluster.sync();   // no CTA leaves while another may still write into its shared memory
}

// One-triangle form for orders up to SYT_MAX_N: the same sums in the same order by one
// CTA.  Warp r forms the column parts of the rows i = r mod 16 (CTA r's in the
// cluster form), a row's dot and the sum of its 16 column parts take four lanes, warp 0
// the sums over all rows and the next reflector while the others update.  Bound by the
// chain of FP64 instructions of a column; the cluster form waits for two cluster barriers
// and three remote accesses as well.  n = 40: 224 -> 169 us.
constexpr int SYT_MAX_N = 64, SYT_LD = SYT_MAX_N + 1, SYT_THREADS = 512;
__global__ void __launch_bounds__(SYT_THREADS) k_sytrd_small(int n, double* A, int lda, double* d, double* e,
                                                             double* tauh) {
  __shared__ double a[SYT_MAX_N * SYT_LD], part[16][SYT_MAX_N], sv[2][SYT_MAX_N], sw[SYT_MAX_N], p[SYT_MAX_N];
  __shared__ double s_tau, s_beta;
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
  for (int t = tid; t < n * n; t += SYT_THREADS) {
    const int i = t / n, c = t - i * n;
    if (c <= i) a[i * SYT_LD + c] = __ldcg(A + (size_t)i * lda + c);
  }
  // Warp 0: the reflector of x (lane holds x0 = x[lane], x1 = x[lane + 32], m entries),
  // its vector to v
  auto reflector = [&](double x0, double x1, int m, double* v) {
    double s = (lane > 0 && lane < m) ? fma(x0, x0, 0.0) : 0.0;
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    if (m > 32) {
      double s1 = (lane + 32 < m) ? fma(x1, x1, 0.0) : 0.0;
      s1 += __shfl_xor_sync(0xffffffffu, s1, 16);
      if (lane >= 16) s = s1;      // entries 32 and on in the upper lanes
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (m > 32) s = __shfl_sync(0xffffffffu, s, 0) + __shfl_sync(0xffffffffu, s, 16);
    const double xf = __shfl_sync(0xffffffffu, x0, 0);
    double tau = 0.0, beta = xf, scale = 0.0;
    if (s > 0.0) {
      beta = -copysign(sqrt(fma(xf, xf, s)), xf);
      const double q = (lane == 1 ? 1.0 : beta - xf) / (lane == 1 ? xf - beta : beta);
      tau = __shfl_sync(0xffffffffu, q, 0);
      scale = __shfl_sync(0xffffffffu, q, 1);
    }
    if (lane == 0) {
      s_tau = tau;
      s_beta = beta;
    }
    if (lane < m) v[lane] = (lane == 0) ? 1.0 : x0 * scale;
    if (lane + 32 < m) v[lane + 32] = x1 * scale;
  };
  __syncthreads();
  if (wid == 0) {
    const int m = n - 1;
    reflector(lane < m ? a[(lane + 1) * SYT_LD] : 0.0, lane + 32 < m ? a[(lane + 33) * SYT_LD] : 0.0, m, sv[0]);
  }
  __syncthreads();
  for (int j = 0; j < n - 2; ++j) {
    const int len = n - j - 1;
    const double* v = sv[j & 1];
    const double tau = s_tau, beta = s_beta;
    // ---- 1: column parts; row dots
    for (int l = lane; l < len; l += 32) {
      const int c = j + 1 + l;
      double acc = 0.0;
      for (int i = (c >= wid) ? c + 16 - ((c - wid) & 15) : wid; i < n; i += 16)
        acc = fma(a[i * SYT_LD + c], v[i - j - 1], acc);
      part[wid][l] = acc;
    }
    const int li = (SYT_THREADS / 32 - 1 - wid) * 8 + (lane >> 2), q = lane & 3;   // row j + 1 + li
    const bool rows = (li & ~7) < len;   // of the whole warp
    double dot = 0.0;
    if (rows) {
      const int cnt = (li < len) ? li + 1 : 0;
      const double* ri = a + (j + 1 + min(li, len - 1)) * SYT_LD + j + 1;
      double f[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int x = q + 4 * m;
        f[m] = (x < cnt) ? fma(ri[x], v[x], 0.0) : 0.0;
        if ((li | 7) >= 32) f[m] = (x + 32 < cnt) ? fma(ri[x + 32], v[x + 32], f[m]) : f[m];
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) f[m] += f[m + 4];
      f[0] += f[2];
      f[1] += f[3];
      dot = f[0] + f[1];
      dot += __shfl_xor_sync(0xffffffffu, dot, 2);
      dot += __shfl_xor_sync(0xffffffffu, dot, 1);
    }
    __syncthreads();
    // ---- 2: p
    if (rows) {
      const int r = min(li, len - 1);
      double s = (part[q][r] + part[q + 8][r]) + (part[q + 4][r] + part[q + 12][r]);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      if (li < len && q == 0) p[li] = (dot + (s + 0.0)) * tau;   // a sum of zeros is +0
    }
    __syncthreads();
    // ---- 3: warp 0: p^T v by the cluster form's shares, w and the next column
    double x0 = 0.0, x1 = 0.0;
    if (wid == 0) {
      const int r = lane & 15;
      const int i0 = (j + 1 > r) ? j + 1 + ((r - j - 1) & 15) : r;   // first row of share r after j
      double kq[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int l = i0 + 16 * u - j - 1;
        kq[u] = 0.0;
        if (16 * u < len) kq[u] = (l < len) ? fma(p[l], v[l], 0.0) : 0.0;
      }
      double kp = kq[0];
      if (len > 32) kp = (kq[0] + kq[2]) + (kq[1] + kq[3]);
      else if (len > 16) kp = kq[0] + kq[1];
      double K = 0.0;
#pragma unroll
      for (int c = 0; c < 16; ++c) K += __shfl_sync(0xffffffffu, kp, c);
      K *= 0.5 * tau;
      const double w0 = p[0] - K * v[0];
      auto next = [&](int l) {   // w[l], returns the updated entry of column j + 1 in row j + 1 + l
        const double vl = v[l], wl = p[l] - K * vl;
        sw[l] = wl;
        return fma(-vl, w0, fma(-wl, 1.0, a[(j + 1 + l) * SYT_LD + j + 1]));
      };
      if (lane == 0) sw[0] = w0;
      if (lane + 1 < len) x0 = next(lane + 1);
      if (len > 33 && lane + 33 < len) x1 = next(lane + 33);
    }
    __syncthreads();
    if (wid == 0 && j + 1 < n - 2) reflector(x0, x1, len - 1, sv[(j + 1) & 1]);
    if ((wid & 3) != 0) {
      for (int l0 = (wid >> 2) * 3 + (wid & 3) - 1; l0 < len; l0 += 12) {
        double* ri = a + (j + 1 + l0) * SYT_LD;
        const double vi = v[l0], wi = sw[l0];
        for (int l = lane; l <= l0; l += 32) ri[j + 1 + l] = fma(-vi, sw[l], fma(-wi, v[l], ri[j + 1 + l]));
        if (lane == 0) ri[j] = vi;
      }
      if (tid == 32) {
        d[j] = a[j * SYT_LD + j];
        e[j] = beta;
        tauh[j] = tau;
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    d[n - 2] = a[(n - 2) * SYT_LD + n - 2];
    e[n - 2] = a[(n - 1) * SYT_LD + n - 2];
    tauh[n - 2] = 0.0;
    d[n - 1] = a[(n - 1) * SYT_LD + n - 1];
    e[n - 1] = 0.0;
    tauh[n - 1] = 0.0;
  }
  for (int t = tid; t < n * n; t += SYT_THREADS) {
    const int i = t / n, c = t - i * n;
    A[(size_t)i * lda + c] = (c <= i) ? a[i * SYT_LD + c] : a[c * SYT_LD + i];
  }
}

static size_t sytrd_lower_smem_bytes(int n, int cs) {
  size_t most = 0;   // packed rows of the rank that holds the most
  for (int rank = 0; rank < cs; ++rank) {
    const int slots = (n - rank + cs - 1) / cs;
    most = std::max(most, (size_t)cs * slots * (slots - 1) / 2 + (size_t)slots * (rank + 1));
  }
  return (3 * (size_t)n + std::max(n, 8) + (size_t)(n + cs - 1) / cs + most) * sizeof(double);
}

// Cluster size of the shared-memory form for order n: 16 when the matrix and the
// work vectors fit in 16 CTAs' shared memory and the device runs such a
// cluster; 0 otherwise.
static size_t sytrd_smem_bytes(int n, int cs) {
  return ((size_t)((n + cs - 1) / cs) * n + 3 * (size_t)n) * sizeof(double);
}
static int sytrd_smem_cluster(int n) {
  static int max_optin = -1;
  static int ok16 = -1;
  if (max_optin < 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  }
  const int cs = 16;
  const size_t need = sytrd_smem_bytes(n, cs);
  if (need + 2048 > (size_t)max_optin) return 0;
  if (ok16 < 0) {
    allow_max_smem((const void*)k_sytrd_cluster_smem);
    cudaFuncSetAttribute((const void*)k_sytrd_cluster_smem, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(SY_THREADS);
    cfg.dynamicSmemBytes = (size_t)max_optin - 2048;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int ncl = 0;
    ok16 = (cudaOccupancyMaxActiveClusters(&ncl, (const void*)k_sytrd_cluster_smem, &cfg) == cudaSuccess && ncl > 0)
               ? 1 : 0;
    cudaGetLastError();
  }
  return ok16 ? cs : 0;
}

// Cluster size of the one-triangle form for order n (16, or 0 when the packed
// rows and work vectors do not fit 16 CTAs' shared memory or the device does
// not run such a cluster).
static int sytrd_lower_cluster(int n) {
  static int max_optin = -1;
  static int ok16 = -1;
  if (max_optin < 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  }
  const int cs = 16;
  if (sytrd_lower_smem_bytes(n, cs) + 2048 > (size_t)max_optin) return 0;
  if (ok16 < 0) {
    allow_max_smem((const void*)k_sytrd_cluster_lower);
    cudaFuncSetAttribute((const void*)k_sytrd_cluster_lower, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(SYL_THREADS);
    cfg.dynamicSmemBytes = (size_t)max_optin - 2048;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int ncl = 0;
    ok16 = (cudaOccupancyMaxActiveClusters(&ncl, (const void*)k_sytrd_cluster_lower, &cfg) == cudaSuccess &&
            ncl > 0) ? 1 : 0;
    cudaGetLastError();
  }
  return ok16 ? cs : 0;
}

// Cluster size for k_sytrd_cluster: 16 where the device allows it, else 8
// (0 = cluster launch unavailable).
static int sytrd_cluster_size(size_t smem) {
  static int cached = -1;
  if (cached >= 0) return cached;
  allow_max_smem((const void*)k_sytrd_cluster);
  cudaFuncSetAttribute((const void*)k_sytrd_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaGetLastError();
  cached = 0;
  for (int cs : {16, 8}) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(SY_THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, (const void*)k_sytrd_cluster, &cfg) == cudaSuccess && ncl > 0) {
      cached = cs;
      break;
    }
    cudaGetLastError();
  }
  return cached;
}

static int sytrd_blocks(int n, size_t smem) {
  static int cached_sms = 0;
  if (!cached_sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&cached_sms, cudaDevAttrMultiProcessorCount, dev);
  }
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sytrd, 256, smem);
  occ = std::max(1, std::min(occ, 2));
  int blocks = cached_sms * occ;
  const int want = (n + 7) / 8;  // 8 warps per CTA, one row per warp is enough
  blocks = std::max(1, std::min(blocks, std::max(want, cached_sms)));
  return std::min(blocks, 4096);
}

// Up to this order the cluster form is faster (the cooperative grid form wins
// once the O(n^3) work needs the whole GPU).
constexpr int SY_CLUSTER_MAX_N = 1024;

// Order of preference: up to order 64 the one-CTA form of the one-triangle sums (64: 44 KB of
// static shared memory, one column chunk of 32 lanes twice); the one-triangle form in cluster shared memory
// (n <= 880); the full-row form (n <= 656, where the device cannot run the
// first); the L2-streaming cluster form; above order 1024 the resident form, then the
// cooperative grid form.  The one-triangle form also leaves more room on its 16 SMs
// for the other problems' kernels of a batch.
static sdp_status sytrd(cudaStream_t st, int n, double* A, EigWork* w) {
  // one CTA forms the cluster form's sums, so it stands in for it only where that runs
  if (n >= 3 && n <= SYT_MAX_N && sytrd_lower_cluster(n) == 16) {
    count_launch();
    ktimer_begin(st, "sytrd");
    k_sytrd_small<<<1, SYT_THREADS, 0, st>>>(n, A, n, w->d, w->e, w->tauh);
    ktimer_end(st, "sytrd", 4.0 / 3.0 * n * (double)n * n, 16.0 * n * (double)n);
    return SDP_OK;
  }
  if (n >= 3 && n <= SY_CLUSTER_MAX_N) {
    const int cs = sytrd_lower_cluster(n);
    if (cs > 0) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(SYL_THREADS);
      cfg.dynamicSmemBytes = sytrd_lower_smem_bytes(n, cs);
      cfg.stream = st;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cs;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int lda = n;
      count_launch();
      ktimer_begin(st, "sytrd");
      cudaError_t err = cudaLaunchKernelEx(&cfg, k_sytrd_cluster_lower, n, A, lda, w->d, w->e, w->tauh);
      ktimer_end(st, "sytrd", 4.0 / 3.0 * n * (double)n * n, 16.0 * n * (double)n);
      if (err == cudaSuccess) return SDP_OK;
      cudaGetLastError();
    }
  }
  if (n >= 3 && n <= SY_CLUSTER_MAX_N) {
    const int cs = sytrd_smem_cluster(n);
    if (cs > 0) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(SY_THREADS);
      cfg.dynamicSmemBytes = sytrd_smem_bytes(n, cs);
      cfg.stream = st;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cs;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int lda = n;
      count_launch();
      ktimer_begin(st, "sytrd");
      cudaError_t err = cudaLaunchKernelEx(&cfg, k_sytrd_cluster_smem, n, A, lda, w->d, w->e, w->tauh);
      ktimer_end(st, "sytrd", 4.0 / 3.0 * n * (double)n * n, 16.0 * n * (double)n);
      if (err == cudaSuccess) return SDP_OK;
      cudaGetLastError();
    }
  }
  if (n <= SY_CLUSTER_MAX_N) {
    const size_t csm = 3 * (size_t)n * sizeof(double);
    const int cs = sytrd_cluster_size(200 * 1024);
    if (cs > 0) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(SY_THREADS);
      cfg.dynamicSmemBytes = csm;
      cfg.stream = st;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cs;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int lda = n;
      count_launch();
      ktimer_begin(st, "sytrd");
      cudaError_t err = cudaLaunchKernelEx(&cfg, k_sytrd_cluster, n, A, lda, w->d, w->e, w->tauh);
      ktimer_end(st, "sytrd", 4.0 / 3.0 * n * (double)n * n, 24.0 * n * (double)n * n / 3.0);
      if (err == cudaSuccess) return SDP_OK;
      cudaGetLastError();
    }
  }
  const size_t smem = 2 * (size_t)n * sizeof(double);
  if (smem > 200 * 1024) return SDP_ERR_UNSUPPORTED;
  allow_max_smem((const void*)k_sytrd);
  cudaMemsetAsync(w->bar, 0, 2 * sizeof(unsigned int), st);
  cudaMemsetAsync(w->flag, 0, sizeof(int), st);
  const int blocks = sytrd_blocks(n, smem);
  int lda = n;
  long long spin = (w->spin_cycles > 0) ? w->spin_cycles : SPIN_CYCLES;
  if (n <= SYR_MAX_N && 8 * blocks >= n) {
    static int sms = 0;
    if (!sms) {
      int dev = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    int rpc = (int)cdiv(n, sms);
    const size_t rsm = sytrd_resident_smem(n, rpc);
    if (rpc <= SYR_WARPS && rsm <= 210 * 1024) {
      allow_max_smem((const void*)k_sytrd_resident);
      // the exchange buffers: vectors that later steps of the eigensolver fill
      void* rargs[] = {&n, &A, &lda, &w->d, &w->e, &w->tauh, &w->p, &w->wsel, &w->es, &w->val, &rpc, &w->bar, &w->flag, &spin};
      count_launch();
      ktimer_begin(st, "sytrd");
      const cudaError_t re = cudaLaunchCooperativeKernel((void*)k_sytrd_resident, dim3(cdiv(n, rpc)), dim3(SYR_THREADS),
                                                         rargs, rsm, st);
      ktimer_end(st, "sytrd", 4.0 / 3.0 * n * (double)n * n, 16.0 * n * (double)n);
      if (re == cudaSuccess) return SDP_OK;
      cudaGetLastError();
    }
  }
  void* args[] = {&n, &A, &lda, &w->d, &w->e, &w->tauh, &w->p, &w->part, &w->bar, &w->flag, &spin};
  count_launch();
  ktimer_begin(st, "sytrd");
  cudaError_t err = cudaLaunchCooperativeKernel((void*)k_sytrd, dim3(blocks), dim3(256), args, smem, st);
  // algorithmic work of the reduction: (4/3) n^3 flops (symmetric matrix-vector
  // product and rank-2 update per column); the trailing block is read twice and
  // written once per column: 3 * 8 * n^3 / 3 bytes
  ktimer_end(st, "sytrd", 4.0 / 3.0 * n * (double)n * n, 24.0 * n * (double)n * n / 3.0);
  return err == cudaSuccess ? SDP_OK : SDP_ERR_CUDA;
}

// ---------------------------------------------------------------------------
// 2. Bisection
// ---------------------------------------------------------------------------
// Number of eigenvalues of T strictly below x, from the signs of the leading
// principal minors p_i(x) = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (Sturm sequence).
// The three-term form needs two FP64 multiply-adds per step and no division,
// which matters on GB300 where every FP64 op of a warp costs many cycles; the
// sequence is rescaled by a power of two every 16 steps to stay in range.
// A zero minor takes the sign opposite to its predecessor.
// Three FP64 instructions a step and nothing else on that pipe: signs, the zero
// test and the range test are integer tests on the bits (an FP64 compare takes
// the pipe as long as a multiply-add; with them the step took 3.6 times as long).
__device__ __forceinline__ bool sturm_neg(double p, bool before) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(p) << 1;
  // zero or NaN: the sign opposite to the predecessor's
  return (u - 1ull >= 0xFFE0000000000000ull) ? !before : __double2hiint(p) < 0;
}
__device__ __forceinline__ int sturm_count(int n, const double* d, const double* e2, double x) {
  double pm = 1.0, p = d[0] - x;
  bool neg = !(p > 0.0);             // sign of p_0 = 1 is +1; zero counts as a change
  int cnt = neg ? 1 : 0;
  int i = 1;
  auto step = [&](int t) {
    const double pn = fma(d[t] - x, p, -e2[t - 1] * pm);
    const bool sn = sturm_neg(pn, neg);
    cnt += (sn != neg) ? 1 : 0;
    neg = sn;
    pm = p;
    p = pn;
  };
  auto rescale = [&]() {
    const unsigned long long m = 0x7FFFFFFFFFFFFFFFull;
    const unsigned long long up = (unsigned long long)__double_as_longlong(p) & m;
    const unsigned long long um = (unsigned long long)__double_as_longlong(pm) & m;
    const unsigned long long ua = up > um ? up : um;
    if (ua > 0x58F0000000000000ull) { p *= 0x1p-400; pm *= 0x1p-400; }                     // above 2^400
    else if (ua < 0x26F0000000000000ull && ua > 0ull) { p *= 0x1p+400; pm *= 0x1p+400; }   // below 2^-400
  };
  for (; i < n && (i & 15) != 0; ++i) step(i);
  if (i < n) {
    step(i);
    rescale();
    ++i;
  }
  for (; i + 15 < n; i += 16) {
#pragma unroll
    for (int u = 0; u < 16; ++u) step(i + u);
    rescale();
  }
  for (; i < n; ++i) step(i);        // fewer than 16 left: no multiple of 16 among them
  return cnt;
}

__device__ void gersh(int n, const double* d, const double* e, double* lo, double* hi) {
  double gl = d[0], gu = d[0];
  for (int i = 0; i < n; ++i) {
    const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < n ? fabs(e[i]) : 0.0);
    gl = fmin(gl, d[i] - r);
    gu = fmax(gu, d[i] + r);
  }
  const double tn = fmax(fabs(gl), fabs(gu));
  const double pad = 2.0 * DBL_EPSILON * tn * n + 4.0 * DBL_MIN;
  *lo = gl - pad;
  *hi = gu + pad;
}

// Gershgorin bounds of a tridiagonal by the whole block (minima and maxima do
// not depend on the order); red: 2 x 32 doubles of shared memory.
__device__ void gersh_block(int n, const double* d, const double* e, double* red, double* lo, double* hi) {
  double gl = d[0], gu = d[0];
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < n ? fabs(e[i]) : 0.0);
    gl = fmin(gl, d[i] - r);
    gu = fmax(gu, d[i] + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    gl = fmin(gl, __shfl_xor_sync(0xffffffffu, gl, o));
    gu = fmax(gu, __shfl_xor_sync(0xffffffffu, gu, o));
  }
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = gl;
    red[32 + (threadIdx.x >> 5)] = gu;
  }
  __syncthreads();
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    gl = fmin(gl, red[w]);
    gu = fmax(gu, red[32 + w]);
  }
  const double tn = fmax(fabs(gl), fabs(gu));
  const double pad = 2.0 * DBL_EPSILON * tn * n + 4.0 * DBL_MIN;
  *lo = gl - pad;
  *hi = gu + pad;
}

__device__ __forceinline__ bool bis_done(double lo, double hi) {
  return hi - lo <= 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + 4.0 * DBL_MIN;
}

// Eigenvalue number idx[t] (or i0 + t; ascending, 0-based) of T for t < cnt, into
// wout[t]; with wfirst != nullptr the first one goes there and the rest to
// wout[0..].  One warp per eigenvalue, 32-point multisection per round (five bits
// per round).  Serial in n: a round is a chain of n dependent multiply-adds, and
// about 12 rounds are needed.  Warps that share an SM share its FP64 pipe, so few
// eigenvalues get one warp per block (wpb = 1; the other warps only stage T).
// An FP64 warp instruction holds its scheduler's pipe for 64 cycles, so a step costs
// 192: n = 565, 565 eigenvalues or 5: 1616 us -> 897 us; n = 2000: 9.8 ms -> 7.0 ms.
__global__ void __launch_bounds__(128) k_stebz(int n, const double* d, const double* e, int cnt, const int* idx,
                                               int i0, double* wout, double* wfirst, int wpb) {
  extern __shared__ double tri[];
  __shared__ double red[64];
  double* sd = tri;
  double* se2 = tri + n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    sd[i] = d[i];
    se2[i] = (i + 1 < n) ? e[i] * e[i] : 0.0;
  }
  double lo, hi;
  gersh_block(n, d, e, red, &lo, &hi);   // its barrier also covers the staging
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int t = blockIdx.x * wpb + warp;
  if (warp >= wpb || t >= cnt) return;
  const int target = idx ? idx[t] : i0 + t;
  for (int round = 0; round < 64 && !bis_done(lo, hi); ++round) {
    const double h = (hi - lo) / 33.0;
    const int c = sturm_count(n, sd, se2, lo + h * (lane + 1));
    const unsigned above = __ballot_sync(0xffffffffu, c > target);
    const int first = above ? __ffs(above) - 1 : 32;
    const double nlo = (first == 0) ? lo : lo + h * first;
    const double nhi = (first == 32) ? hi : lo + h * (first + 1);
    if (nlo == lo && nhi == hi) break;
    lo = nlo;
    hi = nhi;
  }
  if (lane == 0) {
    if (wfirst && t == 0) *wfirst = 0.5 * (lo + hi);
    else wout[wfirst ? t - 1 : t] = 0.5 * (lo + hi);
  }
}

// ---------------------------------------------------------------------------
// 3. Inverse iteration (tridiagonal LU with partial pivoting)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double hash_unif(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ULL;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
  x ^= x >> 31;
  return (double)(x >> 11) * (2.0 / 9007199254740992.0) - 1.0;  // [-1, 1)
}

// Elimination with partial pivoting of V vectors by one warp, four lanes each.
template <int V>
__device__ __forceinline__ void stein_eliminate(int lane, int nmax, const int* sh_s0, const int* sh_n, const double* sh_lam,
                                                const double* __restrict__ dfull, const double* __restrict__ efull,
                                                double* fa, double* fb, double* fc, double* fd, unsigned char* ff) {
  const int v = (lane >> 2) % V, sub = lane & 3;   // lanes past 4 V repeat the first vectors, unstored
  const bool mine = lane < 4 * V && sub == 0;
  const int n = sh_n[v];
  const double* d = dfull + sh_s0[v];
  const double* e = efull + sh_s0[v];
  const double lam = sh_lam[v];
  double ak = (n > 0) ? d[0] - lam : 1.0;
  double bk = (n > 1) ? e[0] : 0.0;
  double ck = bk, dn = (n > 1) ? d[1] : 0.0, en = (n > 2) ? e[1] : 0.0;
  for (int k = 0; k + 1 < nmax; ++k) {
    const bool on = k + 1 < n;
    const double ak1 = dn - lam;
    const double bk1 = en;                               // 0 from row n - 2 on
    const double ckn = en;
    dn = (k + 2 < n) ? d[k + 2] : 0.0;                   // next step's entries on their way
    en = (k + 3 < n) ? e[k + 2] : 0.0;
    const double scale1 = fabs(ak) + fabs(bk);
    const double scale2 = fabs(ck) + fabs(ak1) + fabs(bk1);
    const double num = (sub == 0) ? fabs(ak) : (sub == 1) ? fabs(ck) : (sub == 2) ? ck : ak;
    const double den = (sub == 0) ? scale1 : (sub == 1) ? scale2 : (sub == 2) ? ak : ck;
    const double q = num / den;
    const int b4 = lane & ~3;
    const double q0 = __shfl_sync(0xffffffffu, q, b4), piv2 = __shfl_sync(0xffffffffu, q, b4 + 1);
    const double q2 = __shfl_sync(0xffffffffu, q, b4 + 2), q3 = __shfl_sync(0xffffffffu, q, b4 + 3);
    const double piv1 = (scale1 == 0.0) ? 0.0 : q0;
    if (on) {
      double oa = ak, ob = bk, oc = 0.0, od = 0.0, na, nb = bk1;
      unsigned char fl = 0;
      if (ck == 0.0) {
        na = ak1;
      } else if (piv2 <= piv1) {
        oc = q2;
        na = ak1 - q2 * bk;
      } else {
        fl = 1;
        oa = ck;
        ob = ak1;
        oc = q3;
        na = bk - q3 * ak1;
        if (k + 2 < n) {
          od = bk1;
          nb = -q3 * bk1;
        } else {
          nb = 0.0;
        }
      }
      if (mine) {
        const size_t x = (size_t)k * V + v;
        fa[x] = oa;
        fb[x] = ob;
        fc[x] = oc;
        fd[x] = od;
        ff[x] = fl;
      }
      ak = na;
      bk = nb;
      ck = ckn;
    }
  }
  if (mine && n > 0) fa[(size_t)(n - 1) * V + v] = ak;
}

// Inverse iteration, three solves per vector.  With blocks == nullptr the whole
// tridiagonal is used; otherwise a vector works on the unreduced diagonal block that
// owns its eigenvalue (src[t] is its row, blocks = {blockid, bstart, bend}) and is zero
// outside that block.  A block of 128 threads takes V vectors; what runs along the
// tridiagonal (elimination, substitutions, the sum of squares) runs in lanes of warp
// 0, everything elementwise in all threads.  The elimination's pivot test needs two
// quotients and its multiplier a third: four lanes per vector compute |a|/(|a|+|b|),
// |c|/(|c|+|a'|+|b'|), c/a and a/c side by side and take what the test selects.
// Bound by that serial chain of FP64 instructions (64 cycles of a scheduler's pipe
// each).  Two forms with the same operations in the same order, for the working arrays
// in shared memory and in global memory; a thread per vector through L2 took 4.2 ms at
// n = 565, 22.8 ms at n = 2000 for all vectors, here 1.1 and 4.2 ms.
// Fields, index k, vector v at [(f n + k) V + v]: 0 a (reciprocal pivots), 1 b,
// 2 c (multipliers), 3 d2, 4 y; then n V pivot flags.
constexpr int STEIN_THREADS = 128;
constexpr int STEIN_GL_V = 8;   // vectors per block in global memory, one in shared memory
static size_t stein_sm_bytes(int n) { return (size_t)n * (5 * sizeof(double) + 1) + 16; }
__global__ void __launch_bounds__(STEIN_THREADS) k_stein_sm(int nfull, const double* __restrict__ dfull,
                                                            const double* __restrict__ efull,
                                                            const double* __restrict__ wsel, int cnt,
                                                            double* __restrict__ Eout, int ldE, int tbase,
                                                            const int* __restrict__ src,
                                                            const int* __restrict__ blocks) {
  constexpr int V = 1;
  extern __shared__ double stein_sh[];
  double* fa = stein_sh;
  double* fb = fa + (size_t)nfull * V;
  double* fc = fb + (size_t)nfull * V;
  double* fd = fc + (size_t)nfull * V;
  double* fy = fd + (size_t)nfull * V;
  unsigned char* ff = reinterpret_cast<unsigned char*>(fy + (size_t)nfull * V);
  __shared__ int sh_s0[V], sh_n[V];
  __shared__ double sh_lam[V], sh_tol[V], sh_sc[V];
  __shared__ double sh_max[STEIN_THREADS / 32][V];
  const int t0 = blockIdx.x * V, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < V) {
    const int t = t0 + tid;
    int s0 = 0, s1 = (t < cnt) ? nfull : 0;
    if (blocks && t < cnt) {
      const int b = blocks[src[t]];
      s0 = blocks[nfull + b];
      s1 = blocks[2 * nfull + b];
    }
    sh_s0[tid] = s0;
    sh_n[tid] = s1 - s0;
    sh_lam[tid] = (t < cnt) ? wsel[t] : 0.0;
  }
  __syncthreads();
  int nmax = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) nmax = max(nmax, sh_n[v]);
  // tol from the largest row sum; start vectors
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int n = sh_n[v];
    const double* d = dfull + sh_s0[v];
    const double* e = efull + sh_s0[v];
    double tn = 0.0;
    for (int i = tid; i < n; i += STEIN_THREADS) {
      const double r = fabs(d[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < n ? fabs(e[i]) : 0.0);
      tn = fmax(tn, r);
      fy[(size_t)i * V + v] = hash_unif(((unsigned long long)(tbase + t0 + v) << 32) ^ (unsigned long long)i);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    if (lane == 0) sh_max[warp][v] = tn;
  }
  __syncthreads();
  if (tid < V) {
    double tn = sh_max[0][tid];
    for (int w = 1; w < STEIN_THREADS / 32; ++w) tn = fmax(tn, sh_max[w][tid]);
    sh_tol[tid] = fmax(DBL_EPSILON * tn, DBL_MIN);
  }
  if (warp == 0) stein_eliminate<V>(lane, nmax, sh_s0, sh_n, sh_lam, dfull, efull, fa, fb, fc, fd, ff);
  __syncthreads();
  // reciprocal pivots (tiny pivots replaced by +-tol)
  for (int x = tid; x < nmax * V; x += STEIN_THREADS) {
    const int v = x % V;
    if (x / V >= sh_n[v]) continue;
    double a = fa[x];
    if (fabs(a) < sh_tol[v]) a = (a >= 0.0) ? sh_tol[v] : -sh_tol[v];
    fa[x] = 1.0 / a;
  }
  __syncthreads();
  for (int iter = 0; iter < 3; ++iter) {
    if (warp == 0 && lane < V && sh_n[lane % V] > 0) {
      const int v = lane, n = sh_n[v];
      // forward
      double yp = fy[v];
      {
        double c = 0.0, yn = 0.0;
        unsigned char fl = 0;
        if (n > 1) { c = fc[v]; fl = ff[v]; yn = fy[V + v]; }
        for (int k = 1; k < n; ++k) {
          const double cc = c, yk = yn;
          const bool f = fl != 0;
          if (k + 1 < n) {
            c = fc[(size_t)k * V + v];
            fl = ff[(size_t)k * V + v];
            yn = fy[(size_t)(k + 1) * V + v];
          }
          const double keep = f ? yk : yp, other = f ? yp : yk;
          fy[(size_t)(k - 1) * V + v] = keep;
          yp = other - cc * keep;
        }
        fy[(size_t)(n - 1) * V + v] = yp;
      }
      // backward: U^{-1}.  Each tiny pivot multiplies by up to 1/tol, so a cluster of
      // them can overflow: whenever an entry passes 2^400 the whole vector (solved part
      // and remaining right-hand side alike) is scaled by 2^-400, which keeps the system
      // consistent; the vector is normalised afterwards anyway.
      unsigned long long ymax = 0ull;
      double y1 = 0.0, y2 = 0.0;
      double a = fa[(size_t)(n - 1) * V + v], b = 0.0, d2 = 0.0, yk0 = yp;
      for (int k = n - 1; k >= 0; --k) {
        double tmp = yk0;
        const double ac = a, bc = b, dc = d2;
        if (k > 0) {
          const size_t x = (size_t)(k - 1) * V + v;
          a = fa[x];
          b = fb[x];
          d2 = fd[x];
          yk0 = fy[x];
        }
        if (k + 1 < n) tmp -= bc * y1;
        if (k + 2 < n) tmp -= dc * y2;
        double yk = tmp * ac;
        if ((__double2hiint(yk) & 0x7FFFFFFF) >= 0x58F00000) {   // !(|yk| < 2^400)
          for (int j = 0; j < n; ++j) fy[(size_t)j * V + v] *= 0x1p-400;
          yk0 *= 0x1p-400;
          y1 *= 0x1p-400;
          ymax = (unsigned long long)__double_as_longlong(__longlong_as_double((long long)ymax) * 0x1p-400);
          yk = (tmp * 0x1p-400) * ac;
        }
        fy[(size_t)k * V + v] = yk;
        const unsigned long long u = (unsigned long long)__double_as_longlong(yk) & 0x7FFFFFFFFFFFFFFFull;
        if (u <= 0x7FF0000000000000ull && u > ymax) ymax = u;
        y2 = y1;
        y1 = yk;
      }
      const double ym = __longlong_as_double((long long)ymax);
      sh_sc[v] = (ym > 0.0) ? 1.0 / ym : 1.0;
    }
    __syncthreads();
    for (int x = tid; x < nmax * V; x += STEIN_THREADS)
      if (x / V < sh_n[x % V]) fy[x] = fy[x] * sh_sc[x % V];
    __syncthreads();
    if (warp == 0 && lane < V) {
      const int v = lane, n = sh_n[v];
      double nrm = 0.0;
#pragma unroll 8
      for (int k = 0; k < n; ++k) {
        const double yk = fy[(size_t)k * V + v];
        nrm = fma(yk, yk, nrm);
      }
      sh_sc[v] = 1.0 / sqrt(nrm);
    }
    __syncthreads();
    for (int x = tid; x < nmax * V; x += STEIN_THREADS)
      if (x / V < sh_n[x % V]) fy[x] *= sh_sc[x % V];
    __syncthreads();
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if (t0 + v >= cnt) break;
    double* out = Eout + (size_t)(t0 + v) * ldE;
    const int s0 = sh_s0[v], n = sh_n[v];
    for (int k = tid; k < nfull; k += STEIN_THREADS)
      out[k] = (k >= s0 && k < s0 + n) ? fy[(size_t)(k - s0) * V + v] : 0.0;
  }
}

// Working arrays in global memory: eight vectors per block, whose warp 0 serves them
// side by side, and the chains load some entries ahead.  Four lanes follow a vector's
// chain with the same values, so that they can share a rescaling; the first of them
// stores.  A chain overwrites the entries that it read a batch earlier, and nothing
// keeps four lanes together by itself (the chains of a warp differ in length and in
// their rescalings), so the four meet after every batch of loads -- before the first
// of them stores over it -- and between the passes.
__global__ void __launch_bounds__(STEIN_THREADS) k_stein_gl(int nfull, const double* __restrict__ dfull,
                                                            const double* __restrict__ efull,
                                                            const double* __restrict__ wsel, int cnt,
                                                            double* __restrict__ Eout, int ldE, int tbase,
                                                            const int* __restrict__ src,
                                                            const int* __restrict__ blocks, double* ws) {
  constexpr int V = STEIN_GL_V, CF = 8, CB = 4;   // entries on their way in the chains
  double* fa = ws + (size_t)blockIdx.x * nfull * (5 * V + 1);
  double* fb = fa + (size_t)nfull * V;
  double* fc = fb + (size_t)nfull * V;
  double* fd = fc + (size_t)nfull * V;
  double* fy = fd + (size_t)nfull * V;
  unsigned char* ff = reinterpret_cast<unsigned char*>(fy + (size_t)nfull * V);
  __shared__ int sh_s0[V], sh_n[V];
  __shared__ double sh_lam[V], sh_tol[V], sh_sc[V];
  __shared__ double sh_max[STEIN_THREADS / 32][V];
  const int t0 = blockIdx.x * V, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < V) {
    const int t = t0 + tid;
    int s0 = 0, s1 = (t < cnt) ? nfull : 0;
    if (blocks && t < cnt) {
      const int b = blocks[src[t]];
      s0 = blocks[nfull + b];
      s1 = blocks[2 * nfull + b];
    }
    sh_s0[tid] = s0;
    sh_n[tid] = s1 - s0;
    sh_lam[tid] = (t < cnt) ? wsel[t] : 0.0;
  }
  __syncthreads();
  int nmax = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) nmax = max(nmax, sh_n[v]);
  // tol from the largest row sum; start vectors
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int n = sh_n[v];
    const double* d = dfull + sh_s0[v];
    const double* e = efull + sh_s0[v];
    double tn = 0.0;
    for (int i = tid; i < n; i += STEIN_THREADS) {
      const double r = fabs(d[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < n ? fabs(e[i]) : 0.0);
      tn = fmax(tn, r);
      fy[(size_t)i * V + v] = hash_unif(((unsigned long long)(tbase + t0 + v) << 32) ^ (unsigned long long)i);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    if (lane == 0) sh_max[warp][v] = tn;
  }
  __syncthreads();
  if (tid < V) {
    double tn = sh_max[0][tid];
    for (int w = 1; w < STEIN_THREADS / 32; ++w) tn = fmax(tn, sh_max[w][tid]);
    sh_tol[tid] = fmax(DBL_EPSILON * tn, DBL_MIN);
  }
  if (warp == 0) stein_eliminate<V>(lane, nmax, sh_s0, sh_n, sh_lam, dfull, efull, fa, fb, fc, fd, ff);
  __syncthreads();
  // reciprocal pivots (tiny pivots replaced by +-tol)
  for (int x = tid; x < nmax * V; x += STEIN_THREADS) {
    const int v = x % V;
    if (x / V >= sh_n[v]) continue;
    double a = fa[x];
    if (fabs(a) < sh_tol[v]) a = (a >= 0.0) ? sh_tol[v] : -sh_tol[v];
    fa[x] = 1.0 / a;
  }
  __syncthreads();
  for (int iter = 0; iter < 3; ++iter) {
    if (warp == 0 && sh_n[lane % V] > 0) {
      const int v = lane % V, n = sh_n[v];
      const unsigned four = 0x01010101u << v;   // the lanes of this chain
      const bool stores = lane < V;
      // forward
      double yp = fy[v];
      {
        double c[CF], y[CF];
        bool f[CF];
        auto load = [&](int k0, double* cc, double* yy, bool* fl) {
#pragma unroll
          for (int u = 0; u < CF; ++u) {
            const int k = k0 + u;
            const bool in = k < n;
            cc[u] = in ? fc[(size_t)(k - 1) * V + v] : 0.0;
            yy[u] = in ? fy[(size_t)k * V + v] : 0.0;
            fl[u] = in && ff[(size_t)(k - 1) * V + v] != 0;
          }
        };
        load(1, c, y, f);
        for (int k0 = 1; k0 < n; k0 += CF) {
          double cn[CF], yn[CF];
          bool fn[CF];
          load(k0 + CF, cn, yn, fn);
          __syncwarp(four);   // all four have read up to entry k0 + 2 CF - 1
#pragma unroll
          for (int u = 0; u < CF; ++u) {
            const int k = k0 + u;
            if (k >= n) break;
            const double keep = f[u] ? y[u] : yp, other = f[u] ? yp : y[u];
            if (stores) fy[(size_t)(k - 1) * V + v] = keep;
            yp = other - c[u] * keep;
          }
#pragma unroll
          for (int u = 0; u < CF; ++u) {
            c[u] = cn[u];
            y[u] = yn[u];
            f[u] = fn[u];
          }
        }
        __syncwarp(four);   // a chain of one entry: all four have read it
        if (stores) fy[(size_t)(n - 1) * V + v] = yp;
      }
      __syncwarp(four);     // the forward pass is stored
      // backward
      unsigned long long ymax = 0ull;
      double y1 = 0.0, y2 = 0.0;
      double a[CB], b[CB], d2[CB], y[CB];
      auto load = [&](int k0, double* aa, double* bb, double* dd, double* yy) {
#pragma unroll
        for (int u = 0; u < CB; ++u) {
          const int k = k0 - u;
          const size_t x = (size_t)max(k, 0) * V + v;
          aa[u] = fa[x];
          bb[u] = (k + 1 < n) ? fb[x] : 0.0;
          dd[u] = (k + 1 < n) ? fd[x] : 0.0;
          yy[u] = fy[x];
        }
      };
      load(n - 1, a, b, d2, y);
      for (int k0 = n - 1; k0 >= 0; k0 -= CB) {
        double an[CB], bn[CB], dn[CB], yn[CB];
        load(k0 - CB, an, bn, dn, yn);
        __syncwarp(four);   // all four have read down to entry k0 - 2 CB + 1
#pragma unroll
        for (int u = 0; u < CB; ++u) {
          const int k = k0 - u;
          if (k < 0) break;
          double tmp = y[u];
          if (k + 1 < n) tmp -= b[u] * y1;
          if (k + 2 < n) tmp -= d2[u] * y2;
          double yk = tmp * a[u];
          if ((__double2hiint(yk) & 0x7FFFFFFF) >= 0x58F00000) {   // !(|yk| < 2^400)
            __syncwarp(four);   // what the first has stored in this batch
            for (int j0 = lane / V; j0 < n; j0 += 32) {
              double z[8];
#pragma unroll
              for (int w = 0; w < 8; ++w) z[w] = (j0 + 4 * w < n) ? fy[(size_t)(j0 + 4 * w) * V + v] : 0.0;
#pragma unroll
              for (int w = 0; w < 8; ++w)
                if (j0 + 4 * w < n) fy[(size_t)(j0 + 4 * w) * V + v] = z[w] * 0x1p-400;
            }
            __syncwarp(four);
#pragma unroll
            for (int w = 0; w < CB; ++w) {
              y[w] *= 0x1p-400;
              yn[w] *= 0x1p-400;
            }
            y1 *= 0x1p-400;
            ymax = (unsigned long long)__double_as_longlong(__longlong_as_double((long long)ymax) * 0x1p-400);
            yk = (tmp * 0x1p-400) * a[u];
          }
          if (stores) fy[(size_t)k * V + v] = yk;
          const unsigned long long q = (unsigned long long)__double_as_longlong(yk) & 0x7FFFFFFFFFFFFFFFull;
          if (q <= 0x7FF0000000000000ull && q > ymax) ymax = q;
          y2 = y1;
          y1 = yk;
        }
#pragma unroll
        for (int u = 0; u < CB; ++u) {
          a[u] = an[u];
          b[u] = bn[u];
          d2[u] = dn[u];
          y[u] = yn[u];
        }
      }
      const double ym = __longlong_as_double((long long)ymax);
      if (lane < V) sh_sc[v] = (ym > 0.0) ? 1.0 / ym : 1.0;
    }
    __syncthreads();
    for (int x = tid; x < nmax * V; x += STEIN_THREADS)
      if (x / V < sh_n[x % V]) fy[x] = fy[x] * sh_sc[x % V];
    __syncthreads();
    if (warp == 0 && lane < V) {
      const int v = lane, n = sh_n[v];
      double nrm = 0.0;
#pragma unroll 16
      for (int k = 0; k < n; ++k) {
        const double yk = fy[(size_t)k * V + v];
        nrm = fma(yk, yk, nrm);
      }
      sh_sc[v] = 1.0 / sqrt(nrm);
    }
    __syncthreads();
    for (int x = tid; x < nmax * V; x += STEIN_THREADS)
      if (x / V < sh_n[x % V]) fy[x] *= sh_sc[x % V];
    __syncthreads();
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if (t0 + v >= cnt) break;
    double* out = Eout + (size_t)(t0 + v) * ldE;
    const int s0 = sh_s0[v], n = sh_n[v];
    for (int k = tid; k < nfull; k += STEIN_THREADS)
      out[k] = (k >= s0 && k < s0 + n) ? fy[(size_t)(k - s0) * V + v] : 0.0;
  }
}

// ---------------------------------------------------------------------------
// 5. Back-transformation: row t of E <- Q row t (Q = H_0 ... H_{n-3})
// ---------------------------------------------------------------------------
__global__ void k_ormtr_rows(int n, const double* __restrict__ A, int lda, const double* __restrict__ tauh,
                             double* __restrict__ E, int ldE, int rows) {
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x % 32;
  if (t >= rows) return;
  double* x = E + (size_t)t * ldE;
  for (int j = n - 3; j >= 0; --j) {
    const double tau = tauh[j];
    if (tau == 0.0) continue;
    const double* vj = A + (size_t)j * lda + j + 1;
    const int len = n - j - 1;
    double s = 0.0;
    for (int l = lane; l < len; l += 32) s = fma(vj[l], x[j + 1 + l], s);
    s = wsum(s) * tau;
    for (int l = lane; l < len; l += 32) x[j + 1 + l] -= s * vj[l];
    __syncwarp();
  }
}

// The same with the vectors and the reflectors in shared memory: a warp per vector,
// the warps of a block share the reflector of a step, which cp.async fetches two
// steps ahead.  Same lanes, same sums, same result.  Bound by the FP64 pipe where
// several warps share an SM, by a step's chain (the lane's multiply-adds, the warp
// sum) where they do not; k_ormtr_rows waits for L2 twice a step.
constexpr int ORM_STAGES = 3;
static size_t ormtr_sm_bytes(int n, int warps) { return (size_t)(warps + ORM_STAGES + 1) * n * sizeof(double); }
__global__ void __launch_bounds__(256) k_ormtr_sm(int n, const double* __restrict__ A, int lda,
                                                  const double* __restrict__ tauh, double* __restrict__ E, int ldE,
                                                  int rows) {
  extern __shared__ double orm_sh[];
  const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* x = orm_sh + (size_t)warp * n;
  double* ring = orm_sh + (size_t)nw * n;
  double* st = ring + (size_t)ORM_STAGES * n;
  const int t = blockIdx.x * nw + warp;
  const bool have = t < rows;
  for (int l = lane; l < n; l += 32) x[l] = have ? E[(size_t)t * ldE + l] : 0.0;
  for (int l = threadIdx.x; l < n; l += blockDim.x) st[l] = tauh[l];
  auto fetch = [&](int j, int slot) {
    if (j >= 0) {
      const double* src = A + (size_t)j * lda + j + 1;
      double* dst = ring + (size_t)slot * n;
      for (int l = threadIdx.x; l < n - j - 1; l += blockDim.x)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                         static_cast<uint32_t>(__cvta_generic_to_shared(dst + l))),
                     "l"(src + l)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(n - 3, 0);
  fetch(n - 4, 1);
  int slot = 0;
  for (int j = n - 3; j >= 0; --j) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();   // reflector j is there for every warp, and slot + 2 has been read
    fetch(j - 2, slot >= 1 ? slot - 1 : slot + 2);
    const double tau = st[j];
    if (tau != 0.0) {
      const double* vj = ring + (size_t)slot * n;
      double* xj = x + j + 1;
      const int len = n - j - 1;
      double s = 0.0;
#pragma unroll 4
      for (int l = lane; l < len; l += 32) s = fma(vj[l], xj[l], s);
      s = wsum(s) * tau;
#pragma unroll 4
      for (int l = lane; l < len; l += 32) xj[l] -= s * vj[l];
      __syncwarp();
    }
    slot = (slot == ORM_STAGES - 1) ? 0 : slot + 1;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (have)
    for (int l = lane; l < n; l += 32) E[(size_t)t * ldE + l] = x[l];
}
// Warps per block: about one block per SM (148 of the 152); from 592 vectors on eight, so that every
// scheduler has a second warp to issue while one waits.  Orders whose working set
// does not fit (above 2300 with eight warps, 3500 with four) run k_ormtr_rows.
// All vectors and the top ones of a build together: n = 565 4.0 -> 1.8 ms, n = 2000
// 47 -> 28 ms.
static void ormtr(cudaStream_t st, int n, const double* A, int lda, const double* tauh, double* E, int ldE, int rows) {
  count_launch();
  int nw = (rows > 4 * 148) ? 8 : (rows > 2 * 148) ? 4 : (rows > 148) ? 2 : 1;
  if (nw == 8 && ormtr_sm_bytes(n, nw) > 220 * 1024) nw = 4;
  const size_t smem = ormtr_sm_bytes(n, nw);
  if (smem <= 220 * 1024) {
    allow_max_smem((const void*)k_ormtr_sm);
    k_ormtr_sm<<<cdiv(rows, nw), 32 * nw, smem, st>>>(n, A, lda, tauh, E, ldE, rows);
    return;
  }
  k_ormtr_rows<<<cdiv((size_t)rows * 32, 256), 256, 0, st>>>(n, A, lda, tauh, E, ldE, rows);
}

// Modified Gram-Schmidt over `rows` (<= 32) vectors of length n, one CTA.
__global__ void k_mgs(int n, double* E, int ldE, int rows) {
  __shared__ double red[32];
  __shared__ double s_val;
  for (int a = 0; a < rows; ++a) {
    double* xa = E + (size_t)a * ldE;
    for (int b = 0; b < a; ++b) {
      const double* xb = E + (size_t)b * ldE;
      double s = 0.0;
      for (int i = threadIdx.x; i < n; i += blockDim.x) s = fma(xa[i], xb[i], s);
      s = bsum(s, red);
      if (threadIdx.x == 0) s_val = s;
      __syncthreads();
      const double c = s_val;
      for (int i = threadIdx.x; i < n; i += blockDim.x) xa[i] -= c * xb[i];
      __syncthreads();
    }
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s = fma(xa[i], xa[i], s);
    s = bsum(s, red);
    if (threadIdx.x == 0) s_val = s;
    __syncthreads();
    const double c = 1.0 / sqrt(s_val);
    for (int i = threadIdx.x; i < n; i += blockDim.x) xa[i] *= c;
    __syncthreads();
  }
}

__global__ void k_idx_extremes(int n, int k, int* idx) {
  const int t = threadIdx.x;
  if (t == 0) idx[0] = 0;
  if (t < k) idx[1 + t] = n - k + t;
}

// ---------------------------------------------------------------------------
// Splitting into unreduced blocks.  Where e_i^2 <= eps^2 |d_i d_{i+1}| (+ tiny)
// the off-diagonal is set to zero and T falls apart into independent blocks.
// Equal eigenvalues of different blocks would otherwise share one shift, and
// inverse iteration would return the same null direction for all of them;
// per block, eigenvalues of an unreduced tridiagonal are distinct, the vectors
// of different blocks have disjoint supports and are exactly orthogonal.
// blocks[0..n) = block of each row, blocks[n + b] = first row, blocks[2n + b] =
// one past the last row, blocks[3n] = number of blocks.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_tri_split(int n, const double* __restrict__ d, const double* __restrict__ e,
                                                    double* __restrict__ es, int* __restrict__ blocks) {
  __shared__ int csum[1024];
  const int T = blockDim.x, tid = threadIdx.x;
  const int chunk = (n + T - 1) / T, i0 = tid * chunk, i1 = min(n, i0 + chunk);
  int cnt = 0;
  for (int i = i0; i < i1; ++i) {
    bool split = false;
    if (i + 1 < n) {
      const double e2 = e[i] * e[i];
      split = !(e2 > DBL_EPSILON * DBL_EPSILON * fabs(d[i] * d[i + 1]) + 4.0 * DBL_MIN);
      es[i] = split ? 0.0 : e[i];
    } else {
      es[i] = 0.0;
    }
    const int starts = (i == 0) ? 1 : 0;   // row i starts a block if i == 0 or e_{i-1} split
    cnt += starts;
    (void)split;
  }
  // rows that start a block because the previous off-diagonal split
  for (int i = i0; i < i1; ++i) {
    if (i > 0) {
      const double e2 = e[i - 1] * e[i - 1];
      if (!(e2 > DBL_EPSILON * DBL_EPSILON * fabs(d[i - 1] * d[i]) + 4.0 * DBL_MIN)) ++cnt;
    }
  }
  csum[tid] = cnt;
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int q = 0; q < T; ++q) { const int c = csum[q]; csum[q] = run; run += c; }
    blocks[3 * n] = run;
  }
  __syncthreads();
  int b = csum[tid] - 1;
  for (int i = i0; i < i1; ++i) {
    bool start = (i == 0);
    if (i > 0) {
      const double e2 = e[i - 1] * e[i - 1];
      start = !(e2 > DBL_EPSILON * DBL_EPSILON * fabs(d[i - 1] * d[i]) + 4.0 * DBL_MIN);
    }
    if (start) {
      ++b;
      blocks[n + b] = i;
      if (b > 0) blocks[2 * n + b - 1] = i;
    }
    blocks[i] = b;
  }
  __syncthreads();
  if (tid == 0) blocks[2 * n + blocks[3 * n] - 1] = n;
}

// val[t] = eigenvalue number (t - first row) of the block that owns row t.
__global__ void k_stebz_blk(int n, const double* d, const double* es, const int* __restrict__ blocks, double* val) {
  extern __shared__ double tri[];
  double* sd = tri;
  double* se2 = tri + n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    sd[i] = d[i];
    se2[i] = es[i] * es[i];
  }
  __syncthreads();
  const int lane = threadIdx.x % 32;
  const int t = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  if (t >= n) return;
  const int b = blocks[t], s0 = blocks[n + b], s1 = blocks[2 * n + b], ns = s1 - s0;
  const int target = t - s0;
  if (ns == 1) {
    if (lane == 0) val[t] = sd[s0];
    return;
  }
  double lo, hi;
  gersh(ns, d + s0, es + s0, &lo, &hi);
  for (int round = 0; round < 64 && !bis_done(lo, hi); ++round) {
    const double h = (hi - lo) / 33.0;
    const int c = sturm_count(ns, sd + s0, se2 + s0, lo + h * (lane + 1));
    const unsigned above = __ballot_sync(0xffffffffu, c > target);
    const int first = above ? __ffs(above) - 1 : 32;
    const double nlo = (first == 0) ? lo : lo + h * first;
    const double nhi = (first == 32) ? hi : lo + h * (first + 1);
    if (nlo == lo && nhi == hi) break;
    lo = nlo;
    hi = nhi;
  }
  if (lane == 0) val[t] = 0.5 * (lo + hi);
}

// Global ascending order of the per-block eigenvalues (ties by row).
__global__ void k_rank(int n, const double* __restrict__ val, double* __restrict__ w, int* __restrict__ src) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double v = val[t];
  int r = 0;
  for (int u = 0; u < n; ++u) {
    const double x = val[u];
    r += (x < v) || (x == v && u < t);
  }
  w[r] = v;
  src[r] = t;
}

// ---------------------------------------------------------------------------
// Host drivers
// ---------------------------------------------------------------------------
static int stein_batch(int n) {
  // keep the interleaved workspace near 256 MB
  size_t b = (size_t)(256u << 20) / (6 * sizeof(double) * (size_t)std::max(n, 1));
  b = std::max<size_t>(32, std::min<size_t>(b, (size_t)n));
  return (int)b;
}

size_t eig_work_bytes(int n, bool full) {
  size_t dbl = 7 * (size_t)n + 4096 + 64 + (4 * (size_t)n + 16) / 2 + 8;
  if (full) {
    dbl += (size_t)6 * n * stein_batch(n);
    dbl += (size_t)n * n;  // Gram matrix
    dbl += std::max(potrf_work_doubles(n), trsm_work_doubles(n, n));
  } else {
    dbl += (size_t)6 * n * 64;
  }
  return dbl * sizeof(double) + 64 * sizeof(int) + 256;
}

void eig_work_carve(EigWork* w, void* base, int n, bool full) {
  double* p = (double*)base;
  w->d = p; p += n;
  w->e = p; p += n;
  w->tauh = p; p += n;
  w->p = p; p += n;
  w->wsel = p; p += n;
  w->es = p; p += n;
  w->val = p; p += n;
  w->part = p; p += 4096;
  p += 64;
  w->batch = full ? stein_batch(n) : 64;
  w->ws = p; p += (size_t)6 * n * w->batch;
  if (full) {
    w->G = p; p += (size_t)n * n;
    w->aux = p; p += std::max(potrf_work_doubles(n), trsm_work_doubles(n, n));
  } else {
    w->G = nullptr;
    w->aux = nullptr;
  }
  int* ip = (int*)p;
  w->bar = (unsigned int*)ip; ip += 4;
  w->flag = ip; ip += 4;
  w->info = ip; ip += 4;
  w->blocks = ip; ip += 3 * n + 4;
  w->src = ip; ip += n;
}

// The barrier counters, the timeout flag and the info word start at zero: the
// flag is read after every eigensolver call, also when no grid-barrier kernel
// ran (freshly allocated device memory holds whatever was there before).
void eig_work_clear(cudaStream_t st, EigWork* w) {
  cudaMemsetAsync(w->bar, 0, 12 * sizeof(int), st);   // bar[4], flag[4], info[4]
}

int eig_flag(cudaStream_t st, EigWork* w) {
  int f = 0;
  cudaMemcpyAsync(&f, w->flag, sizeof(int), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return f;
}

static void launch_stebz(cudaStream_t st, int n, const double* d, const double* e, int cnt, const int* idx,
                         int i0, double* out, double* first = nullptr) {
  const size_t smem = 2 * (size_t)n * sizeof(double);
  allow_max_smem((const void*)k_stebz);
  const int wpb = (cnt >= 4 * 148) ? 4 : std::max(1, (int)cdiv(cnt, 148));
  count_launch();
  k_stebz<<<cdiv(cnt, wpb), 128, smem, st>>>(n, d, e, cnt, idx, i0, out, first, wpb);
}

// Splits T into unreduced blocks; returns the number of blocks (host sync).
static int split_blocks(cudaStream_t st, int n, EigWork* w) {
  count_launch();
  k_tri_split<<<1, 1024, 0, st>>>(n, w->d, w->e, w->es, w->blocks);
  int nb = 1;
  cudaMemcpyAsync(&nb, w->blocks + 3 * n, sizeof(int), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return nb;
}

// All eigenvalues ascending (w) and, when blocked, the row of the block that owns each.
static void eigenvalues_all(cudaStream_t st, int n, EigWork* w, int nblocks, double* wout) {
  if (nblocks <= 1) {
    launch_stebz(st, n, w->d, w->e, n, nullptr, 0, wout);
    return;
  }
  allow_max_smem((const void*)k_stebz_blk);
  count_launch(2);
  k_stebz_blk<<<cdiv(n, 4), 128, 2 * (size_t)n * sizeof(double), st>>>(n, w->d, w->es, w->blocks, w->val);
  k_rank<<<cdiv(n, 128), 128, 0, st>>>(n, w->val, wout, w->src);
}

// The shared-memory form takes a vector per block, whose chain fills a scheduler: for up
// to four blocks per SM (as many as there are schedulers, or as fit; n = 565, one vector
// 0.99 ms against 1.31 ms, all of them 1.05 for both; n = 2000, one vector 3.5 against
// 4.7).  More vectors, and orders above 5300, go eight to a block (n = 1000, all of them:
// 1.9 ms, in shared memory 3.6).
static void eigenvectors(cudaStream_t st, int n, EigWork* w, int nblocks, const double* wv, int first, int cnt,
                         double* E) {
  const double* e = (nblocks <= 1) ? w->e : w->es;
  const bool blk = nblocks > 1;
  const size_t need = stein_sm_bytes(n), most = 220 * 1024;
  if (need <= most && cnt <= 148 * (int)std::min<size_t>(4, most / need)) {
    allow_max_smem((const void*)k_stein_sm);
    count_launch();
    k_stein_sm<<<cnt, STEIN_THREADS, need, st>>>(n, w->d, e, wv + first, cnt, E, n, first,
                                                              blk ? w->src + first : nullptr, blk ? w->blocks : nullptr);
    return;
  }
  // blocks whose 5 V + 1 doubles per entry fit in the workspace of 6 per vector
  const int batch = (int)(6ll * w->batch / (5 * STEIN_GL_V + 1)) * STEIN_GL_V;
  for (int t0 = 0; t0 < cnt; t0 += batch) {
    const int c = std::min(batch, cnt - t0);
    count_launch();
    k_stein_gl<<<cdiv(c, STEIN_GL_V), STEIN_THREADS, 0, st>>>(n, w->d, e, wv + first + t0, c, E + (size_t)t0 * n, n,
                                                              first + t0, blk ? w->src + first + t0 : nullptr,
                                                              blk ? w->blocks : nullptr, w->ws);
  }
}

// max over the lower triangle of |G_ij - delta_ij| (non-negative doubles order
// like their bit patterns, so an integer atomicMax takes the maximum)
constexpr double ORTH_TOL = 1e-12;
__global__ void k_gram_err(int n, const double* __restrict__ G, int ldg, unsigned long long* err) {
  double m = 0.0;
  const size_t total = (size_t)n * n;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(t / n), j = (int)(t % n);
    if (j > i) continue;
    double v = fabs(G[(size_t)i * ldg + j] - (i == j ? 1.0 : 0.0));
    if (!(v == v)) v = INFINITY;   // NaN counts as not orthogonal
    m = fmax(m, v);
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(err, (unsigned long long)__double_as_longlong(m));
}

sdp_status eig_full(cudaStream_t st, int n, double* A, double* wout, double* E, EigWork* w) {
  SDP_TRY(sytrd(st, n, A, w));
  const int nb = split_blocks(st, n, w);
  eigenvalues_all(st, n, w, nb, wout);
  eigenvectors(st, n, w, nb, wout, 0, n, E);
  // Up to two Cholesky-QR passes on the rows of E.  Inverse iteration leaves
  // vectors of well separated eigenvalues orthogonal to working accuracy; only
  // tight clusters inside one block lose orthogonality.  Each pass first forms
  // the Gram matrix and stops when max |E E^T - I| is already at rounding level,
  // so the factorisation and the triangular solve run only when needed.
  for (int pass = 0; pass < 2; ++pass) {
    gemm(st, false, true, n, n, n, 1.0, E, n, E, n, 0.0, w->G, n, GEMM_LOWER_C);
    unsigned long long* err = reinterpret_cast<unsigned long long*>(w->part);
    SDP_CK_ST(cudaMemsetAsync(err, 0, sizeof(unsigned long long), st));
    count_launch();
    k_gram_err<<<std::min<unsigned>(cdiv((size_t)n * n, 256), 1024), 256, 0, st>>>(n, w->G, n, err);
    unsigned long long bits = 0;
    SDP_CK_ST(cudaMemcpyAsync(&bits, err, sizeof(bits), cudaMemcpyDeviceToHost, st));
    SDP_CK_ST(cudaStreamSynchronize(st));
    double e;
    std::memcpy(&e, &bits, sizeof(e));
    if (e <= ORTH_TOL) break;
    potrf(st, n, w->G, n, w->info, w->aux);
    trsm_left_lower(st, false, n, n, w->G, n, E, n, w->aux);
  }
  ormtr(st, n, A, n, w->tauh, E, n, n);
  return SDP_OK;
}

sdp_status eig_min(cudaStream_t st, int n, double* A, double* lmin_dev, EigWork* w) {
  SDP_TRY(sytrd(st, n, A, w));
  launch_stebz(st, n, w->d, w->e, 1, nullptr, 0, lmin_dev);
  return SDP_OK;
}

sdp_status eig_extremes(cudaStream_t st, int n, double* A, int k, double* lmin_dev, double* wtop,
                        double* Etop, EigWork* w) {
  if (k < 0 || k > SDP_K_MAX + 1 || k > n) return SDP_ERR_ARG;
  SDP_TRY(sytrd(st, n, A, w));
  const int nb = (k > 0) ? split_blocks(st, n, w) : 1;
  if (nb <= 1) {
    if (k == 0) {
      launch_stebz(st, n, w->d, w->e, 1, nullptr, 0, lmin_dev);
      return SDP_OK;
    }
    int* idx = (int*)w->part;  // small scratch (part is idle here)
    count_launch(1);
    k_idx_extremes<<<1, 128, 0, st>>>(n, k, idx);
    launch_stebz(st, n, w->d, w->e, k + 1, idx, 0, wtop, lmin_dev);   // the smallest and the top k at once
    eigenvectors(st, n, w, 1, wtop, 0, k, Etop);
  } else {
    eigenvalues_all(st, n, w, nb, w->wsel);
    SDP_CK_ST(cudaMemcpyAsync(lmin_dev, w->wsel, sizeof(double), cudaMemcpyDeviceToDevice, st));
    SDP_CK_ST(cudaMemcpyAsync(wtop, w->wsel + n - k, k * sizeof(double), cudaMemcpyDeviceToDevice, st));
    eigenvectors(st, n, w, nb, w->wsel, n - k, k, Etop);
  }
  ormtr(st, n, A, n, w->tauh, Etop, n, k);
  count_launch();
  k_mgs<<<1, 256, 0, st>>>(n, Etop, n, k);
  return SDP_OK;
}

}  // namespace sdpgb
