// Smallest eigenvalue of a dense symmetric matrix by Lanczos, in one
// thread-block cluster (the step-length test of the interior-point method
// needs lambda_min(L^{-1} dX L^{-T}) only, not a full spectrum).
//
// Lanczos with full reorthogonalisation (two classical Gram-Schmidt passes per
// step) builds the tridiagonal T_j = Q_j^T M Q_j.  The Ritz value theta =
// lambda_min(T_j) is never below lambda_min(M), and the residual of its Ritz
// vector is beta_j |s_j| (s the unit eigenvector of T_j for theta, s_j its last
// entry), so some eigenvalue of M lies in [theta - beta_j |s_j|, theta].  The
// iteration stops when that bound is small against |theta| and returns the
// conservative estimate theta - beta_j |s_j|, which can only shorten a step.
//
// The operator is M itself, or M = A1 A2 A3 applied as three products
// (the step length uses L^{-1} dX L^{-T} this way, from the explicit inverse of
// the Cholesky factor, without forming M).
//
// Layout: the LZ_CS CTAs of the cluster split the rows of each product
// w = M q (cyclically, for balance with triangular factors); each CTA writes its slice of w into every CTA's shared memory
// (distributed shared memory), and after one cluster barrier every CTA holds
// the whole w and performs the O(j n) vector work redundantly, so all CTAs
// compute bit-identical q, alpha, beta and take the same branches.  Each CTA
// keeps its own copy of the Lanczos basis in global memory (no cross-CTA
// visibility is needed for it).  One cluster barrier per step; w is double
// buffered so a CTA that runs ahead into step j+1 never overwrites the buffer
// a slower CTA still reads in step j.
#include "internal.cuh"

#include <cooperative_groups.h>

#include <cfloat>

#include <algorithm>
#include <cmath>

namespace cg = cooperative_groups;

namespace sdpgb {

constexpr int LZ_CS = 8;        // CTAs per cluster (portable cluster size)
constexpr int LZ_THREADS = 256;
constexpr int LZ_MAXIT = 120;   // Lanczos steps at most
constexpr int LZ_CHECK = 6;     // convergence test every LZ_CHECK steps

__device__ __forceinline__ double lz_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// block-wide sum; every thread receives the result (red: 32 doubles of smem)
__device__ double lz_block_sum(double v, double* red) {
  v = lz_warp_sum(v);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  return s;
}

// deterministic start vector entry (splitmix64 of the index, mapped to [-1, 1])
__device__ __forceinline__ double lz_start(int i) {
  unsigned long long z = 0x9E3779B97F4A7C15ull * (unsigned long long)(i + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (double)(z >> 11) * 0x1p-52 - 1.0;
}

// Sturm count of T (diagonal a[0..j), nb[i] = -b_i^2 rounded) below x.  Signs, the
// zero test and the range test look at the bits: an FP64 compare would hold the
// pipe as long as a multiply-add.
__device__ int lz_sturm(int j, const double* a, const double* nb, double x) {
  const unsigned long long mag = 0x7FFFFFFFFFFFFFFFull;
  double pm = 1.0, p = a[0] - x;
  bool neg = !(p > 0.0);
  int cnt = neg ? 1 : 0;
  for (int i = 1; i < j; ++i) {
    const double pn = fma(a[i] - x, p, nb[i - 1] * pm);
    const unsigned long long un = (unsigned long long)__double_as_longlong(pn) & mag;
    const bool sn = (un - 1ull >= 0x7FF0000000000000ull) ? !neg : __double2hiint(pn) < 0;   // zero or NaN: a change
    cnt += (sn != neg) ? 1 : 0;
    neg = sn;
    const unsigned long long up = (unsigned long long)__double_as_longlong(p) & mag;
    pm = p;
    p = pn;
    const unsigned long long um = un > up ? un : up;
    if (um > 0x58F0000000000000ull) { p *= 0x1p-400; pm *= 0x1p-400; }                      // above 2^400
    else if (um < 0x26F0000000000000ull && um > 0ull) { p *= 0x1p+400; pm *= 0x1p+400; }    // below 2^-400
  }
  return cnt;
}

// One warp: theta = lambda_min(T_j) by 32-way multisection, then the last
// entry of its unit eigenvector by two steps of inverse iteration (lane 0).
// res[0] = theta, res[1] = |s_last|.  work: 6 LZ_MAXIT doubles.
__device__ void lz_ritz_min(int j, const double* a, const double* b, double* res, double* work) {
  const int lane = threadIdx.x & 31;
  double lo = a[0], hi = a[0];
  for (int i = lane; i < j; i += 32) {
    const double r = (i > 0 ? fabs(b[i - 1]) : 0.0) + (i + 1 < j ? fabs(b[i]) : 0.0);
    lo = fmin(lo, a[i] - r);
    hi = fmax(hi, a[i] + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  double* nb = work + 5 * LZ_MAXIT;   // -b_i^2
  for (int i = lane; i + 1 < j; i += 32) nb[i] = -b[i] * b[i];
  __syncwarp();
  const double pad = 4.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) * j + DBL_MIN;
  lo -= pad;
  hi += pad;
  for (int it = 0; it < 14; ++it) {
    const double x = lo + (hi - lo) * (double)(lane + 1) / 33.0;
    const int c = lz_sturm(j, a, nb, x);
    const unsigned ge = __ballot_sync(0xffffffffu, c >= 1);
    if (ge == 0u) {
      lo = lo + (hi - lo) * 32.0 / 33.0;
    } else {
      const int f = __ffs(ge) - 1;
      const double nh = lo + (hi - lo) * (double)(f + 1) / 33.0;
      const double nl = (f == 0) ? lo : lo + (hi - lo) * (double)f / 33.0;
      lo = nl;
      hi = nh;
    }
    if (hi - lo <= 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi))) break;
  }
  if (lane == 0) {
    const double theta = 0.5 * (lo + hi);
    // inverse iteration: (T - theta I) s = s_prev, Gaussian elimination with
    // partial pivoting on the tridiagonal; the first pass keeps the multipliers
    // and interchanges, the second applies them
    double* s = work;
    double* dd = work + LZ_MAXIT;       // diagonal after elimination
    double* du = work + 2 * LZ_MAXIT;   // first superdiagonal
    double* du2 = work + 3 * LZ_MAXIT;  // second superdiagonal (from pivoting)
    double* ll = work + 4 * LZ_MAXIT;   // multipliers
    unsigned long long sw0 = 0ull, sw1 = 0ull;   // rows interchanged at step i (LZ_MAXIT <= 128)
    const double tiny = fmax(fabs(theta), 1.0) * 1e-300 + DBL_MIN;
    for (int i = 0; i < j; ++i) s[i] = 1.0;
    for (int rep = 0; rep < 2; ++rep) {
      if (rep == 0) {
        // factor rows in place into upper band (dd, du, du2), apply to s
        double cd = a[0] - theta, cu = (j > 1) ? b[0] : 0.0;
        for (int i = 0; i < j; ++i) {
          if (i + 1 < j) {
            const double sub = b[i];
            const double nd = a[i + 1] - theta;
            const double nu = (i + 2 < j) ? b[i + 1] : 0.0;
            if (fabs(cd) >= fabs(sub)) {
              const double piv = (cd != 0.0) ? cd : tiny;
              const double l = sub / piv;
              ll[i] = l;
              dd[i] = piv; du[i] = cu; du2[i] = 0.0;
              s[i + 1] -= l * s[i];
              cd = nd - l * cu;
              cu = nu;
            } else {
              const double l = cd / sub;
              ll[i] = l;
              if (i < 64) sw0 |= 1ull << i;
              else sw1 |= 1ull << (i - 64);
              dd[i] = sub; du[i] = nd; du2[i] = nu;
              const double t = s[i];
              s[i] = s[i + 1];
              s[i + 1] = t - l * s[i];
              cd = cu - l * nd;
              cu = -l * nu;
            }
          } else {
            dd[i] = (cd != 0.0) ? cd : tiny;
          }
        }
      } else {
        for (int i = 0; i + 1 < j; ++i) {
          const bool swp = ((i < 64 ? sw0 >> i : sw1 >> (i - 64)) & 1ull) != 0ull;
          const double l = ll[i], s0 = s[i], s1 = s[i + 1];
          const double keep = swp ? s1 : s0, other = swp ? s0 : s1;
          s[i] = keep;
          s[i + 1] = other - l * keep;
        }
      }
      for (int i = j - 1; i >= 0; --i) {
        double v = s[i];
        if (i + 1 < j) v -= du[i] * s[i + 1];
        if (i + 2 < j) v -= du2[i] * s[i + 2];
        s[i] = v / dd[i];
      }
      double nrm = 0.0;
      for (int i = 0; i < j; ++i) nrm = fmax(nrm, fabs(s[i]));
      const double sc = (nrm > 0.0 && isfinite(nrm)) ? 1.0 / nrm : 0.0;
      for (int i = 0; i < j; ++i) s[i] *= sc;
    }
    double n2 = 0.0;
    for (int i = 0; i < j; ++i) n2 += s[i] * s[i];
    res[0] = theta;
    res[1] = (n2 > 0.0) ? fabs(s[j - 1]) / sqrt(n2) : 1.0;
  }
  __syncwarp();
}

// out = A x for this CTA's rows (row r handled by warp r mod (LZ_CS * warps),
// cyclic over the cluster), each result written into every CTA's `out`
__device__ __forceinline__ void lz_gemv_bcast(cg::cluster_group& cluster, int n, const double* __restrict__ A,
                                              int lda, const double* x, double* out, int rank, int warp,
                                              int lane, int nw) {
  const int stride = LZ_CS * nw;
  for (int r = rank * nw + warp; r < n; r += stride) {
    const double* ar = A + (size_t)r * lda;
    double acc = 0.0;
    for (int c = lane; c < n; c += 32) acc = fma(ar[c], x[c], acc);
    acc = lz_warp_sum(acc);
    if (lane < LZ_CS) {
      double* dst = cluster.map_shared_rank(out, lane);
      dst[r] = acc;
    }
  }
}

// out[0] = conservative lambda_min estimate, out[1] = theta, out[2] = bound,
// out[3] = steps, out[4] = 1 if converged.  Q: LZ_CS * (LZ_MAXIT + 1) * n doubles.
// Converged: bound <= rtol |theta|, or (after 2 LZ_CHECK steps) theta - bound >=
// accept_above (the caller only needs to know that lambda_min is above it).
__global__ void __cluster_dims__(LZ_CS, 1, 1) __launch_bounds__(LZ_THREADS)
    k_lanczos_min(int n, const double* __restrict__ M, const double* __restrict__ A2,
                  const double* __restrict__ A3, int ldm, double rtol, double accept_above,
                  double* __restrict__ Qall, double* __restrict__ out) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ double sm[];
  double* q = sm;                 // n
  double* w0 = sm + n;            // n   (double-buffered product)
  double* w1 = sm + 2 * (size_t)n;
  double* qp = sm + 3 * (size_t)n;  // n   previous q
  double* t1 = sm + 4 * (size_t)n;  // n   A3 q   (three-factor operator)
  double* t2 = sm + 5 * (size_t)n;  // n   A2 A3 q
  __shared__ double alpha[LZ_MAXIT], beta[LZ_MAXIT], cdot[LZ_MAXIT + 1];
  __shared__ double red[32], ritz[2], twork[6 * LZ_MAXIT];
  __shared__ int stop;
  const int rank = (int)cluster.block_rank();
  double* Q = Qall + (size_t)rank * (LZ_MAXIT + 1) * n;
  const int maxit = min(LZ_MAXIT, n);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;

  // q0: the deterministic start vector, normalised (identical in every CTA)
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double v = lz_start(i);
    q[i] = v;
    qp[i] = 0.0;
    s = fma(v, v, s);
  }
  s = lz_block_sum(s, red);
  const double inv0 = 1.0 / sqrt(s);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    q[i] *= inv0;
    Q[i] = q[i];
  }
  if (threadIdx.x == 0) stop = 0;
  double bprev = 0.0, theta = 0.0, bound = INFINITY;
  int steps = 0, conv = 0;
  cluster.sync();

  for (int j = 0; j < maxit; ++j) {
    double* wb = (j & 1) ? w1 : w0;
    if (A2) {
      lz_gemv_bcast(cluster, n, A3, ldm, q, t1, rank, warp, lane, nw);
      cluster.sync();
      lz_gemv_bcast(cluster, n, A2, ldm, t1, t2, rank, warp, lane, nw);
      cluster.sync();
      lz_gemv_bcast(cluster, n, M, ldm, t2, wb, rank, warp, lane, nw);
    } else {
      lz_gemv_bcast(cluster, n, M, ldm, q, wb, rank, warp, lane, nw);
    }
    cluster.sync();
    // alpha_j = q . w ;  w -= alpha q + beta_{j-1} q_{j-1}
    double a = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) a = fma(q[i], wb[i], a);
    a = lz_block_sum(a, red);
    for (int i = threadIdx.x; i < n; i += blockDim.x) wb[i] = wb[i] - a * q[i] - bprev * qp[i];
    __syncthreads();
    // full reorthogonalisation against Q rows 0..j, two passes
    for (int pass = 0; pass < 2; ++pass) {
      for (int t = warp; t <= j; t += nw) {
        const double* qt = Q + (size_t)t * n;
        double c = 0.0;
        for (int i = lane; i < n; i += 32) c = fma(qt[i], wb[i], c);
        c = lz_warp_sum(c);
        if (lane == 0) cdot[t] = c;
      }
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double v = wb[i];
        for (int t = 0; t <= j; ++t) v = fma(-cdot[t], Q[(size_t)t * n + i], v);
        wb[i] = v;
      }
      __syncthreads();
    }
    double b2 = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) b2 = fma(wb[i], wb[i], b2);
    b2 = lz_block_sum(b2, red);
    const double b = sqrt(b2);
    if (threadIdx.x == 0) {
      alpha[j] = a;
      beta[j] = b;
    }
    steps = j + 1;
    __syncthreads();
    const bool invariant = !(b > 1e-14 * fmax(fabs(a), fabs(bprev)) + DBL_MIN);
    if (invariant || steps == maxit || (steps % LZ_CHECK) == 0) {
      if (warp == 0) lz_ritz_min(steps, alpha, beta, ritz, twork);
      __syncthreads();
      theta = ritz[0];
      bound = invariant ? 0.0 : b * ritz[1];
      const bool ok = invariant || bound <= rtol * fabs(theta) ||
                      (steps >= 2 * LZ_CHECK && theta - bound >= accept_above);
      if (threadIdx.x == 0 && (ok || steps == maxit)) stop = 1;
      conv = ok ? 1 : 0;
      __syncthreads();
    }
    if (stop) break;
    // q_{j+1} = w / beta_j
    const double ib = 1.0 / b;
    double* qn = Q + (size_t)(j + 1) * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      qp[i] = q[i];
      const double v = wb[i] * ib;
      q[i] = v;
      qn[i] = v;
    }
    bprev = b;
    __syncthreads();
  }
  if (rank == 0 && threadIdx.x == 0) {
    out[0] = theta - bound;
    out[1] = theta;
    out[2] = bound;
    out[3] = (double)steps;
    out[4] = conv ? 1.0 : 0.0;
  }
  cluster.sync();   // no CTA leaves while another may still write into its shared memory
}

// ---------------------------------------------------------------------------
// The same iteration over the whole GPU (cooperative launch), for orders where 8
// SMs' FP64 pipes bound the three products.  Every sum keeps its order -- a
// row of a product, a reorthogonalisation coefficient and an entry's correction
// are one warp's or one thread's work in either form, the block sums are formed by
// 256 threads in every CTA -- so both forms return the same bits.  Work is dealt
// over all warps and meets in global memory after a grid barrier: three products,
// then per Gram-Schmidt pass the coefficients and the corrected vector (seven
// barriers a step).  For A1 A2 A3 with A1 lower and A3 upper triangular the
// stored zeros are skipped.  The convergence test is a serial computation of tens
// of microseconds, so an extra CTA runs it while the others go on; when it says
// stop, the (at most six) steps done meanwhile are dropped.  Every wait is
// bounded (`spin` cycles of the SM clock; for the testing CTA, without an arrival
// at a barrier): when one runs out, all CTAs leave, and without an accepted
// estimate out[4] = -1.
// ---------------------------------------------------------------------------
constexpr long long LZ_SPIN_CYCLES = 4000000000ll;   // the default, about two seconds
constexpr int LZ_CHECKS = LZ_MAXIT / LZ_CHECK + 2;
struct LzCtl {                 // zeroed before the launch
  unsigned int arrived;        // grid barrier: arrivals so far
  int fail;                    // a wait ran out
  int stop;                    // the test has accepted an estimate
  int halt;                    // workers leave at this step (0: go on), set by CTA 0
  int req[LZ_CHECKS];          // requested tests: steps, + 1024 for an invariant subspace
};
__device__ __forceinline__ int lz_ld(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void lz_st(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// All workers arrive; false when the wait ran out somewhere.
__device__ bool lz_barrier(LzCtl* c, unsigned int target, long long spin) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&c->arrived, 1u);
    const long long t0 = clock64();
    int ok = 1;
    while ((unsigned int)lz_ld(reinterpret_cast<const int*>(&c->arrived)) < target) {
      if (lz_ld(&c->fail)) { ok = 0; break; }
      if (clock64() - t0 > spin) { lz_st(&c->fail, 1); ok = 0; break; }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// y[r] = A[r, :] x, rows dealt over the warps of all workers; shape 0 full, 1 lower, 2 upper
__device__ __forceinline__ void lz_gemv(int n, const double* __restrict__ A, int lda, const double* x, double* y,
                                        int gw, int nwarps, int lane, int shape) {
  for (int r = gw; r < n; r += nwarps) {
    const double* ar = A + (size_t)r * lda;
    const int c0 = (shape == 2) ? (r & ~31) : 0, c1 = (shape == 1) ? min(n, (r & ~31) + 32) : n;
    double acc = 0.0;
#pragma unroll 8
    for (int c = c0 + lane; c < c1; c += 32) acc = fma(ar[c], x[c], acc);
    acc = lz_warp_sum(acc);
    if (lane == 0) __stcg(y + r, acc);
  }
}

__global__ void __launch_bounds__(LZ_THREADS)
    k_lanczos_grid(int n, const double* __restrict__ M, const double* __restrict__ A2, const double* __restrict__ A3,
                   int ldm, double rtol, double accept_above, double* __restrict__ buf, double* __restrict__ out,
                   LzCtl* ctl, long long spin) {
  extern __shared__ double sm[];
  double* q = sm;                   // n   current q
  double* wb = sm + n;              // n   product, then the next direction
  double* qp = sm + 2 * (size_t)n;  // n   previous q
  double* tv = sm + 3 * (size_t)n;  // n   A3 q, A2 A3 q
  __shared__ double red[32], cdot[LZ_MAXIT + 1];
  double* Q = buf;                                     // (LZ_MAXIT + 1) x n
  double* g1 = buf + (size_t)(LZ_MAXIT + 1) * n;       // n each: exchanged vectors
  double* g2 = g1 + n;
  double* g3 = g2 + n;
  double* gc = g3 + n;                                 // 2 x (LZ_MAXIT + 1): coefficients of the two passes
  double* ga = gc + 2 * (LZ_MAXIT + 1);                // alpha, beta
  double* gb = ga + LZ_MAXIT;
  const int G = (int)gridDim.x - 1;                    // workers; the last CTA tests
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int maxit = min(LZ_MAXIT, n);

  if ((int)blockIdx.x == G) {
    __shared__ double alpha[LZ_MAXIT], beta[LZ_MAXIT], ritz[2], twork[6 * LZ_MAXIT];
    __shared__ int s_req;
    for (int ci = 0; ci < LZ_CHECKS; ++ci) {
      if (threadIdx.x == 0) {
        const int* arrivals = reinterpret_cast<const int*>(&ctl->arrived);
        long long t0 = clock64();
        int rq, seen = lz_ld(arrivals);
        while ((rq = lz_ld(&ctl->req[ci])) == 0) {
          if (lz_ld(&ctl->fail)) break;
          if (clock64() - t0 > spin) {
            const int now = lz_ld(arrivals);
            if (now == seen) { lz_st(&ctl->fail, 1); break; }
            seen = now;
            t0 = clock64();
          }
        }
        s_req = rq;
      }
      __syncthreads();
      const int rq = s_req;
      if (rq == 0) {
        if (threadIdx.x == 0) out[4] = -1.0;
        return;
      }
      const int steps = rq & 1023;
      const bool invariant = rq >= 1024;
      for (int i = threadIdx.x; i < steps; i += blockDim.x) {
        alpha[i] = __ldcg(ga + i);
        beta[i] = __ldcg(gb + i);
      }
      __syncthreads();
      if (warp == 0) lz_ritz_min(steps, alpha, beta, ritz, twork);
      __syncthreads();
      const double theta = ritz[0], bound = invariant ? 0.0 : beta[steps - 1] * ritz[1];
      const bool ok = invariant || bound <= rtol * fabs(theta) ||
                      (steps >= 2 * LZ_CHECK && theta - bound >= accept_above);
      if (ok || steps == maxit) {
        if (threadIdx.x == 0) {
          out[0] = theta - bound;
          out[1] = theta;
          out[2] = bound;
          out[3] = (double)steps;
          out[4] = ok ? 1.0 : 0.0;
          lz_st(&ctl->stop, 1);
        }
        return;
      }
      __syncthreads();
    }
    return;
  }

  const int gw = (int)blockIdx.x * (LZ_THREADS / 32) + warp, nwarps = G * (LZ_THREADS / 32);
  const int gt = (int)blockIdx.x * LZ_THREADS + (int)threadIdx.x, nthr = G * LZ_THREADS;
  unsigned int target = 0;
  auto sync = [&]() {
    target += (unsigned)G;
    return lz_barrier(ctl, target, spin);
  };
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double v = lz_start(i);
    q[i] = v;
    qp[i] = 0.0;
    s = fma(v, v, s);
  }
  s = lz_block_sum(s, red);
  const double inv0 = 1.0 / sqrt(s);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    q[i] *= inv0;
    if (blockIdx.x == 0) __stcg(Q + i, q[i]);
  }
  double bprev = 0.0;
  int checks = 0;
  __syncthreads();
  for (int j = 0; j < maxit; ++j) {
    if (A2) {
      lz_gemv(n, A3, ldm, q, g1, gw, nwarps, lane, 2);
      if (!sync()) return;
      for (int i = threadIdx.x; i < n; i += blockDim.x) tv[i] = __ldcg(g1 + i);
      __syncthreads();
      lz_gemv(n, A2, ldm, tv, g2, gw, nwarps, lane, 0);
      if (!sync()) return;
      for (int i = threadIdx.x; i < n; i += blockDim.x) tv[i] = __ldcg(g2 + i);
      __syncthreads();
      lz_gemv(n, M, ldm, tv, g3, gw, nwarps, lane, 1);
    } else {
      lz_gemv(n, M, ldm, q, g3, gw, nwarps, lane, 0);
    }
    if (!sync()) return;
    double a = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      wb[i] = __ldcg(g3 + i);
      a = fma(q[i], wb[i], a);
    }
    a = lz_block_sum(a, red);
    for (int i = threadIdx.x; i < n; i += blockDim.x) wb[i] = wb[i] - a * q[i] - bprev * qp[i];
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
      double* cg_ = gc + pass * (LZ_MAXIT + 1);
      double* gv = pass ? g2 : g1;
      for (int t = gw; t <= j; t += nwarps) {
        const double* qt = Q + (size_t)t * n;
        double c = 0.0;
#pragma unroll 8
        for (int i = lane; i < n; i += 32) c = fma(__ldcg(qt + i), wb[i], c);
        c = lz_warp_sum(c);
        if (lane == 0) __stcg(cg_ + t, c);
      }
      if (!sync()) return;
      for (int t = threadIdx.x; t <= j; t += blockDim.x) cdot[t] = __ldcg(cg_ + t);
      __syncthreads();
      for (int i = gt; i < n; i += nthr) {
        double v = wb[i];
#pragma unroll 8
        for (int t = 0; t <= j; ++t) v = fma(-cdot[t], __ldcg(Q + (size_t)t * n + i), v);
        __stcg(gv + i, v);
      }
      if (pass == 1 && blockIdx.x == 0 && threadIdx.x == 0 && lz_ld(&ctl->stop)) lz_st(&ctl->halt, j + 1);
      if (!sync()) return;
      for (int i = threadIdx.x; i < n; i += blockDim.x) wb[i] = __ldcg(gv + i);
      __syncthreads();
    }
    double b2 = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) b2 = fma(wb[i], wb[i], b2);
    b2 = lz_block_sum(b2, red);
    const double b = sqrt(b2);
    const int steps = j + 1;
    const bool invariant = !(b > 1e-14 * fmax(fabs(a), fabs(bprev)) + DBL_MIN);
    const bool check = invariant || steps == maxit || (steps % LZ_CHECK) == 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      __stcg(ga + j, a);
      __stcg(gb + j, b);
      if (check) {
        __threadfence();
        lz_st(&ctl->req[checks], steps + (invariant ? 1024 : 0));
      }
    }
    checks += check ? 1 : 0;
    if (invariant || steps == maxit) return;
    const int halt = lz_ld(&ctl->halt);   // written before this step's last barrier, for this step or an earlier one
    if (halt != 0 && halt <= steps) return;
    const double ib = 1.0 / b;
    double* qn = Q + (size_t)(j + 1) * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      qp[i] = q[i];
      const double v = wb[i] * ib;
      q[i] = v;
      if (blockIdx.x == 0) __stcg(qn + i, v);
    }
    bprev = b;
    __syncthreads();
  }
}

// Orders from which the whole-GPU form runs.
constexpr int LZ_GRID_MIN_N = 256;

// Basis copies of the cluster form, or one basis, the exchanged vectors and the
// control block of the whole-GPU form.
size_t lanczos_work_doubles(int n) { return (size_t)LZ_CS * (LZ_MAXIT + 1) * n + 8; }

// Launch on st; results land in out_dev[0..4] (device).  spin: bound of a device-side wait
// in SM clock cycles (0: the default).
// Operator M (A2 = A3 = nullptr) or M A2 A3.  Needs 6 n doubles of shared memory per CTA.
bool lanczos_fits(int n) { return n >= 2 && 6 * (size_t)n * sizeof(double) <= 200 * 1024; }

sdp_status lanczos_min(cudaStream_t st, int n, const double* M, const double* A2, const double* A3, int ldm,
                       double rtol, double accept_above, double* work, double* out_dev, long long spin) {
  const size_t smem = 6 * (size_t)n * sizeof(double);
  if (!lanczos_fits(n) || (A2 == nullptr) != (A3 == nullptr)) return SDP_ERR_UNSUPPORTED;
  allow_max_smem((const void*)k_lanczos_min);
  if (n >= LZ_GRID_MIN_N) {
    static int sms = 0;
    if (!sms) {
      int dev = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    // a warp per row, at most one CTA per SM, one SM for the test
    const int G = std::min((n + LZ_THREADS / 32 - 1) / (LZ_THREADS / 32), sms - 1);
    LzCtl* ctl = reinterpret_cast<LzCtl*>(work + lanczos_work_doubles(n) - (sizeof(LzCtl) + 7) / 8);
    const size_t sg = 4 * (size_t)n * sizeof(double);
    if (spin <= 0) spin = LZ_SPIN_CYCLES;
    allow_max_smem((const void*)k_lanczos_grid);
    if (cudaMemsetAsync(ctl, 0, sizeof(LzCtl), st) != cudaSuccess) return SDP_ERR_CUDA;
    void* args[] = {&n, &M, &A2, &A3, &ldm, &rtol, &accept_above, &work, &out_dev, &ctl, &spin};
    count_launch();
    ktimer_begin(st, "lanczos");
    const cudaError_t e = cudaLaunchCooperativeKernel((void*)k_lanczos_grid, dim3(G + 1), dim3(LZ_THREADS), args, sg, st);
    ktimer_end(st, "lanczos", 0.0, 0.0);
    if (e == cudaSuccess) return SDP_OK;
    cudaGetLastError();   // no room for a cooperative grid: the cluster form
  }
  count_launch();
  ktimer_begin(st, "lanczos");
  k_lanczos_min<<<LZ_CS, LZ_THREADS, smem, st>>>(n, M, A2, A3, ldm, rtol, accept_above, work, out_dev);
  ktimer_end(st, "lanczos", 0.0, 0.0);
  return cudaPeekAtLastError() == cudaSuccess ? SDP_OK : SDP_ERR_CUDA;
}

}  // namespace sdpgb
