// The Hessian operator of eq. (hesseqn2), applied matrix-free:
//   V  = sum_j v_j A_j          (gather over the CSR slots of the V pattern)
//   T  = W V                    (sparse-times-dense: T[r, l] = sum_{s in row l} V_ls W[r, s])
//   Hv_i = sum_{(p,q) in A_i} a_pq mult_pq W[p, :] . T[q, :]
// because (W V W)_pq = sum_l W_pl (V W)_lq = W[p, :] . (W V)[q, :] (V, W symmetric).
// T is produced row by row in its final layout, so no transpose is needed, and
// the per-entry dot products read two contiguous rows.
//
// The same CSR machinery serves the IPM: A(X) (op_A_dense), A^T y scattered into
// a dense matrix (scatter_V_dense) and sparse-times-dense products with U or Z.
//
// Reduced precision with the split W = W_l + W_s (W_l = E^T Lambda E, the top-k
// eigenpairs of the preconditioner build): near the optimum W_l holds the k
// eigenvalues of order 1/mu and W_s the rest, so rounding W itself to FP32 or
// BF16 erases W_s.  Instead only W_s V W_s runs in the reduced precision (SpMM
// and SDDMM as above); the other three terms are low rank,
//   (W_l V W_s + W_s V W_l)_pq = sum_l E[l][p] R[l][q] + E[l][q] R[l][p],
//   R = Lambda (E V) W_s  (k x n),
//   (W_l V W_l)_pq = E[:, p]^T Q E[:, q],  Q = Lambda (E V E^T) Lambda  (k x k),
// and are added per stored entry in FP64, so every term keeps a relative error
// of the working precision on its own scale.
#include "internal.cuh"

#include <algorithm>

namespace sdpgb {

static inline unsigned cdiv(size_t a, size_t b) { return (unsigned)((a + b - 1) / b); }

template <typename T> __device__ __forceinline__ float tof(T x);
template <> __device__ __forceinline__ float tof<float>(float x) { return x; }
template <> __device__ __forceinline__ float tof<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

__device__ __forceinline__ double wsum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// K0: V values from v (gather form, no atomics)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void assemble_body(int s, int nnzV, bool single, const int* __restrict__ sptr,
                                              const int* __restrict__ scon, const double* __restrict__ scoef,
                                              const double* __restrict__ v, const double* __restrict__ scale,
                                              double* __restrict__ Vval, const int* __restrict__ sellpos,
                                              double* __restrict__ Vsell, float* __restrict__ Vsell32) {
  if (s >= nnzV) return;
  const int pos = sellpos ? sellpos[s] : 0;
  double acc = 0.0;
  const int c0 = single ? s : sptr[s], c1 = single ? s + 1 : sptr[s + 1];   // one contributor: no list to look up
  for (int c = c0; c < c1; ++c) {
    const int k = scon[c];
    const double f = scale ? scale[k] : 1.0;
    acc = fma(scoef[c] * f, v[k], acc);
  }
  if (Vval) Vval[s] = acc;
  if (Vsell) Vsell[pos] = acc;
  if (Vsell32) Vsell32[pos] = (float)acc;
}
__global__ void k_assemble(int nnzV, bool single, const int* __restrict__ sptr, const int* __restrict__ scon,
                           const double* __restrict__ scoef, const double* __restrict__ v,
                           const double* __restrict__ scale, double* __restrict__ Vval,
                           const int* __restrict__ sellpos, double* __restrict__ Vsell, float* __restrict__ Vsell32) {
  assemble_body(blockIdx.x * blockDim.x + threadIdx.x, nnzV, single, sptr, scon, scoef, v, scale, Vval, sellpos, Vsell,
                Vsell32);
}

void assemble_V(sdp_problem* h, const double* v, const double* scale, double* Vval) {
  count_launch();
  k_assemble<<<cdiv(h->nnzV, 256), 256, 0, h->stream>>>(h->nnzV, h->single, h->sptr, h->scon, h->scoef, v, scale, Vval, nullptr,
                                                        nullptr, nullptr);
}
// V of a Hessian product in the layout of its SpMM; the split form also reads the CSR values.
static void assemble_matvec(sdp_problem* h, const double* v, bool lp) {
  count_launch();
  k_assemble<<<cdiv(h->nnzV, 256), 256, 0, h->stream>>>(h->nnzV, h->single, h->sptr, h->scon, h->scoef, v, nullptr,
                                                        lp ? h->Vval : nullptr, h->sellpos, lp ? nullptr : h->Vsell,
                                                        lp ? h->Vsell32 : nullptr);
}

// ---------------------------------------------------------------------------
// K1: T = W V, R rows of W per CTA staged in shared memory
// ---------------------------------------------------------------------------
// A CTA takes R rows of W in shared memory and all rows of V, a warp 32 rows of V (a
// slice of the sliced-ELL layout, lane = row).  Every entry of T is one thread's sum
// in the row's CSR order, whatever R and the number of warps.
//
// FP64: the FP64 pipe is the bound, one warp instruction per 64 cycles and
// scheduler, so what counts is that all schedulers get the same number of
// entries: slices come by decreasing length and are dealt over the four
// schedulers of the SM (warp number mod 4) there and back, and R is chosen (spmm_rows)
// so that the CTAs fill whole waves of the SMs.  n = 565, 71250 entries: 128 us with
// chunks of eight warps, whose CTAs left a third of the SM time idle.
constexpr int SPMM_UNROLL = 8;
// Slice number it of warp w, of nw (a multiple of 4) warps.
__device__ __forceinline__ int spmm_slice(int w, int nw, int it) {
  const int q = (w >> 2) + it * (nw >> 2);
  return 4 * q + ((q & 1) ? 3 - (w & 3) : (w & 3));
}
static int spmm_threads(int n) {
  const int slices = (n + 31) / 32;
  return 32 * std::max(4, std::min(16, (slices + 3) / 4 * 4));
}
template <int R>
__device__ __forceinline__ void spmm_f64_body(int blk, int n, const int4* __restrict__ sellrow,
                                              const int* __restrict__ sellcol, const double* __restrict__ Vsell,
                                              const double* __restrict__ W, double* __restrict__ T, double* wsh) {
  const int r0 = blk * R, nw = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int rr = 0; rr < R; ++rr)
    for (int c = threadIdx.x; c < n; c += blockDim.x)
      wsh[rr * n + c] = (r0 + rr < n) ? W[(size_t)(r0 + rr) * n + c] : 0.0;
  int t = spmm_slice(w, nw, 0) * 32 + lane;
  int4 row = (t < n) ? sellrow[t] : make_int4(0, 0, 0, 0);   // on its way during the staging
  __syncthreads();
  for (int it = 0;;) {
    if (4 * ((w >> 2) + it * (nw >> 2)) * 32 >= n) break;   // no slice of this group of four left
    const int4 cur = row;
    const bool on = t < n;
    t = spmm_slice(w, nw, ++it) * 32 + lane;
    row = (t < n) ? sellrow[t] : make_int4(0, 0, 0, 0);
    if (!on) continue;
    double acc[R];
#pragma unroll
    for (int rr = 0; rr < R; ++rr) acc[rr] = 0.0;
    const int len = cur.y;
    const int* cp = sellcol + cur.z;
    const double* vp = Vsell + cur.z;
    // eight entries per step: their loads are independent and go out together (the
    // other warps' multiply-adds hide them; loading the next eight ahead as well made
    // the kernel slower where several CTAs share an SM)
    int s = 0;
    for (; s + SPMM_UNROLL <= len; s += SPMM_UNROLL) {
      int col[SPMM_UNROLL];
      double val[SPMM_UNROLL];
#pragma unroll
      for (int u = 0; u < SPMM_UNROLL; ++u) {
        col[u] = cp[32 * (s + u)];
        val[u] = vp[32 * (s + u)];
      }
#pragma unroll
      for (int u = 0; u < SPMM_UNROLL; ++u)
#pragma unroll
        for (int rr = 0; rr < R; ++rr) acc[rr] = fma(val[u], wsh[rr * n + col[u]], acc[rr]);
    }
    if (s < len) {   // fewer than eight left: loads together, an exit after the last (a
                     // multiply-add that is predicated off would hold the FP64 pipe as well)
      int col[SPMM_UNROLL];
      double val[SPMM_UNROLL];
#pragma unroll
      for (int u = 0; u < SPMM_UNROLL - 1; ++u)
        if (s + u < len) {
          col[u] = cp[32 * (s + u)];
          val[u] = vp[32 * (s + u)];
        }
#pragma unroll
      for (int u = 0; u < SPMM_UNROLL - 1; ++u) {
        if (s + u >= len) break;
#pragma unroll
        for (int rr = 0; rr < R; ++rr) acc[rr] = fma(val[u], wsh[rr * n + col[u]], acc[rr]);
      }
    }
#pragma unroll
    for (int rr = 0; rr < R; ++rr)
      if (r0 + rr < n) T[(size_t)(r0 + rr) * n + cur.x] = acc[rr];
  }
}
template <int R>
__global__ void __launch_bounds__(512) k_spmm_wv_f64(int n, const int4* __restrict__ sellrow,
                                                     const int* __restrict__ sellcol,
                                                     const double* __restrict__ Vsell,
                                                     const double* __restrict__ W, double* __restrict__ T) {
  extern __shared__ double wsh[];  // R x n
  spmm_f64_body<R>(blockIdx.x, n, sellrow, sellcol, Vsell, W, T, wsh);
}

// One row of W per CTA and at most one row of V per thread (n <= SPMM_ONE_N): a few
// warps per SM, bound by the latency of the entries' loads.  The first eight are on
// their way during the staging and the next eight during the multiply-adds.  The whole
// product, 75 x 75 with 2400 samples (n = 150): 11.3 us, with the loads of
// spmm_f64_body 15.5; 152 x 152 with 11552: 27.9 and 29.3.
constexpr int SPMM_ONE_N = 512;
__global__ void __launch_bounds__(512) k_spmm_wv_one(int n, const int4* __restrict__ sellrow,
                                                     const int* __restrict__ sellcol,
                                                     const double* __restrict__ Vsell,
                                                     const double* __restrict__ W, double* __restrict__ T) {
  __shared__ double w[SPMM_ONE_N];
  const int r = blockIdx.x, t = spmm_slice(threadIdx.x >> 5, blockDim.x >> 5, 0) * 32 + (threadIdx.x & 31);
  const int4 row = (t < n) ? sellrow[t] : make_int4(0, 0, 0, 0);
  for (int c = threadIdx.x; c < n; c += blockDim.x) w[c] = W[(size_t)r * n + c];
  const int len = row.y;
  const int* cp = sellcol + row.z;
  const double* vp = Vsell + row.z;
  int col[SPMM_UNROLL];
  double val[SPMM_UNROLL];
  auto load = [&](int s, int* cl, double* vl) {
#pragma unroll
    for (int u = 0; u < SPMM_UNROLL; ++u) {
      cl[u] = (s + u < len) ? cp[32 * (s + u)] : 0;
      vl[u] = (s + u < len) ? vp[32 * (s + u)] : 0.0;
    }
  };
  load(0, col, val);
  __syncthreads();
  double acc = 0.0;
  for (int s = 0; s < len; s += SPMM_UNROLL) {
    int col1[SPMM_UNROLL];
    double val1[SPMM_UNROLL];
    load(s + SPMM_UNROLL, col1, val1);
#pragma unroll
    for (int u = 0; u < SPMM_UNROLL; ++u) {
      if (s + u >= len) break;
      acc = fma(val[u], w[col[u]], acc);
    }
#pragma unroll
    for (int u = 0; u < SPMM_UNROLL; ++u) {
      col[u] = col1[u];
      val[u] = val1[u];
    }
  }
  if (t < n) T[(size_t)r * n + row.x] = acc;
}

// The product of small orders and short rows, where launches and latency count: the
// values of V are formed where they are used (every slot has one contributor; the
// place's constraint and coefficient lie in the sliced layout), so the assembly is no
// launch of its own.  One row of W per CTA.  An entry takes two dependent loads here, so
// long rows lose more than the launch is worth.  In a graph, where only the device's
// time counts, n = 100 with 4 / 8 / 12 / 24 entries per row takes 7.6 / 8.4 / 9.5 / 12.4
// us against 7.8 / 8.2 / 8.3 / 9.1 for the assembly and k_spmm_wv_one; launched one by
// one, n = 40 with 10 entries takes 10.3 us against 12.3.  The line lies at 12 entries.
constexpr int SPMM_SMALL_N = 192, SPMM_SMALL_LEN = 12;
__global__ void __launch_bounds__(256) k_spmm_wv_small(int n, const int4* __restrict__ sellrow,
                                                       const int* __restrict__ sellcol,
                                                       const int* __restrict__ sellcon,
                                                       const double* __restrict__ sellcoef,
                                                       const double* __restrict__ v, const double* __restrict__ W,
                                                       double* __restrict__ T) {
  __shared__ double w[SPMM_SMALL_N];
  const int r = blockIdx.x, t = threadIdx.x;
  const int4 row = (t < n) ? sellrow[t] : make_int4(0, 0, 0, 0);
  if (t < n) w[t] = W[(size_t)r * n + t];
  double acc = 0.0;
  for (int s = 0; s < row.y || s == 0; s += SPMM_UNROLL) {
    int col[SPMM_UNROLL];
    double val[SPMM_UNROLL];
#pragma unroll
    for (int u = 0; u < SPMM_UNROLL; ++u)
      if (s + u < row.y) {
        const int e = row.z + 32 * (s + u);
        col[u] = sellcol[e];
        val[u] = fma(sellcoef[e], v[sellcon[e]], 0.0);
      }
    if (s == 0) __syncthreads();
#pragma unroll
    for (int u = 0; u < SPMM_UNROLL; ++u) {
      if (s + u >= row.y) break;
      acc = fma(val[u], w[col[u]], acc);
    }
  }
  if (t < n) T[(size_t)r * n + row.x] = acc;
}

// Rows of the reduced-precision W_s and T: lp_ld(n) entries, and in each full block of 32
// columns those of one lane of the gather (its columns mod 8) side by side, so that a
// lane loads four of its terms at once.  The load pipe bounds the gather: with one term
// per load a wavefront moved 32 bytes.  n = 5024, 631014 constraints, BF16: the product
// 3.02 -> 2.12 ms; n = 593, FP32: 72 -> 70 us.  Every sum keeps its order.
__host__ __device__ __forceinline__ int lp_ld(int n) { return (n + 3) & ~3; }
__device__ __forceinline__ int lp_pos(int n, int c) {
  return (c < (n & ~31)) ? (c & ~31) | ((c & 7) << 2) | ((c >> 3) & 3) : c;
}

// Reduced precision: the R values of W_s that one stored entry of V needs lie side by
// side (column-major staging), read by vector loads; they bound the kernel, so bfloat16
// copies are staged as they are (half the bytes, widened in registers: the same
// float) and V comes as float from the assembly (a conversion from double holds the
// FP64 pipe).  Elements per staged column: padded to an odd number of 16-byte groups
// from 32 bytes on, so that the random columns of a warp's lanes do not all fall on
// the same banks (without it the float form ran 1.4x slower).
template <typename TW> __host__ __device__ constexpr int spmm_lp_stride(int R) {
  return (sizeof(TW) == 4) ? ((R % 4 == 0) ? R + 4 : R) : ((R == 16) ? 24 : R);
}
template <typename TW> __host__ __device__ constexpr size_t spmm_lp_bytes(int R) {   // per column of W
  return sizeof(TW) * spmm_lp_stride<TW>(R);
}
__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }
template <typename TW, int R>
__device__ __forceinline__ void spmm_lp_fma(float val, const TW* w, float* acc) {
  if constexpr (sizeof(TW) == 4 && R % 4 == 0) {
#pragma unroll
    for (int q = 0; q < R / 4; ++q) {
      const float4 w4 = reinterpret_cast<const float4*>(w)[q];
      acc[4 * q + 0] = fmaf(val, w4.x, acc[4 * q + 0]);
      acc[4 * q + 1] = fmaf(val, w4.y, acc[4 * q + 1]);
      acc[4 * q + 2] = fmaf(val, w4.z, acc[4 * q + 2]);
      acc[4 * q + 3] = fmaf(val, w4.w, acc[4 * q + 3]);
    }
  } else if constexpr (sizeof(TW) == 2 && R % 4 == 0) {
#pragma unroll
    for (int q = 0; q < R / 4; q += 2) {
      uint32_t u[4];
      if constexpr (R % 8 == 0) {
        const uint4 x = reinterpret_cast<const uint4*>(w)[q / 2];
        u[0] = x.x; u[1] = x.y; u[2] = x.z; u[3] = x.w;
      } else {
        const uint2 x = reinterpret_cast<const uint2*>(w)[0];
        u[0] = x.x; u[1] = x.y;
      }
#pragma unroll
      for (int e = 0; e < (R % 8 == 0 ? 4 : 2); ++e) {
        acc[4 * q + 2 * e] = fmaf(val, bf_lo(u[e]), acc[4 * q + 2 * e]);
        acc[4 * q + 2 * e + 1] = fmaf(val, bf_hi(u[e]), acc[4 * q + 2 * e + 1]);
      }
    }
  } else {
#pragma unroll
    for (int rr = 0; rr < R; ++rr) acc[rr] = fmaf(val, tof<TW>(w[rr]), acc[rr]);
  }
}
template <typename TW, int R>
__device__ __forceinline__ void spmm_lp_body(int blk, int n, const int4* __restrict__ sellrow,
                                             const int* __restrict__ sellcol, const float* __restrict__ Vsell,
                                             const TW* __restrict__ W, float* __restrict__ T, TW* fsh) {
  constexpr int RS = spmm_lp_stride<TW>(R);
  const int r0 = blk * R, nw = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int rr = 0; rr < R; ++rr)
    for (int c = threadIdx.x; c < n; c += blockDim.x)
      fsh[c * RS + rr] = (r0 + rr < n) ? W[(size_t)(r0 + rr) * lp_ld(n) + lp_pos(n, c)] : (TW)0.f;
  int t = spmm_slice(w, nw, 0) * 32 + lane;
  int4 row = (t < n) ? sellrow[t] : make_int4(0, 0, 0, 0);   // on its way during the staging
  __syncthreads();
  for (int it = 0;;) {
    if (4 * ((w >> 2) + it * (nw >> 2)) * 32 >= n) break;
    const int4 cur = row;
    const bool on = t < n;
    t = spmm_slice(w, nw, ++it) * 32 + lane;
    row = (t < n) ? sellrow[t] : make_int4(0, 0, 0, 0);
    if (!on) continue;
    float acc[R];
#pragma unroll
    for (int rr = 0; rr < R; ++rr) acc[rr] = 0.f;
    const int len = cur.y;
    const int* cp = sellcol + cur.z;
    const float* vp = Vsell + cur.z;
    int col[SPMM_UNROLL];
    float val[SPMM_UNROLL];
#pragma unroll
    for (int u = 0; u < SPMM_UNROLL; ++u) {
      col[u] = (u < len) ? cp[32 * u] : 0;
      val[u] = (u < len) ? vp[32 * u] : 0.f;
    }
    for (int s = 0; s < len; s += SPMM_UNROLL) {
      int col1[SPMM_UNROLL];
      float val1[SPMM_UNROLL];
#pragma unroll
      for (int u = 0; u < SPMM_UNROLL; ++u) {
        const int e = s + SPMM_UNROLL + u;
        col1[u] = (e < len) ? cp[32 * e] : 0;
        val1[u] = (e < len) ? vp[32 * e] : 0.f;
      }
      if (s + SPMM_UNROLL <= len) {
#pragma unroll
        for (int u = 0; u < SPMM_UNROLL; ++u) spmm_lp_fma<TW, R>(val[u], fsh + col[u] * RS, acc);
      } else {
#pragma unroll
        for (int u = 0; u < SPMM_UNROLL - 1; ++u)
          if (s + u < len) spmm_lp_fma<TW, R>(val[u], fsh + col[u] * RS, acc);
      }
#pragma unroll
      for (int u = 0; u < SPMM_UNROLL; ++u) {
        col[u] = col1[u];
        val[u] = val1[u];
      }
    }
#pragma unroll
    for (int rr = 0; rr < R; ++rr)
      if (r0 + rr < n) T[(size_t)(r0 + rr) * lp_ld(n) + lp_pos(n, cur.x)] = acc[rr];
  }
}
template <typename TW, int R>
__global__ void __launch_bounds__(512) k_spmm_wv_lp(int n, const int4* __restrict__ sellrow,
                                                    const int* __restrict__ sellcol,
                                                    const float* __restrict__ Vsell,
                                                    const TW* __restrict__ W, float* __restrict__ T) {
  extern __shared__ __align__(16) unsigned char fsh_raw[];
  spmm_lp_body<TW, R>(blockIdx.x, n, sellrow, sellcol, Vsell, W, T, reinterpret_cast<TW*>(fsh_raw));
}

// ---------------------------------------------------------------------------
// K2: per-constraint gather of W[p,:] . T[q,:]
// ---------------------------------------------------------------------------
// A warp serves SDDMM_G constraints, SDDMM_L = 32 / SDDMM_G lanes each: the
// cross-lane sums then cost log2(SDDMM_L) shuffle-adds per SDDMM_G constraints
// instead of five per constraint, which matters on a GPU whose FP64 pipe is
// the bound; the group's lanes read a row segment of SDDMM_L consecutive
// doubles, and the SDDMM_G groups of a warp read SDDMM_G rows at once.
// With dv != nullptr the kernel also forms dv . Hv (one deterministic grid
// reduction into *dout; PCG's p . Hp), first moving *pro_src to *pro_dst.
constexpr int SDDMM_G = 4;
constexpr int SDDMM_L = 32 / SDDMM_G;
constexpr int SDDMM_PER_BLOCK = (256 / 32) * SDDMM_G;   // constraints per 256-thread block
__device__ __forceinline__ double gsum_d(double v) {
#pragma unroll
  for (int o = SDDMM_L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float gsum_f(float v) {
#pragma unroll
  for (int o = SDDMM_L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ void sddmm_f64_body(int lb, int nb, int n, int m, const int* __restrict__ eptr,
                                               const int* __restrict__ ep, const int* __restrict__ eq,
                                               const double* __restrict__ ecoef, const double* __restrict__ W,
                                               const double* __restrict__ T, double* __restrict__ Hv,
                                               const double* __restrict__ dv, double* dpart, unsigned int* ticket,
                                               double* dout, double* pro_dst, const double* pro_src) {
  const int warp = (lb * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x % 32;
  const int gl = lane % SDDMM_L;
  const int i = warp * SDDMM_G + lane / SDDMM_L;
  const int e0 = (i < m) ? eptr[i] : 0, cnt = (i < m) ? eptr[i + 1] - e0 : 0;
  const int maxcnt = __reduce_max_sync(0xffffffffu, cnt);
  double acc = 0.0;
  for (int t = 0; t < maxcnt; ++t) {
    double s = 0.0;
    if (t < cnt) {
      const double* wp = W + (size_t)ep[e0 + t] * n;
      const double* tq = T + (size_t)eq[e0 + t] * n;
      int l = gl;
      for (; l + 3 * SDDMM_L < n; l += 4 * SDDMM_L) {   // four loads of each row in flight per lane
        const double w0 = wp[l], w1 = wp[l + SDDMM_L], w2 = wp[l + 2 * SDDMM_L], w3 = wp[l + 3 * SDDMM_L];
        const double t0 = tq[l], t1 = tq[l + SDDMM_L], t2 = tq[l + 2 * SDDMM_L], t3 = tq[l + 3 * SDDMM_L];
        s = fma(w0, t0, s);
        s = fma(w1, t1, s);
        s = fma(w2, t2, s);
        s = fma(w3, t3, s);
      }
      for (; l < n; l += SDDMM_L) s = fma(wp[l], tq[l], s);
    }
    s = gsum_d(s);   // every lane of the group holds the dot
    if (t < cnt) acc = fma(ecoef[e0 + t], s, acc);
  }
  if (i < m && gl == 0) Hv[i] = acc;
  if (dv) {
    const double c = (i < m && gl == 0) ? dv[i] * acc : 0.0;
    double tot;
    if (lb_reduce(c, dpart, ticket, &tot, lb, nb)) {
      if (pro_dst) *pro_dst = *pro_src;
      *dout = tot;
    }
  }
}
__global__ void __launch_bounds__(256) k_sddmm_f64(int n, int m, const int* __restrict__ eptr,
                                                   const int* __restrict__ ep, const int* __restrict__ eq,
                                                   const double* __restrict__ ecoef,
                                                   const double* __restrict__ W, const double* __restrict__ T,
                                                   double* __restrict__ Hv, const double* __restrict__ dv,
                                                   double* dpart, unsigned int* ticket, double* dout,
                                                   double* pro_dst, const double* pro_src) {
  sddmm_f64_body(blockIdx.x, gridDim.x, n, m, eptr, ep, eq, ecoef, W, T, Hv, dv, dpart, ticket, dout, pro_dst,
                 pro_src);
}

// ---------------------------------------------------------------------------
// Batched forms (one launch for every problem of a batch; see batch.cu)
// ---------------------------------------------------------------------------
__global__ void kb_assemble(const BDesc* __restrict__ desc, const int* __restrict__ off, int N) {
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active) return;
  const int lb = blockIdx.x - off[i];
  assemble_body(lb * blockDim.x + threadIdx.x, D.nnzV, D.single != 0, D.sptr, D.scon, D.scoef, D.pp, nullptr,
                D.lp ? D.Vval : nullptr, D.sellpos, D.lp ? nullptr : D.Vsell, D.lp ? D.Vsell32 : nullptr);
}
// R rows of W per CTA: chosen per batch by the autotuner (batch.cu); every R
// gives each entry of T by the same sequence of FMAs, so results do not depend on it.
// Two CTAs on an SM (64 registers a thread, no spills), so that one stages its rows of W
// beside the other's multiply-adds.  16 problems of order 181 to 740, cold caches: 547 us
// with R = 2; with one CTA an SM (77 registers for R = 4) 593 us.
template <int R>
__global__ void __launch_bounds__(512, 2) kb_spmm(const BDesc* __restrict__ desc, const int* __restrict__ off, int N) {
  extern __shared__ double wsh[];
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active || D.lp) return;
  spmm_f64_body<R>(blockIdx.x - off[i], D.n, D.sellrow, D.sellcol, D.Vsell, D.W, D.T, wsh);
}
static void launch_kb_spmm(cudaStream_t st, int R, const BDesc* desc, const int* off, int N, int nb, int nmax) {
  const size_t smem = (size_t)R * nmax * sizeof(double);
  const int th = spmm_threads(nmax);
  switch (R) {
    case 1: allow_max_smem((const void*)kb_spmm<1>); kb_spmm<1><<<nb, th, smem, st>>>(desc, off, N); break;
    case 2: allow_max_smem((const void*)kb_spmm<2>); kb_spmm<2><<<nb, th, smem, st>>>(desc, off, N); break;
    case 8: allow_max_smem((const void*)kb_spmm<8>); kb_spmm<8><<<nb, th, smem, st>>>(desc, off, N); break;
    default: allow_max_smem((const void*)kb_spmm<4>); kb_spmm<4><<<nb, th, smem, st>>>(desc, off, N); break;
  }
}
void batch_launch_spmm(cudaStream_t st, int R, const BDesc* desc, const int* off, int N, int nb, int nmax) {
  count_launch();
  if (nb > 0) launch_kb_spmm(st, R, desc, off, N, nb, nmax);
}
bool batch_spmm_fits(int R, int nmax) { return (size_t)R * nmax * sizeof(double) <= 200 * 1024; }
__global__ void __launch_bounds__(256) kb_sddmm(const BDesc* __restrict__ desc, const int* __restrict__ off, int N) {
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active || D.lp) return;
  sddmm_f64_body(blockIdx.x - off[i], off[i + 1] - off[i], D.n, D.m, D.eptr, D.ep, D.eq, D.ecoef, D.W, D.T, D.pq,
                 D.pp, D.part, D.ticket, D.scal + S_PQ, D.scal + S_RZ, D.scal + S_RZN);
}
int batch_blocks_assemble(int nnzV) { return (int)cdiv(nnzV, 256); }
int batch_blocks_spmm(int n, int R) { return (int)cdiv(n, R); }
int batch_blocks_sddmm(int m) { return (int)cdiv(m, SDDMM_PER_BLOCK); }
// nb_sddmm = 0 leaves the gather out (a mixed batch launches it with the
// reduced-precision one, batch_launch_sddmm_mixed)
void batch_launch_matvec(cudaStream_t st, const BDesc* desc, const int* off_asm, const int* off_spmm,
                         const int* off_sddmm, int N, int nb_asm, int nb_spmm, int nb_sddmm, int nmax, int spmm_r) {
  count_launch(nb_sddmm > 0 ? 3 : 2);
  if (nb_asm > 0) kb_assemble<<<nb_asm, 256, 0, st>>>(desc, off_asm, N);
  if (nb_spmm > 0) launch_kb_spmm(st, spmm_r, desc, off_spmm, N, nb_spmm, nmax);
  if (nb_sddmm > 0) kb_sddmm<<<nb_sddmm, 256, 0, st>>>(desc, off_sddmm, N);
}

__device__ __forceinline__ void lp_load4(const float* p, float* w) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  w[0] = x.x;
  w[1] = x.y;
  w[2] = x.z;
  w[3] = x.w;
}
__device__ __forceinline__ void lp_load4(const __nv_bfloat16* p, float* w) {
  const uint2 x = *reinterpret_cast<const uint2*>(p);
  w[0] = __uint_as_float(x.x << 16);
  w[1] = __uint_as_float(x.x & 0xFFFF0000u);
  w[2] = __uint_as_float(x.y << 16);
  w[3] = __uint_as_float(x.y & 0xFFFF0000u);
}
template <typename TW>
__device__ __forceinline__ void sddmm_lp_body(int lb, int nb, int n, int m, const int* __restrict__ eptr,
                                              const int* __restrict__ ep, const int* __restrict__ eq,
                                              const double* __restrict__ ecoef, const TW* __restrict__ W,
                                              const float* __restrict__ T, double* __restrict__ Hv,
                                              const double* __restrict__ dv, double* dpart, unsigned int* ticket,
                                              double* dout, double* pro_dst, const double* pro_src, int k,
                                              const double* __restrict__ E, const float* __restrict__ R,
                                              const double* __restrict__ Q) {
  const int warp = (lb * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x % 32;
  const int gl = lane % SDDMM_L;
  const int i = warp * SDDMM_G + lane / SDDMM_L;
  const int e0 = (i < m) ? eptr[i] : 0, cnt = (i < m) ? eptr[i + 1] - e0 : 0;
  const int maxcnt = __reduce_max_sync(0xffffffffu, cnt);
  double hv = 0.0;
  for (int t = 0; t < maxcnt; ++t) {
    const bool on = t < cnt;
    const int p = on ? ep[e0 + t] : 0, q = on ? eq[e0 + t] : 0;
    float s = 0.f;
    if (on) {
      const TW* wp = W + (size_t)p * lp_ld(n);
      const float* tq = T + (size_t)q * lp_ld(n);
      const int full = n & ~31;
      // steps in flight: with few constraints the loads' latency is the time (FP32, n = 1000,
      // 1000 constraints: 23.6 us with two, 18.6 with four); in BF16 two are as good there
      // and better with many (n = 5024, 631014 constraints: 2.11 against 2.15 ms)
      constexpr int DEPTH = (sizeof(TW) == 4) ? 4 : 2;
#pragma unroll DEPTH
      for (int b = 4 * gl; b < full; b += 32) {   // columns 32 b' + gl, + 8, + 16, + 24
        float w[4];
        lp_load4(wp + b, w);
        const float4 t4 = *reinterpret_cast<const float4*>(tq + b);
        s = fmaf(w[0], t4.x, s);
        s = fmaf(w[1], t4.y, s);
        s = fmaf(w[2], t4.z, s);
        s = fmaf(w[3], t4.w, s);
      }
      for (int l = full + gl; l < n; l += SDDMM_L) s = fmaf(tof<TW>(wp[l]), tq[l], s);
    }
    double v = (double)gsum_f(s);
    if (k > 0) {
      // low-rank terms of the split, in FP64, lane l of the group taking term l
      // (k <= SDDMM_L):  E[l][p] R[l][q] + E[l][q] R[l][p] + E[l][p] (Q E)[l][q]
      double tl = 0.0;
      if (on && gl < k) {
        const int l = gl;
        const double epl = E[(size_t)l * n + p], eql = E[(size_t)l * n + q];
        double qe = 0.0;
        for (int l2 = 0; l2 < k; ++l2) qe = fma(Q[l * k + l2], E[(size_t)l2 * n + q], qe);
        tl = epl * (double)R[(size_t)l * n + q];
        tl = fma(eql, (double)R[(size_t)l * n + p], tl);
        tl = fma(epl, qe, tl);
      }
      v += gsum_d(tl);
    }
    if (on) hv = fma(ecoef[e0 + t], v, hv);
  }
  if (i < m && gl == 0) Hv[i] = hv;
  if (dv) {
    const double c = (i < m && gl == 0) ? dv[i] * hv : 0.0;
    double tot;
    if (lb_reduce(c, dpart, ticket, &tot, lb, nb)) {
      if (pro_dst) *pro_dst = *pro_src;
      *dout = tot;
    }
  }
}
template <typename TW>
__global__ void __launch_bounds__(256) k_sddmm_lp(int n, int m, const int* __restrict__ eptr,
                                                  const int* __restrict__ ep, const int* __restrict__ eq,
                                                  const double* __restrict__ ecoef, const TW* __restrict__ W,
                                                  const float* __restrict__ T, double* __restrict__ Hv,
                                                  const double* __restrict__ dv, double* dpart, unsigned int* ticket,
                                                  double* dout, double* pro_dst, const double* pro_src, int k,
                                                  const double* __restrict__ E, const float* __restrict__ R,
                                                  const double* __restrict__ Q) {
  sddmm_lp_body<TW>(blockIdx.x, gridDim.x, n, m, eptr, ep, eq, ecoef, W, T, Hv, dv, dpart, ticket, dout, pro_dst,
                    pro_src, k, E, R, Q);
}

// Split: G^T[c][l] = (E V)[l][c] = sum_{s in row c} V[c][s] E[l][s] (V symmetric);
// one warp per row c.
__device__ __forceinline__ void split_G_body(int lb, int n, int k, const int* __restrict__ rowptr,
                                             const int* __restrict__ colidx, const double* __restrict__ Vval,
                                             const double* __restrict__ E, double* __restrict__ Gt) {
  const int c = (lb * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (c >= n) return;
  double acc[8];
#pragma unroll
  for (int l = 0; l < 8; ++l) acc[l] = 0.0;
  for (int s = rowptr[c] + lane; s < rowptr[c + 1]; s += 32) {
    const double v = Vval[s];
    const int col = colidx[s];
#pragma unroll
    for (int l = 0; l < 8; ++l)
      if (l < k) acc[l] = fma(v, E[(size_t)l * n + col], acc[l]);
  }
#pragma unroll
  for (int l = 0; l < 8; ++l) {
    if (l >= k) break;
    const double t = wsum_d(acc[l]);
    if (lane == 0) Gt[(size_t)c * k + l] = t;
  }
}
__global__ void k_split_G(int n, int k, const int* __restrict__ rowptr, const int* __restrict__ colidx,
                          const double* __restrict__ Vval, const double* __restrict__ E, double* __restrict__ Gt) {
  split_G_body(blockIdx.x, n, k, rowptr, colidx, Vval, E, Gt);
}

// Split: partial sums of (G W_s)[l][q] over a chunk of rows c (FP32; grid.y = chunk)
constexpr int SPLIT_CHUNKS = 16;
// The chunk's rows of G as float in shared memory: converted once per block (a
// conversion from double holds the FP64 pipe as long as a multiply-add; with one per
// row, term and thread the kernel took three times as long).
constexpr int SPLIT_STAGE = 64;
template <typename TW>
__device__ __forceinline__ void split_R_part_body(int bx, int by, int n, int k, const double* __restrict__ Gt,
                                                  const TW* __restrict__ Ws, float* __restrict__ part) {
  __shared__ float g[SPLIT_STAGE * 8];
  const int q = bx * blockDim.x + threadIdx.x;
  const int rows = (n + SPLIT_CHUNKS - 1) / SPLIT_CHUNKS;
  const int c0 = by * rows, c1 = min(n, c0 + rows);
  float acc[8];
#pragma unroll
  for (int l = 0; l < 8; ++l) acc[l] = 0.f;
  for (int cb = c0; cb < c1; cb += SPLIT_STAGE) {
    const int cnt = min(SPLIT_STAGE, c1 - cb);
    __syncthreads();
    for (int t = threadIdx.x; t < cnt * k; t += blockDim.x) g[(t / k) * 8 + t % k] = (float)Gt[(size_t)cb * k + t];
    __syncthreads();
    if (q < n) {
#pragma unroll 8
      for (int c = 0; c < cnt; ++c) {
        const float w = tof<TW>(Ws[(size_t)(cb + c) * lp_ld(n) + lp_pos(n, q)]);
#pragma unroll
        for (int l = 0; l < 8; ++l)
          if (l < k) acc[l] = fmaf(g[c * 8 + l], w, acc[l]);
      }
    }
  }
  if (q >= n) return;
#pragma unroll
  for (int l = 0; l < 8; ++l)
    if (l < k) part[((size_t)by * k + l) * n + q] = acc[l];
}
template <typename TW>
__global__ void k_split_R_part(int n, int k, const double* __restrict__ Gt, const TW* __restrict__ Ws,
                               float* __restrict__ part) {
  split_R_part_body<TW>(blockIdx.x, blockIdx.y, n, k, Gt, Ws, part);
}
// R[l][q] = lambda_l sum_chunks part;  Q[l][l2] = lambda_l lambda_l2 sum_c G[l][c] E[l2][c]
// (the Q block is formed by the first k * k warps of the grid)
__device__ __forceinline__ void split_R_Q_body(int lb, int n, int k, const float* __restrict__ part,
                                               const double* __restrict__ lam, const double* __restrict__ Gt,
                                               const double* __restrict__ E, float* __restrict__ R,
                                               double* __restrict__ Q) {
  const int t = lb * blockDim.x + threadIdx.x;
  if (t < n * k) {
    const int l = t / n, q = t % n;
    float s = 0.f;
    for (int ch = 0; ch < SPLIT_CHUNKS; ++ch) s += part[((size_t)ch * k + l) * n + q];
    R[t] = (float)(lam[l] * (double)s);
  }
  const int w = t >> 5, lane = t & 31;
  if (w < k * k) {
    const int l = w / k, l2 = w % k;
    double s = 0.0;
    for (int c = lane; c < n; c += 32) s = fma(Gt[(size_t)c * k + l], E[(size_t)l2 * n + c], s);
    s = wsum_d(s);
    if (lane == 0) Q[l * k + l2] = lam[l] * lam[l2] * s;
  }
}
__global__ void k_split_R_Q(int n, int k, const float* __restrict__ part, const double* __restrict__ lam,
                            const double* __restrict__ Gt, const double* __restrict__ E, float* __restrict__ R,
                            double* __restrict__ Q) {
  split_R_Q_body(blockIdx.x, n, k, part, lam, Gt, E, R, Q);
}

// W_s = W - E^T diag(lam) E into Ws (n x n FP64)
__global__ void k_split_Ws(int n, int k, const double* __restrict__ W, const double* __restrict__ E,
                           const double* __restrict__ lam, double* __restrict__ Ws) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)n * n) return;
  const int a = (int)(t / n), b = (int)(t % n);
  double v = W[t];
  for (int l = 0; l < k; ++l) v = fma(-lam[l] * E[(size_t)l * n + a], E[(size_t)l * n + b], v);
  Ws[t] = v;
}

// Batched FP32 forms: the same bodies as the single-problem launches (problems
// in an FP64 sweep return at once).  Each entry of T is one thread's sum in the
// row's CSR order whatever the rows per CTA, so the batched SpMM may take more
// rows of W per CTA than a problem alone and still match it bit for bit: 16 (V is
// read n / 16 times) while the staged rows of the batch's largest problem fit in
// 200 KB of shared memory, fewer for larger orders.
int batch_spmm_lp_rows(int nmax) {
  for (int r = 16; r > 1; r /= 2)
    if (spmm_lp_bytes<float>(r) * nmax <= 200 * 1024) return r;
  return 1;
}
__global__ void __launch_bounds__(256) kb_split_G(const BDesc* __restrict__ desc, const int* __restrict__ off, int N) {
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active || !D.lp || D.ks == 0) return;
  split_G_body(blockIdx.x - off[i], D.n, D.ks, D.rowptr, D.colidx, D.Vval, D.Etop, D.mvG);
}
__global__ void __launch_bounds__(128) kb_split_R_part(const BDesc* __restrict__ desc, const int* __restrict__ off,
                                                       int N) {
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active || !D.lp || D.ks == 0) return;
  const int lb = blockIdx.x - off[i], gx = (D.n + 127) / 128;
  if (D.bf) split_R_part_body<__nv_bfloat16>(lb % gx, lb / gx, D.n, D.ks, D.mvG, D.W16, D.mvPart);
  else split_R_part_body<float>(lb % gx, lb / gx, D.n, D.ks, D.mvG, D.W32, D.mvPart);
}
__global__ void __launch_bounds__(256) kb_split_R_Q(const BDesc* __restrict__ desc, const int* __restrict__ off,
                                                    int N) {
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active || !D.lp || D.ks == 0) return;
  split_R_Q_body(blockIdx.x - off[i], D.n, D.ks, D.mvPart, D.wtop, D.mvG, D.Etop, D.mvR, D.mvQ);
}
template <int R>
__global__ void __launch_bounds__(512) kb_spmm_lp(const BDesc* __restrict__ desc, const int* __restrict__ off, int N) {
  extern __shared__ __align__(16) unsigned char fsh_raw[];
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active || !D.lp) return;
  if (D.bf)
    spmm_lp_body<__nv_bfloat16, R>(blockIdx.x - off[i], D.n, D.sellrow, D.sellcol, D.Vsell32, D.W16, D.T32,
                                   reinterpret_cast<__nv_bfloat16*>(fsh_raw));
  else
    spmm_lp_body<float, R>(blockIdx.x - off[i], D.n, D.sellrow, D.sellcol, D.Vsell32, D.W32, D.T32,
                           reinterpret_cast<float*>(fsh_raw));
}
__global__ void __launch_bounds__(256) kb_sddmm_lp(const BDesc* __restrict__ desc, const int* __restrict__ off,
                                                   int N) {
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active || !D.lp) return;
  if (D.bf)
    sddmm_lp_body<__nv_bfloat16>(blockIdx.x - off[i], off[i + 1] - off[i], D.n, D.m, D.eptr, D.ep, D.eq, D.ecoef,
                                 D.W16, D.T32, D.pq, D.pp, D.part, D.ticket, D.scal + S_PQ, D.scal + S_RZ,
                                 D.scal + S_RZN, D.ks, D.Etop, D.mvR, D.mvQ);
  else
    sddmm_lp_body<float>(blockIdx.x - off[i], off[i + 1] - off[i], D.n, D.m, D.eptr, D.ep, D.eq, D.ecoef, D.W32,
                         D.T32, D.pq, D.pp, D.part, D.ticket, D.scal + S_PQ, D.scal + S_RZ, D.scal + S_RZN, D.ks,
                         D.Etop, D.mvR, D.mvQ);
}
int batch_blocks_split_G(int n) { return (int)cdiv((size_t)n * 32, 256); }
int batch_blocks_split_R(int n) { return (int)cdiv(n, 128) * SPLIT_CHUNKS; }
int batch_blocks_split_Q(int n, int k) { return (int)cdiv(std::max((size_t)n * k, (size_t)k * k * 32), 256); }
int batch_blocks_spmm_lp(int n, int nmax) { return (int)cdiv(n, batch_spmm_lp_rows(nmax)); }
// Both gathers of a mixed batch in one launch: the two forms share the block
// partition (and the reduction groups), so each problem runs the same code as
// in its own launch.
__global__ void __launch_bounds__(256) kb_sddmm_mixed(const BDesc* __restrict__ desc, const int* __restrict__ off,
                                                      int N) {
  const int i = batch_find(off, N, blockIdx.x);
  const BDesc& D = desc[i];
  if (!D.active) return;
  const int lb = blockIdx.x - off[i], nb = off[i + 1] - off[i];
  if (!D.lp)
    sddmm_f64_body(lb, nb, D.n, D.m, D.eptr, D.ep, D.eq, D.ecoef, D.W, D.T, D.pq, D.pp, D.part, D.ticket,
                   D.scal + S_PQ, D.scal + S_RZ, D.scal + S_RZN);
  else if (D.bf)
    sddmm_lp_body<__nv_bfloat16>(lb, nb, D.n, D.m, D.eptr, D.ep, D.eq, D.ecoef, D.W16, D.T32, D.pq, D.pp, D.part,
                                 D.ticket, D.scal + S_PQ, D.scal + S_RZ, D.scal + S_RZN, D.ks, D.Etop, D.mvR, D.mvQ);
  else
    sddmm_lp_body<float>(lb, nb, D.n, D.m, D.eptr, D.ep, D.eq, D.ecoef, D.W32, D.T32, D.pq, D.pp, D.part, D.ticket,
                         D.scal + S_PQ, D.scal + S_RZ, D.scal + S_RZN, D.ks, D.Etop, D.mvR, D.mvQ);
}
void batch_launch_sddmm_mixed(cudaStream_t st, const BDesc* desc, const int* off, int N, int nb) {
  count_launch();
  if (nb > 0) kb_sddmm_mixed<<<nb, 256, 0, st>>>(desc, off, N);
}

void batch_launch_matvec_lp(cudaStream_t st, const BDesc* desc, const int* off_g, const int* off_r,
                            const int* off_q, const int* off_spmm, const int* off_sddmm, int N, int nb_g, int nb_r,
                            int nb_q, int nb_spmm, int nb_sddmm, int nmax, bool with_sddmm) {
  const int R = batch_spmm_lp_rows(nmax);
  const size_t smem = spmm_lp_bytes<float>(R) * nmax;   // the bfloat16 staging needs less
  const int th = spmm_threads(nmax);
  count_launch(with_sddmm ? 5 : 4);
  if (nb_g > 0) kb_split_G<<<nb_g, 256, 0, st>>>(desc, off_g, N);
  if (nb_r > 0) kb_split_R_part<<<nb_r, 128, 0, st>>>(desc, off_r, N);
  if (nb_q > 0) kb_split_R_Q<<<nb_q, 256, 0, st>>>(desc, off_q, N);
  if (nb_spmm > 0) {
    switch (R) {
      case 16: allow_max_smem((const void*)kb_spmm_lp<16>); kb_spmm_lp<16><<<nb_spmm, th, smem, st>>>(desc, off_spmm, N); break;
      case 8: allow_max_smem((const void*)kb_spmm_lp<8>); kb_spmm_lp<8><<<nb_spmm, th, smem, st>>>(desc, off_spmm, N); break;
      case 4: allow_max_smem((const void*)kb_spmm_lp<4>); kb_spmm_lp<4><<<nb_spmm, th, smem, st>>>(desc, off_spmm, N); break;
      case 2: allow_max_smem((const void*)kb_spmm_lp<2>); kb_spmm_lp<2><<<nb_spmm, th, smem, st>>>(desc, off_spmm, N); break;
      default: allow_max_smem((const void*)kb_spmm_lp<1>); kb_spmm_lp<1><<<nb_spmm, th, smem, st>>>(desc, off_spmm, N); break;
    }
  }
  if (with_sddmm && nb_sddmm > 0) kb_sddmm_lp<<<nb_sddmm, 256, 0, st>>>(desc, off_sddmm, N);
}

__device__ __forceinline__ void lp_store(float* y, double x) { *y = (float)x; }
__device__ __forceinline__ void lp_store(__nv_bfloat16* y, double x) { *y = __float2bfloat16_rn((float)x); }
template <typename TW>
__global__ void __launch_bounds__(256) k_lp_copy(int n, const double* __restrict__ W, TW* __restrict__ Wl) {
  const int r = blockIdx.x;
  for (int c = threadIdx.x; c < n; c += 256) lp_store(Wl + (size_t)r * lp_ld(n) + lp_pos(n, c), W[(size_t)r * n + c]);
}
// Reduced-precision copy of W, or of W_s when a preconditioner with top
// eigenpairs is built (the split form); keyed so that a new W or a rebuilt
// preconditioner refreshes it.
sdp_status ensure_lowprec_W(sdp_problem* h, int prec) {
  const int n = h->n;
  const size_t nn = (size_t)n * n, nl = (size_t)n * lp_ld(n);
  if (prec != SDP_FP32 && prec != SDP_BF16) return SDP_OK;
  if (!h->T32) SDP_TRY(h->allocT(&h->T32, nl));
  const bool split = h->pc_valid && h->kpc > 0 && h->Etop && h->KZ && h->kpc <= 8;
  const int64_t key = split ? h->pc_generation : -1;
  bool& valid = (prec == SDP_FP32) ? h->W32_valid : h->W16_valid;
  int64_t& have_key = (prec == SDP_FP32) ? h->W32_key : h->W16_key;
  if (valid && have_key == key) return SDP_OK;
  const double* src = h->W;
  cudaStream_t st = h->stream;
  if (split) {
    count_launch();
    k_split_Ws<<<cdiv(nn, 256), 256, 0, st>>>(n, h->kpc, h->W, h->Etop, h->wtop, h->KZ);
    src = h->KZ;
    if (!h->mv_G) {
      SDP_TRY(h->allocT(&h->mv_G, (size_t)n * 8));
      SDP_TRY(h->allocT(&h->mv_R, (size_t)n * 8));
      SDP_TRY(h->allocT(&h->mv_Q, 64));
      SDP_TRY(h->allocT(&h->mv_part, (size_t)SPLIT_CHUNKS * 8 * n));
    }
  }
  if (prec == SDP_FP32) {
    if (!h->W32) SDP_TRY(h->allocT(&h->W32, nl));
    count_launch();
    k_lp_copy<float><<<n, 256, 0, st>>>(n, src, h->W32);
  } else {
    if (!h->W16) SDP_TRY(h->allocT(&h->W16, nl));
    count_launch();
    k_lp_copy<__nv_bfloat16><<<n, 256, 0, st>>>(n, src, h->W16);
  }
  valid = true;
  have_key = key;
  return SDP_OK;
}

// Rows of W per CTA of the SpMM.  The SM with the most CTAs takes
// ceil(ceil(n / R) / SMs) of them, each as long as its R multiply-adds and a fixed
// share per entry (index, value): the R of the least product, at most 200 KB of
// shared memory.  FP64, 2000 x 2000 with 60000 samples: R = 3, 0.85 ms for the
// SpMM, 90 % of the FP64 pipe.
template <typename Bytes>   // bytes(r): staged bytes per column of W
static int spmm_rows(int n, Bytes bytes, double fixed, const int* cand, int ncand) {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  }
  int best = 1;
  double tb = 1e300;
  for (int i = 0; i < ncand; ++i) {
    const int r = cand[i];
    if (bytes(r) * (size_t)n > 200 * 1024) continue;
    const unsigned per_sm = cdiv(cdiv(n, r), sms);
    const double t = per_sm * (r + fixed) * (per_sm == 1 ? 1.15 : 1.0);   // one CTA alone hides less latency
    if (t < tb) {
      tb = t;
      best = r;
    }
  }
  return best;
}

template <int R>
static void launch_spmm_f64(sdp_problem* h) {
  const size_t smem = (size_t)R * h->n * sizeof(double);
  allow_max_smem((const void*)k_spmm_wv_f64<R>);
  count_launch();
  k_spmm_wv_f64<R><<<cdiv(h->n, R), spmm_threads(h->n), smem, h->stream>>>(h->n, h->sellrow, h->sellcol, h->Vsell, h->W,
                                                                           h->T);
}
static void spmm_f64(sdp_problem* h) {
  static const int cand[8] = {8, 7, 6, 5, 4, 3, 2, 1};
  switch (spmm_rows(h->n, [](int r) { return sizeof(double) * r; }, 0.3, cand, 8)) {
    case 8: launch_spmm_f64<8>(h); break;
    case 7: launch_spmm_f64<7>(h); break;
    case 6: launch_spmm_f64<6>(h); break;
    case 5: launch_spmm_f64<5>(h); break;
    case 4: launch_spmm_f64<4>(h); break;
    case 3: launch_spmm_f64<3>(h); break;
    case 2: launch_spmm_f64<2>(h); break;
    default:
      if (h->n <= SPMM_ONE_N) {
        count_launch();
        k_spmm_wv_one<<<h->n, spmm_threads(h->n), 0, h->stream>>>(h->n, h->sellrow, h->sellcol, h->Vsell, h->W, h->T);
      } else {
        launch_spmm_f64<1>(h);
      }
      break;
  }
}
template <typename TW, int R>
static void launch_spmm_lp(sdp_problem* h, const TW* W) {
  const size_t smem = spmm_lp_bytes<TW>(R) * h->n;
  allow_max_smem((const void*)k_spmm_wv_lp<TW, R>);
  count_launch();
  k_spmm_wv_lp<TW, R><<<cdiv(h->n, R), spmm_threads(h->n), smem, h->stream>>>(h->n, h->sellrow, h->sellcol, h->Vsell32, W,
                                                                              h->T32);
}
template <typename TW>
static void spmm_lp(sdp_problem* h, const TW* W) {
  static const int cand[4] = {8, 4, 2, 1};
  switch (spmm_rows(h->n, [](int r) { return spmm_lp_bytes<TW>(r); }, 4.0, cand, 4)) {
    case 8: launch_spmm_lp<TW, 8>(h, W); break;
    case 4: launch_spmm_lp<TW, 4>(h, W); break;
    case 2: launch_spmm_lp<TW, 2>(h, W); break;
    default: launch_spmm_lp<TW, 1>(h, W); break;
  }
}

sdp_status matvec_impl(sdp_problem* h, const double* v, double* Hv, int prec, double* dot_out, double* pro_dst,
                       const double* pro_src) {
  const double* dv = dot_out ? v : nullptr;
  if (!h->have_W) {
    h->last_error = "hessian_matvec: no scaling matrix W (call sdp_set_W or sdp_ipm_step)";
    return SDP_ERR_ARG;
  }
  const int n = h->n;
  const bool timed = ktimer_on("matvec");
  if (timed) ktimer_begin(h->stream, "matvec");
  if (prec == SDP_FP64) {
    if (h->sellcon && n <= SPMM_SMALL_N && h->nnzV <= SPMM_SMALL_LEN * n) {
      count_launch();
      k_spmm_wv_small<<<n, (n + 31) / 32 * 32, 0, h->stream>>>(n, h->sellrow, h->sellcol, h->sellcon, h->sellcoef, v,
                                                               h->W, h->T);
    } else {
      assemble_matvec(h, v, false);
      spmm_f64(h);
    }
    count_launch();
    k_sddmm_f64<<<cdiv(h->m, SDDMM_PER_BLOCK), 256, 0, h->stream>>>(n, h->m, h->eptr, h->ep, h->eq, h->ecoef,
                                                                     h->W, h->T, Hv, dv, h->pcg_part,
                                                                     h->pcg_ticket, dot_out, pro_dst, pro_src);
  } else if (prec == SDP_FP32 || prec == SDP_BF16) {
    assemble_matvec(h, v, true);
    SDP_TRY(ensure_lowprec_W(h, prec));
    const bool split = (prec == SDP_FP32 ? h->W32_key : h->W16_key) >= 0;
    const int ks = split ? h->kpc : 0;
    if (split) {
      count_launch(3);
      k_split_G<<<cdiv((size_t)n * 32, 256), 256, 0, h->stream>>>(n, ks, h->rowptr, h->colidx, h->Vval, h->Etop,
                                                                    h->mv_G);
      if (prec == SDP_FP32)
        k_split_R_part<float><<<dim3(cdiv(n, 128), SPLIT_CHUNKS), 128, 0, h->stream>>>(n, ks, h->mv_G, h->W32,
                                                                                       h->mv_part);
      else
        k_split_R_part<__nv_bfloat16><<<dim3(cdiv(n, 128), SPLIT_CHUNKS), 128, 0, h->stream>>>(
            n, ks, h->mv_G, h->W16, h->mv_part);
      const size_t th = std::max((size_t)n * ks, (size_t)ks * ks * 32);
      k_split_R_Q<<<cdiv(th, 256), 256, 0, h->stream>>>(n, ks, h->mv_part, h->wtop, h->mv_G, h->Etop, h->mv_R,
                                                        h->mv_Q);
    }
  }
  if (prec == SDP_FP32) {
    spmm_lp<float>(h, h->W32);
    count_launch();
    k_sddmm_lp<float><<<cdiv(h->m, SDDMM_PER_BLOCK), 256, 0, h->stream>>>(
        n, h->m, h->eptr, h->ep, h->eq, h->ecoef, h->W32, h->T32, Hv, dv, h->pcg_part, h->pcg_ticket, dot_out,
        pro_dst, pro_src, h->W32_key >= 0 ? h->kpc : 0, h->Etop, h->mv_R, h->mv_Q);
  } else if (prec == SDP_BF16) {
    spmm_lp<__nv_bfloat16>(h, h->W16);
    count_launch();
    k_sddmm_lp<__nv_bfloat16><<<cdiv(h->m, SDDMM_PER_BLOCK), 256, 0, h->stream>>>(
        n, h->m, h->eptr, h->ep, h->eq, h->ecoef, h->W16, h->T32, Hv, dv, h->pcg_part, h->pcg_ticket, dot_out,
        pro_dst, pro_src, h->W16_key >= 0 ? h->kpc : 0, h->Etop, h->mv_R, h->mv_Q);
  } else if (prec != SDP_FP64) {
    h->last_error = "hessian_matvec: unknown precision";
    return SDP_ERR_ARG;
  }
  if (timed) {
    // algorithmic work: T = W V (2 nnzV n flops), one length-n dot per stored entry;
    // bytes: W read for T, T written, W and T rows read by the gather (4 n^2 s) + sparse data
    const double s = (prec == SDP_FP64) ? 8.0 : (prec == SDP_FP32 ? 4.0 : 3.0);
    const double f = 2.0 * h->nnzV * (double)n + 2.0 * h->nent * (double)n;
    const double by = 4.0 * s * n * (double)n + 12.0 * h->nnzV + 16.0 * h->m;
    ktimer_end(h->stream, "matvec", f, by);
  }
  return SDP_OK;
}

// ---------------------------------------------------------------------------
// Sparse helpers for the IPM and the preconditioner
// ---------------------------------------------------------------------------
// out[i] = alpha * A_i . X + beta * add[i]   (X symmetric)
__global__ void k_opA(int m, const int* __restrict__ eptr, const int* __restrict__ ep,
                      const int* __restrict__ eq, const double* __restrict__ ecoef, int n,
                      const double* __restrict__ X, double* __restrict__ out, double alpha,
                      const double* __restrict__ add, double beta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  double s = 0.0;
  for (int e = eptr[i]; e < eptr[i + 1]; ++e) s = fma(ecoef[e], X[(size_t)ep[e] * n + eq[e]], s);
  out[i] = alpha * s + (add ? beta * add[i] : 0.0);
}
void op_A_dense(sdp_problem* h, const double* X, double* out, double alpha, const double* add, double beta) {
  count_launch();
  k_opA<<<cdiv(h->m, 256), 256, 0, h->stream>>>(h->m, h->eptr, h->ep, h->eq, h->ecoef, h->n, X, out, alpha,
                                                add, beta);
}

// D[row][col] += alpha * Vval[s]  over every slot of the V pattern
__global__ void k_scatter(int n, const int* __restrict__ rowptr, const int* __restrict__ colidx,
                          const double* __restrict__ Vval, double alpha, double* __restrict__ D) {
  const int r = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (r >= n) return;
  for (int s = rowptr[r] + lane; s < rowptr[r + 1]; s += 32) D[(size_t)r * n + colidx[s]] += alpha * Vval[s];
}
void scatter_V_dense(sdp_problem* h, const double* Vval, double alpha, double* D) {
  count_launch();
  k_scatter<<<cdiv((size_t)h->n * 32, 256), 256, 0, h->stream>>>(h->n, h->rowptr, h->colidx, Vval, alpha, D);
}

// out[a, c] = sum_{s in row a} val[s] B[col(s), c]   (c < ncols)
__global__ void k_spmm_rows(int n, const int* __restrict__ rowptr, const int* __restrict__ colidx,
                            const double* __restrict__ val, const double* __restrict__ B, int ldb, int ncols,
                            double* __restrict__ out, int ldo) {
  const int a = blockIdx.y;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncols; c += gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int s = rowptr[a]; s < rowptr[a + 1]; ++s) acc = fma(val[s], B[(size_t)colidx[s] * ldb + c], acc);
    out[(size_t)a * ldo + c] = acc;
  }
}
void spmm_rows(sdp_problem* h, const double* Vval, const double* B, int ldb, int ncols, double* out, int ldo) {
  count_launch();
  const unsigned gx = std::max(1u, std::min(cdiv(ncols, 128), 64u));
  k_spmm_rows<<<dim3(gx, h->n), 128, 0, h->stream>>>(h->n, h->rowptr, h->colidx, Vval, B, ldb, ncols, out, ldo);
}

}  // namespace sdpgb
