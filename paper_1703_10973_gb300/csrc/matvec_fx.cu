// The FP64 Hessian product in fixed point.
//
// The FP64 pipe does two multiply-adds per clock and SM and bounds the sparse products
// of matvec.cu (90 % busy).  The integer multipliers do a 32 x 32 + 64 bit multiply-add
// at many times that rate, so here each row of an operand is scaled by a power of two
// and held as 60-bit integers in two signed limbs,
//   x = (hi 2^30 + lo) 2^(ex - 1081),   |hi| <= 2^29, -2^29 <= lo < 2^29,
// (ex: the largest biased exponent of the row), 59 bits below the row's largest entry
// where FP64 keeps 53 of each.  A product takes three multiply-adds (hi hi, hi lo,
// lo hi; lo lo is below 2^-60 of the largest product), sums are exact in 64 bits for
// FX_TERMS = 16 products, which are then added to a wider pair, and each entry of the
// result is rounded once, by integer instructions.  So the errors are those of the
// scaled inputs, not of the sums: 0.1 to 0.25 of the FMA kernels' error (2-norm, against
// 113-bit sums, scaling matrices of order 210 to 2020).  375 x 190 with 35625 samples:
// 140 -> 63 us for the product, 2000 x 2000 with 60000: 1300 -> 722 us.
// Integer sums are associative: rows per CTA and lanes per constraint change no bit.
// Rows with a NaN or an infinity keep their doubles and are summed in FP64.
#include "internal.cuh"

#include <algorithm>

namespace sdpgb {

static inline unsigned cdiv(size_t a, size_t b) { return (unsigned)((a + b - 1) / b); }

constexpr int FX_TERMS = 16;
constexpr int FX_BAD = 0x7FF;   // largest exponent of a row with infinities or NaN, held as doubles
constexpr int FX_UNROLL = 8;
constexpr size_t FX_SMEM = 192 * 1024;   // for the rows of W
constexpr int FX_MIN_N = 192;   // below: launches and latency are the time (k_spmm_wv_small)

// Biased exponent of x, 1 for zero and subnormals, 0x7FF for infinities and NaN.
__device__ __forceinline__ int fx_exp(double x) { return max(1, (__double2hiint(x) >> 20) & 0x7FF); }
// x 2^(1081 - ex), rounded, in two limbs; fx_exp(x) <= ex.
__device__ __forceinline__ int2 fx_make(double x, int ex) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF);
  const long long m = (b & 0xFFFFFFFFFFFFFll) | (e ? 0x10000000000000ll : 0ll);
  const int sh = max(e, 1) - ex + 6;   // <= 6
  long long q = (sh >= 0) ? (m << sh) : (sh < -54) ? 0 : ((m + (1ll << (-sh - 1))) >> (-sh));
  if (b < 0) q = -q;
  const int lo = (int)((uint32_t)q << 2) >> 2;
  return make_int2((int)((q - lo) >> 30), lo);
}
__device__ __forceinline__ int2 fx_raw(double x) { return make_int2(__double2loint(x), __double2hiint(x)); }
__device__ __forceinline__ double fx_value(int2 q, int ex) {
  return (ex == FX_BAD) ? __hiloint2double(q.y, q.x) : scalbn((double)((long long)q.x * (1ll << 30) + q.y), ex - 1081);
}

__device__ __noinline__ double fx_round_slow(unsigned long long r, int e, bool neg) {   // subnormal or too large
  const double v = scalbn((double)r, e);
  return neg ? -v : v;
}
// (hi 2^32 + lo) 2^e rounded to nearest even.
__device__ __forceinline__ double fx_round(long long hi, long long lo, int e) {
  const long long h2 = hi + (lo >> 32);
  uint32_t l = (uint32_t)lo;
  const bool neg = h2 < 0;
  unsigned long long h = (unsigned long long)h2;
  if (neg) {
    l = 0u - l;
    h = ~h + (l == 0u ? 1ull : 0ull);
  }
  if (h == 0ull && l == 0u) return 0.0;
  unsigned long long m;
  int ex;                 // |value| = m 2^ex (+ the sticky bits below)
  bool sticky = false;
  if (h != 0ull) {
    const int z = __clzll((long long)h);
    if (z <= 32) {
      const unsigned long long ls = (unsigned long long)l << z;
      m = (h << z) | (ls >> 32);
      sticky = (uint32_t)ls != 0u;
    } else {
      m = (h << z) | ((unsigned long long)l << (z - 32));
    }
    ex = 32 - z;
  } else {
    const int z = __clz((int)l);
    m = (unsigned long long)l << (32 + z);
    ex = -32 - z;
  }
  unsigned long long r = m >> 11;
  const uint32_t rem = (uint32_t)m & 0x7FFu;
  if (rem > 0x400u || (rem == 0x400u && (sticky || (r & 1ull)))) r += 1ull;
  const int E = ex + 11 + 52 + 1023 + e;
  const unsigned long long sign = neg ? 0x8000000000000000ull : 0ull;
  if (E > 0 && E < 2046) return __longlong_as_double((long long)((((unsigned long long)(E - 1) << 52) + r) | sign));
  return fx_round_slow(r, ex + 11 + e, neg);
}

// A sum of products: value = s1 2^80 + s0 2^50 after the last flush.
struct FxSum {
  long long hh = 0, cr = 0, s1 = 0, s0 = 0;
  __device__ __forceinline__ void add(int ahi, int alo, int bhi, int blo) {
    hh += (long long)ahi * bhi;
    cr += (long long)ahi * blo;
    cr += (long long)alo * bhi;
  }
  __device__ __forceinline__ void flush() {   // after at most FX_TERMS products
    s1 += hh >> 20;
    s0 += ((hh & 0xFFFFF) << 10) + (cr >> 20);
    hh = cr = 0;
  }
  __device__ __forceinline__ double value(int exa, int exb) const {
    return fx_round(s1 >> 2, s0 + ((s1 & 3) << 30), exa + exb - 2112);
  }
};

// Fixed-point rows of W (n x ld, ld even, zero beyond n), once per W; bound by the
// traffic (n = 4000: 0.1 ms).
__global__ void __launch_bounds__(256) k_fx_rows(int n, int ld, const double* __restrict__ W, int2* __restrict__ Wx,
                                                 int* __restrict__ ex) {
  __shared__ int smx;
  const int r = blockIdx.x;
  const double* w = W + (size_t)r * n;
  if (threadIdx.x == 0) smx = 1;
  __syncthreads();
  int mx = 1;
#pragma unroll 4
  for (int c = threadIdx.x; c < n; c += 256) mx = max(mx, fx_exp(w[c]));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) atomicMax(&smx, mx);
  __syncthreads();
  mx = smx;
  if (threadIdx.x == 0) ex[r] = mx;
#pragma unroll 4
  for (int c = threadIdx.x; c < ld; c += 256) {
    const double x = (c < n) ? w[c] : 0.0;
    Wx[(size_t)r * ld + c] = (mx == FX_BAD) ? fx_raw(x) : fx_make(x, mx);
  }
}

// The entries of V = sum v_j A_j, a warp per row.  An entry is {hi, lo, place of its
// column of W in the product's shared memory}; the G rows of a group lie interleaved.
// Up to FXV_KEEP x 32 entries of a row stay in registers between the search for the
// largest exponent and the split.  Also clears the exponents of T's rows.
constexpr int FXV_KEEP = 8;
__global__ void __launch_bounds__(128) k_fx_v(int n, int R, int split, int lo0, int lo1,
                                              const int* __restrict__ rowptr, const int* __restrict__ colidx,
                                              const int* __restrict__ place, bool single,
                                              const int* __restrict__ sptr, const int* __restrict__ scon,
                                              const double* __restrict__ scoef, const double* __restrict__ v,
                                              int4* __restrict__ E, int* __restrict__ ex, int* __restrict__ exT) {
  const int c = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= n) return;
  const int s0 = rowptr[c], len = rowptr[c + 1] - s0, G = 32 / R, lo = (c < split) ? lo0 : lo1;
  int4* e = E + place[c];
  auto entry = [&](int s) {
    if (single) return fma(scoef[s], v[scon[s]], 0.0);
    double a = 0.0;
    for (int t = sptr[s]; t < sptr[s + 1]; ++t) a = fma(scoef[t], v[scon[t]], a);
    return a;
  };
  double keep[FXV_KEEP];
  int mx = 1;
#pragma unroll
  for (int u = 0; u < FXV_KEEP; ++u) {
    const int s = u * 32 + lane;
    if (s < len) {
      keep[u] = entry(s0 + s);
      mx = max(mx, fx_exp(keep[u]));
    }
  }
  for (int s = FXV_KEEP * 32 + lane; s < len; s += 32) mx = max(mx, fx_exp(entry(s0 + s)));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) {
    ex[c] = mx;
    exT[c] = 1;
  }
  auto put = [&](int s, double x) {
    const int2 q = (mx == FX_BAD) ? fx_raw(x) : fx_make(x, mx);
    const int w = colidx[s0 + s] - lo;
    e[(size_t)s * G] = make_int4(q.x, q.y, (w * R + (w & (R - 1))) * (int)sizeof(int2), 0);
  };
#pragma unroll
  for (int u = 0; u < FXV_KEEP; ++u) {
    const int s = u * 32 + lane;
    if (s < len) put(s, keep[u]);
  }
  for (int s = FXV_KEEP * 32 + lane; s < len; s += 32) put(s, entry(s0 + s));
}

// One entry of T from rows that are held as doubles.
__device__ __noinline__ double fx_spmm_f64(int len, int G, const int4* e, int exv, const uint8_t* w, int xr, int exw) {
  double acc = 0.0;
  for (int s = 0; s < len; ++s) {
    const int4 x = e[(size_t)s * G];
    acc = fma(fx_value(make_int2(x.x, x.y), exv), fx_value(*reinterpret_cast<const int2*>(w + (x.z ^ xr)), exw), acc);
  }
  return acc;
}

// T = W V.  A CTA holds R rows of W over the columns that its rows of V touch, column
// by column, and takes a share of those rows of V; R lanes work on a row of V, each
// for one row of W, so that an entry is a broadcast and the R values of W that it
// needs are one contiguous segment: 3 multiply-adds and 3 shared-memory wavefronts per
// 32 products for R = 16.  (Lanes on different rows of V gather from random columns: 5
// wavefronts.)  The segment's slots are exchanged by the column's low bits, so that the
// staging, along columns, writes without bank conflicts.  The entries of V come by
// asynchronous copies, a chunk of 1 KB per warp ahead of the multiplications (across
// the ends of rows): loaded to registers eight at a time, their latency was most of the
// time.  T goes out transposed (whole segments) and in FP64, its rows' largest
// exponents by atomics.
constexpr int FXP_DEPTH = 2, FXP_WARPS = 16;
constexpr int FXP_CHUNK = 64;   // entries, two per lane
__device__ __forceinline__ void fx_copy16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
template <int R>
__global__ void __launch_bounds__(32 * FXP_WARPS, 2)
    k_fx_spmm(int n, int ld, int2 rng0, int2 rng1, int S0, int S1, int ngrp0, int ngrp1,
              const int2* __restrict__ grp, const int* __restrict__ rid, const int4* __restrict__ E,
              const int* __restrict__ exV, const int* __restrict__ rowptr, const int2* __restrict__ Wx,
              const int* __restrict__ exW, double* __restrict__ Tt, int* __restrict__ exT) {
  constexpr int G = 32 / R;            // rows of V per warp
  constexpr int STEPS = FXP_CHUNK / G;   // entries of each in a chunk
  constexpr int BLOCK = STEPS < FX_TERMS ? STEPS : FX_TERMS;
  extern __shared__ __align__(16) uint8_t fx_smem_raw[];
  __shared__ int smx[R];
  const int r0 = blockIdx.x * R, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int4* ring = reinterpret_cast<int4*>(fx_smem_raw) + w * (FXP_DEPTH * FXP_CHUNK);
  uint8_t* wfx = fx_smem_raw + FXP_WARPS * FXP_DEPTH * FXP_CHUNK * sizeof(int4);   // columns x R limbs
  const uint32_t ring_u = (uint32_t)__cvta_generic_to_shared(ring) + 16u * lane;
  const bool second = (int)blockIdx.y >= S0;
  const int2 rng = second ? rng1 : rng0;
  const int S = second ? S1 : S0, j = (int)blockIdx.y - (second ? S0 : 0);
  const int g0 = second ? ngrp0 : 0, ng = second ? ngrp1 : ngrp0;
  // group of this warp's turn it: by decreasing length, dealt over CTAs and warps there
  // and back; -1 past the end (a turn without a group can only be the last)
  auto group = [&](int it) {
    const int gi = (it * FXP_WARPS + ((it & 1) ? FXP_WARPS - 1 - w : w)) * S + j;
    return gi < ng ? g0 + gi : -1;
  };
  // copies: group pg (its place and length pr), chunk pc; the group after it is on its way
  int pit = 0, pg = group(0), pc = 0, ahead = group(1), slot = 0;
  int2 pr = (pg >= 0) ? grp[pg] : make_int2(0, 0);
  int2 pn = (ahead >= 0) ? grp[ahead] : make_int2(0, 0);
  auto copy = [&]() {   // one chunk; a group of no entries takes one empty chunk
    if (pg >= 0) {
      const int o = pc * FXP_CHUNK + lane, left = pr.y * G;
      if (o < left) fx_copy16(ring_u + 16u * FXP_CHUNK * slot, E + pr.x + o);
      if (o + 32 < left) fx_copy16(ring_u + 16u * FXP_CHUNK * slot + 512u, E + pr.x + o + 32);
      if (++pc * STEPS >= pr.y) {
        pg = ahead;
        pr = pn;
        pc = 0;
        ahead = group(++pit + 1);
        pn = (ahead >= 0) ? grp[ahead] : make_int2(0, 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    slot = (slot + 1 == FXP_DEPTH) ? 0 : slot + 1;
  };
#pragma unroll
  for (int d = 0; d < FXP_DEPTH - 1; ++d) copy();
  if (threadIdx.x < R) smx[threadIdx.x] = 1;
  const int width = rng.y - rng.x;
  for (int i = threadIdx.x; i < width * (R / 4); i += 32 * FXP_WARPS) {
    const int q = i / width, c = i - q * width;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = 4 * q + u;
      const int2 x = (r0 + r < n) ? Wx[(size_t)(r0 + r) * ld + rng.x + c] : make_int2(0, 0);
      reinterpret_cast<int2*>(wfx)[c * R + (r ^ (c & (R - 1)))] = x;
    }
  }
  const int r = lane & (R - 1), g = lane / R, xr = r * (int)sizeof(int2);
  const int exw = (r0 + r < n) ? exW[r0 + r] : 1;
  __syncthreads();
  int mx = 1, use = 0;
  for (int it = 0, gi; (gi = group(it)) >= 0; ++it) {
    const int2 gr = grp[gi];
    const int c = rid[gi * G + g];
    const int exv = (c >= 0) ? exV[c] : 1;
    FxSum f;
    for (int k = 0;; k += STEPS) {
      copy();
      asm volatile("cp.async.wait_group %0;" ::"n"(FXP_DEPTH - 1) : "memory");
      __syncwarp();
      const int4* e = ring + use * FXP_CHUNK + g;
      const int left = gr.y - k;   // of the group's longest row; the others end in zeros
      auto mul = [&](const int4& x) {
        const int2 a = *reinterpret_cast<const int2*>(wfx + (x.z ^ xr));
        f.add(x.x, x.y, a.x, a.y);
      };
#pragma unroll
      for (int b = 0; b < STEPS; b += BLOCK) {
        if (left >= b + BLOCK) {
#pragma unroll
          for (int s = 0; s < BLOCK; ++s) mul(e[(b + s) * G]);
        } else {
#pragma unroll 4
          for (int s = b; s < left; ++s) mul(e[s * G]);
        }
        if (BLOCK == FX_TERMS || (k & STEPS)) f.flush();
      }
      use = (use + 1 == FXP_DEPTH) ? 0 : use + 1;
      __syncwarp();   // the chunk is read: the next copy may take its place
      if (left <= STEPS) break;
    }
    if (BLOCK != FX_TERMS) f.flush();
    if (c >= 0 && r0 + r < n) {
      double t;
      if (exw != FX_BAD && exv != FX_BAD) t = f.value(exw, exv);
      else t = fx_spmm_f64(rowptr[c + 1] - rowptr[c], G, E + gr.x + g, exv, wfx, xr, exw);
      mx = max(mx, fx_exp(t));
      Tt[(size_t)c * n + r0 + r] = t;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  atomicMax(&smx[r], mx);
  __syncthreads();
  if (threadIdx.x < R && r0 + (int)threadIdx.x < n) atomicMax(&exT[r0 + threadIdx.x], smx[threadIdx.x]);
}

// Limbs of T's rows from its transpose, 32 x 32 tiles; columns n .. ld - 1 are zero.
// Bound by the traffic from some 1000 rows on (n = 4000: 50 us).
__global__ void __launch_bounds__(256) k_fx_limbs(int n, int ld, const double* __restrict__ Tt,
                                                  const int* __restrict__ exT, int2* __restrict__ Tx) {
  __shared__ double tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32, x = threadIdx.x & 31, y = threadIdx.x >> 5;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = c0 + y + 8 * u, r = r0 + x;
    tile[y + 8 * u][x] = (c < n && r < n) ? Tt[(size_t)c * n + r] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = r0 + y + 8 * u, c = c0 + x;
    if (r >= n || c >= ld) continue;
    const double t = tile[x][y + 8 * u];
    const int ex = exT[r];
    Tx[(size_t)r * ld + c] = (ex == FX_BAD) ? fx_raw(t) : fx_make(t, ex);
  }
}

// Hv_i = sum over A_i's entries of coef W[p, :] . T[q, :], FXD_L lanes per constraint.
// Bound by the latency and bandwidth of the rows' loads from L2 (constraints in order
// share W[p, :], not T[q, :]).  n = 4000, 60000 constraints: 151 us, with 8 lanes 169 us,
// 32 lanes 149 us (but 22 against 20 us at n = 565); FP64 435 us.
constexpr int FXD_G = 2, FXD_L = 32 / FXD_G;
constexpr int FXD_PER_BLOCK = (256 / 32) * FXD_G;
__device__ __noinline__ double fx_dot_f64(int n, int gl, const int2* w, int exw, const int2* t, int ext) {
  double s = 0.0;
  for (int l = gl; l < n; l += FXD_L) s = fma(fx_value(w[l], exw), fx_value(t[l], ext), s);
  return s;
}
__global__ void __launch_bounds__(256) k_fx_sddmm(int n, int ld, int m, const int* __restrict__ eptr,
                                                  const int* __restrict__ ep, const int* __restrict__ eq,
                                                  const double* __restrict__ ecoef, const int2* __restrict__ Wx,
                                                  const int* __restrict__ exW, const int2* __restrict__ Tx,
                                                  const int* __restrict__ exT, double* __restrict__ Hv,
                                                  const double* __restrict__ dv, double* dpart, unsigned int* ticket,
                                                  double* dout, double* pro_dst, const double* pro_src) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x % 32;
  const int gl = lane % FXD_L;
  const int i = warp * FXD_G + lane / FXD_L;
  const int e0 = (i < m) ? eptr[i] : 0, cnt = (i < m) ? eptr[i + 1] - e0 : 0;
  const int maxcnt = __reduce_max_sync(0xffffffffu, cnt);
  const int pairs = ld / 2;
  double acc = 0.0;
  for (int t = 0; t < maxcnt; ++t) {
    FxSum f;
    double hard = 0.0;
    int exw = 1, ext = 1;
    if (t < cnt) {
      const int p = ep[e0 + t], q = eq[e0 + t];
      exw = exW[p];
      ext = exT[q];
      const int4* wp = reinterpret_cast<const int4*>(Wx + (size_t)p * ld);
      const int4* tq = reinterpret_cast<const int4*>(Tx + (size_t)q * ld);
      int l = gl;
      bool odd = false;
#pragma unroll 2
      for (; l + 3 * FXD_L < pairs; l += 4 * FXD_L) {   // eight products, four loads of each row in flight
        int4 a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          a[u] = wp[l + u * FXD_L];
          b[u] = tq[l + u * FXD_L];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          f.add(a[u].x, a[u].y, b[u].x, b[u].y);
          f.add(a[u].z, a[u].w, b[u].z, b[u].w);
        }
        if (odd) f.flush();
        odd = !odd;
      }
      for (; l < pairs; l += FXD_L) {   // at most six products on top of eight
        const int4 a = wp[l], b = tq[l];
        f.add(a.x, a.y, b.x, b.y);
        f.add(a.z, a.w, b.z, b.w);
      }
      f.flush();
      if (exw == FX_BAD || ext == FX_BAD)
        hard = fx_dot_f64(n, gl, Wx + (size_t)p * ld, exw, Tx + (size_t)q * ld, ext);
    }
#pragma unroll
    for (int o = FXD_L / 2; o > 0; o >>= 1) {
      f.s1 += __shfl_xor_sync(0xffffffffu, f.s1, o);
      f.s0 += __shfl_xor_sync(0xffffffffu, f.s0, o);
    }
    const bool bad = exw == FX_BAD || ext == FX_BAD;
    if (__any_sync(0xffffffffu, bad)) {
#pragma unroll
      for (int o = FXD_L / 2; o > 0; o >>= 1) hard += __shfl_xor_sync(0xffffffffu, hard, o);
    }
    if (t < cnt) acc = fma(ecoef[e0 + t], bad ? hard : f.value(exw, ext), acc);
  }
  if (i < m && gl == 0) Hv[i] = acc;
  if (dv) {
    const double c = (i < m && gl == 0) ? dv[i] * acc : 0.0;
    double tot;
    if (lb_reduce(c, dpart, ticket, &tot, blockIdx.x, gridDim.x)) {
      if (pro_dst) *pro_dst = *pro_src;
      *dout = tot;
    }
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
// Layout of V for the product (at setup, O(n)): two classes of rows, [0, split) and
// [split, n), each with the range of columns that it touches -- for a bipartite pattern
// (completion of a rectangular matrix) that halves the rows of W a CTA has to hold --
// and R, the rows of W per CTA that fit.
void fx_layout(sdp_problem* h, const std::vector<int>& rowptr, const std::vector<int>& colidx,
               const std::vector<int>& rowperm, std::vector<int2>& grp, std::vector<int>& rid, std::vector<int>& place) {
  const int n = h->n;
  h->fx_R = 0;
  if (n <= FX_MIN_N) return;
  std::vector<int2> pre(n + 1, make_int2(n, 0)), suf(n + 1, make_int2(n, 0));   // ranges of the first / last rows
  auto join = [&](int2 a, int c) {
    if (rowptr[c] < rowptr[c + 1])   // columns ascend
      a = make_int2(std::min(a.x, colidx[rowptr[c]]), std::max(a.y, colidx[rowptr[c + 1] - 1] + 1));
    return a;
  };
  for (int c = 0; c < n; ++c) pre[c + 1] = join(pre[c], c);
  for (int c = n - 1; c >= 0; --c) suf[c] = join(suf[c + 1], c);
  auto width = [](int2 a) { return std::max(0, a.y - a.x); };
  int split = n;
  for (int s = 0; s < n; ++s)
    if (std::max(width(pre[s]), width(suf[s])) < std::max(width(pre[split]), width(suf[split]))) split = s;
  h->fx_split = split;
  h->fx_rng[0] = width(pre[split]) ? pre[split] : make_int2(0, 0);
  h->fx_rng[1] = width(suf[split]) ? suf[split] : make_int2(0, 0);
  const size_t widest = std::max({width(pre[split]), width(suf[split]), 1});
  for (int R : {16, 8, 4})
    if (!h->fx_R && widest * R * sizeof(int2) <= FX_SMEM) h->fx_R = R;
  if (!h->fx_R) return;
  const int G = 32 / h->fx_R;
  place.assign(n, 0);
  size_t at = 0;
  for (int cls = 0; cls < 2; ++cls) {
    const size_t first = rid.size() / G;
    int g = 0;
    for (int c : rowperm) {   // by decreasing length
      if ((c < split) != (cls == 0)) continue;
      if (g == 0) {
        const int len = rowptr[c + 1] - rowptr[c];
        grp.push_back(make_int2((int)at, len));
        rid.resize(rid.size() + G, -1);
        at += (size_t)len * G;
      }
      rid[rid.size() - G + g] = c;
      place[c] = grp.back().x + g;
      g = (g + 1) % G;
    }
    h->fx_ngrp[cls] = (int)(rid.size() / G - first);
  }
  if (at > (size_t)INT32_MAX / 2) {
    h->fx_R = 0;
    return;
  }
  h->fx_len = at;
}

// Where the fixed-point form is the faster one (microseconds per product, FP64 / fixed).
// A product costs a third, an entry of T more (rounding, splitting, one more pass):
// at least 12 products per entry (193 with 72 per row: 24.6 / 21.5; 1600, 14 per row:
// 98 / 94; 3000, 7 per row: 244 / 273; 5024, 4 per row: 530 / 585), or
// orders where neither the launches nor the n^2 terms weigh (450, 7 per row: 26.7 /
// 25.5; 1030, 5 per row: 68 / 60; but 193, 9 per row: 18.5 / 20.5).
bool fx_pays(const sdp_problem* h) {
  return h->fx_R > 0 && ((double)h->nnzV + h->nent >= 12.0 * h->n || (h->n >= 300 && h->n <= 1200));
}

// Limbs of the current W (its first call allocates); SDP_ERR_OOM leaves the handle as it was.
sdp_status fx_prepare(sdp_problem* h) {
  const int n = h->n, ld = (n + 1) / 2 * 2;
  if (!h->fx_mem) {
    auto up = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
    const size_t mat = up((size_t)n * ld * sizeof(int2)), ent = up(h->fx_len * sizeof(int4) + 16), exb = up(n * sizeof(int));
    SDP_TRY(h->alloc(&h->fx_mem, 2 * mat + ent + 3 * exb));
    uint8_t* p = static_cast<uint8_t*>(h->fx_mem);
    h->fxW = reinterpret_cast<int2*>(p);
    h->fxT = reinterpret_cast<int2*>(p + mat);
    h->fxE = reinterpret_cast<int4*>(p + 2 * mat);
    h->fx_exW = reinterpret_cast<int*>(p + 2 * mat + ent);
    h->fx_exT = reinterpret_cast<int*>(p + 2 * mat + ent + exb);
    h->fx_exV = reinterpret_cast<int*>(p + 2 * mat + ent + 2 * exb);
    h->fx_valid = false;
    SDP_CK(h, cudaMemsetAsync(h->fxE, 0, ent, h->stream));            // the ends of shorter rows stay zero
  }
  if (!h->fx_valid) {
    count_launch();
    k_fx_rows<<<n, 256, 0, h->stream>>>(n, ld, h->W, h->fxW, h->fx_exW);
    h->fx_valid = true;
  }
  return SDP_OK;
}

static size_t fx_smem(const sdp_problem* h) {
  const int w = std::max(h->fx_rng[0].y - h->fx_rng[0].x, h->fx_rng[1].y - h->fx_rng[1].x);
  return FXP_WARPS * FXP_DEPTH * FXP_CHUNK * sizeof(int4) + std::max((size_t)w, (size_t)1) * h->fx_R * sizeof(int2);
}

// Shares of each class of V's rows: enough CTAs for all SMs, and as few as that takes,
// since each stages its rows of W.  Cycles of the SM with the most CTAs, from 5 per 32
// products and 64 staged bytes per cycle.
static void fx_shares(const sdp_problem* h, int S[2]) {
  const int nb = (int)cdiv(h->n, h->fx_R);
  const size_t smem = fx_smem(h);
  const int occ = smem > 112 * 1024 ? 1 : 2;
  double tb = 1e300;
  const bool two = h->fx_ngrp[0] > 0 && h->fx_ngrp[1] > 0;
  for (int s = 1; s <= 16; ++s) {
    const double ctas = (double)nb * s * (two ? 2 : 1);
    const double one = (h->nnzV / (two ? 2.0 : 1.0) / s) * h->fx_R / 32.0 * 5.0 + smem / 64.0 + 1500.0;
    const double t = std::ceil(ctas / (152.0 * occ)) * occ * one;
    if (t < 0.97 * tb) {
      tb = t;
      S[0] = h->fx_ngrp[0] > 0 ? s : 0;
      S[1] = h->fx_ngrp[1] > 0 ? s : 0;
    }
  }
}
template <int R>
static void launch_fx_spmm(sdp_problem* h, int ld, const int* S) {
  allow_max_smem((const void*)k_fx_spmm<R>);
  count_launch();
  k_fx_spmm<R><<<dim3(cdiv(h->n, R), S[0] + S[1]), 32 * FXP_WARPS, fx_smem(h), h->stream>>>(
      h->n, ld, h->fx_rng[0], h->fx_rng[1], S[0], S[1], h->fx_ngrp[0], h->fx_ngrp[1], h->fx_grp, h->fx_rid,
      h->fxE, h->fx_exV, h->rowptr, h->fxW, h->fx_exW, h->T, h->fx_exT);
}

// Hv = A(W V W); the arguments as for matvec_impl.  Launches only (fx_prepare first).
void fx_matvec(sdp_problem* h, const double* v, double* Hv, double* dot_out, double* pro_dst, const double* pro_src) {
  const int n = h->n, ld = (n + 1) / 2 * 2;
  const bool timed = ktimer_on("matvec");
  if (timed) ktimer_begin(h->stream, "matvec");
  int S[2] = {0, 0};
  fx_shares(h, S);
  count_launch(2);
  k_fx_v<<<cdiv(n, 4), 128, 0, h->stream>>>(n, h->fx_R, h->fx_split, h->fx_rng[0].x, h->fx_rng[1].x, h->rowptr, h->colidx,
                                            h->fx_place, h->single, h->sptr, h->scon, h->scoef, v, h->fxE, h->fx_exV,
                                            h->fx_exT);
  if (S[0] + S[1] > 0) {
    switch (h->fx_R) {
      case 16: launch_fx_spmm<16>(h, ld, S); break;
      case 8: launch_fx_spmm<8>(h, ld, S); break;
      default: launch_fx_spmm<4>(h, ld, S); break;
    }
  }
  k_fx_limbs<<<dim3(cdiv(ld, 32), cdiv(n, 32)), 256, 0, h->stream>>>(n, ld, h->T, h->fx_exT, h->fxT);
  count_launch();
  k_fx_sddmm<<<cdiv(h->m, FXD_PER_BLOCK), 256, 0, h->stream>>>(
      n, ld, h->m, h->eptr, h->ep, h->eq, h->ecoef, h->fxW, h->fx_exW, h->fxT, h->fx_exT, Hv, dot_out ? v : nullptr,
      h->pcg_part, h->pcg_ticket, dot_out, pro_dst, pro_src);
  if (timed) {
    const double f = 2.0 * h->nnzV * (double)n + 2.0 * h->nent * (double)n;
    ktimer_end(h->stream, "matvec", f, 32.0 * n * (double)n + 12.0 * h->nnzV + 16.0 * h->m);
  }
}

}  // namespace sdpgb
