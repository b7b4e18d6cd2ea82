// Low-rank preconditioner of Sec. 3.
//
// Set-up (once per (X, kernel, gamma)): F = RPCholesky(K, r0), K ~= F F^T,
// pivots drawn with probability proportional to the residual diagonal; then
// the rank heuristic of Sec. 3 (smallest r with xi lambda_1 >= lambda_r over
// the eigenvalues of F0^T F0) and truncation to r columns (re-running
// RPCholesky with the same pivot stream reproduces exactly the first r
// columns).  lambda_1 comes from power iteration and the count of eigenvalues
// above xi lambda_1 from the inertia of an LDL^T factorisation of
// F0^T F0 - xi lambda_1 I (Sylvester's law), so no full eigensolver is needed.
//
// Per linear system: Lemma 1,
//   P^{-1} = L^{-1} - L^{-1} U (C + U^T L^{-1} U)^{-1} U^T L^{-1},
//   U = [F 1], C = diag(I_r, 1/gam),
// with the (r+1)^2 core built in FP64, Cholesky-factorised and inverted on the
// device; each apply is two skinny FP64-class products with the FP32 factor.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "kqr_internal.h"
#include "reduce.cuh"
#include "wb_split.cuh"

namespace kqr {

#define GRID_LOOP(i, n) \
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

// ---- weighted Gram of the columns of U = [F, 1] (optional ones column) -----------
// G[a][b] = sum_i U_ai (w_i U_bi), FP64-class on the FP32 pipe.
//
// On the FP64 pipe (2 FMAs per clock and SM) the r^2 n / 2 products of a core cost 21 ms at
// n = 20011, r = 1024, and a conversion of F besides.  Here a product is an FP32 factor (F
// itself, exact) times a double-float (w U, or F of the set-up, as hi + lo): 11 FP32 pipe
// operations with the TwoSum accumulation, 128 lanes per clock and SM instead of 2.  The
// double-float sums run over kCgRows rows only, renormalised every 4, and are then added to FP64 sums.
// Their low part is a plain float sum, whose rounding grows with the rows of a group, where the rounding
// of the FP64 sum that it replaces grows with all rows.  Against 64 bits the apply of such a core errs
// as much as that of an FP64 core, or less, at n = 12000 .. 30000 (geometric means over systems of five
// kinds of diagonal; groups of 32 rows not renormalised: up to 1.7 times as much); at n = 1000 it
// erred two to three times as much.  So up to kCgCompRows rows the low part is summed with its rounding errors
// kept (COMP, 23 operations a product instead of 11), which is at or below FP64's error at every size;
// such a core is small.  w is scaled by the power of two that brings its maximum to [1, 2), so that hi
// and lo stay inside the FP32 range.
//
// Tile: 64 x 64 entries per CTA of 128 threads, 4 x 8 per thread (32 independent chains; the
// operands of a row are 20 shared-memory words for 352 FP32 operations).  The rows are cut into
// chunks so that about two waves of CTAs exist at every (n, r): with a fixed chunk of 4096 rows
// a rank-45 core at n = 2000 ran on 3 CTAs (707 us, now 26).  n = 20011, r = 1024: 21.1 ms
// before, 8.5 ms now; the FP32 pipe alone would take 3.4 ms, the rest is the operand split and
// the FP64 additions (7.2 ms with groups of 32 rows, whose error was larger).
constexpr int kCT = 64;      // core tile
constexpr int kCR = 16;      // rows per shared-memory step
constexpr int kCgRows = 16;  // rows per double-float sum
constexpr int kCgThreads = 128;
constexpr int64_t kCgCompRows = 8192;   // rows up to which the low parts are compensated

// s + e = a + b exactly, s = fl(a + b)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

// T: float (the FP32 factor, weights w; both triangles of G are written) or double (the set-up's FP64 factor, no weights).
template <typename T, bool COMP>
__global__ void __launch_bounds__(kCgThreads, COMP ? 2 : 3)
    core_gram_kernel(const T* __restrict__ F, int64_t ldf, int rr, int ncols, int64_t n, const double* __restrict__ w,
                     const unsigned long long* __restrict__ wmax, double* __restrict__ G, int ntile,
                     int64_t chunk) {
  constexpr bool kPair = sizeof(T) == 8;   // the left operand needs its low part too
  // blockIdx.x enumerates tile pairs (ta <= tb), blockIdx.y row chunks.
  int pair = blockIdx.x, ta = 0;
  while (pair >= ntile - ta) { pair -= ntile - ta; ++ta; }
  const int tb = ta + pair;
  __shared__ __align__(16) float Ah[kCR][kCT + 4];
  __shared__ __align__(16) float Al[kPair ? kCR : 1][kCT + 4];
  __shared__ __align__(16) float Bh[kCR][kCT + 4];
  __shared__ __align__(16) float Bl[kCR][kCT + 4];
  const int tid = threadIdx.x;
  const int la = (tid >> 3) * 4;   // 4 rows of the tile
  const int lb = (tid & 7) * 4;    // columns lb .. lb + 3 and 32 + lb ..
  double scale = 1.0, unscale = 1.0;
  if (wmax) {
    const int ex = (int)((*wmax >> 52) & 0x7ff);   // biased exponent of max w
    if (ex > 0 && ex < 2046) {
      scale = __longlong_as_double((long long)(2046 - ex) << 52);   // 2^(1023 - ex)
      unscale = __longlong_as_double((long long)ex << 52);
    }
  }
  __shared__ float2 wsplit[kCgRows];   // w_i scaled, as hi + lo (float T)
  double tot[4][8];
  float sl[4][8];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      tot[a][b] = 0.0;
      sl[a][b] = 0.f;
    }
  const int64_t i0 = (int64_t)blockIdx.y * chunk;
  const int64_t i1 = min(n, i0 + chunk);
  for (int64_t ig = i0; ig < i1; ig += kCgRows) {
    float sh[4][8], sll[COMP ? 4 : 1][COMP ? 8 : 1];   // sll: what the low sums' roundings left
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        sh[a][b] = 0.f;
        if (COMP) sll[COMP ? a : 0][COMP ? b : 0] = 0.f;
      }
    if (!kPair) {
      __syncthreads();
      if (tid < kCgRows) {
        const double wi = ig + tid < i1 ? (w ? w[ig + tid] * scale : 1.0) : 0.0;
        float hi, lo;
        df_split(wi, hi, lo);
        wsplit[tid] = make_float2(hi, lo);
      }
    }
    for (int64_t ib = ig; ib < min(i1, ig + kCgRows); ib += kCR) {
      __syncthreads();
      // lanes along the rows of a column (F is column-major): 16 rows x 2 columns per warp load
      for (int e = tid; e < kCR * kCT; e += kCgThreads) {
        const int k = e % kCR, c = e / kCR;
        const int64_t i = ib + k;
        const int ca = ta * kCT + c, cb = tb * kCT + c;
        T ua = 0, ub = 0;
        if (i < i1) {
          ua = ca < rr ? F[(size_t)ca * ldf + i] : (T)(ca < ncols ? 1 : 0);
          ub = cb < rr ? F[(size_t)cb * ldf + i] : (T)(cb < ncols ? 1 : 0);
        }
        if (kPair) {
          df_split((double)ua, Ah[k][c], Al[kPair ? k : 0][c]);
          df_split((double)ub, Bh[k][c], Bl[k][c]);
        } else {
          const float2 wi = wsplit[(int)(ib - ig) + k];
          const float u = (float)ub, bh = __fmul_rn(wi.x, u);
          Ah[k][c] = (float)ua;
          Bh[k][c] = bh;
          Bl[k][c] = fmaf(wi.y, u, fmaf(wi.x, u, -bh));
        }
      }
      __syncthreads();
#pragma unroll 2
      for (int k = 0; k < kCR; ++k) {
        if (!COMP && k > 0 && k % 4 == 0) {   // renormalise, so that the low sums' roundings stay small
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) {
              const float v = __fadd_rn(sh[a][b], sl[a][b]);
              sl[a][b] = __fsub_rn(sl[a][b], __fsub_rn(v, sh[a][b]));
              sh[a][b] = v;
            }
        }
        const float4 a4 = *reinterpret_cast<const float4*>(&Ah[k][la]);
        const float4 h0 = *reinterpret_cast<const float4*>(&Bh[k][lb]);
        const float4 h1 = *reinterpret_cast<const float4*>(&Bh[k][32 + lb]);
        const float4 l0 = *reinterpret_cast<const float4*>(&Bl[k][lb]);
        const float4 l1 = *reinterpret_cast<const float4*>(&Bl[k][32 + lb]);
        const float xa[4] = {a4.x, a4.y, a4.z, a4.w};
        float xl[4] = {0.f, 0.f, 0.f, 0.f};
        if (kPair) {
          const float4 q = *reinterpret_cast<const float4*>(&Al[kPair ? k : 0][la]);
          xl[0] = q.x; xl[1] = q.y; xl[2] = q.z; xl[3] = q.w;
        }
        const float yh[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
        const float yl[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) {
            const float p = __fmul_rn(xa[a], yh[b]);
            float e = fmaf(xa[a], yh[b], -p);
            e = fmaf(xa[a], yl[b], e);
            if (kPair) e = fmaf(xl[a], yh[b], fmaf(xl[a], yl[b], e));
            float er;
            sh[a][b] = two_sum(sh[a][b], p, er);
            if (COMP) {
              float g0, g1;
              const float g = two_sum(er, e, g0);
              sl[a][b] = two_sum(sl[a][b], g, g1);
              float& c = sll[COMP ? a : 0][COMP ? b : 0];
              c = __fadd_rn(c, __fadd_rn(g0, g1));
            } else {
              sl[a][b] = __fadd_rn(sl[a][b], __fadd_rn(er, e));
            }
          }
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        // renormalise, so that one FP64 addition takes all but a remainder below half an ulp of it
        const float v = __fadd_rn(sh[a][b], sl[a][b]);
        sl[a][b] = __fsub_rn(sl[a][b], __fsub_rn(v, sh[a][b]));
        if (COMP) sl[a][b] = __fadd_rn(sl[a][b], sll[COMP ? a : 0][COMP ? b : 0]);
        tot[a][b] += (double)v;
      }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const int ra = ta * kCT + la + a, cb = tb * kCT + (b < 4 ? lb + b : 28 + lb + b);
      if (ra < ncols && cb < ncols) {
        const double v = (tot[a][b] + (double)sl[a][b]) * unscale;
        atomicAdd(&G[(size_t)ra * ncols + cb], v);
        if (ta != tb) atomicAdd(&G[(size_t)cb * ncols + ra], v);
      }
    }
}

// wmax (device, nullable): max_i w_i, for the scaling of the weights.
template <typename T>
static cudaError_t core_gram(Handle* h, const T* F, int64_t ldf, int rr, bool ones, const double* w,
                             const unsigned long long* wmax, double* G, cudaStream_t st) {
  const int ncols = rr + (ones ? 1 : 0);
  cudaError_t e = cudaMemsetAsync(G, 0, sizeof(double) * ncols * ncols, st);
  if (e != cudaSuccess) return e;
  const int ntile = (ncols + kCT - 1) / kCT;
  const int pairs = ntile * (ntile + 1) / 2;
  // about 6 CTAs per SM (two waves of 3 resident ones), chunks of a multiple of kCgRows rows
  const int64_t want = ((int64_t)6 * h->num_sms + pairs - 1) / pairs;
  int64_t chunk = (h->n + want - 1) / want;
  chunk = (chunk + kCgRows - 1) / kCgRows * kCgRows;
  const int chunks = (int)((h->n + chunk - 1) / chunk);
  auto kern = h->n <= kCgCompRows ? core_gram_kernel<T, true> : core_gram_kernel<T, false>;
  kern<<<dim3(pairs, chunks), kCgThreads, 0, st>>>(F, ldf, rr, ncols, h->n, w, wmax, G, ntile, chunk);
  h->launches++;
  return cudaGetLastError();
}

__global__ void add_diag_kernel(double* G, int N, double v, double last) {
  GRID_LOOP(i, N) G[i * N + i] += (i == N - 1) ? last : v;
}

// out = 1 / L and the bits of its maximum (non-negative doubles order like their bits).
__global__ void recip_kernel(double* out, const double* L, int64_t n, unsigned long long* __restrict__ wmax) {
  double m = 0.0;
  GRID_LOOP(i, n) {
    const double v = 1.0 / L[i];
    out[i] = v;
    m = fmax(m, v);
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(wmax, (unsigned long long)__double_as_longlong(m));
}

// ---- apply of Lemma 1 -----------------------------------------------------------------
// out = L^{-1} (r - U G^{-1} U^T L^{-1} r): two passes over the FP32 factor F (r n entries each)
// around a product with the (r + 1)^2 core inverse.
//
// What bounds it: reading F twice (80 MB each at n = 20011, r = 1024: from L2, beyond that from
// HBM).  On the FP64 pipe the two passes cost 2 r n FMAs at 2 per clock and SM plus a conversion
// of every F entry at the same rate, 160 and 334 us at that size with the latency of one thread
// per row.  Here every product is FP32 x double-float: L^{-1} r and the core's result are split once
// into hi + lo, after scaling by powers of two (the exponent of ||r|| and of max L^{-1}) that keep both
// parts inside the FP32 range for any r.  Sums are three floats (23 FP32-pipe operations a product: the
// roundings of the low sums are summed too); as double-floats, 11 operations, the apply's error was two
// to three times that of FP64 passes on well-conditioned systems (n = 1000 .. 20000, ranks from 200),
// like this it is FP64's.  Measured (n = 20011, r = 1024): 42 and 37 us (passes in FP64: 160 and 334).
// Sum of three floats, (h + l + ll) += x (yh + yl), x FP32.
struct Sum3 {
  float h = 0.f, l = 0.f, ll = 0.f;
  __device__ __forceinline__ void mac(float x, float yh, float yl) {
    const float p = __fmul_rn(x, yh);
    const float e = fmaf(x, yl, fmaf(x, yh, -p));
    float er, g0, g1;
    h = two_sum(h, p, er);
    const float g = two_sum(er, e, g0);
    l = two_sum(l, g, g1);
    ll = __fadd_rn(ll, __fadd_rn(g0, g1));
  }
  __device__ __forceinline__ void add(float yh, float yl, float yll) {
    float er, e0, e1;
    h = two_sum(h, yh, er);
    l = two_sum(l, yl, e0);
    l = two_sum(l, er, e1);
    ll = __fadd_rn(__fadd_rn(ll, yll), __fadd_rn(e0, e1));
  }
  __device__ __forceinline__ void add_lane(int o) {
    add(__shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, l, o), __shfl_xor_sync(0xffffffffu, ll, o));
  }
  __device__ __forceinline__ double value() const { return (double)h + ((double)l + (double)ll); }
};

// bits of max |r|
__global__ void absmax_kernel(const double* __restrict__ rv, int64_t n, unsigned long long* __restrict__ out) {
  double m = 0.0;
  GRID_LOOP(i, n) m = fmax(m, fabs(rv[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// us = L^{-1} r scaled, as hi + lo (rows >= n: 0); t = 0; the exponent used for r into scal[S_WEXP].
__global__ void __launch_bounds__(256) wb_split_kernel(const double* __restrict__ Linv, const double* __restrict__ rv,
                                                       int64_t n, int64_t ldn, const double* __restrict__ rr,
                                                       int is_max, double* __restrict__ scal, float2* __restrict__ us,
                                                       double* __restrict__ t, int N) {
  const int e = norm_exponent(*rr, is_max != 0);
  const double sr = pow2(-e);
  const double sw = pow2(-max_exponent(*reinterpret_cast<const unsigned long long*>(scal + S_WMAX)));
  GRID_LOOP(i, ldn) {
    float2 v = make_float2(0.f, 0.f);
    if (i < n) df_split((Linv[i] * sw) * (rv[i] * sr), v.x, v.y);
    us[i] = v;
  }
  if (blockIdx.x == 0) {
    for (int c = threadIdx.x; c < N; c += blockDim.x) t[c] = 0.0;
    if (threadIdx.x == 0) scal[S_WEXP] = (double)e;
  }
}

// t[a] += sum_i U_ai (L^{-1} r)_i over `rows` rows (a multiple of 128) and 32 columns of U = [F 1]:
// a warp takes four columns, a lane four consecutive rows per step.
__global__ void __launch_bounds__(256) ut_kernel(const float* __restrict__ F, int64_t ldf, int r,
                                                 const float2* __restrict__ us, const double* __restrict__ scal,
                                                 double* __restrict__ t, int rows) {
  extern __shared__ __align__(16) float su[];   // hi[rows], lo[rows]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * rows;
  const int cnt = (int)min((int64_t)rows, ldf - i0);   // a multiple of 128
  for (int e = threadIdx.x; e < cnt; e += 256) {
    const float2 v = us[i0 + e];
    su[e] = v.x;
    su[rows + e] = v.y;
  }
  __syncthreads();
  const int c0 = blockIdx.y * 32 + warp * 4;
  if (c0 > r) return;
  Sum3 sum[4];
  const float* Fc[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) Fc[c] = F + (size_t)min(c0 + c, r > 0 ? r - 1 : 0) * ldf + i0;
  const float4 one = make_float4(1.f, 1.f, 1.f, 1.f), zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
  for (int k = lane * 4; k < cnt; k += 128) {
    float4 f[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      f[c] = c0 + c < r ? __ldg(reinterpret_cast<const float4*>(Fc[c] + k)) : (c0 + c == r ? one : zero);
    const float4 uh = *reinterpret_cast<const float4*>(su + k);
    const float4 ul = *reinterpret_cast<const float4*>(su + rows + k);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      sum[c].mac(f[c].x, uh.x, ul.x);
      sum[c].mac(f[c].y, uh.y, ul.y);
      sum[c].mac(f[c].z, uh.z, ul.z);
      sum[c].mac(f[c].w, uh.w, ul.w);
    }
  }
  // reduce-scatter: lane bits 4 and 3 select the column, then the lanes of a column are added
  const bool u4 = (lane & 16) != 0, u3 = (lane & 8) != 0;
  auto exchange = [](Sum3& keep, const Sum3& other, bool up, int o) {   // up lanes keep `other`, the rest `keep`
    const Sum3 send = up ? keep : other;
    if (up) keep = other;
    keep.add(__shfl_xor_sync(0xffffffffu, send.h, o), __shfl_xor_sync(0xffffffffu, send.l, o),
             __shfl_xor_sync(0xffffffffu, send.ll, o));
  };
  exchange(sum[0], sum[2], u4, 16);
  exchange(sum[1], sum[3], u4, 16);
  exchange(sum[0], sum[1], u3, 8);
#pragma unroll
  for (int o = 4; o >= 1; o >>= 1) sum[0].add_lane(o);
  const int col = c0 + (u4 ? 2 : 0) + (u3 ? 1 : 0);
  if ((lane & 7) == 0 && col <= r) {
    const int ew = max_exponent(*reinterpret_cast<const unsigned long long*>(scal + S_WMAX));
    atomicAdd(&t[col], (sum[0].value() * pow2((int)scal[S_WEXP])) * pow2(ew));
  }
}

// t2s = Ginv t (N x N times N) scaled by the exponent of r, as hi + lo; one block per output row.
__global__ void gemv_core_kernel(const double* __restrict__ Ginv, const double* __restrict__ t, int N,
                                 const double* __restrict__ scal, float2* __restrict__ t2s) {
  const int a = blockIdx.x;
  double s = 0.0;
  for (int b = threadIdx.x; b < N; b += blockDim.x) s += Ginv[(size_t)a * N + b] * t[b];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double ws[8];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += ws[w];
    float2 q;
    df_split(v * pow2(-(int)scal[S_WEXP]), q.x, q.y);
    t2s[a] = q;
  }
}

// out_i = Linv_i (r_i - (F t2_F)_i - t2_r); rz = r . out (the last block to finish adds the blocks'
// sums).  A CTA takes 32 rows at a time (lane = row), its eight warps an eighth of the columns each.
constexpr int kOutMaxBlocks = 1216;
__global__ void __launch_bounds__(256) woodbury_out_kernel(const float* __restrict__ F, int64_t ldf, int r, int64_t n,
                                                           const double* __restrict__ Linv,
                                                           const double* __restrict__ rv,
                                                           const float2* __restrict__ t2s,
                                                           const double* __restrict__ scal, double* __restrict__ out,
                                                           double* __restrict__ part,
                                                           unsigned int* __restrict__ counter,
                                                           double* __restrict__ rz) {
  extern __shared__ float2 ts[];   // r + 1
  __shared__ float red[2][8][3][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = threadIdx.x; c <= r; c += 256) ts[c] = t2s[c];
  __syncthreads();
  const int per = (r + 7) / 8;
  const int c0 = min(r, warp * per), c1 = min(r, c0 + per);
  const double unscale = pow2((int)scal[S_WEXP]);
  double dot = 0.0;
  int buf = 0;
  for (int64_t base = (int64_t)blockIdx.x * 32; base < n; base += (int64_t)gridDim.x * 32, buf ^= 1) {
    const int64_t i = base + lane;   // < ldf
    const float* Fi = F + i;
    double li = 0.0, ri = 0.0;
    if (warp == 0 && i < n) {
      li = Linv[i];
      ri = rv[i];
    }
    Sum3 sum;
    int c = c0;
    for (; c + 16 <= c1; c += 16) {
      float f[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) f[u] = __ldg(Fi + (size_t)(c + u) * ldf);
#pragma unroll
      for (int u = 0; u < 16; ++u) sum.mac(f[u], ts[c + u].x, ts[c + u].y);
    }
#pragma unroll 4
    for (; c < c1; ++c) sum.mac(__ldg(Fi + (size_t)c * ldf), ts[c].x, ts[c].y);
    red[buf][warp][0][lane] = sum.h;
    red[buf][warp][1][lane] = sum.l;
    red[buf][warp][2][lane] = sum.ll;
    __syncthreads();
    if (warp == 0) {
      sum.h = ts[r].x;
      sum.l = ts[r].y;
      sum.ll = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) sum.add(red[buf][w][0][lane], red[buf][w][1][lane], red[buf][w][2][lane]);
      if (i < n) {
        const double o = li * (ri - sum.value() * unscale);
        out[i] = o;
        dot = fma(ri, o, dot);
      }
    }
  }
  if (!rz) return;
  double dots[1] = {dot}, tot;
  if (grid_sums(dots, part, counter, &tot) && threadIdx.x == 0) *rz = tot;
}

__global__ void __launch_bounds__(256) ident_dot_kernel(const double* __restrict__ rv, double* __restrict__ out,
                                                        int64_t n, double* __restrict__ part,
                                                        unsigned int* __restrict__ counter, double* __restrict__ rz) {
  double dot = 0.0;
  GRID_LOOP(i, n) {
    out[i] = rv[i];
    dot += rv[i] * rv[i];
  }
  if (!rz) return;
  double dots[1] = {dot}, tot;
  if (grid_sums(dots, part, counter, &tot) && threadIdx.x == 0) *rz = tot;
}

// max_i |Lpre_i Linv_i - 1| (relative change of the diagonal since the last build)
__global__ void rel_change_kernel(const double* __restrict__ Lpre, const double* __restrict__ Linv, int64_t n,
                                  unsigned long long* __restrict__ out) {
  double m = 0.0;
  GRID_LOOP(i, n) m = fmax(m, fabs(Lpre[i] * Linv[i] - 1.0));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));  // m >= 0: bit order = value order
}

kqr_status precond_update(Handle* h, const double* Lpre, double gam, double rtol, cudaStream_t st) {
  if (h->core_valid && h->core_gam == gam && h->core_kind == h->opt.precond && h->opt.precond != KQR_PRECOND_NONE) {
    unsigned long long* slot = reinterpret_cast<unsigned long long*>(h->scal + S_COUNT - 2);
    cudaError_t e = cudaMemsetAsync(slot, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return cuda_fail(h, e, "core reuse check");
    rel_change_kernel<<<grid_for(h->n), 256, 0, st>>>(Lpre, h->Linv, h->n, slot);
    h->launches++;
    unsigned long long bits = 0;
    if ((e = cudaMemcpyAsync(&bits, slot, sizeof(bits), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
      return cuda_fail(h, e, "core reuse check");
    double change;
    std::memcpy(&change, &bits, sizeof(change));
    if (change <= rtol) {
      h->core_reuses++;
      return KQR_OK;
    }
  }
  return precond_build(h, Lpre, gam, st);
}

kqr_status precond_build(Handle* h, const double* Lpre, double gam, cudaStream_t st) {
  h->core_valid = false;
  h->core_gam = gam;
  h->core_kind = h->opt.precond;
  h->core_builds++;
  if (h->opt.precond == KQR_PRECOND_NONE) {
    h->core_valid = true;
    return KQR_OK;
  }
  const int N = h->r + 1;
  double* G = h->core;                       // N x N, factor / scratch
  double* W = h->core + (size_t)N * N;       // N x N, L^{-1}
  double* Ginv = W + (size_t)N * N;          // N x N
  cudaError_t e;
  unsigned long long* wmax = reinterpret_cast<unsigned long long*>(h->scal + S_WMAX);
  if ((e = cudaMemsetAsync(wmax, 0, sizeof(*wmax), st)) != cudaSuccess) return cuda_fail(h, e, "core");
  recip_kernel<<<grid_for(h->n), 256, 0, st>>>(h->Linv, Lpre, h->n, wmax);
  h->launches++;
  if ((e = core_gram<float>(h, h->F32, h->ldn, h->r, true, h->Linv, wmax, G, st)) != cudaSuccess) return cuda_fail(h, e, "core");
  add_diag_kernel<<<grid_for(N), 256, 0, st>>>(G, N, 1.0, 1.0 / gam);
  h->launches++;
  int* info = reinterpret_cast<int*>(h->scal + S_COUNT - 1);
  if ((e = spd_inverse(h, G, W, Ginv, N, info, st)) != cudaSuccess) return cuda_fail(h, e, "core inverse");
  int hinfo = 0;
  if ((e = cudaMemcpyAsync(&hinfo, info, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(st)) != cudaSuccess)
    return cuda_fail(h, e, "core inverse info");
  if (hinfo != 0) return fail(h, KQR_BREAKDOWN, "Woodbury core not positive definite at pivot " + std::to_string(hinfo - 1));
  h->core_valid = true;
  return KQR_OK;
}

// out = P^{-1} r with the core built by precond_build for the same Lpre; rz_out (device,
// nullable) receives r^T out.  rr (device, nullable): ||r||^2, for the scaling of the double-float
// parts; without it max |r| is computed here.  split: usplit, t and S_WEXP are there already (the CG
// step kernel left them).
cudaError_t precond_apply(Handle* h, const double* Lpre, const double* rv, double* out, double* rz_out,
                          cudaStream_t st, const double* rr, bool split) {
  (void)Lpre;
  cudaError_t e;
  if (h->opt.precond == KQR_PRECOND_NONE) {
    ident_dot_kernel<<<grid_for(h->n), 256, 0, st>>>(rv, out, h->n, h->red_part, h->red_counter, rz_out);
    h->launches++;
    return cudaGetLastError();
  }
  const int N = h->r + 1;
  const double* Ginv = h->core + 2 * (size_t)N * N;
  double* t = h->tvec;
  float2* t2s = reinterpret_cast<float2*>(h->tvec + N);
  if (!split) {
    const int is_max = rr ? 0 : 1;
    if (!rr) {
      double* slot = h->scal + S_WMAXR;
      if ((e = cudaMemsetAsync(slot, 0, sizeof(double), st)) != cudaSuccess) return e;
      absmax_kernel<<<grid_for(h->n), 256, 0, st>>>(rv, h->n, reinterpret_cast<unsigned long long*>(slot));
      h->launches++;
      rr = slot;
    }
    wb_split_kernel<<<grid_for(h->ldn), 256, 0, st>>>(h->Linv, rv, h->n, h->ldn, rr, is_max, h->scal, h->usplit, t, N);
    h->launches++;
  }
  // rows per CTA of the first pass: about four CTAs per SM, 128 .. 1024 rows
  const int groups = (N + 31) / 32;
  const int64_t want = std::max<int64_t>(1, (int64_t)4 * h->num_sms / groups);
  int64_t rows = (h->ldn / 128 + want - 1) / want * 128;
  rows = std::min<int64_t>(std::max<int64_t>(rows, 128), 1024);
  ut_kernel<<<dim3((unsigned)((h->ldn + rows - 1) / rows), groups), 256, (size_t)rows * 2 * sizeof(float), st>>>(
      h->F32, h->ldn, h->r, h->usplit, h->scal, t, (int)rows);
  gemv_core_kernel<<<N, 256, 0, st>>>(Ginv, t, N, h->scal, t2s);
  const int blocks = (int)std::min<int64_t>((h->n + 31) / 32, kOutMaxBlocks);
  woodbury_out_kernel<<<blocks, 256, (size_t)N * sizeof(float2), st>>>(h->F32, h->ldn, h->r, h->n, h->Linv, rv, t2s,
                                                                       h->scal, out, h->red_part, h->red_counter,
                                                                       rz_out);
  h->launches += 3;
  return cudaGetLastError();
}

WbSplit precond_split(Handle* h) {
  WbSplit w;
  if (h->opt.precond == KQR_PRECOND_NONE) return w;
  w.Linv = h->Linv;
  w.us = h->usplit;
  w.t = h->tvec;
  w.N = h->r + 1;
  return w;
}

// ---- RPCholesky set-up --------------------------------------------------------------
constexpr int kPivChunks = 256;

__global__ void chunk_sum_kernel(const double* __restrict__ d, int64_t n, int64_t chunk, double* __restrict__ out) {
  const int64_t i0 = (int64_t)blockIdx.x * chunk;
  const int64_t i1 = min(n, i0 + chunk);
  double s = 0.0;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) s += d[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double ws[8];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += ws[w];
    out[blockIdx.x] = v;
  }
}

// ---- fused RPCholesky steps ---------------------------------------------------------
// One launch per pivot.  CTA b owns R = blockDim.x rows, one per thread; step t forms column t
// of F for the pivot s = piv[t] chosen by the previous launch, updates the residual diagonal
// and writes its chunk's sum of the new diagonal; the last CTA to finish (a ticket counter, no
// waiting) draws the next pivot from the chunk sums.  state[0] is the stop flag, state[1] the
// number of columns produced, state[2] the ticket counter.
//
// What bounds a step: at large n the FP64 pipe (t + 2 p FMAs per row at 2 per clock and SM;
// the 8 t n bytes of F take two thirds of that), at small n the latency chain of one row and
// of the draw.  So rows are spread one per thread over R = 64 rows per CTA while that fills at
// most one wave (128 beyond), the pivot's residual is d[s] itself (the running diagonal is
// updated by the very operations that would recompute it), and the draw is a scan by all
// threads of the last CTA.  n = 10000, p = 50, t < 100: 141 us a step before (512 rows per
// CTA, one thread scanning them from global memory).
constexpr int kRpcMaxThreads = 128;

static int rpc_rows(const Handle* h) { return h->n <= (int64_t)64 * h->num_sms ? 64 : kRpcMaxThreads; }

// Residual column entry g_i = k(x_i, x_s) - sum_{c<t} F[c][i] F[c][s].
__device__ __forceinline__ double rpc_entry(const double* __restrict__ xc, int64_t ldn, int p, double gamma, int lap,
                                            const double* __restrict__ F, int64_t n, int t, int64_t i,
                                            const double* xs, const double* fs) {
  double dist = 0.0;
#pragma unroll 8
  for (int k = 0; k < p; ++k) {
    const double v = xc[(size_t)k * ldn + i] - xs[k];
    dist = lap ? dist + fabs(v) : fma(v, v, dist);
  }
  double acc = exp(-gamma * dist);
#pragma unroll 16
  for (int c = 0; c < t; ++c) acc -= F[(size_t)c * n + i] * fs[c];
  return acc;
}

// Inclusive sum over the CTA's threads (blockDim.x a multiple of 32, at most kRpcMaxThreads);
// *total receives the sum over all of them.  Contains barriers.
__device__ __forceinline__ double rpc_scan(double v, double* ws, double* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  __syncthreads();
  if (lane == 31) ws[warp] = v;
  __syncthreads();
  double base = 0.0, all = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    if (w < warp) base += ws[w];
    all += ws[w];
  }
  *total = all;
  return base + v;
}

// Pivot draw by the last CTA: the smallest s with running sum of d > u * sum(d), among the
// rows with d > 0 (the scan's rounding must not select an exhausted row).  Chunk sums first
// (threads take contiguous runs of them), then the rows of the chosen chunk.
__device__ void rpc_pick(const double* d, const double* csum, int64_t n, int nchunks, double u, long long* piv_out,
                         double* val_out, int* state) {
  __shared__ double ws[kRpcMaxThreads / 32];
  __shared__ int first;
  __shared__ int chunk_sh;
  __shared__ double run_sh;
  const int T = blockDim.x, tid = threadIdx.x;
  const int per = (nchunks + T - 1) / T;
  const int c0 = min(nchunks, tid * per), c1 = min(nchunks, c0 + per);
  double mine = 0.0;
#pragma unroll 4
  for (int c = c0; c < c1; ++c) mine += __ldcg(csum + c);
  double total;
  const double incl = rpc_scan(mine, ws, &total);
  if (!(total > 0.0)) {
    if (tid == 0) {
      *piv_out = -1;
      state[0] = 1;
    }
    return;
  }
  const double target = u * total;
  if (tid == 0) {
    first = T;
    chunk_sh = nchunks - 1;
    run_sh = -INFINITY;   // stays if rounding left the target past the last chunk: no row qualifies
  }
  __syncthreads();
  if (c1 > c0 && incl > target) atomicMin(&first, tid);
  __syncthreads();
  if (tid == first) {
    double run = incl - mine;
    int c = c0;
    for (; c < c1 - 1; ++c) {
      const double cs = __ldcg(csum + c);
      if (run + cs > target) break;
      run += cs;
    }
    chunk_sh = c;
    run_sh = run;
  }
  __syncthreads();
  const int64_t row = (int64_t)chunk_sh * T + tid;
  const double dv = row < n ? __ldcg(d + row) : 0.0;
  double dummy;
  const double at = run_sh + rpc_scan(dv, ws, &dummy);
  if (tid == 0) first = T;
  __syncthreads();
  if (dv > 0.0 && at > target) atomicMin(&first, tid);
  __syncthreads();
  if (first < T) {
    if (tid == first) {
      *piv_out = row;
      *val_out = dv;
    }
  } else if (tid == 0) {   // rounding left the target past the last positive entry: take the last positive one
    int64_t q = n - 1;
    while (q > 0 && !(__ldcg(d + q) > 0.0)) --q;
    *piv_out = q;
    *val_out = __ldcg(d + q);
  }
}

__device__ __forceinline__ void rpc_chunk_sum_and_ticket(double local, double* csum, const double* d, int64_t n,
                                                         int nchunks, const double* u, int t, int r0,
                                                         long long* piv, double* pval, int* state) {
  __shared__ double cs_ws[kRpcMaxThreads / 32];
  __shared__ int last;
  for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
  if ((threadIdx.x & 31) == 0) cs_ws[threadIdx.x >> 5] = local;
  __threadfence();   // this thread's d and F entry before the ticket
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += cs_ws[w];
    csum[blockIdx.x] = v;
    __threadfence();
    last = atomicAdd(state + 2, 1) == nchunks - 1;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    if (threadIdx.x == 0) {
      state[2] = 0;
      state[1] = t + 1;
    }
    if (t + 1 < r0) rpc_pick(d, csum, n, nchunks, u[t + 1], piv + t + 1, pval + t + 1, state);
  }
}

// d = diag(K) = 1 and the draw of the first pivot.
__global__ void __launch_bounds__(kRpcMaxThreads) rpc_init_kernel(double* __restrict__ d, int64_t n, int nchunks,
                                                                 double* __restrict__ csum,
                                                                 const double* __restrict__ u, int r0,
                                                                 long long* __restrict__ piv,
                                                                 double* __restrict__ pval, int* __restrict__ state) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double local = 0.0;
  if (i < n) {
    d[i] = 1.0;   // k(x, x) = 1 for the RBF and Laplacian kernels
    local = 1.0;
  }
  rpc_chunk_sum_and_ticket(local, csum, d, n, nchunks, u, -1, r0, piv, pval, state);
}

__global__ void __launch_bounds__(kRpcMaxThreads) rpc_step_kernel(const double* __restrict__ xc, int64_t ldn, int p,
                                                              double gamma, int lap, double* F,
                                                              double* __restrict__ d, int64_t n, int t, int r0,
                                                              int nchunks, double* __restrict__ csum,
                                                              const double* __restrict__ u,
                                                              long long* __restrict__ piv,
                                                              double* __restrict__ pval, int* __restrict__ state) {
  if (*(volatile int*)state) return;   // an earlier step stopped the factorization
  const long long s = piv[t];
  const double gs = pval[t];   // residual at the pivot
  if (!(gs > 0.0)) {           // it vanished: stop with t columns
    if (blockIdx.x == 0 && threadIdx.x == 0) state[0] = 1;
    return;
  }
  extern __shared__ double sm[];
  double* fs = sm;            // F[c][s], c < t
  double* xs = sm + t;        // x_s
  for (int c = threadIdx.x; c < t; c += blockDim.x) fs[c] = F[(size_t)c * n + s];
  for (int k = threadIdx.x; k < p; k += blockDim.x) xs[k] = xc[(size_t)k * ldn + s];
  __syncthreads();
  const double inv = 1.0 / sqrt(gs);
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double local = 0.0;
  if (i < n) {
    const double f = rpc_entry(xc, ldn, p, gamma, lap, F, n, t, i, xs, fs) * inv;
    F[(size_t)t * n + i] = f;
    const double di = fmax(d[i] - f * f, 0.0);
    d[i] = di;
    local = di;
  }
  rpc_chunk_sum_and_ticket(local, csum, d, n, nchunks, u, t, r0, piv, pval, state);
}

// FP64 factor [r][n] -> FP32 factor [r][ldn], zero in the padding rows.
__global__ void to_float_kernel(const double* __restrict__ src, float* __restrict__ dst, int64_t n, int64_t ldn,
                                int r) {
  GRID_LOOP(e, (int64_t)r * ldn) {
    const int64_t c = e / ldn, i = e % ldn;
    dst[e] = i < n ? (float)src[c * n + i] : 0.f;
  }
}

__global__ void dres_kernel(const float* __restrict__ F, int64_t ldf, int r, int64_t n, double* __restrict__ dres) {
  GRID_LOOP(i, n) {
    double s = 0.0;
    for (int c = 0; c < r; ++c) {
      const double f = (double)F[(size_t)c * ldf + i];
      s += f * f;
    }
    dres[i] = fmax(1.0 - s, 0.0);   // k(x, x) = 1 for the RBF and Laplacian kernels
  }
}

__global__ void floor_kernel(double* __restrict__ d, int64_t n, double nu) { GRID_LOOP(i, n) d[i] = fmax(d[i], nu); }

// lambda_1 of the SPD matrix A (N x N) by power iteration (single CTA).
__global__ void __launch_bounds__(512) power_iter_kernel(const double* __restrict__ A, int N, double* __restrict__ x,
                                                         double* __restrict__ y, int iters, double* __restrict__ lam) {
  __shared__ double red[16];
  __shared__ double cur;
  for (int i = threadIdx.x; i < N; i += blockDim.x) x[i] = 1.0 / sqrt((double)N) * (1.0 + 1e-3 * (i % 7));
  __syncthreads();
  double prev = 0.0;
  for (int it = 0; it < iters; ++it) {
    double loc = 0.0;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      double s = 0.0;
      for (int k = 0; k < N; ++k) s += A[(size_t)i * N + k] * x[k];
      y[i] = s;
      loc += s * s;
    }
    for (int o = 16; o > 0; o >>= 1) loc += __shfl_xor_sync(0xffffffffu, loc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = loc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double v = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w];
      cur = sqrt(v);
    }
    __syncthreads();
    const double nv = cur;
    for (int i = threadIdx.x; i < N; i += blockDim.x) x[i] = y[i] / nv;
    __syncthreads();
    if (fabs(nv - prev) <= 1e-15 * nv) break;
    prev = nv;
  }
  if (threadIdx.x == 0) *lam = cur;
}

// Number of negative pivots of the LDL^T factorisation (no pivoting) of A - c I,
// i.e. the number of eigenvalues of A below c (single CTA, A overwritten).
__global__ void __launch_bounds__(1024) inertia_kernel(double* A, int N, double c, int* neg) {
  __shared__ double dj;
  __shared__ int cnt;
  if (threadIdx.x == 0) cnt = 0;
  for (int i = threadIdx.x; i < N; i += blockDim.x) A[(size_t)i * N + i] -= c;
  __syncthreads();
  for (int j = 0; j < N; ++j) {
    if (threadIdx.x == 0) {
      double d = A[(size_t)j * N + j];
      if (d == 0.0) d = 1e-300;
      if (d < 0.0) ++cnt;
      dj = d;
    }
    __syncthreads();
    const double invd = 1.0 / dj;
    // trailing update A_ik -= A_ij A_kj / d_j for j < k <= i (lower), one warp per row
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = j + 1 + (int)(threadIdx.x >> 5); i < N; i += nw) {
      const double aij = A[(size_t)i * N + j] * invd;
      for (int k = j + 1 + lane; k <= i; k += 32) A[(size_t)i * N + k] -= aij * A[(size_t)k * N + j];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *neg = cnt;
}

kqr_status rpcholesky_setup(Handle* h, const double* uniforms) {
  const int64_t n = h->n;
  int r0 = h->opt.rank0 > 0 ? h->opt.rank0 : (int)std::ceil(std::sqrt((double)n));
  if (r0 > n) r0 = (int)n;
  if (r0 > 1024) r0 = 1024;
  h->r0 = r0;
  cudaStream_t st = h->stream;
  cudaError_t e;
  const size_t fbytes = sizeof(double) * (size_t)r0 * n;
  double* F64 = (double*)dev_alloc(h, fbytes);
  double* d = (double*)dev_alloc(h, sizeof(double) * n);
  double* csum = (double*)dev_alloc(h, sizeof(double) * (kPivChunks + 8));
  int* bad = (int*)dev_alloc(h, sizeof(int) * 2);
  auto cleanup = [&]() {
    dev_free(h, F64); dev_free(h, d); dev_free(h, csum); dev_free(h, bad);
  };
  if (!F64 || !d || !csum || !bad) {
    cleanup();
    return fail(h, KQR_OOM, "RPCholesky workspace");
  }
  // Pivot uniforms: given, or a splitmix64 stream from the seed.
  std::vector<double> u(r0);
  if (uniforms) {
    for (int t = 0; t < r0; ++t) u[t] = uniforms[t];
  } else {
    uint64_t x = h->opt.seed;
    for (int t = 0; t < r0; ++t) {
      x += 0x9E3779B97F4A7C15ull;
      uint64_t z = x;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z ^= z >> 31;
      u[t] = (double)(z >> 11) * (1.0 / 9007199254740992.0);
    }
  }
  const int64_t chunk = (n + kPivChunks - 1) / kPivChunks;
  const int nchunks = (int)((n + chunk - 1) / chunk);
  const int rrows = rpc_rows(h);
  const int rchunks = (int)((n + rrows - 1) / rrows);
  double* u_dev = (double*)dev_alloc(h, sizeof(double) * (r0 + 1));
  double* rsum = (double*)dev_alloc(h, sizeof(double) * (rchunks + 1));
  double* piv_val = (double*)dev_alloc(h, sizeof(double) * (r0 + 1));
  long long* piv_all = (long long*)dev_alloc(h, sizeof(long long) * (r0 + 1));
  int* state = (int*)dev_alloc(h, sizeof(int) * 4);
  auto cleanup2 = [&]() { dev_free(h, u_dev); dev_free(h, rsum); dev_free(h, piv_val); dev_free(h, piv_all); dev_free(h, state); };
  if (!u_dev || !rsum || !piv_val || !piv_all || !state) {
    cleanup2();
    cleanup();
    return fail(h, KQR_OOM, "RPCholesky workspace");
  }
  const size_t smem = sizeof(double) * ((size_t)r0 + h->p);
  if (smem > 48 * 1024 &&
      (e = cudaFuncSetAttribute(rpc_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) {
    cleanup2();
    cleanup();
    return cuda_fail(h, e, "RPCholesky shared memory (p too large)");
  }
  // All r0 steps are queued back to back; the device decides the pivots and when to stop.
  if ((e = cudaMemcpyAsync(u_dev, u.data(), sizeof(double) * r0, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
      (e = cudaMemsetAsync(state, 0, sizeof(int) * 4, st)) != cudaSuccess ||
      (e = cudaMemsetAsync(piv_all, 0xff, sizeof(long long) * (r0 + 1), st)) != cudaSuccess) {
    cleanup2();
    cleanup();
    return cuda_fail(h, e, "RPCholesky start");
  }
  rpc_init_kernel<<<rchunks, rrows, 0, st>>>(d, n, rchunks, rsum, u_dev, r0, piv_all, piv_val, state);
  h->launches++;
  for (int t = 0; t < r0; ++t) {
    rpc_step_kernel<<<rchunks, rrows, smem, st>>>(h->xc64, h->ldn, (int)h->p, h->gamma, h->kind == KQR_LAPLACIAN,
                                                  F64, d, n, t, r0, rchunks, rsum, u_dev, piv_all, piv_val, state);
    h->launches++;
  }
  int hstate[4] = {0, 0, 0, 0};
  std::vector<long long> hpiv(r0 + 1);
  if ((e = cudaGetLastError()) != cudaSuccess ||
      (e = cudaMemcpyAsync(hstate, state, sizeof(int) * 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(hpiv.data(), piv_all, sizeof(long long) * (r0 + 1), cudaMemcpyDeviceToHost, st)) !=
          cudaSuccess ||
      (e = cudaStreamSynchronize(st)) != cudaSuccess) {
    cleanup2();
    cleanup();
    return cuda_fail(h, e, "RPCholesky steps");
  }
  cleanup2();
  h->pivots.clear();
  const int t = hstate[1];
  for (int q = 0; q < t; ++q) h->pivots.push_back(hpiv[q]);
  const int rr0 = t;  // columns actually produced
  h->r0 = rr0;
  int r = rr0;
  if (h->opt.adaptive_rank && rr0 > 1) {
    // Rank heuristic on F0^T F0 (rr0 x rr0).
    double* A = (double*)dev_alloc(h, sizeof(double) * (size_t)rr0 * rr0 + sizeof(double) * (2 * rr0 + 4));
    if (!A) {
      cleanup();
      return fail(h, KQR_OOM, "rank heuristic workspace");
    }
    double* xw = A + (size_t)rr0 * rr0;
    double* yw = xw + rr0;
    double* lam1 = yw + rr0;
    core_gram<double>(h, F64, n, rr0, false, nullptr, nullptr, A, st);
    power_iter_kernel<<<1, 512, 0, st>>>(A, rr0, xw, yw, 2000, lam1);
    h->launches++;
    double hl1 = 0.0;
    if ((e = cudaMemcpyAsync(&hl1, lam1, sizeof(double), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess) {
      dev_free(h, A);
      cleanup();
      return cuda_fail(h, e, "power iteration");
    }
    inertia_kernel<<<1, 1024, 0, st>>>(A, rr0, h->opt.xi * hl1, bad + 1);
    h->launches++;
    int neg = 0;
    if ((e = cudaMemcpyAsync(&neg, bad + 1, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess) {
      dev_free(h, A);
      cleanup();
      return cuda_fail(h, e, "inertia");
    }
    dev_free(h, A);
    const int above = rr0 - neg;           // eigenvalues > xi lambda_1
    r = above + 1 <= rr0 ? above + 1 : rr0;
  }
  h->r = r;
  dev_free(h, h->F32); dev_free(h, h->dres); dev_free(h, h->core); dev_free(h, h->tvec); dev_free(h, h->Linv);
  dev_free(h, h->usplit);
  h->core_valid = false;
  h->F32 = (float*)dev_alloc(h, sizeof(float) * ((size_t)r * h->ldn + 1));
  h->dres = (double*)dev_alloc(h, sizeof(double) * n);
  const int N = r + 1;
  h->core = (double*)dev_alloc(h, sizeof(double) * 3 * (size_t)N * N);
  h->tvec = (double*)dev_alloc(h, sizeof(double) * 2 * N);
  h->Linv = (double*)dev_alloc(h, sizeof(double) * n);
  h->usplit = (float2*)dev_alloc(h, sizeof(float2) * h->ldn);
  if (!h->F32 || !h->dres || !h->core || !h->tvec || !h->Linv || !h->usplit) {
    cleanup();
    return fail(h, KQR_OOM, "preconditioner buffers");
  }
  if (r > 0) {
    to_float_kernel<<<grid_for((int64_t)r * h->ldn), 256, 0, st>>>(F64, h->F32, n, h->ldn, r);
    h->launches++;
  }
  dres_kernel<<<grid_for(n), 256, 0, st>>>(h->F32, h->ldn, r, n, h->dres);
  h->launches++;
  // Floor the residual diagonal at 0.1 of its mean: it is 0 at the pivots, and
  // L + dres must stay away from 0 for a well-conditioned Woodbury core.
  chunk_sum_kernel<<<nchunks, 256, 0, st>>>(h->dres, n, chunk, csum);
  h->launches++;
  std::vector<double> hsum(nchunks);
  if ((e = cudaMemcpyAsync(hsum.data(), csum, sizeof(double) * nchunks, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(st)) != cudaSuccess) {
    cleanup();
    return cuda_fail(h, e, "residual diagonal");
  }
  double tot = 0.0;
  for (double v : hsum) tot += v;
  h->dres_mean = tot / (double)n;
  floor_kernel<<<grid_for(n), 256, 0, st>>>(h->dres, n, 0.1 * tot / (double)n);
  h->launches++;
  e = cudaStreamSynchronize(st);
  cleanup();
  if (e != cudaSuccess) return cuda_fail(h, e, "RPCholesky finish");
  return KQR_OK;
}

}  // namespace kqr
