// Inverse of the symmetric positive definite Woodbury core (N <= 1025, FP64) over all SMs:
// G = L L^T, W = L^{-1}, G^{-1} = W^T W.
//
// What bounds it: this part's FP64 pipe gives 2 FMAs per clock and SM (0.63 T/s over the
// chip) at a latency of 65 cycles, so one CTA can neither fill the chip nor hide the chain
// of pivots.  The work is therefore cut into 32 x 32 blocks, one CTA's registers for the
// serial parts and one CTA per output block for the products:
//   1. per block column k: every CTA of the panel kernel factors the 32 x 32 pivot block
//      again (the CTAs do the same at the same time, which costs nothing and saves a launch)
//      together with its own 32 rows below it; the update kernel subtracts L_ik L_jk^T from
//      the blocks to the right (lower half only);
//   2. the inverses of all diagonal blocks in one launch, then doubling: blocks of s rows are
//      joined pairwise, W_21 = -W_22 (L_21 W_11), s = 32, 64, ... (two launches per doubling,
//      zero blocks skipped);
//   3. W^T W, lower blocks and their mirror images.
// 1.8e8 FMAs per part at N = 1025 are 0.29 ms of the FP64 pipe; the pivot chain of part 1
// (33 panels of 36 us) is the longer one.  Measured at N = 1025, summed launch times: panels
// 1.19, updates 0.71, joins 1.18, W^T W 0.56 ms = 3.7 ms, where one CTA each for the factor
// (62.8 ms) and the inverse (84.7 ms) and an untiled W^T W (1.0 ms) took 148.5 ms before.
#include "kqr_internal.h"

namespace kqr {

namespace {

constexpr int kB = 32;            // block edge
constexpr int kMmThreads = 128;   // a 32 x 32 output block: 4 x 2 entries per thread

// Block (rows r0.., columns c0..) of the row-major N x N matrix A into shared memory, zero
// outside the matrix.
__device__ __forceinline__ void load_block(const double* __restrict__ A, int N, int r0, int c0,
                                           double (*s)[kB + 1]) {
  for (int e = threadIdx.x; e < kB * kB; e += blockDim.x) {
    const int r = e / kB, c = e % kB;
    s[r][c] = (r0 + r < N && c0 + c < N) ? A[(size_t)(r0 + r) * N + c0 + c] : 0.0;
  }
}

// The same in two halves, so that the next block's global loads are in flight while the
// current one is multiplied (kMmThreads threads).
constexpr int kBlockRegs = kB * kB / kMmThreads;
__device__ __forceinline__ void fetch_block(const double* A, int N, int r0, int c0, double (&q)[kBlockRegs]) {
#pragma unroll
  for (int u = 0; u < kBlockRegs; ++u) {
    const int e = threadIdx.x + u * kMmThreads, r = r0 + e / kB, c = c0 + e % kB;
    q[u] = (r < N && c < N) ? A[(size_t)r * N + c] : 0.0;
  }
}
__device__ __forceinline__ void put_block(const double (&q)[kBlockRegs], double (*s)[kB + 1]) {
#pragma unroll
  for (int u = 0; u < kBlockRegs; ++u) {
    const int e = threadIdx.x + u * kMmThreads;
    s[e / kB][e % kB] = q[u];
  }
}

// acc += X Y with X[i][k] = TX ? sx[k][i] : sx[i][k] and Y[k][j] = TY ? sy[j][k] : sy[k][j].
template <bool TX, bool TY>
__device__ __forceinline__ void block_mm(const double (*sx)[kB + 1], const double (*sy)[kB + 1], double (&acc)[4][2]) {
  const int ty = (threadIdx.x >> 4) * 4, tx = (threadIdx.x & 15) * 2;
#pragma unroll 4
  for (int k = 0; k < kB; ++k) {
    double x[4], y[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = TX ? sx[k][ty + i] : sx[ty + i][k];
#pragma unroll
    for (int j = 0; j < 2; ++j) y[j] = TY ? sy[tx + j][k] : sy[k][tx + j];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) acc[i][j] = fma(x[i], y[j], acc[i][j]);
  }
}

// 1 / sqrt(d) from the FP32 estimate (relative error about 2^-22) and one cubic step: a chain of
// four FP64 operations instead of the library's longer one (65 cycles each on this part).
__device__ __forceinline__ double rsqrt_fast(double d) {
  if (!(d > 1e-35 && d < 1e35)) return rsqrt(d);
  const double y = (double)rsqrtf((float)d);
  const double e = fma(-d * y, y, 1.0);
  return fma(fma(0.375, e, 0.5), e * y, y);
}

// Block column k: CTA 0 writes the pivot block's factor to L, CTA b >= 1 the solved block
// L_ik = A_ik L_kk^{-T} of block row k + b.  G holds the updated matrix and is only read
// (a CTA may still be reading the pivot block when another one is done).
//
// Right-looking, lane = row of the pivot block and of the CTA's own block; warp w of the four
// holds their columns w, w + 4, ..., because one warp alone gets a quarter of the SM's FP64
// pipe (an FMA every 64 cycles).  Step j: the warp that owns column j scales it and publishes
// the multipliers; every warp updates its columns right of j, in both blocks.
constexpr int kPanelWarps = 4, kPanelCols = kB / kPanelWarps;
__global__ void __launch_bounds__(kPanelWarps * 32) chol_panel_kernel(const double* __restrict__ G,
                                                                      double* __restrict__ L, int N, int k,
                                                                      int* __restrict__ info) {
  __shared__ double sa[kB][kB + 1], sb[kB][kB + 1];
  __shared__ double mult[2][2][kB];   // [step parity][block][row]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c0 = k * kB;
  const int r0 = (k + blockIdx.x) * kB;
  const bool own = blockIdx.x > 0;
  load_block(G, N, c0, c0, sa);
  if (own) load_block(G, N, r0, c0, sb);
  __syncthreads();
  double a[kPanelCols], b[kPanelCols];
#pragma unroll
  for (int q = 0; q < kPanelCols; ++q) {
    const int j = q * kPanelWarps + w;
    a[q] = c0 + lane < N ? sa[lane][j] : (lane == j ? 1.0 : 0.0);
    b[q] = own ? sb[lane][j] : 0.0;
  }
#pragma unroll
  for (int j = 0; j < kB; ++j) {
    const int qj = j / kPanelWarps, wj = j % kPanelWarps, par = j & 1;
    if (w == wj) {
      double d = __shfl_sync(0xffffffffu, a[qj], j);
      if (!(d > 0.0)) {   // not positive definite: report, go on with 1
        if (!own && lane == 0 && *info == 0) *info = c0 + j + 1;
        d = 1.0;
      }
      const double ri = rsqrt_fast(d);
      a[qj] = lane == j ? d * ri : a[qj] * ri;
      b[qj] *= ri;
      mult[par][0][lane] = a[qj];
      mult[par][1][lane] = b[qj];
    }
    __syncthreads();
    const double la = mult[par][0][lane], lb = mult[par][1][lane];
#pragma unroll
    for (int q = j / kPanelWarps; q < kPanelCols; ++q) {
      const int c = q * kPanelWarps + w;
      if (c > j) {
        const double m = mult[par][0][c];
        a[q] = fma(-la, m, a[q]);
        if (own) b[q] = fma(-lb, m, b[q]);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kPanelCols; ++q) {
    const int j = q * kPanelWarps + w;
    if (own) sb[lane][j] = b[q];
    else sa[lane][j] = j <= lane ? a[q] : 0.0;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kB * kB; e += blockDim.x) {
    const int r = e / kB, c = e % kB;
    if (r0 + r < N && c0 + c < N) L[(size_t)(r0 + r) * N + c0 + c] = own ? sb[r][c] : sa[r][c];
  }
}

// Block pair (i, j), i >= j, number t of the lower triangle in row order.
__device__ __forceinline__ void tri_pair(int t, int* i, int* j) {
  int r = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((r + 1) * (r + 2) / 2 <= t) ++r;
  while (r * (r + 1) / 2 > t) --r;
  *i = r;
  *j = t - r * (r + 1) / 2;
}

// G_ij -= L_ik L_jk^T over the blocks i >= j > k.
__global__ void __launch_bounds__(kMmThreads) chol_update_kernel(double* __restrict__ G, const double* __restrict__ L,
                                                                 int N, int k) {
  __shared__ double sx[kB][kB + 1], sy[kB][kB + 1];
  int i, j;
  tri_pair(blockIdx.x, &i, &j);
  const int r0 = (k + 1 + i) * kB, c0 = (k + 1 + j) * kB;
  load_block(L, N, r0, k * kB, sx);
  load_block(L, N, c0, k * kB, sy);
  __syncthreads();
  double acc[4][2] = {};
  block_mm<false, true>(sx, sy, acc);
  const int ty = (threadIdx.x >> 4) * 4, tx = (threadIdx.x & 15) * 2;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b)
      if (r0 + ty + a < N && c0 + tx + b < N) G[(size_t)(r0 + ty + a) * N + c0 + tx + b] -= acc[a][b];
}

// Inverses of the diagonal blocks of L into W: column `lane` of the inverse in a lane, its rows
// w, w + 4, ... in warp w (four warps for the FP64 pipe, as in the panel), right-looking.
__global__ void __launch_bounds__(kPanelWarps * 32) tri_diag_inverse_kernel(const double* __restrict__ L, int N,
                                                                            double* __restrict__ W) {
  __shared__ double s[kB][kB + 1];
  __shared__ double row[2][kB];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, c0 = blockIdx.x * kB;
  load_block(L, N, c0, c0, s);
  __syncthreads();
  double w[kPanelCols];
#pragma unroll
  for (int q = 0; q < kPanelCols; ++q) w[q] = q * kPanelWarps + wp == lane ? 1.0 : 0.0;
  const double inv = c0 + lane < N ? 1.0 / s[lane][lane] : 1.0;
#pragma unroll
  for (int k = 0; k < kB; ++k) {
    const int qk = k / kPanelWarps;
    if (wp == k % kPanelWarps) {
      w[qk] *= __shfl_sync(0xffffffffu, inv, k);
      row[k & 1][lane] = w[qk];
    }
    __syncthreads();
    const double wk = row[k & 1][lane];
#pragma unroll
    for (int q = k / kPanelWarps; q < kPanelCols; ++q) {
      const int i = q * kPanelWarps + wp;
      if (i > k) w[q] = fma(-s[i][k], wk, w[q]);
    }
  }
  if (c0 + lane < N)
#pragma unroll
    for (int q = 0; q < kPanelCols; ++q) {
      const int i = q * kPanelWarps + wp;
      if (c0 + i < N) W[(size_t)(c0 + i) * N + c0 + lane] = w[q];
    }
}

// One half of a doubling step from blocks of `sb` block rows: output block (i, j) of the
// lower-left square of a pair.  FIRST: T = L_21 W_11 (k from j on); else W_21 = -W_22 T
// (k up to i).
template <bool FIRST>
__global__ void __launch_bounds__(kMmThreads) tri_join_kernel(const double* X, const double* Y, double* out, int N,
                                                              int sb) {
  __shared__ double sx[kB][kB + 1], sy[kB][kB + 1];
  const int base = blockIdx.z * 2 * sb;                 // first block row of the pair
  const int i = base + sb + blockIdx.y, j = base + blockIdx.x;
  if (i * kB >= N) return;
  const int k0 = FIRST ? j : base + sb, k1 = FIRST ? base + sb : i + 1;
  double acc[4][2] = {};
  double qx[kBlockRegs], qy[kBlockRegs];
  fetch_block(X, N, i * kB, k0 * kB, qx);
  fetch_block(Y, N, k0 * kB, j * kB, qy);
  for (int k = k0; k < k1; ++k) {
    __syncthreads();
    put_block(qx, sx);
    put_block(qy, sy);
    __syncthreads();
    if (k + 1 < k1) {
      fetch_block(X, N, i * kB, (k + 1) * kB, qx);
      fetch_block(Y, N, (k + 1) * kB, j * kB, qy);
    }
    block_mm<false, false>(sx, sy, acc);
  }
  const int ty = (threadIdx.x >> 4) * 4, tx = (threadIdx.x & 15) * 2;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int r = i * kB + ty + a, c = j * kB + tx + b;
      if (r < N && c < N) out[(size_t)r * N + c] = FIRST ? acc[a][b] : -acc[a][b];
    }
}

// Ginv = W^T W: lower block (i, j) over the block rows k >= i, and its mirror image.
__global__ void __launch_bounds__(kMmThreads) wtw_kernel(const double* __restrict__ W, int N, int nb,
                                                         double* __restrict__ Ginv) {
  __shared__ double sx[kB][kB + 1], sy[kB][kB + 1];
  int i, j;
  tri_pair(blockIdx.x, &i, &j);
  double acc[4][2] = {};
  double qx[kBlockRegs], qy[kBlockRegs];
  fetch_block(W, N, i * kB, i * kB, qx);
  fetch_block(W, N, i * kB, j * kB, qy);
  for (int k = i; k < nb; ++k) {
    __syncthreads();
    put_block(qx, sx);
    put_block(qy, sy);
    __syncthreads();
    if (k + 1 < nb) {
      fetch_block(W, N, (k + 1) * kB, i * kB, qx);
      fetch_block(W, N, (k + 1) * kB, j * kB, qy);
    }
    block_mm<true, false>(sx, sy, acc);
  }
  const int ty = (threadIdx.x >> 4) * 4, tx = (threadIdx.x & 15) * 2;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int r = i * kB + ty + a, c = j * kB + tx + b;
      if (r < N && c < N) {
        Ginv[(size_t)r * N + c] = acc[a][b];
        Ginv[(size_t)c * N + r] = acc[a][b];
      }
    }
}

}  // namespace

// G (N x N row-major, lower half read; overwritten) -> Ginv = G^{-1} (both halves) and
// W = L^{-1} (lower blocks; above the diagonal blocks W is not written).  *info (device):
// 0, or the first pivot that was not positive, counted from 1.  Enqueues only.
cudaError_t spd_inverse(Handle* h, double* G, double* W, double* Ginv, int N, int* info, cudaStream_t st) {
  const int nb = (N + kB - 1) / kB;
  cudaError_t e = cudaMemsetAsync(info, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  double* L = Ginv;   // the factor lives in Ginv until W^T W overwrites it
  for (int k = 0; k < nb; ++k) {
    const int below = nb - k - 1;
    chol_panel_kernel<<<1 + below, kPanelWarps * 32, 0, st>>>(G, L, N, k, info);
    h->launches++;
    if (below > 0) {
      chol_update_kernel<<<below * (below + 1) / 2, kMmThreads, 0, st>>>(G, L, N, k);
      h->launches++;
    }
  }
  tri_diag_inverse_kernel<<<nb, kPanelWarps * 32, 0, st>>>(L, N, W);
  h->launches++;
  for (int sb = 1; sb < nb; sb *= 2) {
    const dim3 grid(sb, sb, (nb + 2 * sb - 1) / (2 * sb));
    tri_join_kernel<true><<<grid, kMmThreads, 0, st>>>(L, W, G, N, sb);     // T into G, which is free by now
    tri_join_kernel<false><<<grid, kMmThreads, 0, st>>>(W, G, W, N, sb);
    h->launches += 2;
  }
  wtw_kernel<<<nb * (nb + 1) / 2, kMmThreads, 0, st>>>(W, N, nb, Ginv);
  h->launches++;
  return cudaGetLastError();
}

}  // namespace kqr
