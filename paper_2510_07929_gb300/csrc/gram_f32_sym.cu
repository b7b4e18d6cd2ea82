// Symmetric FP32 Gram product u = K v (one right-hand side).
//
// K is symmetric, so each off-diagonal 128 x 128 tile K_IJ (J > I) is formed
// once and used twice: u_I += K_IJ v_J (row sums) and u_J += K_IJ^T v_I
// (column sums).  Diagonal tiles give row sums only.  This halves the kernel
// entries formed per product (n^2/2 + O(n) instead of n^2).
//
// Work units are (row tile I, column tiles [J0, J1)) with J0 >= I, about 64
// per resident CTA, listed in a table built once per problem; a CTA TMA-loads
// its row tile once and double-buffers the column tiles as in the plain
// kernel.  Column sums are reduced across the 16 row groups of the CTA through
// shared memory (double-buffered by tile parity) and added to the output with
// FP32 atomics, as are the unit's row sums at the end; the order of those
// additions is not fixed, so results vary in the last bits between runs.
#include <cmath>
#include <vector>

#include "kqr_internal.h"
#include "ptx.cuh"
#include "reduce.cuh"

namespace kqr {

enum { SYM_RBF = 0, SYM_LAP = 1, SYM_LAP_MIX = 2 };

// ---- Laplacian distances on two pipes (SYM_LAP_MIX) --------------------------------------
// A feature's |x_i - x_j| costs two FP32 operations (a difference and an addition), 128 lanes a clock
// and SM, or one 64-lane integer sum of absolute differences of the fixed-point coordinates hq =
// round(xs 2^G) of the FP64-class layout.  The first p_int features go to the integer pipe, the others
// to the FP32 one (differences as packed f32x2, which halves their issue slots); half of the warps of
// every scheduler take the integer features first and the other half last, so that both pipes work.
// A thread's 64 sums change type between the two: integer sums are below 2^30 (the choice of G), FP32
// sums are rounded to the 2^-G grid.  The integer unit turned out to share much of the FP32 lanes' time
// (busy 53 and 42 % together): n = 200000, p = 50 takes 50.9 ms, 61.5 with all features in FP32.
__device__ __forceinline__ uint64_t lap_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}

__device__ __forceinline__ void lap_int(const int32_t* HI, const int32_t* HJ, int n, int ty, int tx,
                                        unsigned (&A)[8][8]) {
#pragma unroll 2
  for (int k = 0; k < n; ++k) {
    const int4 a0 = *reinterpret_cast<const int4*>(HI + k * kTile + ty * 8);
    const int4 a1 = *reinterpret_cast<const int4*>(HI + k * kTile + ty * 8 + 4);
    const int4 b0 = *reinterpret_cast<const int4*>(HJ + k * kTile + tx * 8);
    const int4 b1 = *reinterpret_cast<const int4*>(HJ + k * kTile + tx * 8 + 4);
    const int ha[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const int hb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) A[a][b] = __sad(ha[a], hb[b], A[a][b]);
  }
}

__device__ __forceinline__ void lap_f32(const float* XI, const float* XJ, int n, int ty, int tx, float (&d)[8][8]) {
  const uint64_t mone = lap_pack(-1.f, -1.f);
#pragma unroll 2
  for (int k = 0; k < n; ++k) {
    const float4 a0 = *reinterpret_cast<const float4*>(XI + k * kTile + ty * 8);
    const float4 a1 = *reinterpret_cast<const float4*>(XI + k * kTile + ty * 8 + 4);
    const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(XJ + k * kTile + tx * 8);
    const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(XJ + k * kTile + tx * 8 + 4);
    const float xa[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const uint64_t xb[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const uint64_t aa = lap_pack(xa[a], xa[a]);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        uint64_t t;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(t) : "l"(xb[b]), "l"(mone), "l"(aa));
        float t0, t1;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(t0), "=f"(t1) : "l"(t));
        d[a][2 * b] += fabsf(t0);
        d[a][2 * b + 1] += fabsf(t1);
      }
    }
  }
}

template <int KIND>
__global__ void __launch_bounds__(kThreads, 2)
    gram_f32_sym_kernel(const __grid_constant__ CUtensorMap tm, const float* __restrict__ nrm,
                        const float* __restrict__ v32, const int4* __restrict__ units, float* __restrict__ acc, int p,
                        const __grid_constant__ CUtensorMap tm_int, int p_int, float grid, float grid_inv,
                        int* __restrict__ err) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* XI = reinterpret_cast<float*>(smem_raw);
  float* XJ0 = XI + p * kTile;
  float* XJ1 = XJ0 + p * kTile;
  float* colred = XJ1 + p * kTile;        // 2 buffers x 4 row-group warps x 128 columns
  float* rowred = colred + 2 * 4 * kTile; // 2 column-group warps x 128 rows
  uint64_t* bars = reinterpret_cast<uint64_t*>(rowred + 2 * kTile);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ty = (warp >> 1) * 4 + (lane >> 3);
  const int tx = (warp & 1) * 8 + (lane & 7);
  const int4 unit = units[blockIdx.x];
  const int row0 = unit.x * kTile;
  const int jt0 = unit.y, jt1 = unit.z;
  const uint32_t bytes = (uint32_t)p * kTile * 4u;

  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    mbar_init(&bars[2], 1);
    fence_mbar_init();
  }
  __syncthreads();
  // one tile: p rows of 128 coordinates; SYM_LAP_MIX: the p_int fixed-point rows, then the FP32 ones
  auto load_tile = [&](float* dst, int c0, uint64_t* bar) {
    mbar_arrive_expect_tx(bar, bytes);
    if (KIND == SYM_LAP_MIX) {
      tma_load_2d(dst, &tm_int, c0, 0, bar);
      tma_load_2d(dst + p_int * kTile, &tm, c0, p_int, bar);
    } else {
      tma_load_2d(dst, &tm, c0, 0, bar);
    }
  };
  if (tid == 0) {
    load_tile(XI, row0, &bars[0]);
    load_tile(XJ0, jt0 * kTile, &bars[1]);
  }
  float va[8], ni[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    va[a] = __ldg(v32 + row0 + ty * 8 + a);
    ni[a] = (KIND == SYM_RBF) ? __ldg(nrm + row0 + ty * 8 + a) : 0.f;
  }
  float racc[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) racc[a] = 0.f;
  if (!mbar_wait_bounded(&bars[0], 0, err)) {
    if (tid == 0) tile_drain(bars, 1, err);
    return;
  }

  for (int t = jt0; t < jt1; ++t) {
    const int q = t - jt0;
    const int s = q & 1;
    float* XJ = s ? XJ1 : XJ0;
    if (tid == 0 && t + 1 < jt1) {
      const int ns = (q + 1) & 1;
      load_tile(ns ? XJ1 : XJ0, (t + 1) * kTile, &bars[1 + ns]);
    }
    const int col0 = t * kTile + tx * 8;
    float vb[8], nj[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      vb[b] = __ldg(v32 + col0 + b);
      nj[b] = (KIND == SYM_RBF) ? __ldg(nrm + col0 + b) : 0.f;
    }
    if (!mbar_wait_bounded(&bars[1 + s], (uint32_t)((q >> 1) & 1), err)) {
      if (tid == 0) tile_drain(bars, min(q + 2, jt1 - jt0), err);
      return;
    }

    float d[8][8];
    if (KIND == SYM_LAP_MIX) {
      const int32_t* HI = reinterpret_cast<const int32_t*>(XI);
      const int32_t* HJ = reinterpret_cast<const int32_t*>(XJ);
      unsigned A[8][8];
      if (warp & 4) {
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) d[a][b] = 0.f;
        lap_f32(XI + p_int * kTile, XJ + p_int * kTile, p - p_int, ty, tx, d);
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) A[a][b] = __float2uint_rn(d[a][b] * grid_inv);
        lap_int(HI, HJ, p_int, ty, tx, A);
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) d[a][b] = __uint2float_rn(A[a][b]) * grid;
      } else {
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) A[a][b] = 0u;
        lap_int(HI, HJ, p_int, ty, tx, A);
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) d[a][b] = __uint2float_rn(A[a][b]) * grid;
        lap_f32(XI + p_int * kTile, XJ + p_int * kTile, p - p_int, ty, tx, d);
      }
    } else {
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) d[a][b] = 0.f;
#pragma unroll 2
      for (int k = 0; k < p; ++k) {
        const float4 a0 = *reinterpret_cast<const float4*>(XI + k * kTile + ty * 8);
        const float4 a1 = *reinterpret_cast<const float4*>(XI + k * kTile + ty * 8 + 4);
        const float4 b0 = *reinterpret_cast<const float4*>(XJ + k * kTile + tx * 8);
        const float4 b1 = *reinterpret_cast<const float4*>(XJ + k * kTile + tx * 8 + 4);
        const float xa[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float xb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) {
            if (KIND == SYM_LAP)
              d[a][b] += fabsf(xa[a] - xb[b]);
            else
              d[a][b] = fmaf(xa[a], xb[b], d[a][b]);
          }
      }
    }
    float cs[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) cs[b] = 0.f;
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const float arg = (KIND != SYM_RBF) ? -d[a][b] : fmaf(2.f, d[a][b], -(ni[a] + nj[b]));
        const float e = ex2_approx(arg);
        racc[a] = fmaf(e, vb[b], racc[a]);
        cs[b] = fmaf(e, va[a], cs[b]);
      }
    const bool offdiag = (t != unit.x);   // uniform over the CTA
    float* cr = colred + s * (4 * kTile);
    if (offdiag) {
      // column sums: reduce over the 4 row groups of the warp, then the 4 row-group warps
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        cs[b] += __shfl_xor_sync(0xffffffffu, cs[b], 8);
        cs[b] += __shfl_xor_sync(0xffffffffu, cs[b], 16);
      }
      if ((lane >> 3) == 0) {
#pragma unroll
        for (int b = 0; b < 8; ++b) cr[(warp >> 1) * kTile + tx * 8 + b] = cs[b];
      }
    }
    __syncthreads();
    if (offdiag && tid < kTile) {
      const float c = cr[tid] + cr[kTile + tid] + cr[2 * kTile + tid] + cr[3 * kTile + tid];
      atomicAdd(acc + t * kTile + tid, c);
    }
  }

  // row sums: reduce over the 8 lanes of a row group, then the 2 column-group warps
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    float v = racc[a];
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    racc[a] = v;
  }
  if ((lane & 7) == 0) {
#pragma unroll
    for (int a = 0; a < 8; ++a) rowred[(warp & 1) * kTile + ty * 8 + a] = racc[a];
  }
  __syncthreads();
  if (tid < kTile) atomicAdd(acc + row0 + tid, rowred[tid] + rowred[kTile + tid]);
}

// v (FP64, n) -> v32 [ldn] zero padded; acc [ldn] zeroed; optional sum of v.
__global__ void __launch_bounds__(256) sym_prep_kernel(const double* __restrict__ V, float* __restrict__ v32,
                                                       double* __restrict__ acc, int64_t n, int64_t ldn,
                                                       double* __restrict__ part, unsigned int* __restrict__ counter,
                                                       double* __restrict__ sum_out) {
  double s[1] = {0.0};
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ldn; i += (int64_t)gridDim.x * blockDim.x) {
    const double x = i < n ? V[i] : 0.0;
    v32[i] = (float)x;
    acc[i] = 0.0;
    s[0] += x;
  }
  if (!sum_out) return;
  double tot;
  if (grid_sums(s, part, counter, &tot) && threadIdx.x == 0) *sum_out = tot;
}

// out = acc (+ gam sum_p + L p), *dot_out = p . out, raw_out = acc.
template <typename T>
__global__ void __launch_bounds__(256) sym_finish_kernel(const T* __restrict__ acc, int64_t n,
                                                         double* __restrict__ out, GramEpilogue ep,
                                                         double* __restrict__ part,
                                                         unsigned int* __restrict__ counter) {
  double dot[1] = {0.0};
  const double add = ep.L ? (ep.gam_dev ? *ep.gam_dev : ep.gam) * (ep.sum_p ? *ep.sum_p : 0.0) : 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double s = (double)acc[i];
    if (ep.raw_out) ep.raw_out[i] = s;
    if (ep.L) s += add + ep.L[i] * ep.pvec[i];
    out[i] = s;
    if (ep.dot_out) dot[0] += ep.pvec[i] * s;
  }
  if (!ep.dot_out) return;
  double tot;
  if (grid_sums(dot, part, counter, &tot) && threadIdx.x == 0) *ep.dot_out = tot;
}

static size_t sym_smem_bytes(int p) {
  return ((size_t)3 * p * kTile + 2 * 4 * kTile + 2 * kTile) * sizeof(float) + 4 * sizeof(uint64_t);
}

// Work-unit table: for each row tile I, column tiles [J0, J1) with I <= J0,
// chunks of C tiles, C chosen for ~64 units per resident CTA.
cudaError_t sym_units_ensure(Handle* h, cudaStream_t st) {
  const int T = (int)(h->ldn / kTile);
  if (h->sym_units && h->sym_T == T) return cudaSuccess;
  const int64_t pairs = (int64_t)T * (T + 1) / 2;
  const int64_t target = (int64_t)64 * 2 * h->num_sms;
  int C = (int)((pairs + target - 1) / target);
  if (C < 1) C = 1;
  std::vector<int4> u;
  for (int I = 0; I < T; ++I)
    for (int J0 = I; J0 < T; J0 += C) u.push_back(make_int4(I, J0, J0 + C < T ? J0 + C : T, 0));
  dev_free(h, h->sym_units);
  h->sym_nunits = (int)u.size();
  h->sym_T = T;
  return dev_upload(h, u.data(), u.size() * sizeof(int4), st, reinterpret_cast<void**>(&h->sym_units));
}

cudaError_t gram_f32_sym(Handle* h, const double* V, double* U, const GramEpilogue* ep, cudaStream_t st) {
  cudaError_t e = sym_units_ensure(h, st);
  if (e != cudaSuccess) return e;
  float* v32;
  double* sums;
  if ((e = sym_buffers(h, &v32, &sums)) != cudaSuccess) return e;
  GramEpilogue none;
  const GramEpilogue& g = ep ? *ep : none;
  if (!g.prepped && (e = sym_prep(h, V, v32, sums, const_cast<double*>(g.sum_p), st)) != cudaSuccess) return e;
  float* acc = reinterpret_cast<float*>(sums);
  const size_t smem = sym_smem_bytes((int)h->p);
  prof_mark(h, 0, true, st);
  const bool mix = h->kind == KQR_LAPLACIAN && h->lap_int > 0;
  auto kern = mix ? gram_f32_sym_kernel<SYM_LAP_MIX>
                  : (h->kind == KQR_LAPLACIAN ? gram_f32_sym_kernel<SYM_LAP> : gram_f32_sym_kernel<SYM_RBF>);
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<h->sym_nunits, kThreads, smem, st>>>(mix ? h->tm_lap_f32 : h->tm_xs32, h->nrm32, v32, h->sym_units, acc,
                                              (int)h->p, h->tm_lap_int, h->lap_int, std::ldexp(1.f, -h->grid_G),
                                              std::ldexp(1.f, h->grid_G), h->err_flag);
  prof_mark(h, 0, false, st);
  h->launches++;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return sym_finish(h, acc, false, U, g, st);
}

}  // namespace kqr

namespace kqr {

cudaError_t sym_buffers(Handle* h, float** v32, double** acc) {
  const size_t need = (size_t)h->ldn * (sizeof(float) + sizeof(double));
  if (h->v32_cap < need) {
    dev_free(h, h->v32);
    h->v32 = (float*)dev_alloc(h, need);
    h->v32_cap = h->v32 ? need : 0;
    if (!h->v32) return cudaErrorMemoryAllocation;
  }
  *v32 = h->v32;
  *acc = reinterpret_cast<double*>(h->v32 + h->ldn);   // ldn is a multiple of 128
  return cudaSuccess;
}

// v -> FP32 copy and zeroed sums (and 1^T v into *sum_out if given), for products that accumulate
// with atomics (symmetric tiles, stored K).
cudaError_t sym_prep(Handle* h, const double* V, float* v32, double* acc, double* sum_out, cudaStream_t st) {
  sym_prep_kernel<<<grid_for(h->ldn), 256, 0, st>>>(V, v32, acc, h->n, h->ldn, h->red_part, h->red_counter, sum_out);
  h->launches++;
  return cudaGetLastError();
}

// out = acc (+ the CG operator's terms of g).
cudaError_t sym_finish(Handle* h, const void* acc, bool f64, double* U, const GramEpilogue& g, cudaStream_t st) {
  if (f64)
    sym_finish_kernel<double><<<grid_for(h->n), 256, 0, st>>>((const double*)acc, h->n, U, g, h->red_part, h->red_counter);
  else
    sym_finish_kernel<float><<<grid_for(h->n), 256, 0, st>>>((const float*)acc, h->n, U, g, h->red_part, h->red_counter);
  h->launches++;
  return cudaGetLastError();
}

}  // namespace kqr
