// RBF Gram product U = K V with the cross term on the tcgen05 tensor cores.
//
// K_ij = exp2(2 xs_i . xs_j - |xs_i|^2 - |xs_j|^2) (Sec. 1 RBF kernel, with
// xs = sqrt(gamma log2 e)(x - mean)).  The 128 x 128 tile of dot products
// xs_I xs_J^T is a dense contraction over p: it runs as tcgen05.mma kind::tf32
// (M = N = 128, K = 8 per instruction) from shared-memory tiles that TMA loads
// with the 128-byte swizzle, into an FP32 accumulator in tensor memory (two
// 128-column buffers, so the MMAs of tile q overlap the epilogue of tile q-1).
// FP32 accuracy comes from splitting xs = hi + lo into TF32 parts and summing
// hi.hi + hi.lo + lo.hi (the lo.lo term is below FP32 rounding); one term
// (hi.hi) gives the TF32 product.
//
// One CTA = 8 warps = 256 threads; thread t serves TMEM lane t mod 128 (row
// t mod 128 of the tile) over column half t / 128, reads its 64 accumulators
// with tcgen05.ld and accumulates exp2(...) v_j in registers (four independent
// chains per right-hand side, so the FFMAs do not serialise); the two halves
// of a row are added once at the end.  Thread 0 issues the TMA copies and the
// MMAs.  Column tiles are split over
// gridDim.y; per-split row sums are added in FP64 by a second kernel.
// Every mbarrier wait is bounded; on a timeout the CTA records the error,
// stops issuing work, waits (bounded) for its own copies and MMAs and frees
// its tensor memory.
#include <algorithm>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "kqr_internal.h"
#include "ptx.cuh"

namespace kqr {

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] B[smem]^T, tf32 inputs, FP32 accumulate.
__device__ __forceinline__ void umma_tf32(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// D[tmem] (+)= A[smem] B[smem]^T, kind::f16: bf16 or fp16 inputs as the instruction
// descriptor says (A and B of the same type), FP32 accumulate.
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// 32 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// A load of 16 columns, and the wait that makes its registers valid (it waits for all of the thread's loads).
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15])::"memory");
}

// Waits for all tensor-memory loads of this thread; a load of 8 columns without the wait.
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// Untiled bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16).
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Shared-memory matrix descriptor: K-major operand in the canonical 128-byte
// swizzled layout (8-row groups 1024 bytes apart), tcgen05 version bits 0b001.
__device__ __forceinline__ uint64_t umma_desc_sw128(const void* p) {
  const uint32_t a = smem_u32(p);
  uint64_t d = (uint64_t)((a & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;              // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;    // stride byte offset
  d |= (uint64_t)1 << 46;              // fixed 0b001
  d |= (uint64_t)2 << 61;              // 128-byte swizzle
  return d;
}

constexpr uint32_t kAtomBytes = 128 * 128;   // 128 rows x 128 bytes (32 tf32 of K)

template <int M, int NTERMS>
__global__ void __launch_bounds__(256, 1)
    gram_rbf_tc_kernel(const __grid_constant__ CUtensorMap tm_hi, const __grid_constant__ CUtensorMap tm_lo,
                       const float* __restrict__ nrm, const float* __restrict__ v32, float* __restrict__ part,
                       int ksteps, int katoms, int ldn, int tiles_per_split, int col_tiles, int fold_rows,
                       int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~static_cast<uintptr_t>(1023));
  const uint32_t tb = (uint32_t)katoms * kAtomBytes;   // one operand tile
  unsigned char* XIh = base;
  unsigned char* XIl = XIh + tb;
  unsigned char* XJh[2] = {XIl + tb, XIl + 3 * tb};
  unsigned char* XJl[2] = {XIl + 2 * tb, XIl + 4 * tb};
  float* s_nrm = reinterpret_cast<float*>(XIl + 5 * tb);   // [2][128]
  float* s_v = s_nrm + 2 * 128;                             // [2][128 * M]
  float* s_red = s_v + 2 * 128 * M;                         // [128 * M] second-half row sums
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_red + 128 * M);  // 0: XI, 1-2: stages, 3-4: MMA buffers
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 5);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5;
  const int row = tid & 127, half = tid >> 7;
  const int row0 = blockIdx.x * 128;
  const int split = blockIdx.y;
  const int jt0 = split * tiles_per_split;
  const int jt1 = min(col_tiles, jt0 + tiles_per_split);
  const int nt = jt1 - jt0;
  const uint32_t load_bytes = (NTERMS == 3 ? 2u : 1u) * tb;

  if (warp == 0) {
    tmem_alloc(tmem_slot, 256);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int i = 0; i < 5; ++i) mbar_init(&bars[i], 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto load_tile = [&](unsigned char* dh, unsigned char* dl, int row, uint64_t* bar) {
    mbar_arrive_expect_tx(bar, load_bytes);
    for (int a = 0; a < katoms; ++a) {
      tma_load_2d(dh + a * kAtomBytes, &tm_hi, a * 32, row, bar);
      if (NTERMS == 3) tma_load_2d(dl + a * kAtomBytes, &tm_lo, a * 32, row, bar);
    }
  };
  if (tid == 0) {
    load_tile(XIh, XIl, row0, &bars[0]);
    if (nt > 0) load_tile(XJh[0], XJl[0], jt0 * 128, &bars[1]);
    if (nt > 1) load_tile(XJh[1], XJl[1], (jt0 + 1) * 128, &bars[2]);
  }
  // K_ij = exp2(2 g_ij - n_j) exp2(-n_i): with fold_rows the row factor exp2(-n_i)
  // multiplies the finished row sums instead of every entry (the host enables it
  // only when max n_i is small enough that exp2(2 g - n_j) <= exp2(n_i) cannot overflow).
  const float ni = nrm[row0 + row];
  const float ni_in = fold_rows ? 0.f : ni;
  float racc[M][4];
#pragma unroll
  for (int c = 0; c < M; ++c)
#pragma unroll
    for (int u = 0; u < 4; ++u) racc[c][u] = 0.f;
  // kind::tf32, FP32 accumulate, A and B K-major, N = 128, M = 128
  // FP32 accumulate, A and B K-major, N = 128, M = 128; operands TF32 (kind::tf32) or bf16 (kind::f16)
  const uint32_t idesc = (1u << 4) | (NTERMS == 0 ? (1u << 7) | (1u << 10) : (2u << 7) | (2u << 10)) |
                         ((128u >> 3) << 17) | ((128u >> 4) << 24);

  for (int q = 0; q <= nt; ++q) {
    if (q < nt && tid < 128) {
      const int col = (jt0 + q) * 128 + tid;
      s_nrm[(q & 1) * 128 + tid] = __ldg(nrm + col);
#pragma unroll
      for (int c = 0; c < M; ++c) s_v[(q & 1) * 128 * M + tid * M + c] = __ldg(v32 + (size_t)col * M + c);
    }
    if (q < nt && tid == 0) {
      bool ok = true;
      if (q == 0) ok = mbar_wait_bounded(&bars[0], 0, err);
      if (ok) ok = mbar_wait_bounded(&bars[1 + (q & 1)], (uint32_t)((q >> 1) & 1), err);
      if (ok) {
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)((q & 1) * 128);
        const unsigned char* bh = XJh[q & 1];
        const unsigned char* bl = XJl[q & 1];
        for (int k = 0; k < ksteps; ++k) {
          const uint32_t off = (uint32_t)(k >> 2) * kAtomBytes + (uint32_t)(k & 3) * 32u;
          if (NTERMS == 0) umma_f16(d, umma_desc_sw128(XIh + off), umma_desc_sw128(bh + off), idesc, k > 0 ? 1u : 0u);
          else umma_tf32(d, umma_desc_sw128(XIh + off), umma_desc_sw128(bh + off), idesc, k > 0 ? 1u : 0u);
          if (NTERMS == 3) {
            umma_tf32(d, umma_desc_sw128(XIh + off), umma_desc_sw128(bl + off), idesc, 1u);
            umma_tf32(d, umma_desc_sw128(XIl + off), umma_desc_sw128(bh + off), idesc, 1u);
          }
        }
        umma_commit(&bars[3 + (q & 1)]);
      } else {
        *abort_flag = 1;
      }
    }
    if (q >= 1) {
      const int pq = q - 1;
      const int b = pq & 1;
      // the lanes agree on the outcome: the loads from tensor memory are operations of the whole warp
      if (__all_sync(0xffffffffu, mbar_wait_bounded(&bars[3 + b], (uint32_t)((pq >> 1) & 1), err))) {
        tc_fence_after();
        const uint32_t tbase = tmem + (uint32_t)(b * 128 + half * 64) + ((uint32_t)((warp & 3) * 32) << 16);
        const float* nj = s_nrm + b * 128 + half * 64;
        const float* vj = s_v + (b * 128 + half * 64) * M;
#pragma unroll 1
        for (int c4 = 0; c4 < 2; ++c4) {
          float g[32];
          tmem_ld32(tbase + (uint32_t)(c4 * 32), g);
#pragma unroll
          for (int j4 = 0; j4 < 8; ++j4) {
            const float4 n4 = *reinterpret_cast<const float4*>(nj + c4 * 32 + j4 * 4);
            const float nn[4] = {n4.x + ni_in, n4.y + ni_in, n4.z + ni_in, n4.w + ni_in};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int jj = j4 * 4 + u;
              const int col = c4 * 32 + jj;
              const float e = ex2_approx(fmaf(2.f, g[jj], -nn[u]));
#pragma unroll
              for (int c = 0; c < M; ++c) racc[c][u] = fmaf(e, vj[col * M + c], racc[c][u]);
            }
          }
        }
      } else {
        *abort_flag = 1;
      }
      tc_fence_before();
    }
    __syncthreads();
    if (*abort_flag) {
      // no copy and no MMA of this CTA in flight when its tensor memory is freed (bounded); without an
      // abort every one of them has been waited for
      if (tid == 0) {
        tile_drain(bars, min(nt, max(2, q + 1)), err);
        mma_drain(bars + 3, max(0, q - 1), min(q + 1, nt), err);
      }
      break;
    }
    // Stage (q + 1) & 1 held tile q - 1, whose MMAs completed above: refill it with tile q + 1.
    if (tid == 0 && q >= 1 && q + 1 < nt) load_tile(XJh[(q + 1) & 1], XJl[(q + 1) & 1], (jt0 + q + 1) * 128, &bars[1 + ((q + 1) & 1)]);
  }
  float rs[M];
  const float rowf = fold_rows ? ex2_approx(-ni) : 1.f;
#pragma unroll
  for (int c = 0; c < M; ++c) rs[c] = ((racc[c][0] + racc[c][1]) + (racc[c][2] + racc[c][3])) * rowf;
  if (half == 1) {
#pragma unroll
    for (int c = 0; c < M; ++c) s_red[row * M + c] = rs[c];
  }
  tc_fence_before();
  __syncthreads();
  if (half == 0) {
#pragma unroll
    for (int c = 0; c < M; ++c) part[((size_t)split * ldn + row0 + row) * M + c] = rs[c] + s_red[row * M + c];
  }
  if (warp == 0) tmem_dealloc(tmem, 256);
}

// xs32 (feature-major [p][ldn]) -> row-major TF32 parts [ldn][Kp], zero padded.
__global__ void tf32_split_kernel(const float* __restrict__ xs32, int64_t ldn, int p, int Kp, float* __restrict__ hi,
                                  float* __restrict__ lo) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ldn * Kp; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / Kp;
    const int k = (int)(e % Kp);
    const float x = k < p ? xs32[(size_t)k * ldn + i] : 0.f;
    uint32_t h, l;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(h) : "f"(x));
    const float r = x - __uint_as_float(h);
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(l) : "f"(r));
    hi[e] = __uint_as_float(h);
    lo[e] = __uint_as_float(l);
  }
}

__global__ void tc_to_f32_kernel(const double* __restrict__ V, float* __restrict__ v32, int64_t n, int64_t ldn, int m,
                                 int M, double* __restrict__ sum_out) {
  double s = 0.0;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < ldn * M;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx / M;
    const int c = (int)(idx % M);
    const double x = (i < n && c < m) ? V[i * m + c] : 0.0;
    v32[idx] = (float)x;
    if (c == 0) s += x;
  }
  if (sum_out) {
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double ws[32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
      atomicAdd(sum_out, t);
    }
  }
}

// out = sum of split partials (+ gam sum_p + L p for the CG operator); dot_out += p . out.
__global__ void tc_reduce_kernel(const float* __restrict__ part, int splits, int64_t ldn, int M, int m, int64_t n,
                                 double* __restrict__ out, GramEpilogue ep) {
  double dot = 0.0;
  const double sump = ep.sum_p ? *ep.sum_p : 0.0;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n * m;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = idx / m;
    const int c = (int)(idx % m);
    double s = 0.0;
    for (int sp = 0; sp < splits; ++sp) s += (double)part[((size_t)sp * ldn + row) * M + c];
    if (ep.raw_out) ep.raw_out[idx] = s;
    if (ep.L) s += (ep.gam_dev ? *ep.gam_dev : ep.gam) * sump + ep.L[row] * ep.pvec[row];
    out[idx] = s;
    if (ep.dot_out) dot += ep.pvec[row] * s;
  }
  if (ep.dot_out) {
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    __shared__ double ws[32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = dot;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
      atomicAdd(ep.dot_out, t);
    }
  }
}

static size_t tc_smem(int katoms, int M) {
  return 1024 + (size_t)6 * katoms * kAtomBytes + (2 * 128 + 3 * 128 * (size_t)M) * sizeof(float) + 5 * 8 + 16;
}

bool make_tmap_rowmajor_sw128(CUtensorMap* tm, void* base, int64_t ldn, int Kp);

// Prepares the TF32 row-major copies and their tensor maps (once per problem).
cudaError_t rbf_tc_prepare(Handle* h) {
  if (h->tc_hi) return cudaSuccess;
  const int Kp = h->p <= 32 ? 32 : 64;
  const size_t bytes = (size_t)h->ldn * Kp * sizeof(float);
  h->tc_hi = (float*)dev_alloc(h, bytes);
  h->tc_lo = (float*)dev_alloc(h, bytes);
  if (!h->tc_hi || !h->tc_lo) return cudaErrorMemoryAllocation;
  h->tc_Kp = Kp;
  // Fold the row factor exp2(-n_i) out of the entries when every n_i < 60:
  // then exp2(2 g - n_j) <= exp2(n_i) < 2^60 stays finite in FP32.
  {
    std::vector<float> nrm((size_t)h->ldn);
    cudaError_t e2 = cudaMemcpy(nrm.data(), h->nrm32, nrm.size() * sizeof(float), cudaMemcpyDeviceToHost);
    if (e2 != cudaSuccess) return e2;
    float mx = 0.f;
    for (float v : nrm) mx = v > mx ? v : mx;
    h->tc_fold_rows = mx < 60.f ? 1 : 0;
  }
  tf32_split_kernel<<<grid_for(h->ldn * Kp), 256, 0, h->stream>>>(h->xs32, h->ldn, (int)h->p, Kp, h->tc_hi, h->tc_lo);
  h->launches++;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (!make_tmap_rowmajor_sw128(&h->tm_tc_hi, h->tc_hi, h->ldn, Kp) ||
      !make_tmap_rowmajor_sw128(&h->tm_tc_lo, h->tc_lo, h->ldn, Kp))
    return cudaErrorInvalidValue;
  return cudaStreamSynchronize(h->stream);
}

// xs32 (feature-major [p][ldn]) -> the fp16 operands of the symmetric FP32-class tiles,
// row-major [ldn][W] halves: per row A' = [hi | hi | lo] and B' = [hi | lo | hi] over the
// p features (hi = fp16 round-to-nearest of x, lo = that of x - hi), zero beyond 3p.
// A'_j . B'_i = hi_j.hi_i + hi_j.lo_i + lo_j.hi_i, the three-term product of the TF32
// form with the same 11-bit parts, as one contraction of length 3p.
__global__ void f16_split_kernel(const float* __restrict__ xs32, int64_t ldn, int p, int W, __half* __restrict__ a,
                                 __half* __restrict__ b) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ldn * W; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / W;
    const int k = (int)(e % W);
    __half va = __float2half_rn(0.f), vb = va;
    if (k < 3 * p) {
      const int seg = k / p;
      const float x = xs32[(size_t)(k % p) * ldn + i];
      const __half hi = __float2half_rn(x);
      const __half lo = __float2half_rn(x - __half2float(hi));
      va = seg == 2 ? lo : hi;
      vb = seg == 1 ? lo : hi;
    }
    a[e] = va;
    b[e] = vb;
  }
}

// Prepares the fp16 operands of the symmetric FP32-class tiles (once per problem).  Used
// only with folded row factors (every n_i < 60, so |xs| < 8: far inside the fp16 range; a
// lo part below 2^-14 loses bits as a subnormal, an absolute error of at most 2^-25 per
// part, below FP32 rounding of the cross term) and 3p <= 128.
static cudaError_t rbf_f16_prepare(Handle* h) {
  if (h->tc_a16) return cudaSuccess;
  const int katoms = (int)((3 * h->p + 63) / 64);
  const int W = 64 * katoms;
  const size_t bytes = (size_t)h->ldn * W * sizeof(__half);
  h->tc_a16 = (float*)dev_alloc(h, bytes);
  h->tc_b16 = (float*)dev_alloc(h, bytes);
  if (!h->tc_a16 || !h->tc_b16) return cudaErrorMemoryAllocation;
  h->tc16_katoms = katoms;
  f16_split_kernel<<<grid_for(h->ldn * W), 256, 0, h->stream>>>(h->xs32, h->ldn, (int)h->p, W,
                                                                 reinterpret_cast<__half*>(h->tc_a16),
                                                                 reinterpret_cast<__half*>(h->tc_b16));
  h->launches++;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // a row of W halves is W / 2 FP32 words: the same 128-byte swizzled boxes as the TF32 parts
  if (!make_tmap_rowmajor_sw128(&h->tm_tc_a16, h->tc_a16, h->ldn, W / 2) ||
      !make_tmap_rowmajor_sw128(&h->tm_tc_b16, h->tc_b16, h->ldn, W / 2))
    return cudaErrorInvalidValue;
  return cudaStreamSynchronize(h->stream);
}

template <int M, int NT>
static cudaError_t launch_tc(Handle* h, int splits, int tps, int ksteps, cudaStream_t st) {
  const int katoms = NT == 0 ? 1 : h->tc_Kp / 32;
  const size_t smem = tc_smem(katoms, M);
  auto kern = gram_rbf_tc_kernel<M, NT>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int row_tiles = (int)(h->ldn / kTile);
  prof_mark(h, 0, true, st);
  kern<<<dim3(row_tiles, splits), 256, smem, st>>>(NT == 0 ? h->tm_tc_bf : h->tm_tc_hi, h->tm_tc_lo, h->nrm32,
                                                   h->v32, h->part, ksteps,
                                                   katoms, (int)h->ldn, tps, row_tiles, h->tc_fold_rows,
                                                   h->err_flag);
  prof_mark(h, 0, false, st);
  h->launches++;
  return cudaGetLastError();
}

// row-major bf16 copy [ldn][64] of xs32 (feature-major), round to nearest, zero padded.
__global__ void bf16_copy_kernel(const float* __restrict__ xs32, int64_t ldn, int p,
                                 __nv_bfloat16* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ldn * 64; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / 64;
    const int k = (int)(e % 64);
    out[e] = __float2bfloat16_rn(k < p ? xs32[(size_t)k * ldn + i] : 0.f);
  }
}

bool make_tmap_rowmajor_bf16_sw128(CUtensorMap* tm, void* base, int64_t ldn);

static cudaError_t rbf_bf16_prepare(Handle* h) {
  if (h->tc_bf) return cudaSuccess;
  h->tc_bf = (__nv_bfloat16*)dev_alloc(h, (size_t)h->ldn * 64 * sizeof(__nv_bfloat16));
  if (!h->tc_bf) return cudaErrorMemoryAllocation;
  bf16_copy_kernel<<<grid_for(h->ldn * 64), 256, 0, h->stream>>>(h->xs32, h->ldn, (int)h->p, h->tc_bf);
  h->launches++;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (!make_tmap_rowmajor_bf16_sw128(&h->tm_tc_bf, h->tc_bf, h->ldn)) return cudaErrorInvalidValue;
  return cudaStreamSynchronize(h->stream);
}

// U = K V on the tensor cores; nt = 3: FP32 class (TF32 hi.hi + hi.lo + lo.hi), 1: TF32 (hi.hi),
// 0: bf16 (one term, K = 16 per instruction).
static cudaError_t rbf_tc_product(Handle* h, const double* V, double* U, int m, int nt, const GramEpilogue* ep,
                                  cudaStream_t st) {
  cudaError_t e = rbf_tc_prepare(h);
  if (e != cudaSuccess) return e;
  if (nt == 0 && (e = rbf_bf16_prepare(h)) != cudaSuccess) return e;
  const int M = m <= 1 ? 1 : (m <= 2 ? 2 : (m <= 4 ? 4 : 8));
  const int row_tiles = (int)(h->ldn / kTile), col_tiles = row_tiles;
  const int katoms = nt == 0 ? 1 : h->tc_Kp / 32;
  const int resident = tc_smem(katoms, M) * 2 <= 228 * 1024 ? 2 : 1;
  const int target = 8 * resident * h->num_sms;
  int s = (target + row_tiles - 1) / row_tiles;
  if (s < 1) s = 1;
  if (s > col_tiles) s = col_tiles;
  const int tps = (col_tiles + s - 1) / s;
  const int splits = (col_tiles + tps - 1) / tps;
  const size_t vb = (size_t)h->ldn * M * sizeof(float) * 2;
  if (h->v32_cap < vb) {
    dev_free(h, h->v32);
    h->v32 = (float*)dev_alloc(h, vb);
    h->v32_cap = h->v32 ? vb : 0;
    if (!h->v32) return cudaErrorMemoryAllocation;
  }
  const size_t pb = (size_t)splits * h->ldn * M * sizeof(float);
  if (h->part_cap < pb) {
    dev_free(h, h->part);
    h->part = (float*)dev_alloc(h, pb);
    h->part_cap = h->part ? pb : 0;
    if (!h->part) return cudaErrorMemoryAllocation;
  }
  GramEpilogue none;
  const GramEpilogue& g = ep ? *ep : none;
  double* sum_out = g.sum_p ? const_cast<double*>(g.sum_p) : nullptr;
  if (sum_out && (e = cudaMemsetAsync(sum_out, 0, sizeof(double), st)) != cudaSuccess) return e;
  tc_to_f32_kernel<<<grid_for(h->ldn * M), 256, 0, st>>>(V, h->v32, h->n, h->ldn, m, M, sum_out);
  h->launches++;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int ksteps = nt == 0 ? (int)((h->p + 15) / 16) : (int)((h->p + 7) / 8);
  if (nt == 0) {
    switch (M) {
      case 1: e = launch_tc<1, 0>(h, splits, tps, ksteps, st); break;
      case 2: e = launch_tc<2, 0>(h, splits, tps, ksteps, st); break;
      case 4: e = launch_tc<4, 0>(h, splits, tps, ksteps, st); break;
      default: e = launch_tc<8, 0>(h, splits, tps, ksteps, st); break;
    }
  } else if (nt == 3) {
    switch (M) {
      case 1: e = launch_tc<1, 3>(h, splits, tps, ksteps, st); break;
      case 2: e = launch_tc<2, 3>(h, splits, tps, ksteps, st); break;
      case 4: e = launch_tc<4, 3>(h, splits, tps, ksteps, st); break;
      default: e = launch_tc<8, 3>(h, splits, tps, ksteps, st); break;
    }
  } else {
    switch (M) {
      case 1: e = launch_tc<1, 1>(h, splits, tps, ksteps, st); break;
      case 2: e = launch_tc<2, 1>(h, splits, tps, ksteps, st); break;
      case 4: e = launch_tc<4, 1>(h, splits, tps, ksteps, st); break;
      default: e = launch_tc<8, 1>(h, splits, tps, ksteps, st); break;
    }
  }
  if (e != cudaSuccess) return e;
  if (g.dot_out && (e = cudaMemsetAsync(g.dot_out, 0, sizeof(double), st)) != cudaSuccess) return e;
  tc_reduce_kernel<<<grid_for(h->n * m), 256, 0, st>>>(h->part, splits, h->ldn, M, m, h->n, U, g);
  h->launches++;
  return cudaGetLastError();
}

// ---- symmetric tiles for one right-hand side ------------------------------------------
// K is symmetric, so each off-diagonal 128 x 128 tile K_JI (J > I) is formed once on the
// tensor cores and used twice: u_J += K_JI v_I and u_I += K_JI^T v_J.  The MMA computes
// D = X_J X_I^T, so TMEM lane l is row j = J*128 + l and TMEM column c is i = I*128 + c.
//
// Operands (NTERMS): 3 = TF32 parts hi.hi + hi.lo + lo.hi, three MMAs per K = 8 step;
// 16 = the same three products from fp16 parts concatenated along K (A' = [hi | hi | lo]
// for J, B' = [hi | lo | hi] for I), one chain of ceil(3p / 16) MMAs of K = 16; 1 = TF32
// hi.hi alone (the TF32 product).
//
// What bounds it: one ex2 per entry, 32 lanes per clock and SM, 512 cycles a tile; the issue
// slots come next (2.5 per entry: the exponent's FFMA and the two sums' FFMAs are packed
// f32x2, one slot for two entries).  The rest of a tile has to hide behind that, so:
//   - one persistent CTA per SM walks an equal share of the tiles, with no set-up or drain
//     between tiles (units of 60 tiles spent a seventh of their time on it).  Tiles are
//     ordered by rows 0, T-1, 1, T-2, ... of the upper triangle, so that short rows, where
//     the row tile changes often, are spread over the CTAs;
//   - 16 epilogue warps take their tiles at their own pace (warp w: TMEM lanes
//     32 (w mod 4) .. + 31, 32 columns of I), four accumulators of 128 columns in tensor
//     memory.  A warp's 32 columns are read in halves of 16, each while the half before it is
//     worked on, the first half of the next tile included (0.36 ms without);
//   - one warp issues the copies and another the MMAs, each with running stage indexes and
//     descriptors and converged, an elected lane issuing: the thread that did both computed
//     for longer than the tile's epilogue takes (0.80 ms), two threads in branches of their
//     own took 0.45 ms.
// n = 50000, p = 20 (fp16 operands): 0.31 ms a product, 0.50 ms with 16 warps on tiles of 60-tile
// units and a CTA-wide barrier per tile; 0.127 ms is the ex2 unit's share.
// Per element a thread forms e = exp2(2 xs_j.xs_i - n_j [- n_i]) and adds e w_i to its row
// j's sum and e v_j to column i's sum, which stays in a register while the row tile I is the
// same, so the exchange across the warp's 32 rows happens once per I.  With FOLD (every
// n < 60) exp2(-n_i) is folded into w_i = v_i exp2(-n_i) and into the column results.  Row
// sums per tile and column sums per I go to FP64 sums with atomics (FP32 ones, added to
// a thousand times per row, were the largest error of the product).
// Every wait is bounded; on a timeout the CTA records the error, drains its own copies
// and MMAs (bounded) and frees its tensor memory.
constexpr int kSymEpi = 16;                         // epilogue warps
constexpr int kSymCols = 32;                       // columns of tile I per warp
static_assert(kSymEpi * 32 * kSymCols == kTile * kTile, "the warps cover a tile");
constexpr int kSymThreads = (kSymEpi + 2) * 32;    // + copy warp + MMA warp
constexpr int kSymBufs = 4;                        // TMEM accumulators of 128 columns
constexpr int kSymMaxStages = 8;

__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Walk over the order of tiles: row pair k = rows k and T - 1 - k, T + 1 tiles together (the middle
// row of an odd T alone).  I, J: the current tile; left: tiles of this row from here on.
struct SymWalk {
  int T, k, I, J, left;
  bool second;
  __device__ __forceinline__ SymWalk(int64_t t, int T_) : T(T_) {
    k = (int)(t / (T + 1));
    const int off = (int)(t - (int64_t)k * (T + 1));
    second = off >= T - k;
    I = second ? T - 1 - k : k;
    J = I + (second ? off - (T - k) : off);
    left = T - J;
  }
  // to the next tile; true if it begins another row
  __device__ __forceinline__ bool next() {
    ++J;
    if (--left) return false;
    if (second) ++k;
    second = !second;
    I = second ? T - 1 - k : k;
    J = I;
    left = T - I;
    return true;
  }
};

template <int NTERMS, bool FOLD>
__global__ void __launch_bounds__(kSymThreads, 1)
    gram_rbf_tc_sym_kernel(const __grid_constant__ CUtensorMap tm_hi, const __grid_constant__ CUtensorMap tm_lo,
                           const float* __restrict__ nrm, const float* __restrict__ v32, double* __restrict__ acc, int T,
                           int ksteps, int katoms, int nibuf, int nstage, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~static_cast<uintptr_t>(1023));
  const uint32_t tb = (uint32_t)katoms * kAtomBytes;
  const uint32_t sb = (NTERMS == 3 ? 2u : 1u) * tb;   // one tile: hi part, then (NTERMS = 3) lo part
  unsigned char* xj = base + nibuf * sb;              // nibuf (1 or 2) row tiles I, then nstage tiles J
  float* s_w = reinterpret_cast<float*>(xj + (size_t)nstage * sb);   // [kSymEpi][kSymCols] column factors of each warp
  float* s_ni = s_w + 512;                                           // [kSymEpi][kSymCols] n_i (without FOLD)
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_ni + 512);
  uint64_t* full_i = &bars[0];                        // [2] row tile landed
  uint64_t* full_j = &bars[2];                        // [nstage] X_J stage landed
  uint64_t* mma_done = &bars[2 + kSymMaxStages];      // [kSymBufs] MMAs of TMEM buffer b completed
  uint64_t* tmem_free = mma_done + kSymBufs;          // [kSymBufs] all warps have read TMEM buffer b
  uint64_t* stage_free = tmem_free + kSymBufs;        // [nstage] the MMAs that read the stage completed
  uint64_t* i_free = stage_free + kSymMaxStages;      // [2] the MMAs that read the row tile completed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(i_free + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int64_t total = (int64_t)T * (T + 1) / 2;
  const int64_t t0 = total * blockIdx.x / gridDim.x;
  const int nt = (int)(total * (blockIdx.x + 1) / gridDim.x - t0);

  if (warp == kSymEpi) {
    tmem_alloc(tmem_slot, 128 * kSymBufs);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int k = 0; k < 2; ++k) {
      mbar_init(&full_i[k], 1);
      mbar_init(&i_free[k], 1);
    }
    for (int s = 0; s < nstage; ++s) {
      mbar_init(&full_j[s], 1);
      mbar_init(&stage_free[s], 1);
    }
    for (int b = 0; b < kSymBufs; ++b) {
      mbar_init(&mma_done[b], 1);
      mbar_init(&tmem_free[b], kSymEpi);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == kSymEpi) {
    // ---- copies, in the order of the MMAs (converged warp, one elected lane)
    if (nt > 0) {
      const bool elected = elect_one();
      // with fp16 operands tm_hi maps A' (the J rows) and tm_lo maps B' (the I rows)
      auto load_tile = [&](unsigned char* dst, int row_tile, const CUtensorMap* hi, uint64_t* bar) {
        if (!elected) return;
        mbar_arrive_expect_tx(bar, sb);
        for (int a = 0; a < katoms; ++a) {
          tma_load_2d(dst + a * kAtomBytes, hi, a * 32, row_tile * 128, bar);
          if (NTERMS == 3) tma_load_2d(dst + tb + a * kAtomBytes, &tm_lo, a * 32, row_tile * 128, bar);
        }
      };
      SymWalk w(t0, T);
      int s = 0, ib = 0, q = 0, ki = 0;
      uint32_t ph = 1, iph = 1;    // parity of the free barriers: the first use of a buffer does not wait
      bool fresh = true, ok = true;
      for (; q < nt; ++q) {
        if (fresh) {
          ok = __all_sync(0xffffffffu, mbar_wait_bounded(&i_free[ib], iph, err));
          if (!ok) break;
          load_tile(base + (size_t)ib * sb, w.I, NTERMS == 16 ? &tm_lo : &tm_hi, &full_i[ib]);
          __syncwarp();
          ++ki;
          if (++ib == nibuf) {
            ib = 0;
            iph ^= 1;
          }
        }
        ok = __all_sync(0xffffffffu, *abort_flag == 0 && mbar_wait_bounded(&stage_free[s], ph, err));
        if (!ok) break;
        load_tile(xj + (size_t)s * sb, w.J, &tm_hi, &full_j[s]);
        __syncwarp();
        if (++s == nstage) {
          s = 0;
          ph ^= 1;
        }
        fresh = w.next();
      }
      if (!ok) *abort_flag = 1;
      // the CTA must not exit with a copy in flight: wait (bounded) for the last one of every buffer
      for (int k = ki > nibuf ? ki - nibuf : 0; k < ki; ++k)
        mbar_wait_bounded(&full_i[k % nibuf], (uint32_t)((k / nibuf) & 1), err);
      for (int t = q > nstage ? q - nstage : 0; t < q; ++t)
        mbar_wait_bounded(&full_j[t % nstage], (uint32_t)((t / nstage) & 1), err);
    }
  } else if (warp == kSymEpi + 1) {
    // ---- MMAs: the warp stays converged, so that indexes and descriptors are uniform values; one
    // elected lane issues (issued from a branch of one lane an MMA took hundreds of cycles)
    if (nt > 0) {
      const bool elected = elect_one();
      // FP32 accumulate, A and B K-major, N = 128, M = 128; operands TF32 (format 2) or fp16 (0)
      const uint32_t idesc = (1u << 4) | (NTERMS == 16 ? 0u : (2u << 7) | (2u << 10)) | ((128u >> 3) << 17) |
                             ((128u >> 4) << 24);
      const uint64_t desc_i = umma_desc_sw128(base), desc_j = umma_desc_sw128(xj);
      const uint32_t dhi = (uint32_t)(desc_i >> 32), t16 = tb / 16u, s16 = sb / 16u;
      auto dsc = [&](uint32_t lo) { return ((uint64_t)dhi << 32) | lo; };
      SymWalk w(t0, T);
      int s = 0, ib = 0, b = 0, q = 0;
      uint32_t ph = 0, iph = 0, fph = 1;
      uint32_t aj = (uint32_t)desc_j, bi = (uint32_t)desc_i;
      bool fresh = true, ok = true;
      for (; q < nt; ++q) {
        if (fresh) ok = mbar_wait_bounded(&full_i[ib], iph, err);
        // TMEM buffer b last held tile q - kSymBufs: every warp must have read it out
        ok = ok && mbar_wait_bounded(&tmem_free[b], fph, err) && mbar_wait_bounded(&full_j[s], ph, err);
        if (!__all_sync(0xffffffffu, ok && *abort_flag == 0)) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(b * 128);
        if (elected) {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (k < ksteps) {
              const uint32_t off = ((uint32_t)(k >> 2) * kAtomBytes + (uint32_t)(k & 3) * 32u) / 16u;
              if (NTERMS == 16) umma_f16(d, dsc(aj + off), dsc(bi + off), idesc, k > 0 ? 1u : 0u);
              else umma_tf32(d, dsc(aj + off), dsc(bi + off), idesc, k > 0 ? 1u : 0u);
              if (NTERMS == 3) {
                umma_tf32(d, dsc(aj + off), dsc(bi + t16 + off), idesc, 1u);
                umma_tf32(d, dsc(aj + t16 + off), dsc(bi + off), idesc, 1u);
              }
            }
          }
          if (w.left == 1) umma_commit(&i_free[ib]);   // the row ends: committed before the last waits below
          umma_commit(&mma_done[b]);
          umma_commit(&stage_free[s]);
        }
        __syncwarp();
        if (++b == kSymBufs) {
          b = 0;
          fph ^= 1;
        }
        aj += s16;
        if (++s == nstage) {
          s = 0;
          ph ^= 1;
          aj = (uint32_t)desc_j;
        }
        fresh = w.next();
        if (fresh && q + 1 < nt) {
          bi += s16;
          if (++ib == nibuf) {
            ib = 0;
            iph ^= 1;
            bi = (uint32_t)desc_i;
          }
        }
      }
      if (q < nt) *abort_flag = 1;
      // let the MMAs and commits in flight finish (bounded) before the tensor memory is freed
      if (q > 0) {
        mbar_wait_bounded(&mma_done[(q - 1) % kSymBufs], (uint32_t)(((q - 1) / kSymBufs) & 1), err);
        mbar_wait_bounded(&stage_free[(q - 1) % nstage], (uint32_t)(((q - 1) / nstage) & 1), err);
      }
    }
  } else if (nt > 0) {
    const int lq = warp & 3, cq = warp >> 2;
    float* wq = s_w + warp * kSymCols;
    float* nq = s_ni + warp * kSymCols;
    uint64_t cacc[kSymCols / 2];   // column sums of tile I over this warp's 32 rows, across the tiles of this I
    const uint64_t two = pack2(2.f, 2.f);
    SymWalk w(t0, T);
    int I = -1;
    bool fresh = true, ok = true;
    const int lrow = lq * 32 + lane;
    float n_nx = __ldg(nrm + w.J * 128 + lrow);
    float v_nx = w.J == w.I ? 0.f : __ldg(v32 + w.J * 128 + lrow);   // the diagonal tile gives row sums only
    // column sums: reduce-scatter each 32 over the warp's 32 rows, so that lane l ends with column l
    auto flush = [&]() {
      float ch[32];
#pragma unroll
      for (int c = 0; c < 16; ++c) unpack2(cacc[c], ch[2 * c], ch[2 * c + 1]);
#pragma unroll
      for (int wd = 16; wd >= 1; wd >>= 1) {
        const bool up = (lane & wd) != 0;
#pragma unroll
        for (int i = 0; i < wd; ++i) {
          const float keep = up ? ch[i + wd] : ch[i], send = up ? ch[i] : ch[i + wd];
          ch[i] = keep + __shfl_xor_sync(0xffffffffu, send, wd);
        }
      }
      const float f = FOLD ? ex2_approx(-nq[lane]) : 1.f;
      atomicAdd(acc + I * 128 + cq * kSymCols + lane, (double)(ch[0] * f));
    };
    const uint32_t tcol = tmem + (uint32_t)(cq * kSymCols) + ((uint32_t)(lq * 32) << 16);
    uint32_t ph = 0;
    int b = 0;
    // the accumulators come in halves of 16 columns, each loaded while the half before it is worked on
    uint32_t g0[16], g1[16];
    auto wait_tile = [&]() {
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(&mma_done[b], ph, err));
      if (!ok) {
        *abort_flag = 1;
        return;
      }
      tc_fence_after();
      tmem_ld16_nowait(tcol + (uint32_t)(b * 128), g0);
    };
    wait_tile();
    for (int q = 0; q < nt && ok; ++q) {
      if (fresh) {
        if (I >= 0) flush();
        I = w.I;
        __syncwarp();
        const float n_i = __ldg(nrm + I * 128 + cq * kSymCols + lane);
        wq[lane] = __ldg(v32 + I * 128 + cq * kSymCols + lane) * (FOLD ? ex2_approx(-n_i) : 1.f);
        nq[lane] = n_i;
        __syncwarp();
#pragma unroll
        for (int c = 0; c < kSymCols / 2; ++c) cacc[c] = 0ull;
      }
      const int jrow = w.J * 128 + lrow;
      const float n_j = n_nx, v_j = v_nx;
      fresh = w.next();
      if (q + 1 < nt) {
        n_nx = __ldg(nrm + w.J * 128 + lrow);
        v_nx = fresh ? 0.f : __ldg(v32 + w.J * 128 + lrow);   // a row begins with its diagonal tile
      }
      const uint64_t nj2 = pack2(-n_j, -n_j), vj2 = pack2(v_j, v_j);
      uint64_t racc[2] = {0ull, 0ull};
      auto half = [&](const uint32_t (&g)[16], auto half_tag) {
        constexpr int hh = decltype(half_tag)::value;
#pragma unroll
        for (int c4 = 0; c4 < 4; ++c4) {
          const float4 w4 = *reinterpret_cast<const float4*>(wq + hh * 16 + c4 * 4);
          float4 n4;
          if (!FOLD) n4 = *reinterpret_cast<const float4*>(nq + hh * 16 + c4 * 4);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int c = c4 * 2 + u;
            uint64_t off = nj2;
            if (!FOLD) off = add2(nj2, u ? pack2(-n4.z, -n4.w) : pack2(-n4.x, -n4.y));
            float e0, e1;
            unpack2(fma2(pack2(__uint_as_float(g[2 * c]), __uint_as_float(g[2 * c + 1])), two, off), e0, e1);
            const uint64_t e = pack2(ex2_approx(e0), ex2_approx(e1));
            racc[u] = fma2(e, u ? pack2(w4.z, w4.w) : pack2(w4.x, w4.y), racc[u]);
            cacc[hh * 8 + c] = fma2(e, vj2, cacc[hh * 8 + c]);
          }
        }
      };
      tmem_wait16(g0);
      tmem_ld16_nowait(tcol + (uint32_t)(b * 128 + 16), g1);
      half(g0, std::integral_constant<int, 0>{});
      tmem_wait16(g1);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tmem_free[b]);
      if (++b == kSymBufs) {
        b = 0;
        ph ^= 1;
      }
      if (q + 1 < nt) wait_tile();
      half(g1, std::integral_constant<int, 1>{});
      float r0, r1;
      unpack2(add2(racc[0], racc[1]), r0, r1);
      atomicAdd(acc + jrow, (double)(r0 + r1));
    }
    if (__all_sync(0xffffffffu, ok && *abort_flag == 0)) flush();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kSymEpi) tmem_dealloc(tmem, 128 * kSymBufs);
}

// Row-tile buffers and J stages: 2 + 8 (tiles of 16 KB; 4: 0.33 ms), 2 + 3 (32 KB), 1 + 2 (64 KB).
static void tc_sym_stages(size_t tile_bytes, int* nibuf, int* nstage) {
  *nibuf = tile_bytes <= 32 * 1024 ? 2 : 1;
  *nstage = tile_bytes <= 16 * 1024 ? kSymMaxStages : (tile_bytes <= 32 * 1024 ? 3 : 2);
}

static size_t tc_sym_smem(size_t tile_bytes) {
  int ni, ns;
  tc_sym_stages(tile_bytes, &ni, &ns);
  return 1024 + (size_t)(ni + ns) * tile_bytes + 2 * 512 * sizeof(float) +
         (4 + 2 * kSymMaxStages + 2 * kSymBufs) * sizeof(uint64_t) + 16;
}

// m = 1 RBF product on symmetric tensor-core tiles; nt = 3: FP32 class (fp16 parts when
// the row factors fold and 3p <= 128, else TF32 parts), 1: TF32.
static cudaError_t rbf_tc_sym_product(Handle* h, const double* V, double* U, int nt, const GramEpilogue* ep,
                                      cudaStream_t st) {
  cudaError_t e = rbf_tc_prepare(h);
  if (e != cudaSuccess) return e;
  float* v32;
  double* acc;
  if ((e = sym_buffers(h, &v32, &acc)) != cudaSuccess) return e;
  GramEpilogue none;
  const GramEpilogue& g = ep ? *ep : none;
  if (!g.prepped && (e = sym_prep(h, V, v32, acc, const_cast<double*>(g.sum_p), st)) != cudaSuccess) return e;
  const bool f16 = nt == 3 && h->tc_fold_rows && 3 * h->p <= 128;
  if (f16 && (e = rbf_f16_prepare(h)) != cudaSuccess) return e;
  const int katoms = f16 ? h->tc16_katoms : h->tc_Kp / 32;
  const int ksteps = f16 ? (int)((3 * h->p + 15) / 16) : (int)((h->p + 7) / 8);
  const size_t tile = (size_t)(!f16 && nt == 3 ? 2 : 1) * katoms * kAtomBytes;
  const size_t smem = tc_sym_smem(tile);
  int nibuf, nstage;
  tc_sym_stages(tile, &nibuf, &nstage);
  auto kern = f16 ? gram_rbf_tc_sym_kernel<16, true>
                  : nt == 3 ? (h->tc_fold_rows ? gram_rbf_tc_sym_kernel<3, true> : gram_rbf_tc_sym_kernel<3, false>)
                            : (h->tc_fold_rows ? gram_rbf_tc_sym_kernel<1, true> : gram_rbf_tc_sym_kernel<1, false>);
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return e;
  const int T = (int)(h->ldn / kTile);
  const int grid = (int)std::min<int64_t>(h->num_sms, (int64_t)T * (T + 1) / 2);
  prof_mark(h, 0, true, st);
  kern<<<grid, kSymThreads, smem, st>>>(f16 ? h->tm_tc_a16 : h->tm_tc_hi, f16 ? h->tm_tc_b16 : h->tm_tc_lo, h->nrm32,
                                        v32, acc, T, ksteps, katoms, nibuf, nstage, h->err_flag);
  prof_mark(h, 0, false, st);
  h->launches++;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return sym_finish(h, acc, true, U, g, st);
}

// ---- several right-hand sides, FP32 class (p <= 32) -------------------------------------
// u_I += K_IJ V_J for M = 2, 4 or 8 vectors, all n^2 entries, row sums only (deterministic).  A
// step is 256 rows (two row tiles, one after the other in tensor memory) x 128 columns.
//
// What bounds it: the FFMAs with the vectors, 4 issue slots per entry at M = 8 as packed f32x2
// over column pairs (the even and odd columns' sums are separate chains), beside 1.5 for the
// exponent and the ex2, and the broadcast loads of V, which serve two rows of a thread each.
// n = 19999, p = 8, M = 8: 257 us; the plain kernel (one row per thread, unpacked, a CTA-wide
// barrier per tile and one thread of the epilogue computing descriptors for 3 ksteps MMAs) 602 us.
// Loading 4-column chunks ahead of their use gave nothing (260 us).
// One persistent CTA per SM walks an equal share of the steps (row pairs in order, all columns of
// a pair); copies and MMAs are issued by a warp each; 16 epilogue warps: warp w has TMEM lanes
// 32 (w mod 4) .. + 31 and columns 32 (w / 4) .. + 31.  Sums of a step's 32 columns start at zero
// and are added to per-thread totals in shared memory, which keeps FP32 chains short.  A CTA's
// sums for a row pair go to its own partial (slot = CTA minus the pair's first CTA); a second
// kernel adds the partials in FP64.
constexpr int kMtEpi = 16;
constexpr int kMtThreads = (kMtEpi + 2) * 32;
constexpr int kMtStages = 3;

__host__ __device__ __forceinline__ int mt_cta_of(int64_t step, int64_t total, int grid) {
  return (int)(((step + 1) * grid - 1) / total);   // the CTA whose share [total b / grid, ...) holds the step
}

template <int M>
__global__ void __launch_bounds__(kMtThreads, 1)
    gram_rbf_tc_multi_kernel(const __grid_constant__ CUtensorMap tm_hi, const __grid_constant__ CUtensorMap tm_lo,
                             const float* __restrict__ nrm, const float* __restrict__ vp, float* __restrict__ part,
                             int ksteps, int64_t ldn, int T, int fold_rows, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~static_cast<uintptr_t>(1023));
  constexpr uint32_t kTile16 = kAtomBytes / 16u;
  constexpr uint32_t kStage = 2 * kAtomBytes;              // hi, lo
  constexpr uint32_t kVBytesM = 128u * M * 4u;
  unsigned char* xj = base + 4 * kAtomBytes;               // row tiles: hi 0, lo 0, hi 1, lo 1
  unsigned char* cst = xj + kMtStages * kStage;            // [stage]: 128 norms, 128 x M of V in column pairs
  constexpr uint32_t kCst = 512u + kVBytesM;
  float4* tot = reinterpret_cast<float4*>(cst + kMtStages * kCst);   // [2 M / 4][512]
  uint64_t* bars = reinterpret_cast<uint64_t*>(tot + (2 * M / 4) * 512);
  uint64_t* full_i = bars;
  uint64_t* i_free = bars + 1;
  uint64_t* full_j = bars + 2;                  // [kMtStages]
  uint64_t* stage_free = full_j + kMtStages;    // [kMtStages] MMAs done and constants read
  uint64_t* mma_done = stage_free + kMtStages;  // [2]
  uint64_t* tmem_free = mma_done + 2;           // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tmem_free + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int pairs = (T + 1) / 2;
  const int64_t total = (int64_t)pairs * T;
  const int64_t t0 = total * blockIdx.x / gridDim.x;
  const int nt = (int)(total * (blockIdx.x + 1) / gridDim.x - t0);

  if (warp == kMtEpi) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(full_i, 1);
    mbar_init(i_free, 1);
    for (int s = 0; s < kMtStages; ++s) {
      mbar_init(&full_j[s], 1);
      mbar_init(&stage_free[s], 1 + kMtEpi);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&mma_done[b], 1);
      mbar_init(&tmem_free[b], kMtEpi);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  int P = (int)(t0 / T), J = (int)(t0 % T);   // row pair and column tile of the first step

  if (warp == kMtEpi) {
    // ---- copies (converged warp, one elected lane)
    if (nt > 0) {
      const bool elected = elect_one();
      int s = 0, q = 0, ki = 0;
      uint32_t ph = 1;
      bool ok = true;
      for (; q < nt; ++q) {
        if (q == 0 || J == 0) {
          if (ki > 0) ok = __all_sync(0xffffffffu, mbar_wait_bounded(i_free, (uint32_t)((ki - 1) & 1), err));
          if (!ok) break;
          if (elected) {
            mbar_arrive_expect_tx(full_i, 4 * kAtomBytes);
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {   // rows beyond ldn read as zero
              tma_load_2d(base + hh * kStage, &tm_hi, 0, (2 * P + hh) * 128, full_i);
              tma_load_2d(base + hh * kStage + kAtomBytes, &tm_lo, 0, (2 * P + hh) * 128, full_i);
            }
          }
          __syncwarp();
          ++ki;
        }
        ok = __all_sync(0xffffffffu, *abort_flag == 0 && mbar_wait_bounded(&stage_free[s], ph, err));
        if (!ok) break;
        if (elected) {
          mbar_arrive_expect_tx(&full_j[s], kStage + kCst);
          tma_load_2d(xj + s * kStage, &tm_hi, 0, J * 128, &full_j[s]);
          tma_load_2d(xj + s * kStage + kAtomBytes, &tm_lo, 0, J * 128, &full_j[s]);
          bulk_copy(cst + s * kCst, nrm + J * 128, 512u, &full_j[s]);
          bulk_copy(cst + s * kCst + 512, vp + (size_t)J * 128 * M, kVBytesM, &full_j[s]);
        }
        __syncwarp();
        if (++s == kMtStages) {
          s = 0;
          ph ^= 1;
        }
        if (++J == T) {
          J = 0;
          ++P;
        }
      }
      if (!ok) *abort_flag = 1;
      if (ki > 0) mbar_wait_bounded(full_i, (uint32_t)((ki - 1) & 1), err);
      for (int t = q > kMtStages ? q - kMtStages : 0; t < q; ++t)
        mbar_wait_bounded(&full_j[t % kMtStages], (uint32_t)((t / kMtStages) & 1), err);
    }
  } else if (warp == kMtEpi + 1) {
    // ---- MMAs (converged warp, one elected lane, as in the symmetric kernel)
    if (nt > 0) {
      const bool elected = elect_one();
      // FP32 accumulate, TF32 A and B, K-major, N = 128, M = 128
      const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
      const uint64_t desc_i = umma_desc_sw128(base), desc_j = umma_desc_sw128(xj);
      const uint32_t dhi = (uint32_t)(desc_i >> 32);
      auto dsc = [&](uint32_t lo) { return ((uint64_t)dhi << 32) | lo; };
      int s = 0, b = 0, q = 0, ki = 0;
      uint32_t ph = 0, fph = 1;
      bool ok = true;
      for (; q < nt; ++q) {
        if (q == 0 || J == 0) {
          ok = mbar_wait_bounded(full_i, (uint32_t)(ki & 1), err);
          ++ki;
        }
        ok = ok && mbar_wait_bounded(&tmem_free[b], fph, err) && mbar_wait_bounded(&full_j[s], ph, err);
        if (!__all_sync(0xffffffffu, ok && *abort_flag == 0)) break;
        tc_fence_after();
        const uint32_t bj = (uint32_t)desc_j + (uint32_t)s * (2 * kTile16);
        if (elected) {
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const uint32_t d = tmem + (uint32_t)(b * 256 + hh * 128);
            const uint32_t ai = (uint32_t)desc_i + (uint32_t)hh * (2 * kTile16);
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (k < ksteps) {
                umma_tf32(d, dsc(ai + k * 2u), dsc(bj + k * 2u), idesc, k > 0 ? 1u : 0u);
                umma_tf32(d, dsc(ai + k * 2u), dsc(bj + kTile16 + k * 2u), idesc, 1u);
                umma_tf32(d, dsc(ai + kTile16 + k * 2u), dsc(bj + k * 2u), idesc, 1u);
              }
          }
          umma_commit(&stage_free[s]);
          if (J + 1 == T && q + 1 < nt) umma_commit(i_free);
          umma_commit(&mma_done[b]);
        }
        __syncwarp();
        if (++J == T) {
          J = 0;
          ++P;
        }
        b ^= 1;
        if (b == 0) fph ^= 1;
        if (++s == kMtStages) {
          s = 0;
          ph ^= 1;
        }
      }
      if (q < nt) *abort_flag = 1;
      if (q > 0) mbar_wait_bounded(&mma_done[(q - 1) & 1], (uint32_t)(((q - 1) >> 1) & 1), err);
    }
  } else if (nt > 0) {
    // ---- epilogue
    const int lq = warp & 3, cg = warp >> 2;
    const uint32_t lane_off = (uint32_t)(lq * 32) << 16;
    const uint64_t two = pack2(2.f, 2.f);
    const int lrow = lq * 32 + lane;
    float ni[2] = {0.f, 0.f};       // row norms, inside the exponent unless the row factors fold
    auto row_norms = [&](int pair) {
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const int64_t row = (int64_t)pair * 256 + hh * 128 + lrow;
        ni[hh] = !fold_rows && row < ldn ? __ldg(nrm + row) : 0.f;
      }
    };
    auto zero_totals = [&]() {
#pragma unroll
      for (int e = 0; e < 2 * M / 4; ++e) tot[e * 512 + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // the totals of the four column groups, added in a fixed order, to this CTA's partial of the pair
    auto flush = [&](int pair) {
      const int slot = blockIdx.x - mt_cta_of((int64_t)pair * T, total, gridDim.x);
      asm volatile("bar.sync 1, 512;" ::: "memory");
      for (int e = tid; e < 256 * M; e += kMtEpi * 32) {
        const int row = e / M, c = e % M;
        const int idx = (row >> 7) * M + c, t = ((row >> 5) & 3) * 32 + (row & 31);
        float v = 0.f;
#pragma unroll
        for (int g = 0; g < 4; ++g) v += reinterpret_cast<const float*>(tot + (idx >> 2) * 512 + g * 128 + t)[idx & 3];
        const int64_t gr = (int64_t)pair * 256 + row;
        if (gr < ldn) {
          if (fold_rows) v *= ex2_approx(-__ldg(nrm + gr));
          part[((size_t)slot * ldn + gr) * M + c] = v;
        }
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
    };
    row_norms(P);
    zero_totals();
    bool ok = true;
    int s = 0, b = 0;
    uint32_t ph = 0, mph = 0;
    for (int q = 0; q < nt; ++q) {
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full_j[s], ph, err) && mbar_wait_bounded(&mma_done[b], mph, err))) {
        ok = false;
        *abort_flag = 1;
      }
      if (ok) {
        tc_fence_after();
        const float* nj = reinterpret_cast<const float*>(cst + s * kCst) + cg * 32;
        const float* vj = reinterpret_cast<const float*>(cst + s * kCst + 512) + cg * 32 * M;
        uint64_t acc[2][M];   // even and odd columns' sums of this step
#pragma unroll
        for (int hh = 0; hh < 2; ++hh)
#pragma unroll
          for (int c = 0; c < M; ++c) acc[hh][c] = 0ull;
#pragma unroll 1
        for (int ch = 0; ch < 4; ++ch) {
          uint32_t g[2][8];
          tmem_ld8_nowait(tmem + (uint32_t)(b * 256 + cg * 32 + ch * 8) + lane_off, g[0]);
          tmem_ld8_nowait(tmem + (uint32_t)(b * 256 + 128 + cg * 32 + ch * 8) + lane_off, g[1]);
          tmem_wait_ld();
          if (ch == 3) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tmem_free[b]);
          }
#pragma unroll
          for (int c2 = 0; c2 < 4; ++c2) {
            const int col = ch * 8 + 2 * c2;
            const float2 n2 = *reinterpret_cast<const float2*>(nj + col);
            uint64_t e[2];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              float e0, e1;
              unpack2(fma2(pack2(__uint_as_float(g[hh][2 * c2]), __uint_as_float(g[hh][2 * c2 + 1])), two,
                           pack2(-(n2.x + ni[hh]), -(n2.y + ni[hh]))),
                      e0, e1);
              e[hh] = pack2(ex2_approx(e0), ex2_approx(e1));
            }
#pragma unroll
            for (int c = 0; c < M; c += 2) {
              const float4 v = *reinterpret_cast<const float4*>(vj + col * M + 2 * c);
#pragma unroll
              for (int hh = 0; hh < 2; ++hh) {
                acc[hh][c] = fma2(e[hh], pack2(v.x, v.y), acc[hh][c]);
                acc[hh][c + 1] = fma2(e[hh], pack2(v.z, v.w), acc[hh][c + 1]);
              }
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&stage_free[s]);
        float sums[2 * M];
#pragma unroll
        for (int hh = 0; hh < 2; ++hh)
#pragma unroll
          for (int c = 0; c < M; ++c) {
            float a0, a1;
            unpack2(acc[hh][c], a0, a1);
            sums[hh * M + c] = a0 + a1;
          }
#pragma unroll
        for (int e = 0; e < 2 * M / 4; ++e) {
          float4 t = tot[e * 512 + tid];
          t.x += sums[4 * e];
          t.y += sums[4 * e + 1];
          t.z += sums[4 * e + 2];
          t.w += sums[4 * e + 3];
          tot[e * 512 + tid] = t;
        }
        b ^= 1;
        if (b == 0) mph ^= 1;
        if (++s == kMtStages) {
          s = 0;
          ph ^= 1;
        }
      }
      // every warp comes here for every step, also after a timeout: the flush has barriers
      if (++J == T || q + 1 == nt) {
        flush(P);
        if (J == T) {
          J = 0;
          ++P;
        }
        if (q + 1 < nt) {
          row_norms(P);
          zero_totals();
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kMtEpi) tmem_dealloc(tmem, 512);
}

// V (n x m) -> FP32 in column-pair order of the rows: vp[(i / 2) 2 M + 2 c + (i mod 2)], zero padded.
__global__ void mt_prep_kernel(const double* __restrict__ V, float* __restrict__ vp, int64_t n, int64_t ldn, int m,
                               int M) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ldn * M; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / (2 * M) * 2 + (e & 1);
    const int c = (int)(e % (2 * M)) >> 1;
    vp[e] = (i < n && c < m) ? (float)V[i * m + c] : 0.f;
  }
}

// out = sum of the pair's partials, in FP64.
__global__ void mt_reduce_kernel(const float* __restrict__ part, int64_t ldn, int T, int grid, int M, int m, int64_t n,
                                 double* __restrict__ out) {
  const int64_t total = (int64_t)((T + 1) / 2) * T;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * m; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / m, pair = row >> 8;
    const int c = (int)(e % m);
    const int slots = mt_cta_of(pair * T + T - 1, total, grid) - mt_cta_of(pair * T, total, grid) + 1;
    double s = 0.0;
    for (int q = 0; q < slots; ++q) s += (double)part[((size_t)q * ldn + row) * M + c];
    out[e] = s;
  }
}

template <int M>
static cudaError_t launch_multi(Handle* h, int grid, int ksteps, cudaStream_t st) {
  const size_t smem = 1024 + 4 * kAtomBytes + kMtStages * (2 * kAtomBytes + 512 + 128 * M * 4) +
                      (size_t)(2 * M / 4) * 512 * 16 + (2 + 2 * kMtStages + 4) * 8 + 16;
  auto kern = gram_rbf_tc_multi_kernel<M>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  prof_mark(h, 0, true, st);
  kern<<<grid, kMtThreads, smem, st>>>(h->tm_tc_hi, h->tm_tc_lo, h->nrm32, h->v32, h->part, ksteps, h->ldn,
                                       (int)(h->ldn / kTile), h->tc_fold_rows, h->err_flag);
  prof_mark(h, 0, false, st);
  h->launches++;
  return cudaGetLastError();
}

// From this many row tiles on: 256 x 128 steps leave most SMs without work below (n = 1000, M = 8:
// 24.9 us a call, 23.2 with the plain kernel; n = 2000: 25.6 against 31.4).
constexpr int kMtMinTiles = 12;

// FP32-class product with 2 to 8 right-hand sides, p <= 32 (one 128-byte atom per row and part).
static cudaError_t rbf_tc_multi_product(Handle* h, const double* V, double* U, int m, cudaStream_t st) {
  cudaError_t e = rbf_tc_prepare(h);
  if (e != cudaSuccess) return e;
  const int M = m <= 2 ? 2 : (m <= 4 ? 4 : 8);
  const int T = (int)(h->ldn / kTile);
  const int64_t total = (int64_t)((T + 1) / 2) * T;
  const int grid = (int)std::min<int64_t>(h->num_sms, total);
  // CTAs that share a row pair: at most its T steps over the shortest share, plus the two cut ones
  const int64_t slots = std::min<int64_t>(grid, T / (total / grid) + 2);
  const size_t vb = (size_t)h->ldn * M * sizeof(float);
  if (h->v32_cap < vb) {
    dev_free(h, h->v32);
    h->v32 = (float*)dev_alloc(h, vb);
    h->v32_cap = h->v32 ? vb : 0;
    if (!h->v32) return cudaErrorMemoryAllocation;
  }
  const size_t pb = (size_t)slots * h->ldn * M * sizeof(float);
  if (h->part_cap < pb) {
    dev_free(h, h->part);
    h->part = (float*)dev_alloc(h, pb);
    h->part_cap = h->part ? pb : 0;
    if (!h->part) return cudaErrorMemoryAllocation;
  }
  mt_prep_kernel<<<grid_for(h->ldn * M), 256, 0, st>>>(V, h->v32, h->n, h->ldn, m, M);
  h->launches++;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int ksteps = (int)((h->p + 7) / 8);
  switch (M) {
    case 2: e = launch_multi<2>(h, grid, ksteps, st); break;
    case 4: e = launch_multi<4>(h, grid, ksteps, st); break;
    default: e = launch_multi<8>(h, grid, ksteps, st); break;
  }
  if (e != cudaSuccess) return e;
  mt_reduce_kernel<<<grid_for(h->n * m), 256, 0, st>>>(h->part, h->ldn, T, grid, M, m, h->n, U);
  h->launches++;
  return cudaGetLastError();
}

cudaError_t gram_rbf_tc(Handle* h, const double* V, double* U, int m, bool three_terms, const GramEpilogue* ep,
                        cudaStream_t st) {
  if (m == 1 && h->opt.symmetric_gram) return rbf_tc_sym_product(h, V, U, three_terms ? 3 : 1, ep, st);
  if (m >= 2 && three_terms && !ep && h->p <= 32 && h->ldn >= kMtMinTiles * kTile)
    return rbf_tc_multi_product(h, V, U, m, st);
  return rbf_tc_product(h, V, U, m, three_terms ? 3 : 1, ep, st);
}

cudaError_t gram_rbf_tc_bf16(Handle* h, const double* V, double* U, int m, cudaStream_t st) {
  return rbf_tc_product(h, V, U, m, 0, nullptr, st);
}

}  // namespace kqr
