// FP64-class RBF Gram products u = K V with the cross term on the tcgen05 tensor cores
// (p <= 32, every |xs_i|^2 < 28).
//
// K_ij = 2^-E_ij, E_ij = |xs_i|^2 + |xs_j|^2 - 2 xs_i . xs_j with xs = sqrt(gamma log2 e)(x - mean).
// Each coordinate is an integer H = rint(xs 2^59), cut into seven balanced base-512 digits
// d_6 .. d_0 (|d| <= 256, exact in bf16, stored as d 2^(9 s - 59) 2^10, so that the sums come out in
// units the epilogue can convert without a multiplication).  The product of digits s and t has weight
// 2^(9 (s + t) - 118) in the cross term.  The 28 digit pairs with s + t >= 6 are taken; the first level
// dropped is at most 6 p 2^16 2^-73 = 2^-49.4 at p = 32 (digits all of magnitude 256 and of one sign;
// about 2^-54 for digits without correlation).  They run as kind::f16 MMAs (bf16
// A and B, FP32 accumulators in tensor memory), grouped by level l = s + t so that the sums the
// exponent needs exactly are exact integers below 2^24 units:
//   A = levels 12 + 11 (|sum| <= |xs_i||xs_j| < 28 = 2^23.8 units of 2^-19),
//   B = level 10 and C = level 9 (at most 4 p 2^16 <= 2^23 units),
//   D = levels 8 + 7 + 6 (at most 5 p 2^16 2^-46 = 2^-22.7 and a little, so an FP32 rounding is up to
//   2^-47; about 2^-26 and 2^-50 for digits without correlation).
// The epilogue adds them to the norms (two int32 words and a float per point) in fixed point:
// integer part, 12-bit table index (4096-entry double-float table of 2^-(k/4096)) and a remainder
// below 2^-12, whose exponential needs one float polynomial; entry and sums are double-float.
// Measured entry error about 2e-15 relative.
//
// What bounds it: issue slots and the FP32 pipe of the epilogue, about 75 instructions per entry with
// row sums and 94 with the column sums (p no longer enters: the 56 MMAs of a 128 x 64 tile run beside
// it, from unrolled code with precomputed descriptors; a loop that built them cost the issuing thread
// 40 instructions per MMA among 16 busy warps and made the MMAs the bound).  For one vector each
// off-diagonal tile serves its rows and its columns (n(n+1)/2 entries); for several, an entry is formed
// once per pass over K and added to every vector's row sums.  Measured: one vector, n = 50000, p = 20:
// 3.86 ms (3.80 with plain atomics, whose results differed from run to run), before 20.9 ms; eight vectors, n = 10007, p = 8: 0.62 ms, before
// 4.38 ms.  Before: int64 sums of squared differences on the CUDA cores (6 operations per entry and
// feature, all n^2 entries, columns one after another).
//
// One CTA per SM: warps 0..15 are the epilogue (warp w: TMEM lanes 32 (w mod 4) .. + 31 = rows of
// tile I, columns 16 (w / 4) .. + 15 of the 64-column tile J), lane 0 of warp 16 issues TMA copies
// and MMAs.  Two accumulator sets of 256 columns fill tensor memory; three stages of J digits and
// point constants.  Row sums stay in registers over the unit; column sums are reduced across the
// warp's 32 rows.  For one vector both go to the result by atomics whose sums do not depend on their
// order (OrderFree below), so that the product is the same in every run.  Every wait is bounded; on a timeout the CTA records
// the error.  In any case it waits (bounded) for its own copies and MMAs before it frees its tensor
// memory.
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include <cuda_bf16.h>

#include "ht_units.h"
#include "kqr_internal.h"
#include "ptx.cuh"

namespace kqr {

namespace {

constexpr int kDigits = 7;
constexpr int kDigitBits = 9;
constexpr int kFracBits = 59;
constexpr float kMaxNorm = 28.f;
constexpr int kTabBits = 12;
constexpr int kJCols = 64;
constexpr int kStages = 3;
constexpr int kEpiWarps = 16;
constexpr int kThreadsHt = (kEpiWarps + 1) * 32;
constexpr uint32_t kIAtom = 128 * 128;       // 128 rows x 128 bytes
constexpr uint32_t kJAtom = kJCols * 128;
constexpr uint32_t kTabBytes = (1u << kTabBits) * 8u;

__device__ __forceinline__ void ht_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void ht_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void ht_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void ht_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void ht_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void ht_mma(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void ht_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// The MMAs of one 128 x 64 tile into the accumulator set at d; alo, blo: low descriptor words of
// the I tile and of the J stage.  KS: 16-feature steps per digit (digits of 32 KS bytes, 4 / KS per
// 128-byte atom).  All offsets are compile-time constants.
template <int KS>
__device__ __forceinline__ void ht_issue_tile(uint32_t d, uint32_t alo, uint32_t blo, uint32_t hi, uint32_t idesc) {
  constexpr int kPer = 4 / KS;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int top = 2 * (kDigits - 1);
    const int l1 = g == 0 ? top : top - 1 - g, l0 = g == 0 ? top - 1 : (g == 3 ? top - 6 : top - 1 - g);
    bool first = true;
#pragma unroll
    for (int l = l1; l >= l0; --l)
#pragma unroll
      for (int si = kDigits - 1; si >= 0; --si) {
        const int sj = l - si;
        if (sj < 0 || sj >= kDigits) continue;
#pragma unroll
        for (int k = 0; k < KS; ++k) {
          const uint32_t a = alo + ((uint32_t)(si / kPer) * 16384u + (uint32_t)(si % kPer) * (KS * 32u) + k * 32u) / 16u;
          const uint32_t b = blo + ((uint32_t)(sj / kPer) * 8192u + (uint32_t)(sj % kPer) * (KS * 32u) + k * 32u) / 16u;
          ht_mma(d + (uint32_t)(g * 64), ((uint64_t)hi << 32) | a, ((uint64_t)hi << 32) | b, idesc, first ? 0u : 1u);
          first = false;
        }
      }
  }
}

// 8 consecutive 32-bit columns of this thread's TMEM lane (no wait).
__device__ __forceinline__ void ht_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void ht_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// K-major operand in the 128-byte swizzled layout (8-row groups 1024 bytes apart).
__device__ __forceinline__ uint64_t ht_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ void ht_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// (sh, sl) += (yh, yl) without renormalising sl.
__device__ __forceinline__ void ht_add(float& sh, float& sl, float yh, float yl) {
  const float s = __fadd_rn(sh, yh);
  const float bb = __fsub_rn(s, sh);
  const float er = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(yh, bb));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(er, yl));
}
// The same with the lows added to one another first: swapping the operands gives the same bits.
__device__ __forceinline__ void ht_add_even(float& sh, float& sl, float yh, float yl) {
  const float s = __fadd_rn(sh, yh);
  const float bb = __fsub_rn(s, sh);
  const float er = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(yh, bb));
  sh = s;
  sl = __fadd_rn(__fadd_rn(sl, yl), er);
}
// (ph, pl) = (kh + kl) (vh + vl)
__device__ __forceinline__ void ht_mul(float kh, float kl, float vh, float vl, float& ph, float& pl) {
  ph = __fmul_rn(kh, vh);
  float l = fmaf(kh, vh, -ph);
  l = fmaf(kh, vl, l);
  pl = fmaf(kl, vh, l);
}

constexpr int kScaleBits = 10;                                         // digits carry 2^10, sums 2^20
constexpr float kMagicC = 1.5f * 8388608.f / 16384.f;                  // 1.5 2^23 2^(20 - 34)
constexpr double kLn2 = 0.693147180559945309417;

struct EntryConst {
  float c1, c2;        // ln2 2^-33 as hi + lo
};

// The entry from its four cross-term sums, times the power of two with the bits `one`; ci, cj: point
// constants (see ht_prep_kernel).
__device__ __forceinline__ void ht_entry(float ga, float gb, float gc, float gd, int ni, int nj, int fi, int fj,
                                         float li, float lj, EntryConst ec, int one, const unsigned char* tab,
                                         float& kh, float& kl) {
  const int ta = __float2int_rn(ga);                       // 2 x cross term, units of 2^-19
  const int tb = __float2int_rn(gb * 16384.f);             // 2 x cross term, units of 2^-33
  const float u = __fadd_rn(gc, kMagicC);                  // gc rounded to a cross term of 2^-34
  const float lc = __fsub_rn(gc, __fsub_rn(u, kMagicC));   // the rest, exact
  const float w = fmaf(-2.f * (float)kLn2 / 1048576.f, __fadd_rn(lc, gd), __fadd_rn(li, lj));   // times ln 2
  const int J = (fi + fj - __float_as_int(u)) - tb;        // units of 2^-33
  const int T = (ni + nj - ta) + (J >> 14);                // units of 2^-19
  const float rem = __fsub_rn(__int_as_float((((T & 127) << 14) + 0x4B000000) | (J & 0x3fff)), 8388608.f);
  const float2 t = *reinterpret_cast<const float2*>(tab + ((T >> 4) & 0x7ff8));
  const float sc = __int_as_float(one - (T & (int)0xfff80000) * 16);
  // 2^-(rem 2^-33) e^-w = 1 - y, y = x + ...
  const float x = __fmul_rn(rem, ec.c1);
  float e = fmaf(rem, ec.c1, -x);
  e = fmaf(rem, ec.c2, e);
  const float om = __fsub_rn(1.f, x);
  e = fmaf(w, om, e);
  const float y = fmaf(-__fmul_rn(x, x), fmaf(x, -1.f / 6.f, 0.5f), e);
  const float z = __fmul_rn(t.x, x);
  float zl = fmaf(t.x, x, -z);
  zl = fmaf(t.x, y, zl);
  const float h = __fsub_rn(t.x, z);
  const float er = __fsub_rn(__fsub_rn(t.x, h), z);
  const float l = __fsub_rn(fmaf(t.y, om, er), zl);
  kh = __fmul_rn(h, sc);
  kl = __fmul_rn(l, sc);
}

// Sums that come out the same whatever the order of their atomics.  An addend a is cut on fixed grids:
// h1, a multiple of g1 = 2^(e0 - 52), h2 of g2, ..., each plane collecting its own.  2^e0 bounds
// sum_j |K_ij v_j| (from n max |v|), so every partial sum of the h1 is a multiple of g1 below 2^53 g1:
// exact, hence without an order.  What the first cut leaves of an addend is below g1; with 2^(la - 1) of
// them the sums of the rest stay below 2^(e2 - 1), e2 = e0 - 52 + la, and the second grid is
// g2 = 2^(e2 - 52); the later cuts leave half a step, so the grids then lie 53 - la bits apart.
// Entries go down to 2^-112, addends carry 48 bits: four planes lose nothing that the addends carry.
//
// The first cut clears mantissa bits (FP64 operations have a latency of 65 cycles, and a warp would
// wait for two more).  An addend of 2^e2 and more ends on the second grid by itself, its last bit being
// at least 2^(e2 - 52): two atomics, one FP64 subtraction.  Smaller ones, by a vote of the warp, are cut
// further.
//
// The entries are formed times 2^k, k such that max |v| 2^k comes to 2^60 (0 <= k <= 120), which costs
// nothing (it is part of the entry's exponent) and keeps entry times vector inside the FP32 range down
// to the smallest entries; the finishing kernel takes the factor out.
// Layout: planes 0 and 1 of element i at [2 i], [2 i + 1], planes 2 and 3 the same way 2 ldn further.
constexpr int kPlanes = 4;
struct OrderFree {
  int e0, e2, k, la;
  __device__ __forceinline__ OrderFree(unsigned long long vmax, int log2n, int la_) : la(la_) {
    const int field = (int)(vmax >> 52);
    const int ex = field > 0 ? field - 1022 : 0;         // max |v| < 2^ex (below 2^-1022 it is zero in FP32)
    k = min(120, max(0, 60 - ex));
    e0 = ex + k + log2n + 1;
    e2 = e0 - 52 + la;
  }
  // a rounded towards zero to a multiple of g1
  __device__ __forceinline__ double first(double a) const {
    const int t = min(63, max(0, e0 + 1023 - ((__double2hiint(a) >> 20) & 0x7ff)));
    return __longlong_as_double(__double_as_longlong(a) & (t > 52 ? 0ll : -1ll << t));
  }
  // a is zero or not below 2^e2
  __device__ __forceinline__ bool two_planes(double a) const {
    const int hi = __double2hiint(a) & 0x7fffffff;
    return hi == 0 || hi >= (e2 + 1023) << 20;
  }
  static __device__ __forceinline__ double power(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }
  // a rounded to the grid of m = 1.5 2^e; r: the rest, exact
  static __device__ __forceinline__ double cut(double a, double m, double& r) {
    const double h = __dsub_rn(__dadd_rn(a, m), m);
    r = __dsub_rn(a, h);
    return h;
  }
  // the second to fourth plane of what the first cut left; p: the element of the second
  static __device__ __noinline__ void rest(double* p, int64_t ldn, double r1, int e2, int la) {
    double r2, r3, r4;
    const double m2 = 1.5 * power(e2), step = power(la - 53);
    atomicAdd(p, cut(r1, m2, r2));
    atomicAdd(p + 2 * ldn - 1, cut(r2, m2 * step, r3));
    atomicAdd(p + 2 * ldn, cut(r3, m2 * step * step, r4));
  }
};

}  // namespace

// units[b] = {row tile I, first and end 64-column tile, partial index}.  SYM (M = 1): each unit's
// tiles start at or right of the diagonal, results into the kPlanes planes of out with atomics
// (vmax[0]: bits of max |v|, vmax[1] receives those of 2^-k; log2n, la: base-2 logarithms, rounded up, of
// n and of twice the addends of an element); else row sums over the unit's columns into
// out[partial][ldn][M].
template <int M, bool SYM, int KS>
__global__ void __launch_bounds__(kThreadsHt, 1)
    gram_rbf_high_tc_kernel(const __grid_constant__ CUtensorMap tm_i, const __grid_constant__ CUtensorMap tm_j,
                            const int4* __restrict__ cst, const float2* __restrict__ vhl,
                            const float2* __restrict__ table, const int4* __restrict__ units, double* __restrict__ out,
                            int64_t ldn, float c1, float c2, unsigned long long* __restrict__ vmax, int log2n, int la,
                            int* __restrict__ err) {
  constexpr int katoms = KS == 1 ? 2 : 4;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(base);
  const uint32_t i_bytes = (uint32_t)katoms * kIAtom, j_bytes = (uint32_t)katoms * kJAtom;
  const uint32_t off_j = i_bytes;
  const uint32_t off_cst = off_j + kStages * j_bytes;                        // int4 [stage][64]
  const uint32_t off_v = off_cst + kStages * kJCols * 16u;                   // float2 [stage][64][M]
  const uint32_t off_tab = off_v + kStages * kJCols * M * 8u;
  unsigned char* tab = base + off_tab;
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + off_tab + kTabBytes);
  uint64_t* full_i = bars;
  uint64_t* full_j = bars + 1;                  // [kStages] digits, constants and v landed
  uint64_t* stage_free = full_j + kStages;      // [kStages] all epilogue warps are done with the stage
  uint64_t* mma_done = stage_free + kStages;    // [2]
  uint64_t* tmem_free = mma_done + 2;           // [2] all epilogue warps have read the accumulators
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tmem_free + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = M == 1 ? warp_index() : tid >> 5, lane = tid & 31;
  const int4 unit = units[blockIdx.x];
  const int ti = unit.x, jt0 = unit.y, nt = unit.z - unit.y;

  if (warp == kEpiWarps) {
    ht_alloc(tmem_slot, 512);
    ht_relinquish();
  }
  if (tid == 0) {
    mbar_init(full_i, 1);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full_j[s], 1);
      mbar_init(&stage_free[s], kEpiWarps);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&mma_done[b], 1);
      mbar_init(&tmem_free[b], kEpiWarps);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  for (int e = tid; e < (1 << kTabBits); e += kThreadsHt) reinterpret_cast<float2*>(tab)[e] = table[e];
  ht_fence_before();
  __syncthreads();
  ht_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == kEpiWarps) {
    // Copies and MMAs.  M = 1: the warp stays converged, so that indexes and descriptors are uniform
    // values, and one elected lane issues (n = 50000: 3.79 ms then, 4.32 with a branch of one lane); with
    // several vectors one lane does it all, which measured faster (M = 8, n = 10007: 0.62 against 0.64).
    constexpr bool kConverged = M == 1;
    if (kConverged || lane == 0) {
      const bool elected = !kConverged || elect_one();
      auto agree = [](bool ok) { return kConverged ? (bool)__all_sync(0xffffffffu, ok) : ok; };
      auto join = []() {
        if (kConverged) __syncwarp();
      };
      auto load_j = [&](int q) {
        const int s = q % kStages;
        const int col0 = (jt0 + q) * kJCols;
        if (!elected) return;
        mbar_arrive_expect_tx(&full_j[s], j_bytes + kJCols * 16u + kJCols * M * 8u);
        for (int a = 0; a < katoms; ++a)
          tma_load_2d(base + off_j + s * j_bytes + a * kJAtom, &tm_j, a * 32, col0, &full_j[s]);
        ht_bulk(base + off_cst + s * kJCols * 16u, cst + col0, kJCols * 16u, &full_j[s]);
        ht_bulk(base + off_v + s * kJCols * M * 8u, vhl + (size_t)col0 * M, kJCols * M * 8u, &full_j[s]);
      };
      // FP32 accumulate, bf16 A and B, both K-major, N = 64, M = 128
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
      const uint64_t i_desc = ht_desc(sbase), j_desc = ht_desc(sbase + off_j);
      int loaded = 0, issued = 0;
      bool ok = true;
      if (elected) {
        mbar_arrive_expect_tx(full_i, i_bytes);
        for (int a = 0; a < katoms; ++a) tma_load_2d(base + a * kIAtom, &tm_i, a * 32, ti * 128, full_i);
      }
      for (; loaded < nt && loaded < kStages; ++loaded) load_j(loaded);
      for (int q = 0; q < nt && ok; ++q) {
        const int s = q % kStages, b = q & 1;
        if (q == 0) ok = mbar_wait_bounded(full_i, 0, err);
        if (ok) ok = mbar_wait_bounded(&full_j[s], (uint32_t)((q / kStages) & 1), err);
        if (ok && q >= 2) ok = *abort_flag == 0 && mbar_wait_bounded(&tmem_free[b], (uint32_t)(((q >> 1) - 1) & 1), err);
        ok = agree(ok);
        if (!ok) break;
        ht_fence_after();
        if (elected) {
          ht_issue_tile<KS>(tmem + (uint32_t)(b * 256), (uint32_t)i_desc, (uint32_t)j_desc + s * (j_bytes / 16u),
                            (uint32_t)(i_desc >> 32), idesc);
          ht_commit(&mma_done[b]);
        }
        join();
        issued = q + 1;
        // the stage that held tile q - 2 takes tile q + 1: waiting for a later stage here would hold the
        // next tile's MMAs back until the epilogue of tile q - 1 is over
        if (q >= 2 && loaded < nt) {
          ok = *abort_flag == 0 && mbar_wait_bounded(&stage_free[(q - 2) % kStages], (uint32_t)(((q - 2) / kStages) & 1), err);
          ok = agree(ok);
          if (ok) {
            load_j(loaded);
            ++loaded;
          }
          join();
        }
      }
      if (!ok) *abort_flag = 1;
      // The CTA does not free its tensor memory or exit with a copy or an MMA of its own in flight, also
      // when it was an epilogue warp that gave up, after the last tile was issued (bounded waits, done
      // already when nothing went wrong).
      mbar_wait_bounded(full_i, 0, err);
      for (int q = loaded > kStages ? loaded - kStages : 0; q < loaded; ++q)
        mbar_wait_bounded(&full_j[q % kStages], (uint32_t)((q / kStages) & 1), err);
      if (issued > 0) mbar_wait_bounded(&mma_done[(issued - 1) & 1], (uint32_t)(((issued - 1) >> 1) & 1), err);
    }
  } else {
    const int lq = warp & 3, cg = warp >> 2;
    const int i = ti * 128 + lq * 32 + lane;
    const int4 ci = cst[i];
    const float li = __int_as_float(ci.z);
    float2 vi = make_float2(0.f, 0.f);
    if (SYM) vi = vhl[i];
    const EntryConst ec{c1, c2};
    const OrderFree sums(SYM ? *vmax : 0ull, log2n, la);
    const int one = SYM ? 0x3F800000 + (sums.k << 23) : 0x3F800000;
    if (SYM && blockIdx.x == 0 && tid == 0) vmax[1] = (unsigned long long)(1023 - sums.k) << 52;
    float sh[M], sl[M];
#pragma unroll
    for (int m = 0; m < M; ++m) sh[m] = sl[m] = 0.f;
    const uint32_t lane_off = (uint32_t)(lq * 32) << 16;
    for (int q = 0; q < nt; ++q) {
      const int s = q % kStages, b = q & 1;
      const bool ok = __all_sync(0xffffffffu, *abort_flag == 0 &&
                                                  mbar_wait_bounded(&mma_done[b], (uint32_t)((q >> 1) & 1), err) &&
                                                  mbar_wait_bounded(&full_j[s], (uint32_t)((q / kStages) & 1), err));
      if (!ok) {
        *abort_flag = 1;
        break;
      }
      ht_fence_after();
      const int4* cj = reinterpret_cast<const int4*>(base + off_cst + s * kJCols * 16u) + cg * 16;
      const float2* vj = reinterpret_cast<const float2*>(base + off_v + s * kJCols * M * 8u) + cg * 16 * M;
      const int j0 = (jt0 + q) * kJCols + cg * 16;
      auto halves = [&](auto diag_tag) {
        constexpr bool DIAG = decltype(diag_tag)::value;
        float c0h = 0.f, c0l = 0.f;   // column sums of the first half
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          uint32_t g[4][8];
          const uint32_t tcol = tmem + (uint32_t)(b * 256 + cg * 16 + h * 8) + lane_off;
#pragma unroll
          for (int a = 0; a < 4; ++a) ht_ld8(tcol + (uint32_t)(a * 64), g[a]);
          ht_wait_ld();
          if (h == 1) {
            ht_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tmem_free[b]);
          }
          float ch[SYM ? 8 : 1], cl[SYM ? 8 : 1];
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int4 k = cj[h * 8 + c];
            float kh, kl;
            ht_entry(__uint_as_float(g[0][c]), __uint_as_float(g[1][c]), __uint_as_float(g[2][c]),
                     __uint_as_float(g[3][c]), ci.x, k.x, ci.y, k.y, li, __int_as_float(k.z), ec, one, tab, kh, kl);
            if (DIAG && j0 + h * 8 + c < i) kh = kl = 0.f;   // the entry belongs to its mirror image
#pragma unroll
            for (int m = 0; m < M; ++m) {
              const float2 v = vj[(h * 8 + c) * M + m];
              float ph, pl;
              ht_mul(kh, kl, v.x, v.y, ph, pl);
              ht_add(sh[m], sl[m], ph, pl);
            }
            if (SYM) {
              if (DIAG && j0 + h * 8 + c <= i) kh = kl = 0.f;
              ht_mul(kh, kl, vi.x, vi.y, ch[SYM ? c : 0], cl[SYM ? c : 0]);
            }
          }
          // renormalise: sl stays below an ulp of sh, so its additions round at 2^-48 of the sum
#pragma unroll
          for (int m = 0; m < M; ++m) {
            const float v = __fadd_rn(sh[m], sl[m]);
            sl[m] = __fsub_rn(sl[m], __fsub_rn(v, sh[m]));
            sh[m] = v;
          }
          if (SYM) {
            // sums over the warp's 32 rows: lane bits 4, 3, 2 select one of the 8 columns
#pragma unroll
            for (int wd = 4; wd >= 1; wd >>= 1) {
              const int o = wd * 4;
              const bool up = (lane & o) != 0;
#pragma unroll
              for (int c = 0; c < wd; ++c) {
                const float gh = __shfl_xor_sync(0xffffffffu, up ? ch[c] : ch[c + wd], o);
                const float gl = __shfl_xor_sync(0xffffffffu, up ? cl[c] : cl[c + wd], o);
                if (up) {
                  ch[c] = ch[c + wd];
                  cl[c] = cl[c + wd];
                }
                ht_add(ch[c], cl[c], gh, gl);
              }
            }
            // The first half waits for the second: lane bit 1 selects the half, bit 0 the plane, so that 16
            // columns go out in one operation of 32 lanes.  Both lanes of a pair end with the same bits.
            if (h == 0) {
              c0h = ch[0];
              c0l = cl[0];
            } else {
              const bool up = (lane & 2) != 0;
              const float gh = __shfl_xor_sync(0xffffffffu, up ? c0h : ch[0], 2);
              const float gl = __shfl_xor_sync(0xffffffffu, up ? c0l : cl[0], 2);
              float sh2 = up ? ch[0] : c0h, sl2 = up ? cl[0] : c0l;
              ht_add(sh2, sl2, gh, gl);
              ht_add_even(sh2, sl2, __shfl_xor_sync(0xffffffffu, sh2, 1), __shfl_xor_sync(0xffffffffu, sl2, 1));
              const double a = (double)sh2 + (double)sl2;
              const double h1 = sums.first(a), r1 = __dsub_rn(a, h1);
              const bool rest = (lane & 1) != 0;
              double* p = out + 2 * (j0 + (up ? 8 : 0) + (lane >> 2)) + (lane & 1);
              if (__all_sync(0xffffffffu, sums.two_planes(a)) || !rest) atomicAdd(p, rest ? r1 : h1);
              else OrderFree::rest(p, ldn, r1, sums.e2, sums.la);
            }
          }
        }
      };
      if (SYM && (jt0 + q) * kJCols < ti * 128 + 128) halves(std::true_type{});
      else halves(std::false_type{});
      __syncwarp();
      if (lane == 0) mbar_arrive(&stage_free[s]);
    }
    // the four column groups' row sums meet in shared memory (the J stages are free: every copy has
    // landed and every MMA has completed) and are added in a fixed order
    double* red = reinterpret_cast<double*>(base + off_j);   // [4][128][M]
#pragma unroll
    for (int m = 0; m < M; ++m) red[((size_t)cg * 128 + lq * 32 + lane) * M + m] = (double)sh[m] + (double)sl[m];
    asm volatile("bar.sync 1, 512;" ::: "memory");
    if (*abort_flag == 0) {
      for (int e = tid; e < 128 * M; e += kEpiWarps * 32) {
        const double v = (red[e] + red[128 * M + e]) + (red[2 * 128 * M + e] + red[3 * 128 * M + e]);
        if (SYM) {
          double* p = out + 2 * (ti * 128 + e);
          const double h1 = sums.first(v);
          const double r1 = __dsub_rn(v, h1);
          atomicAdd(p, h1);
          if (sums.two_planes(v)) atomicAdd(p + 1, r1);
          else OrderFree::rest(p + 1, ldn, r1, sums.e2, sums.la);
        } else out[((size_t)unit.w * ldn + ti * 128) * M + e] = v;
      }
    }
  }
  ht_fence_before();
  __syncthreads();
  ht_fence_after();
  if (warp == kEpiWarps) ht_dealloc(tmem, 512);
}

// Digits (row-major [ldn][W] bf16, digit s of feature k at s * kf + k) and point constants:
// |x|^2 of the rounded coordinates = x 2^-19 + y 2^-33 + z / ln 2 with int x, int y (plus the
// magic constant's bits, which the epilogue subtracts) and float z.  nmax: bits of the largest norm.
__global__ void ht_prep_kernel(const double* __restrict__ xc, int64_t ldn, int p, double scale, int kf, int W,
                               __nv_bfloat16* __restrict__ dig, int4* __restrict__ cst, unsigned int* __restrict__ nmax) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ldn; i += (int64_t)gridDim.x * blockDim.x) {
    double nh = 0.0, nl = 0.0;
    __nv_bfloat16* row = dig + (size_t)i * W;
    for (int k = 0; k < kf; ++k) {
      double xs = k < p ? scale * xc[(size_t)k * ldn + i] : 0.0;
      xs = fmin(fmax(xs, -7.9), 7.9);   // such a point's norm rules this layout out anyway
      const double Hd = rint(ldexp(xs, kFracBits));
      long long H = (long long)Hd;
      const double x = ldexp(Hd, -kFracBits);
      const double sq = x * x, sqe = fma(x, x, -sq);
      const double s = nh + sq, bb = s - nh;
      nl += ((nh - (s - bb)) + (sq - bb)) + sqe;
      nh = s;
      for (int d = 0; d < kDigits; ++d) {
        long long v = H;
        if (d < kDigits - 1) {
          v = ((H + 256) & 511) - 256;
          H = (H - v) >> kDigitBits;
        }
        row[d * kf + k] = __float2bfloat16_rn((float)ldexp((double)v, kDigitBits * d - kFracBits + kScaleBits));
      }
    }
    for (int e = kDigits * kf; e < W; ++e) row[e] = __float2bfloat16_rn(0.f);
    const double tot = nh + nl;
    atomicMax(nmax, __float_as_uint((float)tot));
    double hi = floor(ldexp(nh, 19));
    double r = (nh - ldexp(hi, -19)) + nl;                 // [-2^-52, 2^-19)
    const double mid = floor(ldexp(r, 33));
    r -= ldexp(mid, -33);
    cst[i] = make_int4((int)hi, (int)mid + (__float_as_int(kMagicC) >> 1), __float_as_int((float)(r * kLn2)), 0);
  }
}

// V (n x m) -> (hi, lo) floats [ldn][M], zero padded.  One vector: the planes of the sums zeroed, and
// the bits of max |v| into *vmax (zero before; NaN orders above all).
__global__ void __launch_bounds__(256) ht_split_kernel(const double* __restrict__ V, float2* __restrict__ out,
                                                       double* __restrict__ acc, int64_t n, int64_t ldn, int m, int M,
                                                       unsigned long long* __restrict__ vmax) {
  unsigned long long mx = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ldn * M; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / M;
    const int c = (int)(e % M);
    const double x = (i < n && c < m) ? V[i * m + c] : 0.0;
    const float hi = (float)x;
    out[e] = make_float2(hi, (float)(x - (double)hi));
    if (acc) {
#pragma unroll
      for (int k = 0; k < kPlanes; ++k) acc[k * ldn + i] = 0.0;
      mx = max(mx, (unsigned long long)__double_as_longlong(fabs(x)));
    }
  }
  if (!acc) return;
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(vmax, mx);
}

// out[i][c] = sum over the partials.  One vector (vmax not null): they are the planes, added from the
// finest on, times vmax[1]; vmax[0] goes back to zero for the next product.
__global__ void ht_finish_kernel(const double* __restrict__ part, int parts, int64_t ldn, int M, int m, int64_t n,
                                 double* __restrict__ out, unsigned long long* __restrict__ vmax) {
  if (vmax && blockIdx.x == 0 && threadIdx.x == 0) *vmax = 0ull;
  const double unscale = vmax ? __longlong_as_double((long long)vmax[1]) : 1.0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * m; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / m;
    const int c = (int)(e % m);
    double s = 0.0;
    if (vmax) s = ((part[2 * (ldn + i) + 1] + part[2 * (ldn + i)]) + part[2 * i + 1]) + part[2 * i];
    else
      for (int q = 0; q < parts; ++q) s += part[((size_t)q * ldn + i) * M + c];
    out[e] = s * unscale;
  }
}

bool make_tmap_2d_f32_sw128(CUtensorMap* tm, void* base, int64_t inner, int64_t outer, int64_t row_bytes,
                            int box_inner, int box_outer);

// Once per problem; h->ht_state: 0 not prepared, 1 ready, -1 this problem keeps the CUDA-core kernels
// (norms too large, or no memory for the digits: 256 or 512 bytes a row that those kernels do without).
static cudaError_t ht_prepare(Handle* h) {
  if (h->ht_state) return cudaSuccess;
  const int kf = h->p <= 16 ? 16 : 32;
  const int W = kf == 16 ? 128 : 256;   // whole 128-byte atoms of 64 bf16
  cudaStream_t st = h->stream;
  h->ht_dig = dev_alloc(h, (size_t)h->ldn * W * 2);
  h->ht_cst = (int4*)dev_alloc(h, (size_t)h->ldn * sizeof(int4));
  h->ht_table = (float2*)dev_alloc(h, kTabBytes);
  unsigned int* nmax = (unsigned int*)dev_alloc(h, 16);
  cudaError_t e = cudaSuccess;
  if (!h->ht_dig || !h->ht_cst || !h->ht_table || !nmax) e = cudaErrorMemoryAllocation;
  unsigned int bits = 0;
  if (e == cudaSuccess) {
    std::vector<float2> tab(1 << kTabBits);
    for (int k = 0; k < (1 << kTabBits); ++k) {
      const double t = std::exp2(-(double)k / (double)(1 << kTabBits));
      const float hi = (float)t;
      tab[k] = make_float2(hi, (float)(t - (double)hi));
    }
    e = cudaMemcpyAsync(h->ht_table, tab.data(), kTabBytes, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(nmax, 0, 4, st);
    if (e == cudaSuccess) {
      ht_prep_kernel<<<grid_for(h->ldn, 64), 64, 0, st>>>(h->xc64, h->ldn, (int)h->p, std::sqrt(h->gamma / std::log(2.0)),
                                                         kf, W, (__nv_bfloat16*)h->ht_dig, h->ht_cst, nmax);
      h->launches++;
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bits, nmax, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  dev_free(h, nmax);
  float mx;
  static_assert(sizeof(mx) == sizeof(bits), "");
  memcpy(&mx, &bits, 4);
  bool usable = e == cudaSuccess && mx < kMaxNorm;
  if (usable && (!make_tmap_2d_f32_sw128(&h->tm_ht_i, h->ht_dig, W / 2, h->ldn, (int64_t)W * 2, 32, 128) ||
                 !make_tmap_2d_f32_sw128(&h->tm_ht_j, h->ht_dig, W / 2, h->ldn, (int64_t)W * 2, 32, kJCols)))
    usable = false;
  if (!usable) {
    dev_free(h, h->ht_dig);
    dev_free(h, h->ht_cst);
    dev_free(h, h->ht_table);
    h->ht_dig = nullptr;
    h->ht_cst = nullptr;
    h->ht_table = nullptr;
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      e = cudaSuccess;
    }
    if (e == cudaSuccess) h->ht_state = -1;
    return e;
  }
  h->ht_state = 1;
  return cudaSuccess;
}

// The work list of the one-vector (sym) or of the several-vector products, made at its first use.
static cudaError_t ht_units(Handle* h, bool sym, cudaStream_t st) {
  Handle::HtWork& w = h->ht_work[sym ? 0 : 1];
  if (w.units) return cudaSuccess;
  const int T = (int)(h->ldn / kTile);
  const HtList l = sym ? ht_list_symmetric(T, h->num_sms) : ht_list_rows(T, h->num_sms);
  static_assert(sizeof(HtUnit) == sizeof(int4), "the kernel reads a unit as an int4");
  w.n = (int)l.units.size();
  w.parts = l.parts;
  return dev_upload(h, l.units.data(), l.units.size() * sizeof(int4), st, reinterpret_cast<void**>(&w.units));
}

static size_t ht_smem(int katoms, int M) {
  return 1024 + (size_t)katoms * kIAtom + (size_t)kStages * (katoms * kJAtom + kJCols * 16 + kJCols * M * 8) + kTabBytes +
         (1 + 2 * kStages + 4) * 8 + 16;
}

static unsigned long long* ht_vmax(Handle* h) { return reinterpret_cast<unsigned long long*>(h->scal + S_HTMAX); }

static int log2_up(int64_t x) {
  int k = 0;
  while (((int64_t)1 << k) < x) ++k;
  return k;
}

// Addends that an element of the one-vector sums gets at most: four warps' column sums from every row
// tile above, and one from each unit of its own row tile (at most one per column tile).
static int64_t ht_addends(const Handle* h) { return 6 * (h->ldn / kTile) + 8; }

template <int M, bool SYM>
static cudaError_t ht_launch(Handle* h, const float2* vhl, double* out, cudaStream_t st) {
  const size_t smem = ht_smem(h->p <= 16 ? 2 : 4, M);
  auto kern = h->p <= 16 ? gram_rbf_high_tc_kernel<M, SYM, 1> : gram_rbf_high_tc_kernel<M, SYM, 2>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const double c = kLn2 * std::ldexp(1.0, -33);
  const float c1 = (float)c, c2 = (float)(c - (double)c1);
  const Handle::HtWork& w = h->ht_work[SYM ? 0 : 1];
  prof_mark(h, 1, true, st);
  kern<<<w.n, kThreadsHt, smem, st>>>(h->tm_ht_i, h->tm_ht_j, h->ht_cst, vhl, h->ht_table, w.units, out, h->ldn, c1, c2,
                                      SYM ? ht_vmax(h) : nullptr, log2_up(h->n), log2_up(2 * ht_addends(h)), h->err_flag);
  prof_mark(h, 1, false, st);
  h->launches++;
  return cudaGetLastError();
}

static cudaError_t ht_buffer(Handle* h, float** buf, size_t* cap, size_t bytes) {
  if (*cap >= bytes) return cudaSuccess;
  dev_free(h, *buf);
  *buf = (float*)dev_alloc(h, bytes);
  *cap = *buf ? bytes : 0;
  return *buf ? cudaSuccess : cudaErrorMemoryAllocation;
}

// Scratch of the product of m vectors: the FP32 pairs of V (and, for one vector, the sums) in v32, the
// partial sums of several in part.
static cudaError_t ht_scratch(Handle* h, int m, int M, cudaStream_t st) {
  const bool sym = m == 1;
  cudaError_t e = ht_units(h, sym, st);
  if (e != cudaSuccess) return e;
  const size_t vbytes = (size_t)h->ldn * M * sizeof(float2) + (sym ? (size_t)kPlanes * h->ldn * sizeof(double) : 0);
  if ((e = ht_buffer(h, &h->v32, &h->v32_cap, vbytes)) != cudaSuccess || sym) return e;
  return ht_buffer(h, &h->part, &h->part_cap, (size_t)h->ht_work[1].parts * h->ldn * M * sizeof(double));
}

static int ht_columns(int m) { return m <= 1 ? 1 : (m <= 2 ? 2 : (m <= 4 ? 4 : 8)); }

// Whether the tensor-core product of m vectors serves this problem: RBF, p <= 32, norms below 28
// (kernel values against the data's mean above 2^-28), options.symmetric_gram and rbf_tensor_cores on,
// and memory for its layout and scratch, which are made here.  Anything else keeps the CUDA-core
// kernels of gram_high.cu, which need less memory.
cudaError_t high_tc_ready(Handle* h, int m, cudaStream_t st, bool* ready) {
  *ready = false;
  if (h->kind != KQR_RBF || h->p > 32 || !h->opt.symmetric_gram || !h->opt.rbf_tensor_cores) return cudaSuccess;
  cudaError_t e = ht_prepare(h);
  if (e != cudaSuccess || h->ht_state < 0) return e;
  e = ht_scratch(h, m, ht_columns(m), st);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return cudaSuccess;
  }
  *ready = e == cudaSuccess;
  return e;
}

// After high_tc_ready(h, m, ...) said so.
cudaError_t gram_high_tc(Handle* h, const double* V, double* U, int m, cudaStream_t st) {
  const bool sym = m == 1;
  const int M = ht_columns(m), parts = h->ht_work[sym ? 0 : 1].parts;
  cudaError_t e;
  float2* vhl = reinterpret_cast<float2*>(h->v32);
  double* acc = sym ? reinterpret_cast<double*>(vhl + h->ldn * M) : reinterpret_cast<double*>(h->part);
  ht_split_kernel<<<grid_for(h->ldn * M), 256, 0, st>>>(V, vhl, sym ? acc : nullptr, h->n, h->ldn, m, M,
                                                         sym ? ht_vmax(h) : nullptr);
  h->launches++;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  switch (M) {
    case 1: e = ht_launch<1, true>(h, vhl, acc, st); break;
    case 2: e = ht_launch<2, false>(h, vhl, acc, st); break;
    case 4: e = ht_launch<4, false>(h, vhl, acc, st); break;
    default: e = ht_launch<8, false>(h, vhl, acc, st); break;
  }
  if (e != cudaSuccess) return e;
  ht_finish_kernel<<<grid_for(h->n * m), 256, 0, st>>>(acc, parts, h->ldn, M, m, h->n, U, sym ? ht_vmax(h) : nullptr);
  h->launches++;
  return cudaGetLastError();
}

void high_tc_free(Handle* h) {
  dev_free(h, h->ht_dig);
  dev_free(h, h->ht_cst);
  dev_free(h, h->ht_table);
  for (Handle::HtWork& w : h->ht_work) dev_free(h, w.units);
}

}  // namespace kqr
