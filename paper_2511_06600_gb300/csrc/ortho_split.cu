// FP64 Gram matrix and triangular apply of CholQR2 (Algorithm 1 step 4) on the
// tensor cores, by error-free splitting (Ozaki, Ogita, Oishi and Rump 2012):
// every FP64 value is written as a sum of 7-bit signed digits on a common
// scale, the digits' products are summed exactly by BF16 MMAs with FP32
// accumulators, and the digit levels are put together in integers.
//
// Why: FP64 arithmetic runs at 2 multiply-adds per clock and SM on this chip
// (0.63 T/s in all), 1/2000 of the BF16 tensor rate.  The Gram matrix needs
// n K^2 / 2 multiply-adds and the apply as many: 50,851 rows of K = 160 took
// 1.63 and 2.73 ms per pass with FP64 instructions, both bound by that pipe.
// A product of two 53-bit numbers takes 43 (Gram, 8 digits) or 45 (apply, 9
// digits) digit products, which the tensor cores do in a few per cent of that:
// 0.19 and 0.27 ms now, bound by writing the digits.  Against 113-bit
// arithmetic Q's error per unit column is 0.35 to 0.7 of the FP64 kernels'
// (0.95e-16 for 2.1e-16 on a Krylov basis of 9,999 x 64).
//
// Digits.  A column of scale 2^E (|x| < 2^E for all its entries, from the
// largest exponent in it) has x = 2^(E - 6) sum_j d_j 2^(-7j), |d_j| <= 64,
// j < D, rounded to nearest at the last digit: 55 bits below 2^E with D = 8,
// 62 with D = 9.  A digit times a power of two is exact in BF16, a product of
// digits is at most 2^12, and a sum of N (g + 1) products of level g = i + j
// stays below 2^24 units, where FP32 sums are exact, for N (g + 1) <= 4096.
//  - Gram: rows are summed in windows of 512, so levels 0..6 are exact; level 8
//    joins level 7 (its products d_4 d_4 are positive on the diagonal, and
//    leaving the level out costs 2^-57 (max / rms)^2 of a column's squared
//    norm: 1.6e-14 where an entry is 48 times the rms).  A window leaves TMEM
//    as two 64-bit integers per entry, which add up exactly over windows and
//    CTAs, so the result does not depend on the grid.  The error, 2^-56 of the
//    columns' scales per row and so 2^-55 of their norms, is that of the
//    triangular factor: it multiplies the rows of Q, and their differences,
//    from the right.
//  - apply: K <= 512 products per entry; levels 0..5 exact in six accumulators,
//    levels 6..8 (weights 2^-42 and less) in a seventh, whose FP32 rounding is
//    2^-66 of the scale.  Rows of V are scaled too, by the power of two that
//    brings their largest entry (in units of its column's scale) to 2^0: a row is
//    as accurate as any other, however small it is beside the columns' largest
//    (62 bits of its largest entry; an error of 2^-60 of the row, where the
//    rounding of R^-1 leaves 2^-53 of it).  The mean is subtracted in the same
//    integers, before the one rounding to FP64.  Within a row, an output below
//    2^-20 of its scale (the largest that |V| |R^-1| can be there), which would
//    keep less than 40 bits, is formed again by FP64 multiply-adds, unless one of
//    its products reaches that line by itself, so that FP64 would round at it as
//    well.  On Krylov bases that is one output in 10^5 (at 2^-11 one in 100 and 80
//    us at 50,851 x 160, for accuracy that the rounding of R^-1 hides).  Rows'
//    scales, the exact means and this line took the apply there from 221 us per
//    pass to 270.
// An entry that is not finite makes its column's mean and its Gram row and
// column NaN (the column is then dropped by the elimination) and, as with FP64
// arithmetic, whose products with the mean-free column are NaN in every row, all
// rows of the output NaN from the 64-column block on that reads the column.
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>

#include "internal.h"
#include "umma.cuh"

namespace hef {

namespace {

using namespace umma;

constexpr int kSpThreads = 512;   // converter (and epilogue) threads: 16 warps
constexpr int kSpConv = kSpThreads / 32;
constexpr int kSpHalf = 32;       // rows (Gram) or basis values (apply) per stage
constexpr int kSpWindow = 512;    // Gram: rows summed before the accumulators are drained
constexpr int kSpN = 64;          // output columns per job: 8 levels x 64 = the 512 TMEM columns
constexpr int kGD = 8, kAD = 9;   // digits: Gram, apply
constexpr int kAExact = 6;        // apply: levels with an accumulator of their own
constexpr uint32_t kSpWait = 1u << 20;
constexpr int kNotFinite = 0x7ff;

// D[tmem] (+)= A B^T over 16 values, kind::f16 with BF16 inputs (K-major).
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// K-major operand of 32 BF16 values per row in the 64-byte swizzle: rows 64 B
// apart, 8-row groups 512 B apart, 16-byte chunk c of row r at c ^ ((r / 2) % 4).
__device__ __forceinline__ uint64_t desc_k_sw64(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1u << 16) | ((uint64_t)(512u >> 4) << 32) |
         ((uint64_t)1u << 46) | ((uint64_t)4u << 61);
}
__device__ __forceinline__ uint32_t sw64_offset(int row, int chunk) {
  return (uint32_t)(row * 64 + ((chunk ^ ((row >> 1) & 3)) * 16));
}

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

template <int D>
struct Digits {
  static constexpr int kShift = 7 * D - 54;  // 53-bit mantissa -> 7 D - 1 bits
  static constexpr uint64_t kBias =
      64ull * ((D == 9 ? 0x7fffffffffffffffull : (1ull << (7 * D)) - 1) / 127ull);
};

// round(x 2^(7D - 1 - E)) plus 64 in every digit, for the FP64 bits `b` of x
// and the scale as the difference `d` >= 0 between the scale's exponent field
// and x's own (x's field taken as 1 when it is 0).
template <int D>
__device__ __forceinline__ uint64_t biased_int(uint64_t b, int scale_field) {
  const int f = (int)(b >> 52) & 0x7ff;
  const uint64_t mant = (b & 0xfffffffffffffull) | (f ? 1ull << 52 : 0ull);
  const int d = min(scale_field - max(f, 1), 63);
  const uint64_t x = (((mant << (Digits<D>::kShift + 1)) >> d) + 1) >> 1;
  const uint64_t s = (uint64_t)((int64_t)b >> 63);
  return ((x ^ s) - s) + Digits<D>::kBias;
}

// Digit j (0 = most significant) of two values times 2^(-7 j), as packed BF16:
// 128 + (d + 64) is 0x4300 | (d + 64) in BF16.
template <int D>
__device__ __forceinline__ uint32_t digit_pair(uint64_t a, uint64_t b, int j) {
  const int s = 7 * (D - 1 - j);
  const uint32_t m = j == 0 ? 0xffu : 0x7fu;  // the top digit reaches 128
  const uint32_t w = 0x43004300u | ((uint32_t)(a >> s) & m) | (((uint32_t)(b >> s) & m) << 16);
  const int e = 7 * j;
  const uint32_t one = (uint32_t)(127 - e) << 7, off = 0x8000u | ((uint32_t)(134 - e) << 7) | 0x40u;
  const uint32_t one2 = one | (one << 16), off2 = off | (off << 16);
  const __nv_bfloat162 r = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&w),
                                   *reinterpret_cast<const __nv_bfloat162*>(&one2),
                                   *reinterpret_cast<const __nv_bfloat162*>(&off2));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// Largest exponent field of every column (exps: K ints, zero on entry).  Bound
// by the read of V: a row's values by consecutive threads.
constexpr int kExpRows = 8;  // rows a thread loads at once
__global__ void __launch_bounds__(512) k_col_exps(const double* __restrict__ V, long long ldv, int n,
                                                  int K, int* __restrict__ exps) {
  __shared__ int sm[512];
  const int rpi = 512 / K;  // rows per round (K <= 512)
  const int c = threadIdx.x % K, r = threadIdx.x / K;
  sm[threadIdx.x] = 0;
  __syncthreads();
  if (r < rpi) {
    uint32_t best = 0;
    for (long long row = (long long)blockIdx.x * rpi * kExpRows + r; row < n;
         row += (long long)gridDim.x * rpi * kExpRows) {
      uint32_t h[kExpRows];
#pragma unroll
      for (int u = 0; u < kExpRows; ++u) {
        const long long q = row + (long long)u * rpi;
        h[u] = q < n ? (uint32_t)__double2hiint(__ldg(V + q * ldv + c)) & 0x7fffffffu : 0u;
      }
#pragma unroll
      for (int u = 0; u < kExpRows; ++u) best = max(best, h[u]);
    }
    atomicMax(&sm[c], (int)(best >> 20));
  }
  __syncthreads();
  if (threadIdx.x < K && sm[threadIdx.x] > 0) atomicMax(exps + threadIdx.x, sm[threadIdx.x]);
}

// ---------------------------------------------------------------- Gram

struct GramSplitArgs {
  const double* V;
  long long ldv;
  int n, K, Kc;       // Kc: columns of the partials (K and the ones column, padded)
  int rows_per_cta;   // a multiple of 64
  const int* exps;
  long long* hi;      // chunks x K x Kc: levels 0-3, units 2^-33 of the scales
  long long* lo;      // levels 4-7, units 2^-61
  int* err;
};

// Column blocks of the upper triangle: row block bi (128 basis columns) with
// column blocks bj (64) from 2 bi on.
__device__ __forceinline__ void gram_job(int job, int nbj, int& bi, int& bj) {
  bi = 0;
  while (job >= nbj - 2 * bi) job -= nbj - 2 * bi, ++bi;
  bj = 2 * bi + job;
}

// One CTA: rows [r0, r1) of its chunk, one job: columns [128 bi, +128) against
// [64 bj, +64).  Per stage of 32 rows the 16 converter warps turn 8 rows of a
// column per thread into its 8 digits, one 16-byte store each into the digit's
// K-major tile (a quarter warp meets eight distinct bank groups); the 17th
// warp's thread issues, per 16 rows and A digit i, the MMAs against the stacked
// B digits 0..7-i, whose accumulators (levels i..7) are contiguous too (12 MMAs
// of up to 256 columns instead of 36), and the seven products of level 8.  Two
// stages (the halves of 128-byte rows), handed over by mbarriers.  Conversion,
// about 60 integer operations per value, is repeated by the jobs that share a
// column; it and the MMAs (1.4 us per stage) bound the kernel.
__global__ void __launch_bounds__(kSpThreads + 32, 1) k_gram_split(GramSplitArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t conv[2], empty[2], drained;
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nbj = (a.K + kSpN) / kSpN;  // blocks of the K + 1 columns
  int bi, bj;
  gram_job(blockIdx.y, nbj, bi, bj);
  const int i0 = 128 * bi, j0 = kSpN * bj;
  const int Nj = min(kSpN, (a.K + 1 - j0 + 15) & ~15);
  const bool within = bj <= 2 * bi + 1;  // B's columns are among A's
  constexpr uint32_t a_tile = 128u * 128u;
  const uint32_t b_tile = (uint32_t)Nj * 128u;
  unsigned char* At = base;
  unsigned char* Bt = base + kGD * a_tile;
  if (warp == 0) tmem_alloc(&tmem_slot, 512);
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) mbar_init(&conv[q], kSpConv), mbar_init(&empty[q], 1);
    mbar_init(&drained, kSpConv);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // columns past the basis: zero once
  for (uint32_t e = tid; e < (kGD * (a_tile + b_tile)) / 16; e += blockDim.x)
    reinterpret_cast<uint4*>(base)[e] = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const long long r0 = (long long)blockIdx.x * a.rows_per_cta;
  const long long r1 = min((long long)a.n, r0 + a.rows_per_cta);
  const int nhalf = r1 > r0 ? (int)((r1 - r0 + kSpHalf - 1) / kSpHalf) : 0;
  constexpr int kWin = kSpWindow / kSpHalf;  // stages per window
  bool ok = true;
  // stage h uses half h % 2 for the (h / 2)-th time; window h / kWin
  if (warp == kSpConv) {
    if (lane == 0) {
      int h = 0;
      for (; h < nhalf; ++h) {
        const int s = h & 1;
        const bool first = h % kWin == 0;
        if (first && h > 0 && !(ok = mbar_wait(&drained, (uint32_t)(h / kWin - 1) & 1u, kSpWait))) break;
        if (!(ok = mbar_wait(&conv[s], (uint32_t)(h >> 1) & 1u, kSpWait))) break;
        tc_fence_after();
        const uint32_t id1 = idesc_bf16(128, Nj), id256 = idesc_bf16(128, 256);
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          const uint32_t ko = (uint32_t)(4 * s + 2 * ks) * 16u;
          const uint64_t dA = desc_k_sw128(smem_u32(At) + ko), dB = desc_k_sw128(smem_u32(Bt) + ko);
#pragma unroll
          for (int i = 0; i < kGD; ++i) {
            const uint64_t da = dA + (uint64_t)((i * a_tile) >> 4);
            const uint32_t acc = (first && ks == 0 && i == 0) ? 0u : 1u;
            const uint32_t d = tmem + (uint32_t)(Nj * i);
            const int width = Nj * (kGD - i);
            if (width > 256) {
              mma_bf16(d, da, dB, id256, acc);
              mma_bf16(d + 256u, da, dB + (256u * 128u >> 4), idesc_bf16(128, width - 256), acc);
            } else {
              mma_bf16(d, da, dB, idesc_bf16(128, width), acc);
            }
            if (i > 0)  // level 8
              mma_bf16(tmem + (uint32_t)(Nj * (kGD - 1)), da, dB + ((uint32_t)(kGD - i) * b_tile >> 4), id1, 1u);
          }
        }
        mma_commit(&empty[s]);
      }
      // MMAs in flight finish before TMEM may be released
      for (int q = max(0, h - 2); q < h; ++q) mbar_wait(&empty[q & 1], (uint32_t)(q >> 1) & 1u, kSpWait);
    }
  } else {
    // this thread's column of A and of B (when B is not within A), row octets
    const int oct = tid >> 7, ca = tid & 127, cb = tid & 63, octb = (tid >> 6) & 3;
    const int colA = i0 + ca, colB = j0 + cb;
    const bool doA = colA < a.K;
    const bool doB = !within && tid < 256 && cb < Nj && colB < a.K;
    const bool ones = tid < 256 && cb < Nj && colB == a.K;
    const int sa = doA ? max(a.exps[colA], 1) : 1, sb = doB ? max(a.exps[colB], 1) : 1;
    const int inb = colA - j0;  // A's column as a column of B
    const bool toB = within && doA && inb >= 0 && inb < Nj;
    auto off128 = [](int row, int chunk) {  // 128-byte swizzle
      return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((chunk ^ (row & 7)) * 16));
    };
    uint64_t xa[8], xb[8];
    const double* pa = a.V + (r0 + 8 * oct) * a.ldv + colA;
    const double* pb = a.V + (r0 + 8 * octb) * a.ldv + colB;
    auto load = [&](int h) {
      const int left = (int)(r1 - r0) - h * kSpHalf;  // rows left at this stage
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        xa[u] = doA && 8 * oct + u < left ? (uint64_t)__double_as_longlong(__ldg(pa + u * a.ldv)) : 0ull;
        xb[u] = doB && 8 * octb + u < left ? (uint64_t)__double_as_longlong(__ldg(pb + u * a.ldv)) : 0ull;
      }
      pa += kSpHalf * a.ldv;
      pb += kSpHalf * a.ldv;
    };
    if (nhalf > 0) load(0);
    for (int h = 0; h < nhalf; ++h) {
      const int s = h & 1;
      if (h >= 2) ok = mbar_wait(&empty[s], (uint32_t)((h >> 1) - 1) & 1u, kSpWait);
      if (!(ok = __all_sync(0xffffffffu, ok))) break;
      if (doA) {
#pragma unroll
        for (int u = 0; u < 8; ++u) xa[u] = biased_int<kGD>(xa[u], sa);
        unsigned char* wa = At + off128(ca, 4 * s + oct);
        unsigned char* wb = Bt + off128(toB ? inb : 0, 4 * s + oct);
#pragma unroll
        for (int j = 0; j < kGD; ++j) {
          uint4 w;
          w.x = digit_pair<kGD>(xa[0], xa[1], j);
          w.y = digit_pair<kGD>(xa[2], xa[3], j);
          w.z = digit_pair<kGD>(xa[4], xa[5], j);
          w.w = digit_pair<kGD>(xa[6], xa[7], j);
          *reinterpret_cast<uint4*>(wa + j * a_tile) = w;
          if (toB) *reinterpret_cast<uint4*>(wb + j * b_tile) = w;
        }
      }
      if (doB) {
#pragma unroll
        for (int u = 0; u < 8; ++u) xb[u] = biased_int<kGD>(xb[u], sb);
        unsigned char* wb = Bt + off128(cb, 4 * s + octb);
#pragma unroll
        for (int j = 0; j < kGD; ++j) {
          uint4 w;
          w.x = digit_pair<kGD>(xb[0], xb[1], j);
          w.y = digit_pair<kGD>(xb[2], xb[3], j);
          w.z = digit_pair<kGD>(xb[4], xb[5], j);
          w.w = digit_pair<kGD>(xb[6], xb[7], j);
          *reinterpret_cast<uint4*>(wb + j * b_tile) = w;
        }
      }
      if (ones) {  // 1 = 64 2^(-6): top digit 64 (0x4280) on this chunk's rows, scale 2^0
        const int left = (int)(r1 - r0) - h * kSpHalf - 8 * octb;
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          w[u] = (2 * u < left ? 0x4280u : 0u) | (2 * u + 1 < left ? 0x42800000u : 0u);
        *reinterpret_cast<uint4*>(Bt + off128(cb, 4 * s + octb)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&conv[s]);
      if (h + 1 < nhalf) load(h + 1);
      if (h + 1 < nhalf && (h + 1) % kWin != 0) continue;
      // drain the window: every MMA done (the commit covers the earlier ones),
      // then TMEM -> integers -> this chunk's partial sums
      ok = mbar_wait(&empty[s], (uint32_t)(h >> 1) & 1u, kSpWait);
      if (!(ok = __all_sync(0xffffffffu, ok))) break;
      tc_fence_after();
      const bool start = h < kWin;
      const int i = i0 + (warp & 3) * 32 + lane;
      for (int c8 = warp >> 2; c8 < Nj / 8; c8 += kSpConv / 4) {
        // level g holds multiples of 2^(-7 g) (the last one after rounding);
        // four levels at a time, within the registers of 17 warps
        const bool use = i < a.K && j0 + c8 * 8 + 7 >= i;
        const size_t at = ((size_t)blockIdx.x * a.K + i) * a.Kc + j0 + c8 * 8;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          float L[4][8];
#pragma unroll
          for (int g = 0; g < 4; ++g)
            tmem_ld8(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((4 * half + g) * Nj + c8 * 8), L[g]);
          tmem_wait_ld();
          long long* out = (half ? a.lo : a.hi) + at;
          if (use) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              long long v = 0;
#pragma unroll
              for (int g = 0; g < 4; ++g)
                v = v * 128 + __float2int_rn(L[g][u] * (float)(1ull << (7 * (4 * half + g))));
              out[u] = start ? v : out[u] + v;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&drained);
    }
  }
  if (!ok) atomicExch(a.err, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// G (K x K, FP64) and c (K): the chunks' integers summed (exactly, so in any
// order), then rounded to FP64 (each half, where it passes 2^53, and their sum)
// and put on the columns' scales.
__global__ void __launch_bounds__(256) k_gram_split_reduce(const long long* __restrict__ hi,
                                                           const long long* __restrict__ lo, int K,
                                                           int Kc, int nchunk,
                                                           const int* __restrict__ exps, double* G,
                                                           double* c) {
  __shared__ long long red[2][8][32];
  const int e = threadIdx.x & 31, sub = threadIdx.x >> 5;
  const long long total = (long long)K * (K + 1);
  const size_t stride = (size_t)K * Kc;
  for (long long base = (long long)blockIdx.x * 32; base < total; base += (long long)gridDim.x * 32) {
    const long long idx = base + e;
    const int i = (int)(idx / (K + 1)), j = (int)(idx % (K + 1));
    const bool act = idx < total && i <= j;
    long long h = 0, l = 0;
    if (act) {
      const size_t at = (size_t)i * Kc + j;
#pragma unroll 4
      for (int q = sub; q < nchunk; q += 8) {
        h += __ldcg(hi + at + q * stride);
        l += __ldcg(lo + at + q * stride);
      }
    }
    red[0][sub][e] = h;
    red[1][sub][e] = l;
    __syncthreads();
    if (sub == 0 && act) {
#pragma unroll
      for (int u = 1; u < 8; ++u) h += red[0][u][e], l += red[1][u][e];
      const int fi = exps[i], fj = j < K ? exps[j] : 1022;  // ones: scale 2^0
      double v = fma((double)h, 268435456.0, (double)l);
      v = scalbn(v, max(fi, 1) + max(fj, 1) - 2 * 1022 - 61);
      if (fi == kNotFinite || fj == kNotFinite) v = __longlong_as_double(0x7ff8000000000000ll);
      if (j < K) {
        G[(size_t)i * K + j] = v;
        G[(size_t)j * K + i] = v;
      } else {
        c[i] = v;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- apply

// Stages (32 basis values) that feed output block J: R^-1 is upper triangular.
__host__ __device__ __forceinline__ int split_stages(int J, int K) {
  const int last = kSpN * (J + 1) < K ? kSpN * (J + 1) : K;
  return (last + kSpHalf - 1) / kSpHalf;
}
__host__ __device__ __forceinline__ int split_width(int J, int K) {
  const int left = K - kSpN * J;
  return left >= kSpN ? kSpN : (left + 15) & ~15;
}
// Bytes of the B image before block J: per stage, 9 digit tiles of width(J)
// rows of 64 bytes.
__host__ __device__ __forceinline__ size_t split_image(int J, int K) {
  size_t b = 0;
  for (int q = 0; q < J; ++q) b += (size_t)split_stages(q, K) * kAD * split_width(q, K) * 64;
  return b;
}

// What an output column needs besides its digits: its values are
// (sum - mean) 2^exp with the sum in units of level 5 and the mean of the
// column m = (mu^T R^-1)_j split into an integer and a remainder of those units.
// tag = 64 exp + the number of bits of |mean|, or kNanCol: a column that the
// output's block reads has no finite mean.
struct __align__(32) SplitCol {
  long long mean;
  float mean_lo;
  int tag;
  double m;
};
constexpr int kNanCol = INT_MIN;
constexpr int kColExp0 = -2 * 1022 - 12 - 7 * (kAExact - 1);  // exp of a column of R^-1 of scale 2^0
// Columns below 2^(kTinyField - 1022): their squares underflow, so the
// elimination has dropped them and R^-1 does not read them.
constexpr int kTinyField = 256;
constexpr int kWeakBits = 27;  // 2^-20 of the scale in units of level 5

// The B operand's digits, laid out as the apply's stages take them: column j of
// diag(2^E) R^-1 (the columns' scales moved into R^-1) on its own scale 2^F.
// A warp per column.
__global__ void k_split_rinv(const double* __restrict__ Rinv, const double* __restrict__ mu,
                             const int* __restrict__ exps, int K, int Kp,
                             unsigned char* __restrict__ image, SplitCol* __restrict__ cols) {
  const int lane = threadIdx.x & 31;
  const int j = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nJ = (K + kSpN - 1) / kSpN;
  if (j >= kSpN * (nJ - 1) + split_width(nJ - 1, K)) return;
  const int J = j / kSpN, jl = j % kSpN, Nj = split_width(J, K);
  const int nst = split_stages(J, K);
  int F = 1;
  if (j < K) {
    const int iend = min(kSpN * (J + 1), K);
    bool nan = false;
    for (int i = lane; i < iend; i += 32) {
      const double r = i <= j ? Rinv[(size_t)i * Kp + j] : 0.0;
      const int f = exp_field(r);
      if (r != 0.0) F = max(F, max(f, 1) + max(exps[i], 1));
      nan |= exp_field(mu[i]) == kNotFinite || f == kNotFinite;
    }
    F = __reduce_max_sync(0xffffffffu, F);
    nan = __any_sync(0xffffffffu, nan);
    // m to more than FP64's precision: the outputs of refine_weak take the means
    // off before their products, and must not differ from the others by a
    // rounding of m.  |mu_i r| < 2^(F - 2 1022), so the parts of the products on
    // the grid of `big` sum exactly, and the rest is 2^-43 of them.
    const int fb = F - 2 * 1022 + 10 + 1023;
    const double big = fb > 100 && fb < 2000 ? __hiloint2double(fb << 20, 0) : 0.0;
    double hi = 0.0, lo = 0.0;
    for (int i = lane; i <= j; i += 32) {
      const double a = mu[i], r = Rinv[(size_t)i * Kp + j], p = __dmul_rn(a, r);
      const double top = __dadd_rn(__dadd_rn(p, big), -big);
      hi += top;
      lo += (p - top) + fma(a, r, -p);
    }
    hi = warp_sum(hi);
    lo = warp_sum(lo);
    if (lane == 0) {
      // |m| <= K 2^F 2^(-2 1022), as |mu_i| < 2^(E_i): |u| < 2^57
      const int e = F + kColExp0;
      const double u = nan ? 0.0 : scalbn(hi, -e), r = rint(u);
      const double rest = nan ? 0.0 : (u - r) + scalbn(lo, -e), r2 = rint(rest);
      const long long mean = (long long)r + (long long)r2;
      cols[j] = SplitCol{mean, (float)(rest - r2),
                         nan ? kNanCol : 64 * e + 64 - __clzll(llabs(mean)), hi + lo};
    }
  }
  unsigned char* tile = image + split_image(J, K);
  for (int st = 0; st < nst; ++st, tile += (size_t)kAD * Nj * 64) {
    const int i = st * kSpHalf + lane;
    uint64_t x = Digits<kAD>::kBias;
    if (j < K && i <= j) {
      const uint64_t b = (uint64_t)__double_as_longlong(Rinv[(size_t)i * Kp + j]);
      // biased_int compares the scale with the value's own field
      if (b << 1) x = biased_int<kAD>(b, F - max(exps[i], 1));
    }
    const uint32_t at = sw64_offset(jl, lane >> 3) + (lane & 7) * 2;
#pragma unroll
    for (int d = 0; d < kAD; ++d)
      *reinterpret_cast<uint16_t*>(tile + (size_t)d * Nj * 64 + at) =
          (uint16_t)digit_pair<kAD>(x, x, d);
  }
}

struct ApplySplitArgs {
  double* V;
  long long ldv;
  int n, K;
  const int* exps;
  const unsigned char* image;
  const SplitCol* cols;
  const double* Rinv;  // row stride Kp
  int Kp;
  const double* mu;
  int* out_exps;  // largest exponent field of every output column, or null
  int* err;
};

// (d + m) 2^e rounded to FP64, for an integer |d| < 2^62 and a small |m|
// (in 62-bit integers: a 64-bit conversion and no FP64 arithmetic, which would
// take four operations on a pipe of two per clock).
// `plain` becomes false when the result is outside FP64's normal range.
__device__ __forceinline__ double scaled(long long d, float m, int e, bool& plain) {
  const unsigned long long mag = (unsigned long long)(d < 0 ? -d : d);
  const int s = min(max(__clzll((long long)mag) - 2, 0), 40);
  const long long t = (d << s) + __float2ll_rn(m * __int_as_float((127 + s) << 23));
  const double v = __ll2double_rn(t);
  const int hi = __double2hiint(v), f = ((hi >> 20) & 0x7ff) + e - s;
  plain = plain && (t == 0 || (f >= 1 && f <= 2046));
  return __hiloint2double(t == 0 ? 0 : hi + ((e - s) << 20), __double2loint(v));
}
// The same anywhere in FP64's range.
__device__ __noinline__ double to_double(long long d, float m, int e) {
  bool plain = true;
  const double v = scaled(d, m, 0, plain);
  return scalbn(v, e);
}

// The column's mean (mean + mean_lo) 2^s, in units of a row whose scale is 2^-s
// of the columns', as an integer and a remainder, for s <= kPlainShift and a mean
// of at most 61 - s bits: what almost every output takes.
constexpr int kPlainShift = 21;
__device__ __forceinline__ void shift_mean(const SplitCol& c, int s, long long& mean, float& rest) {
  const float x = c.mean_lo * __int_as_float((127 + s) << 23);  // at most 2^20: rounded by a magic sum
  const float t = x + 12582912.0f;
  mean = (c.mean << s) + (__float_as_int(t) - 0x4b400000);
  rest = x - (t - 12582912.0f);
}

// An output (sum h + l in units of a row of scale 2^rs, minus the mean) without
// those limits; weak: below the line of refine_weak.
__device__ __noinline__ double odd_output(const SplitCol& c, long long h, float l, int rs, bool& weak) {
  if (c.tag == kNanCol) return __longlong_as_double(0x7ff8000000000000ll);
  const int s = -rs, e = c.tag >> 6, bits = c.tag & 63;
  const float x = scalbnf(c.mean_lo, s);
  // a mean of 2^5 times what the row's own sum can be, or more
  if (!(fabsf(x) < 0x1p60f) || (bits > 0 && bits + s > 61)) return to_double(h, l, e + rs) - c.m;
  const long long i = __float2ll_rn(x), d = h - (bits > 0 ? c.mean << s : 0) - i;
  weak = llabs(d) < (1ll << kWeakBits);
  return to_double(d, l - (x - __ll2float_rn(i)), e + rs);
}

// The mark of a row of zeros (isolated vertices: a few per cent of a netlist's),
// whose scale is 2^0.
constexpr int kZeroRow = 1;

// Outputs of a warp's 32 rows (lane = row, from row0) and columns jb + u whose
// bit u is set in `weak`: formed again in FP64 where no product of theirs
// reaches the line (see the head of the file); `shift`: the row's scale.  Eight
// lanes per output, four outputs of different rows at a time.
__device__ __forceinline__ void refine_weak(const ApplySplitArgs& a, long long row0, int jb, int shift,
                                            unsigned weak, double (&v)[8]) {
  const int lane = threadIdx.x & 31, grp = lane >> 3, sub = lane & 7;
  while (const unsigned todo = __ballot_sync(0xffffffffu, weak != 0)) {
    unsigned t = todo;
    for (int q = 0; q < grp; ++q) t &= t - 1;
    const bool have = t != 0;
    const int src = have ? __ffs(t) - 1 : 0;
    const int j = jb + max(__ffs(__shfl_sync(0xffffffffu, weak, src)) - 1, 0);
    const double* vr = a.V + (row0 + src) * a.ldv;
    const double* rc = a.Rinv + j;
    int top = 0;  // a product is at least 2^(top - 2047)
    if (have) {
#pragma unroll 4
      for (int i = sub; i <= j; i += 8) {
        const int fv = exp_field(vr[i]), fr = exp_field(rc[(size_t)i * a.Kp]);
        if (fv >= exp_field(a.mu[i]) + 2 && fr > 0) top = max(top, fv + fr);
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    const int rs = __shfl_sync(0xffffffffu, shift, src);
    const int redo = have && top < (a.cols[j].tag >> 6) + rs + kWeakBits + 2047;
    double s = 0.0;
    if (__any_sync(0xffffffffu, redo)) {
      if (redo) {
#pragma unroll 4
        for (int i = sub; i <= j; i += 8) s = fma(vr[i] - a.mu[i], rc[(size_t)i * a.Kp], s);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    // the first four rows that had one take theirs
    const int rank = __popc(todo & ((1u << lane) - 1u));
    const double got = __shfl_sync(0xffffffffu, s, (rank & 3) * 8);
    const int take = __shfl_sync(0xffffffffu, redo, (rank & 3) * 8);
    if (weak != 0 && rank < 4) {
      const int u0 = __ffs(weak) - 1;
      weak &= weak - 1;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (take && u == u0) v[u] = got;
    }
  }
}

// Q = (V - 1 mu^T) R^-1 = V R^-1 - 1 (mu^T R^-1) in place, a tile of 128 rows
// per step; output blocks of 64 columns from the last to the first (a column is
// overwritten after every later block has read it).  Per stage of 32 basis
// values the 16 converter warps write the digit tiles of V (8 values of a row
// per thread: one 16-byte store per digit, a warp covering 512 contiguous
// bytes), a bulk copy by the 18th warp brings the digit tiles of R^-1, and the
// 17th warp's thread issues the MMAs: levels 0..5 stacked like the Gram's,
// levels 6..8 into the seventh accumulator.  Two stages; the converters also
// drain a finished block, so conversion, MMAs (1.8 us per stage) and the
// drain's 64-bit conversions share the time.
__global__ void __launch_bounds__(kSpThreads + 64, 1) k_apply_split(ApplySplitArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t conv[2], full[2], empty[2], drained, rows[4];
  __shared__ uint32_t tmem_slot;
  __shared__ int colmax[512], shifts[2][128];  // row scales of this and the next tile
  __shared__ __align__(16) int scales[512];    // exponent fields of the columns' scales
  constexpr uint32_t a_tile = 128u * 64u, a_stage = kAD * a_tile, b_stage = kAD * kSpN * 64u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) tmem_alloc(&tmem_slot, 512);
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) mbar_init(&conv[q], kSpConv), mbar_init(&full[q], 1), mbar_init(&empty[q], 1);
    mbar_init(&drained, kSpConv);
    for (int q = 0; q < 4; ++q) mbar_init(&rows[q], kSpConv / 4);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int q = tid; q < 512; q += blockDim.x) {
    const int e = q < a.K ? a.exps[q] : 0;
    scales[q] = e >= kTinyField ? e : 2 * 0x7ff + 64;  // all digits 0, whatever the row's scale
    colmax[q] = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int ntiles = (a.n + 127) / 128;
  const int nJ = (a.K + kSpN - 1) / kSpN;
  bool ok = true;
  uint32_t g = 0;    // stages so far; stage g uses buffer g % 2 for the (g / 2)-th time
  uint32_t blk = 0;  // output blocks so far (MMA warp)
  if (warp == kSpConv + 1) {
    if (lane == 0) {  // B producer
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x)
        for (int J = nJ - 1; J >= 0 && ok; --J) {
          const int nst = split_stages(J, a.K);
          const uint32_t b_bytes = (uint32_t)(kAD * split_width(J, a.K) * 64);
          const unsigned char* img = a.image + split_image(J, a.K);
          for (int st = 0; st < nst; ++st) {
            const int s = (int)(g & 1u);
            if (g >= 2 && !(ok = mbar_wait(&empty[s], ((g >> 1) - 1) & 1u, kSpWait))) break;
            mbar_arrive_expect_tx(&full[s], b_bytes);
            bulk_g2s(base + (size_t)s * (a_stage + b_stage) + a_stage, img + (size_t)st * b_bytes, b_bytes, &full[s]);
            ++g;
          }
        }
      // copies still landing finish before the CTA may leave
      for (uint32_t q = g > 2 ? g - 2 : 0; q < g; ++q) mbar_wait(&full[q & 1u], (q >> 1) & 1u, kSpWait);
    }
  } else if (warp == kSpConv) {
    if (lane == 0) {  // MMA issue
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x)
        for (int J = nJ - 1; J >= 0 && ok; --J, ++blk) {
          const int nst = split_stages(J, a.K), Nj = split_width(J, a.K);
          const uint32_t b_tile = (uint32_t)Nj * 64u;
          if (blk > 0 && !(ok = mbar_wait(&drained, (blk - 1) & 1u, kSpWait))) break;
          for (int st = 0; st < nst; ++st) {
            const int s = (int)(g & 1u);
            if (!(ok = mbar_wait(&conv[s], (g >> 1) & 1u, kSpWait) &&
                       mbar_wait(&full[s], (g >> 1) & 1u, kSpWait)))
              break;
            tc_fence_after();
            const uint32_t sA = smem_u32(base + (size_t)s * (a_stage + b_stage)), sB = sA + a_stage;
            const int nks = min(2, (a.K - st * kSpHalf + 15) / 16);
            const uint32_t id1 = idesc_bf16(128, Nj), id256 = idesc_bf16(128, 256);
            for (int ks = 0; ks < nks; ++ks) {
              const uint64_t dA = desc_k_sw64(sA + (uint32_t)ks * 32u), dB = desc_k_sw64(sB + (uint32_t)ks * 32u);
              const uint32_t start = (st > 0 || ks > 0) ? 1u : 0u;
#pragma unroll
              for (int i = 0; i < kAD; ++i) {
                const uint64_t da = dA + (uint64_t)((i * a_tile) >> 4);
                const uint32_t acc = i == 0 ? start : 1u;
                if (i < kAExact) {
                  const uint32_t d = tmem + (uint32_t)(Nj * i);
                  const int width = Nj * (kAExact - i);
                  if (width > 256) {
                    mma_bf16(d, da, dB, id256, acc);
                    mma_bf16(d + 256u, da, dB + (256u * 64u >> 4), idesc_bf16(128, width - 256), acc);
                  } else {
                    mma_bf16(d, da, dB, idesc_bf16(128, width), acc);
                  }
                }
#pragma unroll
                for (int j = (kAExact - i > 0 ? kAExact - i : 0); j < kAD - i; ++j)
                  mma_bf16(tmem + (uint32_t)(Nj * kAExact), da, dB + (j * b_tile >> 4), id1,
                           (i == 0 && j == kAExact) ? start : 1u);
              }
            }
            mma_commit(&empty[s]);
            ++g;
          }
        }
      // MMAs in flight finish before TMEM may be released
      for (uint32_t q = g > 2 ? g - 2 : 0; q < g; ++q) mbar_wait(&empty[q & 1u], (q >> 1) & 1u, kSpWait);
    }
  } else {
    const int r = tid >> 2, chunk = tid & 3;  // this thread's row of the tile, 8 values
    const uint32_t my = sw64_offset(r, chunk);
    uint64_t x[8];
    int sc[8];
    uint32_t stored = 0;  // rounds of the drain so far
    int shift = 0;        // scale of this thread's row: its largest entry beside its column's
    auto row_shift = [&](int tile) {
      const long long row = (long long)tile * 128 + r;
      int top = -0x7ff;
      uint64_t any = 0;
      if (a.K <= kSpHalf) {  // the whole row is in the four threads' stage
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          any |= x[u];
          top = max(top, max((int)(x[u] >> 52) & 0x7ff, 1) - sc[u]);
        }
      } else if (row < a.n) {  // 16 bytes of it at a time, eight loads in flight
        const double2* p = reinterpret_cast<const double2*>(a.V + row * a.ldv);
        const int np = a.K / 2;
#pragma unroll 8
        for (int c = chunk; c < np; c += 4) {
          const double2 x = p[c];
          const int2 e = *reinterpret_cast<const int2*>(scales + 2 * c);
          any |= (uint64_t)__double_as_longlong(x.x) | (uint64_t)__double_as_longlong(x.y);
          top = max(top, max(max(exp_field(x.x), 1) - e.x, max(exp_field(x.y), 1) - e.y));
        }
        if ((a.K & 1) && chunk == 0) {
          const double x = a.V[row * a.ldv + a.K - 1];
          any |= (uint64_t)__double_as_longlong(x);
          top = max(top, max(exp_field(x), 1) - scales[a.K - 1]);
        }
      }
      if (any << 1 == 0) top = -0x7ff;
      top = max(top, __shfl_xor_sync(0xffffffffu, top, 1));
      top = max(top, __shfl_xor_sync(0xffffffffu, top, 2));
      return top == -0x7ff ? kZeroRow : top;
    };
    auto load = [&](int tile, int st) {
      const long long row = (long long)tile * 128 + r;
      const int c = st * kSpHalf + 8 * chunk;
      const double* p = a.V + row * a.ldv + c;  // rows are 16-byte aligned, c even
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        double2 v = make_double2(0.0, 0.0);
        if (row < a.n) {
          if (c + u + 1 < a.K) v = *reinterpret_cast<const double2*>(p + u);
          else if (c + u < a.K) v.x = p[u];
        }
        x[u] = (uint64_t)__double_as_longlong(v.x);
        x[u + 1] = (uint64_t)__double_as_longlong(v.y);
      }
#pragma unroll
      for (int u = 0; u < 8; u += 4) {
        const int4 e = *reinterpret_cast<const int4*>(scales + c + u);
        sc[u] = e.x, sc[u + 1] = e.y, sc[u + 2] = e.z, sc[u + 3] = e.w;
      }
    };
    if ((int)blockIdx.x < ntiles) load(blockIdx.x, 0);
    int buf = 0;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, buf ^= 1) {
      // read by the drains, after the MMAs of stages that follow this
      shift = row_shift(tile);
      if (chunk == 0) shifts[buf][r] = shift;
      shift = min(shift, 0);
      for (int J = nJ - 1; J >= 0 && ok; --J) {
        const int nst = split_stages(J, a.K), Nj = split_width(J, a.K);
        for (int st = 0; st < nst; ++st, ++g) {
          const int s = (int)(g & 1u);
          if (g >= 2) ok = mbar_wait(&empty[s], ((g >> 1) - 1) & 1u, kSpWait);
          if (!(ok = __all_sync(0xffffffffu, ok))) break;
          // (an entry that is not finite has its column's scale: some digits,
          // which reach outputs that are NaN by their kNanCol)
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = biased_int<kAD>(x[u], sc[u] + shift);
          unsigned char* As = base + (size_t)s * (a_stage + b_stage) + my;
#pragma unroll
          for (int j = 0; j < kAD; ++j) {
            uint4 w;
            w.x = digit_pair<kAD>(x[0], x[1], j);
            w.y = digit_pair<kAD>(x[2], x[3], j);
            w.z = digit_pair<kAD>(x[4], x[5], j);
            w.w = digit_pair<kAD>(x[6], x[7], j);
            *reinterpret_cast<uint4*>(As + j * a_tile) = w;
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(&conv[s]);
          // next stage: columns that no output block written so far has
          // touched, or the next tile's rows
          if (st + 1 < nst) load(tile, st + 1);
          else if (J > 0) load(tile, 0);
          else if (tile + (int)gridDim.x < ntiles) load(tile + gridDim.x, 0);
        }
        if (!ok) break;
        // block complete: TMEM -> FP64 -> V
        ok = mbar_wait(&empty[(g - 1) & 1u], ((g - 1) >> 1) & 1u, kSpWait);
        if (!(ok = __all_sync(0xffffffffu, ok))) break;
        tc_fence_after();
        const int q4 = warp & 3;
        const long long row = (long long)tile * 128 + q4 * 32 + lane;
        const int mark = shifts[buf][q4 * 32 + lane], rs = min(mark, 0);
        const bool zero_row = mark == kZeroRow;
        // rounds of four column octets, one per warp of these rows, from the last
        // to the first; a round is stored when all four have read what they need
        // of the rows (columns up to their own)
        for (int round = (Nj / 8 - 1) / 4; round >= 0; --round) {
          const int c8 = 4 * round + (warp >> 2);
          const bool on = c8 < Nj / 8;  // warp-uniform
          const int jb = J * kSpN + c8 * 8;
          double v[8];
          if (on) {
            long long h[8];  // levels 0..5; level l holds multiples of 2^(-7 l)
            float low[8];    // levels 6..8
            const uint32_t at = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(c8 * 8);
#pragma unroll
            for (int half = 0; half < 2; ++half) {  // within the registers of 18 warps
              float L[3][8];
#pragma unroll
              for (int l = 0; l < 3; ++l) tmem_ld8(at + (uint32_t)((3 * half + l) * Nj), L[l]);
              if (half) tmem_ld8(at + (uint32_t)(kAExact * Nj), low);
              tmem_wait_ld();
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                if (!half) h[u] = 0;
#pragma unroll
                for (int l = 0; l < 3; ++l)
                  h[u] = h[u] * 128 + __float2int_rn(L[l][u] * (float)(1ull << (7 * (3 * half + l))));
              }
            }
            unsigned weak = 0, odd = 0;
            const int s = min(-rs, kPlainShift);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              low[u] *= (float)(1ull << (7 * (kAExact - 1)));
              v[u] = 0.0;
              if (jb + u < a.K) {
                const SplitCol col = a.cols[jb + u];
                long long mean;
                float rest;
                shift_mean(col, s, mean, rest);
                const long long d = h[u] - mean;
                bool plain = -rs <= kPlainShift && (col.tag & 63) + s <= 61 && col.tag != kNanCol;
                v[u] = scaled(d, low[u] - rest, (col.tag >> 6) + rs, plain);
                // (not where R^-1's column is zero)
                if (((unsigned long long)(d + (1ll << kWeakBits)) >> (kWeakBits + 1)) == 0 &&
                    col.tag >= 64 * (2 + kColExp0))
                  weak |= 1u << u;
                if (!plain) odd |= 1u << u;
              }
            }
            if (__any_sync(0xffffffffu, odd != 0)) {
#pragma unroll
              for (int u = 0; u < 8; ++u)
                if ((odd >> u) & 1u) {
                  bool w = false;
                  v[u] = odd_output(a.cols[jb + u], h[u], low[u], rs, w);
                  weak = (weak & ~(1u << u)) | ((w ? 1u : 0u) << u);
                }
            }
            refine_weak(a, row - lane, jb, rs, row < a.n && !zero_row ? weak : 0u, v);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&rows[q4]);
          ok = mbar_wait(&rows[q4], stored++ & 1u, kSpWait);
          if (!(ok = __all_sync(0xffffffffu, ok))) break;
          if (!on) continue;
          if (row < a.n) {
            double* dst = a.V + row * a.ldv + jb;
#pragma unroll
            for (int u = 0; u < 8; u += 2) {
              if (jb + u + 1 < a.K) *reinterpret_cast<double2*>(dst + u) = make_double2(v[u], v[u + 1]);
              else if (jb + u < a.K) dst[u] = v[u];
            }
          }
          if (a.out_exps) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int top = __reduce_max_sync(0xffffffffu, row < a.n ? (__double2hiint(v[u]) >> 20) & 0x7ff : 0);
              if (lane == 0 && jb + u < a.K && top > colmax[jb + u]) atomicMax(&colmax[jb + u], top);
            }
          }
        }
        if (!ok) break;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&drained);
      }
    }
  }
  if (!ok) atomicExch(a.err, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (a.out_exps)
    for (int j = tid; j < a.K; j += blockDim.x)
      if (colmax[j] > 0) atomicMax(a.out_exps + j, colmax[j]);
  if (warp == 0) tmem_dealloc(tmem, 512);
}

int gram_jobs(int K) {
  const int nbj = (K + kSpN) / kSpN;
  int jobs = 0;
  for (int bi = 0; 128 * bi < K; ++bi) jobs += nbj - 2 * bi;
  return jobs;
}

}  // namespace

// Chunks of rows of the Gram: about one CTA per SM over all jobs, chunks of
// whole 64-row slabs.
int split_chunks(long long n, int K) {
  const int want = std::max(1, num_sms() / gram_jobs(K));
  return (int)std::max(1ll, std::min<long long>(want, (n + 63) / 64));
}

size_t carve_split(Carver& cv, long long n, int K, SplitWs* w) {
  const int Kc = (K + 1 + 15) & ~15;
  const size_t part = (size_t)split_chunks(n, K) * K * Kc;
  w->hi = cv.take<long long>(part);
  w->lo = cv.take<long long>(part);
  w->exps = cv.take<int>(2 * (size_t)K);
  w->cols = cv.take<unsigned char>((size_t)K * sizeof(SplitCol));
  w->image = cv.take<unsigned char>(split_image((K + kSpN - 1) / kSpN, K));
  return cv.bytes();
}

hef_status split_col_exps(const double* V, long long ldv, long long n, int K, const SplitWs& w,
                          cudaStream_t st) {
  HEF_CHECK_CUDA(cudaMemsetAsync(w.exps, 0, 2 * (size_t)K * sizeof(int), st));
  const long long rounds = (n + (512 / K) * kExpRows - 1) / ((512 / K) * kExpRows);
  HEF_LAUNCH("k_col_exps", st, k_col_exps<<<(int)std::min<long long>(rounds, 4ll * num_sms()), 512, 0, st>>>(
                                   V, ldv, (int)n, K, w.exps));
  HEF_CHECK_LAUNCH();
  return HEF_OK;
}

hef_status gram_split(const double* V, long long ldv, long long n, int K, const int* exps,
                      const SplitWs& w, double* G, double* c, int* err, cudaStream_t st) {
  GramSplitArgs a;
  a.V = V;
  a.ldv = ldv;
  a.n = (int)n;
  a.K = K;
  a.Kc = (K + 1 + 15) & ~15;
  const int chunks = split_chunks(n, K);
  a.rows_per_cta = (int)(((n + chunks - 1) / chunks + 63) / 64 * 64);
  a.exps = exps;
  a.hi = w.hi;
  a.lo = w.lo;
  a.err = err;
  const int used = (int)((n + a.rows_per_cta - 1) / a.rows_per_cta);  // chunks with rows
  const size_t smem = 1024 + (size_t)kGD * (128 + kSpN) * 128;
  HEF_ENSURE_SMEM(k_gram_split, (int)smem);
  HEF_LAUNCH("k_gram_split", st, k_gram_split<<<dim3(used, gram_jobs(K)), kSpThreads + 32, smem, st>>>(a));
  HEF_LAUNCH("k_gram_split_reduce", st,
             k_gram_split_reduce<<<(int)std::min<long long>(((long long)K * (K + 1) + 31) / 32, 8ll * num_sms()),
                                   256, 0, st>>>(w.hi, w.lo, K, a.Kc, used, exps, G, c));
  HEF_CHECK_LAUNCH();
  return HEF_OK;
}

hef_status apply_split(double* V, long long ldv, long long n, int K, const double* Rinv, int Kp,
                       const double* mu, const int* exps, int* out_exps, const SplitWs& w, int* err,
                       cudaStream_t st) {
  HEF_LAUNCH("k_split_rinv", st, k_split_rinv<<<(((K + 15) & ~15) * 32 + 255) / 256, 256, 0, st>>>(
                                     Rinv, mu, exps, K, Kp, w.image,
                                     reinterpret_cast<SplitCol*>(w.cols)));
  ApplySplitArgs a;
  a.V = V;
  a.ldv = ldv;
  a.n = (int)n;
  a.K = K;
  a.exps = exps;
  a.image = w.image;
  a.cols = reinterpret_cast<const SplitCol*>(w.cols);
  a.Rinv = Rinv;
  a.Kp = Kp;
  a.mu = mu;
  a.out_exps = out_exps;
  a.err = err;
  const size_t smem = 1024 + 2 * (size_t)kAD * (128 + kSpN) * 64;
  HEF_ENSURE_SMEM(k_apply_split, (int)smem);
  const int grid = (int)std::min<long long>((n + 127) / 128, num_sms());
  HEF_LAUNCH("k_apply_split", st, k_apply_split<<<grid, kSpThreads + 64, smem, st>>>(a));
  HEF_CHECK_LAUNCH();
  return HEF_OK;
}

}  // namespace hef
