// FP64 products on the tensor cores ("digit engine"), sm_103a.
//
// GB300 has two FP64 FMA units per SM (1.1 TFLOP/s for the whole GPU), so a
// plain FP64 product is bound by them at any shape.  Here every FP64 operand is
// cut into eight signed base-256 digits, every row of A and every column of B
// relative to the power of two above its own largest magnitude (62 bits:
// elements within 2^-9 of the largest are represented exactly) -- the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication", Numer. Algorithms 59 (2012), with digits in place of
// floating-point slices (Mukunoki et al., "DGEMM using tensor cores", ISC 2020).
// A digit is an integer in [-128, 127], exact in FP16; a product of two digits is
// below 2^14, and the
// digit products of one weight (i + j = l <= 7) over 128 values of K stay below
// 2^24, so the tensor cores' FP32 accumulation of them is exact.  The 36 digit
// products with i + j <= 7 go to eight accumulators, one per weight.  What is
// dropped is at most 7 2^-62 of the two powers of two, 28 2^-62 of max|a_m|
// max|b_n| (largest magnitudes of the output's row and column); with the cut of
// both operands 2^-57 max|a_m| max|b_n| per term at most.  Every 128 values of K
// the accumulators are combined into a 96-bit integer per output, which is
// rounded to FP64 once at the end: the result carries one rounding instead of
// one per term.  One power of two per operand would lose rows that are small as
// a whole (2^-40 below the largest: 3e-6 of their products) and costs less: FP64
// sweep at chi = 128 24.48 ms, now 24.83; gradient of a torus at chi = 64 3.48,
// now 3.58; measurement of a Heisenberg chain at chi = 128 3.24, now 3.30; close
// product of 96 x 80 x 10007 53.4 us, now 54.0.  (In a sum of several groups, whose
// scales differ by output, 8 % of the product; else 0 to 1 %.)
//
// One CTA owns a 128 x BN output tile (BN 64 or 32); two stages of 32 K values.
// Warps 0-15 load FP64 operands (any strides), cut them into digits with integer
// operations and write them to shared memory in the K-major 64-byte-swizzle
// layout; digits that oz_prepare_kernel left in memory (small operands that many
// tiles read) arrive as one bulk copy per stage, started by a thread of warp 17;
// one thread of warp 16 issues the MMAs.  The digits of B are stacked along N, so
// that one MMA multiplies A's digit i with B's digits 0 .. 7 - i and adds each
// product to the accumulator of its weight: TMEM columns (i + j) BN .. of the
// same instruction.  All waits are bounded, as in the other tensor-core kernels.
//
// What bounds it (clocks of a 128 x 64 tile, K = 128): the four stages' MMAs take
// 12.5 k -- 9.2 k at the tensor rate, the rest is shared memory, which feeds them
// 106 bytes a clock beside the next stage's stores -- the combination of the
// accumulators 7 k (100 instructions per output), first loads and start 4 k; a
// stage that converts both operands takes 6 k, half of it its loads.  128 x 64
// because eight accumulators of 64 columns fill TMEM.  Sixteen converter warps
// (eight before: 2 warps a scheduler, an instruction every third clock): FP64
// sweep at chi = 128 25.29 -> 25.05 ms, FP64 gradient of a torus at chi = 64 3.61 ->
// 3.46 ms, measurement 3.35 -> 3.23 ms.  Measured on a GB300 (P = n = 128, with the
// preparation): F X of 128 x 128 by 128 x 16384 35 us (the FP64 kernel 547), the
// environment's five such products in one 160 us (2674), three close products over
// K = 16384 126 us (1931), the Gram matrix of 128 x 16384 55 us (449).  Converting
// both operands in every tile with BF16 digits, which take two operations more a
// pair, and combining by eight converting instructions per output took 55, 186,
// 123 and 59 (all with one power of two per operand, which now takes 35, 147, 126
// and 55); loads whose 16-byte pieces are consecutive over four threads (K permuted
// in a stage) took 5 % more than eight consecutive values per thread.
// Relative error against extended precision 4e-17 to 2e-16 where the
// FP64 kernel has 2e-16 to 2e-15.
//
// A row or column of a tile with an infinity or NaN, or whose range would leave
// the normal FP64 numbers, makes the CTA compute its tile with plain FP64 FMAs
// instead, so that the result is what the FP64 kernel gives.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <utility>

#include <cuda_fp16.h>

#include "common.h"
#include "f64_bits.cuh"
#include "oz_rule.h"

namespace ttn {

namespace {

constexpr int kOD = 8;              // digits per operand
constexpr int kOConv = 512;         // converter threads
constexpr int kOThreads = kOConv + 128;   // and the warpgroup of the MMA and image warps
constexpr int kOWork = kOConv / 32; // converter warps; the MMA warp follows them, then the image warp
constexpr long kOWait = 1L << 22;
constexpr int kOBlocks = 24;        // 16-column blocks of a CTA of the streamed kernel at most

// Magnitudes of an operand's rows (columns of B): the word (the high word of |x|,
// at least 1 for a nonzero x) of the largest value of a row among 2^len_log2
// values of K, part by part: word off + ((b0 s0 + b1 s1) parts + part) rows + row.
// img >= 0: the operand's digits are ready in memory (oz_prepare_kernel), cut
// under the largest value of the whole row (one part), block (batch, row tile, K
// slice of 32) at byte img + ((batch nrt + row tile) nks + slice) of the block
// size, laid out as a stage of shared memory.  chunk0, chunks: the group's chunks
// of K among all; whole: rows are cut under their value over all of K (a group
// with ready digits), else over the chunks that a CTA sums.
struct OzOperand {
  int off, parts, len_log2, rows, s0, s1, nrt, nks, chunk0, chunks, whole;
  long long img;
};
struct OzParams {
  const unsigned* words;
  const uint8_t* images;
  OzOperand a[kMaxGroups], b[kMaxGroups];
  int total_chunks;
  int blocks, nb16;                 // streamed kernel: 16-column blocks in all and per row tile
  long wait;                        // tries of a wait before it expires
  int* err;                         // raised by an expired wait; null: the outputs it leaves become NaN
};

struct AbsItem {
  const double* p;
  long long s_mn, s_k0, s_k1, s_b0, s_b1, img;
  int mn, k0_log2, k, n0, n1, parts, len_log2, off, blocks_before, nrt, nks, rt;
};
constexpr int kAbsBlocks = 512;     // blocks that a pass over an operand is divided into
// A row's exponent is kOBias + the biased exponent of the power of two above its
// largest value, or 0 for a row of zeros.  (The sum of a row's and a column's fits
// 15 bits, and pairs of sums are added and compared 16 bits each; the bias keeps
// the sums with a row or column of zeros below all others.)
constexpr int kOBias = 10000;
struct AbsParams {
  AbsItem it[2 * kMaxGroups];
  int n;
  unsigned* words;
  uint8_t* images;
  const int* skip;
  int skip_when_zero;
};
static_assert(sizeof(AbsParams) < 32000, "kernel parameter");

__device__ __forceinline__ int word_exponent(unsigned w) { return w ? static_cast<int>(w >> 20) + kOBias : 0; }
// The exponent that a row's values are cut under (a row of zeros: any, its digits
// are zero).
__device__ __forceinline__ int cut_exponent(int e) { return e ? e - kOBias : 1023; }

__device__ __forceinline__ unsigned mag_word(double x) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(x)) & 0x7FFFFFFFu;
  return hi | (__double2loint(x) != 0 ? 1u : 0u);
}

// The eight digits of x as bytes (digit + 128; the most significant digit in
// the highest byte), for |x| below 2^(emax - 1022): x / 2^(emax - 1084), cut
// to an integer, plus 128 in every byte.
__device__ __forceinline__ void digit_bytes(double x, int emax, uint32_t& lo, uint32_t& hi) {
  const uint32_t h = static_cast<uint32_t>(__double2hiint(x)), l = static_cast<uint32_t>(__double2loint(x));
  const int e = (h >> 20) & 0x7FF;
  const uint32_t mh = (h & 0xFFFFFu) | 0x100000u;
  unsigned long long v = (static_cast<unsigned long long>(__funnelshift_l(l, mh, 9)) << 32) | (l << 9);
  v >>= min(emax - e, 63);                      // a subnormal x (e = 0) is far below the cut
  const long long s = static_cast<int>(h) >> 31;
  v = (v ^ s) + (0x8080808080808080ull - s);
  lo = static_cast<uint32_t>(v);
  hi = static_cast<uint32_t>(v >> 32);
}

// Two digits (bytes b of w0 and w1, each digit + 128) as an FP16 pair: the
// byte in the low mantissa bits of 1024 is 1024 + digit + 128, less 1152.
template <int b>
__device__ __forceinline__ uint32_t digit_pair(uint32_t w0, uint32_t w1) {
  const uint32_t t = __byte_perm(w0, w1, 0x0400 + 0x0101 * b);
  const uint32_t y = (t & 0x00FF00FFu) | 0x64006400u, z = 0x64806480u;
  const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&y), *reinterpret_cast<const __half2*>(&z));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// Eight consecutive K values of row r -> 16-byte chunk c (of four) of every
// digit tile: rows of 64 bytes, 64-byte swizzle, tiles `stride` bytes apart.
__device__ __forceinline__ void store_digits(const double* v, int emax, uint8_t* tile, int r, int c, int stride) {
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) digit_bytes(v[q], emax, lo[q], hi[q]);
  uint8_t* p = tile + r * 64 + ((c ^ ((r >> 1) & 3)) << 4);
#define TTN_OZ_DIGIT(d, w, b)                                                              \
  *reinterpret_cast<uint4*>(p + (d) * stride) =                                            \
      make_uint4(digit_pair<b>(w[0], w[1]), digit_pair<b>(w[2], w[3]),                     \
                 digit_pair<b>(w[4], w[5]), digit_pair<b>(w[6], w[7]));
  TTN_OZ_DIGIT(0, hi, 3) TTN_OZ_DIGIT(1, hi, 2) TTN_OZ_DIGIT(2, hi, 1) TTN_OZ_DIGIT(3, hi, 0)
  TTN_OZ_DIGIT(4, lo, 3) TTN_OZ_DIGIT(5, lo, 2) TTN_OZ_DIGIT(6, lo, 1) TTN_OZ_DIGIT(7, lo, 0)
#undef TTN_OZ_DIGIT
}

// Row and 16-byte chunk of converter task `task` of a stage (4 chunks per row):
// K contiguous: eight rows by four chunks per warp (a row's 64 bytes of a digit
// are consecutive); MN contiguous: 32 consecutive rows of one chunk per warp.
// Both fill the 32 banks in every store phase.
template <int ROWS>
__device__ __forceinline__ void task_pos(int task, bool kfast, int& r, int& c) {
  const int w = task >> 5, lane = task & 31;
  if (kfast) {
    r = w * 8 + (lane >> 2);
    c = lane & 3;
  } else {
    r = (w % (ROWS / 32)) * 32 + lane;
    c = w / (ROWS / 32);
  }
}

// Eight consecutive K values (k a multiple of 8) of a row that starts at
// `base`; zeros outside.
__device__ __forceinline__ void load8(long long s_mn, long long s_k0, long long s_k1, int k0_log2,
                                      const double* base, int row, bool row_ok, int k, int K, bool vec, double* v) {
  if (!row_ok || k >= K) {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = 0.0;
    return;
  }
  const int k0 = k & ((1 << k0_log2) - 1), k1 = k >> k0_log2;
  const double* p = base + row * s_mn + k0 * s_k0 + static_cast<long long>(k1) * s_k1;
  if (k + 8 <= K) {
    if (vec) {
#pragma unroll
      for (int q = 0; q < 8; q += 2) {
        const double2 t = *reinterpret_cast<const double2*>(p + q);
        v[q] = t.x;
        v[q + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = p[q * s_k0];
    }
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = k + q < K ? p[q * s_k0] : 0.0;
  }
}

// The digits of one stage block (ROWS rows from r0, 32 K values from k) of a
// small operand into memory, by the whole block; words: its rows' magnitudes.
template <int ROWS>
__device__ __forceinline__ void image_block(const AbsItem& it, const double* p, int r0, int k, const unsigned* words,
                                            uint8_t* out) {
  const bool kf = it.s_k0 == 1;
  const bool vec = kf && (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ((it.s_mn | it.s_k1) & 1) == 0;
#pragma unroll 1
  for (int task = threadIdx.x; task < ROWS * 4; task += 256) {
    int r, c;
    task_pos<ROWS>(task, kf, r, c);
    double v[8];
    load8(it.s_mn, it.s_k0, it.s_k1, it.k0_log2, p, r0 + r, r0 + r < it.mn, k + 8 * c, it.k, vec, v);
    store_digits(v, cut_exponent(word_exponent(words[r])), out, r, c, ROWS * 64);
  }
}

// words[r] = the largest magnitude word of row r0 + r over K values k_lo .. k_hi
// - 1, for R rows (32, 64 or 128); words hold 0 before.  K contiguous: a warp per
// row, lanes along K, KS steps of K and 16 / KS rows at a time; else lanes along
// the rows and the warps share K.  Sixteen loads in flight per thread.  kFull: all
// rows are there, the K values are whole steps of one run of K0 -- without the
// index arithmetic and the tests per value, which take three times the
// instructions of the loads and maxima.
template <int KS, bool kFull>
__device__ __forceinline__ void rows_kfast(const AbsItem& it, const double* p, int r0, int R, int k_lo, int k_hi,
                                           unsigned* words) {
  constexpr int kRows = 16 / KS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kmask = (1 << it.k0_log2) - 1;
  const double* pf = p + (k_lo & kmask) + static_cast<long long>(k_lo >> it.k0_log2) * it.s_k1 - k_lo + r0 * it.s_mn;
#pragma unroll 1
  for (int r = warp; r < R; r += 8 * kRows) {
    unsigned m[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) m[i] = 0u;
#pragma unroll 1
    for (int k = k_lo + lane; k < k_hi; k += 32 * KS) {
      double v[kRows][KS];
      if constexpr (kFull) {
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          const double* pr = pf + (r + 8 * i < R ? r + 8 * i : r) * it.s_mn + k;   // (a short tile: a row again)
#pragma unroll
          for (int q = 0; q < KS; ++q) v[i][q] = pr[32 * q];
        }
      } else {
#pragma unroll
        for (int q = 0; q < KS; ++q) {
          const int kk = k + 32 * q;
          const bool in = kk < k_hi;
          const double* pk = p + (in ? (kk & kmask) + static_cast<long long>(kk >> it.k0_log2) * it.s_k1 : 0);
#pragma unroll
          for (int i = 0; i < kRows; ++i)
            v[i][q] = in && r + 8 * i < R && r0 + r + 8 * i < it.mn ? pk[(r0 + r + 8 * i) * it.s_mn] : 0.0;
        }
      }
#pragma unroll
      for (int i = 0; i < kRows; ++i)
#pragma unroll
        for (int q = 0; q < KS; ++q) m[i] = max(m[i], mag_word(v[i][q]));
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      m[i] = __reduce_max_sync(0xffffffffu, m[i]);
      if (lane == 0 && r + 8 * i < R) words[r + 8 * i] = m[i];
    }
  }
}
template <bool kFull>
__device__ __forceinline__ void rows_mnfast(const AbsItem& it, const double* p, int r0, int R, int k_lo, int k_hi,
                                            unsigned* words) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kmask = (1 << it.k0_log2) - 1;
  const int groups = R >> 5, rg = warp % groups, step = 8 / groups;
  const int row = r0 + rg * 32 + lane;
  if (!kFull && row >= it.mn) return;
  const double* pr = p + row * it.s_mn;
  unsigned m = 0;
#pragma unroll 1
  for (int k = k_lo + warp / groups; k < k_hi; k += 16 * step) {
    double v[16];
    const double* pk = pr + (k & kmask) * it.s_k0 + static_cast<long long>(k >> it.k0_log2) * it.s_k1;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      if constexpr (kFull) {
        v[q] = *pk;
        pk += step * it.s_k0;
      } else {
        const int kk = k + q * step;
        v[q] = kk < k_hi ? pr[(kk & kmask) * it.s_k0 + static_cast<long long>(kk >> it.k0_log2) * it.s_k1] : 0.0;
      }
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) m = max(m, mag_word(v[q]));
  }
  atomicMax(&words[rg * 32 + lane], m);
}
__device__ __forceinline__ void row_magnitudes(const AbsItem& it, const double* p, int r0, int R, int k_lo, int k_hi,
                                               unsigned* words) {
  const int nk = k_hi - k_lo;
  const bool full = r0 + R <= it.mn && ((k_lo ^ (k_hi - 1)) >> it.k0_log2) == 0;
  if (it.s_k0 != 1) {
    if (full && nk % (4096 / R) == 0) rows_mnfast<true>(it, p, r0, R, k_lo, k_hi, words);
    else rows_mnfast<false>(it, p, r0, R, k_lo, k_hi, words);
  } else if (nk > 64) {
    if (full && nk % 128 == 0) rows_kfast<4, true>(it, p, r0, R, k_lo, k_hi, words);
    else rows_kfast<4, false>(it, p, r0, R, k_lo, k_hi, words);
  } else if (nk > 32) {
    if (full && nk == 64) rows_kfast<2, true>(it, p, r0, R, k_lo, k_hi, words);
    else rows_kfast<2, false>(it, p, r0, R, k_lo, k_hi, words);
  } else {
    rows_kfast<1, false>(it, p, r0, R, k_lo, k_hi, words);
  }
}

// Before a product: the magnitudes of its operands' rows, and the digits of the
// small operands that many of its tiles read.
//   without an image: a block per 32 to 128 rows of a batch and part of K;
//   with one: a block per stage block; each scans its (few, short) rows.
// Bound by the read of the operands (from L2 when they were just produced): 20 us
// for five operands of 128 x 16384 from DRAM, 9 to 11 for one.  Five blocks a SM: at
// four (80 registers instead of 48) the five operands' product took 1 % longer.
__global__ void __launch_bounds__(256, 5) oz_prepare_kernel(const AbsParams ap) {
  pdl_wait();
  pdl_trigger();
  if (ap.skip && ((*ap.skip != 0) != (ap.skip_when_zero != 0))) return;
  int i = 0;
  while (i + 1 < ap.n && static_cast<int>(blockIdx.x) >= ap.it[i + 1].blocks_before) ++i;
  const AbsItem& it = ap.it[i];
  const int u = blockIdx.x - it.blocks_before;
  const bool image = it.img >= 0;
  const int inner = image ? it.nks : it.parts;       // K slices, or parts of K
  const int rt = (u / inner) % it.nrt, ks = u % inner, batch = u / (inner * it.nrt);
  const int b0 = batch % it.n0, b1 = batch / it.n0;
  const double* p = it.p + b0 * it.s_b0 + static_cast<long long>(b1) * it.s_b1;
  const int r0 = rt * it.rt;
  const int k_lo = image ? 0 : ks << it.len_log2, k_hi = image ? it.k : min(it.k, k_lo + (1 << it.len_log2));
  __shared__ unsigned words[kOBM];
  if (threadIdx.x < kOBM) words[threadIdx.x] = 0u;
  __syncthreads();
  const int rows = it.mn - r0;
  row_magnitudes(it, p, r0, min(it.rt, rows <= 32 ? 32 : (rows <= 64 ? 64 : 128)), k_lo, k_hi, words);
  __syncthreads();
  if (static_cast<int>(threadIdx.x) < it.rt && r0 + static_cast<int>(threadIdx.x) < it.mn && (!image || ks == 0))
    ap.words[it.off + (static_cast<long long>(batch) * it.parts + (image ? 0 : ks)) * it.mn + r0 + threadIdx.x] =
        words[threadIdx.x];
  if (!image) return;
  uint8_t* out = ap.images + it.img + static_cast<long long>(u) * kOD * it.rt * 64;
  if (it.rt == 128) image_block<128>(it, p, r0, ks * kOBK, words, out);
  else if (it.rt == 64) image_block<64>(it, p, r0, ks * kOBK, words, out);
  else image_block<32>(it, p, r0, ks * kOBK, words, out);
}

__device__ __forceinline__ uint32_t osmem(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool omb_wait(uint64_t* bar, uint32_t parity, const volatile int* abort_flag,
                                         long tries = kOWait) {
  const uint32_t a = osmem(bar);
  for (long it = 0; it < tries; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    if (abort_flag && *abort_flag) return false;
  }
  return false;
}
__device__ __forceinline__ void omb_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(osmem(bar)), "r"(count));
}
__device__ __forceinline__ void omb_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(osmem(bar)) : "memory");
}
__device__ __forceinline__ void omb_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(osmem(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(osmem(bar))
               : "memory");
}
__device__ __forceinline__ void ocommit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(osmem(bar))
      : "memory");
}
// K-major, 64-byte swizzle: rows of 64 bytes, 8-row atoms every 512 bytes.
__device__ __forceinline__ uint64_t odesc(uint32_t saddr) {
  return static_cast<uint64_t>((saddr >> 4) & 0x3FFF) | (1ull << 16) |
         (static_cast<uint64_t>(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}
__device__ __forceinline__ void omma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}
// D = F32, A and B FP16, both K-major.
__host__ __device__ constexpr uint32_t oidesc(int N) {
  return (1u << 4) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(kOBM >> 4) << 24);
}

// A sum of digit products of a row with exponent ea and a column with exponent
// eb is an integer times 2^(ea + eb - kOScale).
constexpr int kOScale = 2 * kOBias + 2 * 1022 + 68;

// The 96-bit integer (a2 a1 a0, two's complement) times 2^scale, rounded to
// FP64 (the caller has checked that the result is zero or a normal number).  A
// negative value is complemented without the one: a unit of 2^scale, 2^-68 of
// the powers of two above the row's and the column's largest values, below the
// dropped digit products.
__device__ __forceinline__ double to_double(uint32_t a0, uint32_t a1, uint32_t a2, int scale) {
  const uint32_t neg = static_cast<uint32_t>(static_cast<int>(a2) >> 31);
  a0 ^= neg; a1 ^= neg; a2 ^= neg;
  int e = scale + 1022 + 95;
  if (a2 == 0u) {
    a2 = a1; a1 = a0; a0 = 0u; e -= 32;
    if (a2 == 0u) { a2 = a1; a1 = 0u; e -= 32; }
  }
  const int n = __clz(a2);
  const uint32_t t1 = __funnelshift_l(a1, a2, n), t0 = __funnelshift_l(a0, a1, n);
  const unsigned long long t = (static_cast<unsigned long long>(t1) << 32) | t0;
  const unsigned long long m = (t >> 11) + ((t0 >> 10) & 1u);
  const uint32_t hi = static_cast<uint32_t>(m >> 32) + (static_cast<uint32_t>(e - n) << 20);
  return __hiloint2double(a2 ? static_cast<int>(hi | (neg & 0x80000000u)) : 0, static_cast<int>(static_cast<uint32_t>(m)));
}

// Output (or split-K partial) of one element.
__device__ __forceinline__ double* out_ptr(const GemmDesc& d, int b, int b0, int b1, int split, int m, int n) {
  if (d.splits > 1)
    return d.partial + ((static_cast<long long>(split) * d.B0 * d.B1 + b) * d.M + m) * d.N + n;
  return static_cast<double*>(d.C) + b0 * d.sc_b0 + static_cast<long long>(b1) * d.sc_b1 + m * d.sc_m + n * d.sc_n;
}

// Plain FP64 tile over the CTA's chunks (operands with infinities or NaN, or a
// range that the digits do not cover).
__device__ __noinline__ void plain_tile(const GemmDesc& d, int b, int b0, int b1, int split, int m0, int n0, int bn,
                                        int c_lo, int c_hi) {
  for (int e = threadIdx.x; e < kOBM * bn; e += kOThreads) {
    const int m = m0 + e / bn, n = n0 + e % bn;
    if (m >= d.M || n >= d.N) continue;
    double acc = 0.0;
    int c = 0;
    for (int g = 0; g < d.ngroups; ++g) {
      const Group& G = d.g[g];
      const int nc = (G.K + kOChunk - 1) / kOChunk;
      const int k_lo = min(G.K, max(0, c_lo - c) * kOChunk), k_hi = min(G.K, max(0, c_hi - c) * kOChunk);
      c += nc;
      const double* pa = static_cast<const double*>(G.a.p) + b0 * G.a.s_b0 + static_cast<long long>(b1) * G.a.s_b1 + m * G.a.s_mn;
      const double* pb = static_cast<const double*>(G.b.p) + b0 * G.b.s_b0 + static_cast<long long>(b1) * G.b.s_b1 + n * G.b.s_mn;
      for (int k = k_lo; k < k_hi; ++k) {
        const int k0 = k & ((1 << G.k0_log2) - 1), k1 = k >> G.k0_log2;
        acc = fma(pa[k0 * G.a.s_k0 + static_cast<long long>(k1) * G.a.s_k1],
                  pb[k0 * G.b.s_k0 + static_cast<long long>(k1) * G.b.s_k1], acc);
      }
    }
    double* out = out_ptr(d, b, b0, b1, split, m, n);
    *out = acc;
    if (d.c32 && d.splits <= 1) d.c32[out - static_cast<double*>(d.C)] = static_cast<float>(acc);
  }
}

// The accumulators of four columns (two columns): levels l, `cols` columns
// apart.  (The registers hold them after ld_wait.)
__device__ __forceinline__ void ld_levels(uint32_t taddr, int cols, uint32_t (&r)[kOD][2]) {
#pragma unroll
  for (int l = 0; l < kOD; ++l)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];"
                 : "=r"(r[l][0]), "=r"(r[l][1])
                 : "r"(taddr + l * cols));
}
__device__ __forceinline__ void ld_levels(uint32_t taddr, int cols, uint32_t (&r)[kOD][4]) {
#pragma unroll
  for (int l = 0; l < kOD; ++l)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3])
                 : "r"(taddr + l * cols));
}
// The loads of r are complete (r as operands: nothing reads it before).
template <int NC>
__device__ __forceinline__ void ld_wait(uint32_t (&r)[kOD][NC]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int l = 0; l < kOD; ++l)
#pragma unroll
    for (int j = 0; j < NC; ++j) asm volatile("" : "+r"(r[l][j]));
}

// Combine the columns' accumulators into 96-bit integers.
template <int NC>
__device__ __forceinline__ void combine(const uint32_t (&r)[kOD][NC], uint32_t (&v)[NC][3]) {
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    // levels 0 to 2 are at most 2^22 (digit 0 is at most 64): their integers sit
    // in the low bits of x + 1.5 2^23; the others take the converting
    // instruction, a quarter of the rate of an addition
    int L[kOD];
#pragma unroll
    for (int l = 0; l < 3; ++l) L[l] = __float_as_int(__uint_as_float(r[l][j]) + 12582912.f) - 0x4B400000;
#pragma unroll
    for (int l = 3; l < kOD; ++l) L[l] = __float2int_rn(__uint_as_float(r[l][j]));
    // (both inner sums fit 32 bits: 2^27 and 2^30 + 2^23)
    const long long H = static_cast<long long>(L[0] * 256 + L[1]) * (1 << 16) + (L[2] * 256 + L[3]);
    const long long Q = static_cast<long long>(L[4]) * (1 << 24) + (static_cast<long long>(L[5]) * (1 << 16) +
                        (static_cast<long long>(L[6]) * 256 + L[7]));
    const long long hi = H + static_cast<int>(Q >> 32);
    v[j][0] = static_cast<uint32_t>(Q);
    v[j][1] = static_cast<uint32_t>(hi);
    v[j][2] = static_cast<uint32_t>(hi >> 32);
  }
}

// The 96-bit integer v shifted right by 0 <= sh <= 63.
__device__ __forceinline__ void shift96(uint32_t (&v)[3], uint32_t sh) {
  const uint32_t sg = static_cast<uint32_t>(static_cast<int>(v[2]) >> 31);
  const bool w = sh >= 32u;
  const uint32_t a0 = w ? v[1] : v[0], a1 = w ? v[2] : v[1], a2 = w ? sg : v[2];
  v[0] = __funnelshift_r(a0, a1, sh);
  v[1] = __funnelshift_r(a1, a2, sh);
  v[2] = static_cast<uint32_t>(static_cast<int>(a2) >> (sh & 31u));
}

// Whether the digits do not cover a tile whose nonzero rows and columns have
// exponents within [range[0], range[1]] and [range[2], range[3]]: its results
// could leave the normal numbers.
__device__ __forceinline__ bool plain_range(const int* range) {
  return range[1] && range[3] &&
         (range[1] + range[3] - kOScale > 900 || range[0] + range[2] - kOScale < -1000);
}
// The exponents of 32 rows (one per lane) into a range, by lane 0.
__device__ __forceinline__ void add_range(int* range, int e) {
  const int hi = __reduce_max_sync(0xffffffffu, e), lo = __reduce_min_sync(0xffffffffu, e ? e : 0x7FFF);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&range[0], lo);
    atomicMax(&range[1], hi);
  }
}
// Rows with infinities, NaN or so small values that their digits would be
// subnormal: the tile is left to plain FP64.
__device__ __forceinline__ bool plain_row(int e) { return e >= kOBias + 0x7FF || (e && e < kOBias + 80); }

// kMulti: several groups (their sums are shifted to a common scale); without, the
// same code at run time took 2 to 4 % of a product of one group.
template <int BN, bool kMulti>
__global__ void __launch_bounds__(kOThreads, 1) gemm_oz_kernel(const GemmDesc d, const OzParams op) {
  pdl_wait();
  pdl_trigger();
  constexpr int kA = kOBM * 64, kB = BN * 64;      // bytes of one digit tile of a stage
  constexpr int kStage = kOD * (kA + kB);
  constexpr int kPart = BN / 4;                    // columns per flush warp
  constexpr int kCols = kOD * BN;                  // TMEM columns
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  __shared__ __align__(8) uint64_t full_bar[2], empty_bar[2], done_bar, free_bar, drain_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  // exponents of the tile's rows and columns, group by group, and their range
  constexpr int kRB = (kOBM + BN) / 32;
  __shared__ __align__(16) short ea[kMaxGroups][kOBM], eb[kMaxGroups][BN];
  __shared__ int range[4], plain_flag;

  if (desc_skipped(d)) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_n = (d.N + BN - 1) / BN;
  const int tm = blockIdx.x / tiles_n, tn = blockIdx.x % tiles_n;
  const int b = blockIdx.y, b0 = b % d.B0, b1 = b / d.B0;
  const int split = blockIdx.z;
  const int m0 = tm * kOBM, n0 = tn * BN;
  const int c_lo = static_cast<int>(static_cast<long long>(op.total_chunks) * split / d.splits);
  const int c_hi = static_cast<int>(static_cast<long long>(op.total_chunks) * (split + 1) / d.splits);

  if (warp == kOWork) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(osmem(&tmem_slot)), "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // first chunk of the CTA: group g0, K offset kfirst
  int g0 = 0, kfirst = 0;
  {
    int c = c_lo;
    while (g0 < d.ngroups) {
      const int nc = (d.g[g0].K + kOChunk - 1) / kOChunk;
      if (c < nc) break;
      c -= nc;
      ++g0;
    }
    kfirst = c * kOChunk;
  }
  const int nchunks = c_hi - c_lo;

  // converter state: the values of the next stage (loaded before the operands'
  // magnitudes arrive), their rows and chunks, the position after them
  const int t = threadIdx.x;
  constexpr int kATasks = kOBM * 4 / kOConv;                     // 1
  double va[kATasks][8], vb[8];
  int g = g0, k = kfirst;                                        // next stage to load
  const double *pa = nullptr, *pb = nullptr;
  bool avec = false, bvec = false, a_on = false, b_on = false;
  int ar[kATasks], ac[kATasks], br = 0, bc = 0;
  auto enter = [&]() {
    const Group& G = d.g[g];
    pa = static_cast<const double*>(G.a.p) + b0 * G.a.s_b0 + static_cast<long long>(b1) * G.a.s_b1;
    pb = static_cast<const double*>(G.b.p) + b0 * G.b.s_b0 + static_cast<long long>(b1) * G.b.s_b1;
    const bool akf = G.a.s_k0 == 1, bkf = G.b.s_k0 == 1;
    a_on = op.a[g].img < 0;
    b_on = op.b[g].img < 0 && t < BN * 4;
    avec = akf && ((reinterpret_cast<uintptr_t>(pa) & 15) == 0) && ((G.a.s_mn | G.a.s_k1) & 1) == 0;
    bvec = bkf && ((reinterpret_cast<uintptr_t>(pb) & 15) == 0) && ((G.b.s_mn | G.b.s_k1) & 1) == 0;
#pragma unroll
    for (int q = 0; q < kATasks; ++q) task_pos<kOBM>(t + q * kOConv, akf, ar[q], ac[q]);
    task_pos<BN>(t, bkf, br, bc);
  };
  auto load_a = [&](int q) {
    const Group& G = d.g[g];
    load8(G.a.s_mn, G.a.s_k0, G.a.s_k1, G.k0_log2, pa, m0 + ar[q], m0 + ar[q] < d.M, k + 8 * ac[q], G.K, avec, va[q]);
  };
  auto load_b = [&]() {
    const Group& G = d.g[g];
    load8(G.b.s_mn, G.b.s_k0, G.b.s_k1, G.k0_log2, pb, n0 + br, n0 + br < d.N, k + 8 * bc, G.K, bvec, vb);
  };
  if (warp < kOWork && nchunks > 0) {
    enter();
    if (b_on) load_b();
    if (a_on) {
#pragma unroll
      for (int q = 0; q < kATasks; ++q) load_a(q);
    }
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      omb_init(&full_bar[s], kOConv + 1);
      omb_init(&empty_bar[s], 1);
    }
    omb_init(&done_bar, 1);
    omb_init(&drain_bar, 1);
    omb_init(&free_bar, kOConv);
    abort_flag = 0;
    range[0] = range[2] = 0x7FFF;
    range[1] = range[3] = 0;
    plain_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
#pragma unroll 1
  for (int u = warp; u < d.ngroups * kRB; u += kOThreads / 32) {
    const int gi = u / kRB, q = u - gi * kRB;
    const bool isb = q >= kOBM / 32;
    const OzOperand& o = isb ? op.b[gi] : op.a[gi];
    const int q_lo = max(0, c_lo - o.chunk0), q_hi = min(o.chunks, c_hi - o.chunk0);   // chunks of the group
    int p_lo = 0, p_hi = q_lo < q_hi ? o.parts : 0;
    if (!o.whole && q_lo < q_hi) {
      p_lo = q_lo * kOChunk >> o.len_log2;
      p_hi = min(p_hi, ((q_hi * kOChunk - 1) >> o.len_log2) + 1);
    }
    const int r = (isb ? q - kOBM / 32 : q) * 32 + lane, row = (isb ? n0 : m0) + r;
    unsigned m = 0u;
    if (row < o.rows) {
      const unsigned* w = op.words + o.off + static_cast<long long>(b0 * o.s0 + b1 * o.s1) * o.parts * o.rows + row;
#pragma unroll 4
      for (int j = p_lo; j < p_hi; ++j) m = max(m, __ldcg(w + static_cast<long long>(j) * o.rows));
    }
    const int e = word_exponent(m);
    if (isb) eb[gi][r] = static_cast<short>(e);
    else ea[gi][r] = static_cast<short>(e);
    if (plain_row(e)) plain_flag = 1;
    add_range(&range[isb ? 2 : 0], e);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  const bool plain = plain_flag || plain_range(range);
  if (plain) plain_tile(d, b, b0, b1, split, m0, n0, BN, c_lo, c_hi);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  volatile int* abort_v = &abort_flag;

  // registers: five warpgroups of 96 at launch -> 32 for the MMA warp's, 112 for
  // the four of the converters (4 x 112 + 32 = 5 x 96)
  if (plain) {
    // (the tile is done)
  } else if (warp >= kOWork) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (warp == kOWork && lane == 0) {
      // ---- MMA issuer ----
      bool ok = true;
      int g = g0, k = kfirst, it = 0;
      const uint32_t base = osmem(smem);
      for (int c = 0; c < nchunks && ok; ++c) {
        if (c > 0 && !omb_wait(&free_bar, (c - 1) & 1, abort_v, op.wait)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int kend = min(d.g[g].K, k + kOChunk);
        const int nst = (kend - k + kOBK - 1) / kOBK;
        for (int st = 0; st < nst; ++st, ++it) {
          const int s = it & 1;
          if (!omb_wait(&full_bar[s], (it >> 1) & 1, abort_v, op.wait)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = base + s * kStage, sb = sa + kOD * kA;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
#pragma unroll
            for (int i = 0; i < kOD; ++i) {
              const uint64_t ad = odesc(sa + i * kA + j * 32);
              const uint32_t acc = (st > 0 || j > 0 || i > 0) ? 1u : 0u;
              // digits 0 .. 7 - i of B in pieces of at most 256 columns
#pragma unroll
              for (int n = 0; n < (kOD - i) * BN; n += 256) {
                constexpr int kMaxN = 256;
                const int nn = (kOD - i) * BN - n < kMaxN ? (kOD - i) * BN - n : kMaxN;
                omma(tmem + i * BN + n, ad, odesc(sb + n * 64 + j * 32), oidesc(nn), acc);
              }
            }
          }
          ocommit(&empty_bar[s]);
        }
        ocommit(&done_bar);
        k += kOChunk;
        if (k >= d.g[g].K) { ++g; k = 0; }
      }
      if (!ok) {
        *abort_v = 1;
        if (op.err) atomicOr(op.err, 1);
        // the MMAs issued so far must be complete before TMEM is freed
        ocommit(&drain_bar);
        omb_wait(&drain_bar, 0, nullptr);
      }
    } else if (warp == kOWork + 1 && lane == 0) {
      // ---- ready digits: one bulk copy per operand and stage ----
      bool ok = true;
      int g = g0, k = kfirst, it = 0;
      const uint32_t base = osmem(smem);
      for (int c = 0; c < nchunks && ok; ++c) {
        const int kend = min(d.g[g].K, k + kOChunk);
        const OzOperand &oa = op.a[g], &ob = op.b[g];
        for (int ks = k / kOBK; ks * kOBK < kend; ++ks, ++it) {
          const int s = it & 1;
          if (it >= 2 && !omb_wait(&empty_bar[s], ((it >> 1) - 1) & 1, abort_v, op.wait)) { ok = false; break; }
          const uint32_t bytes = (oa.img >= 0 ? kOD * kA : 0) + (ob.img >= 0 ? kOD * kB : 0);
          if (!bytes) { omb_arrive(&full_bar[s]); continue; }
          omb_expect(&full_bar[s], bytes);
          if (oa.img >= 0)
            bulk_load(base + s * kStage,
                      op.images + oa.img +
                          ((static_cast<long long>(b0 * oa.s0 + b1 * oa.s1) * oa.nrt + tm) * oa.nks + ks) * (kOD * kA),
                      kOD * kA, &full_bar[s]);
          if (ob.img >= 0)
            bulk_load(base + s * kStage + kOD * kA,
                      op.images + ob.img +
                          ((static_cast<long long>(b0 * ob.s0 + b1 * ob.s1) * ob.nrt + tn) * ob.nks + ks) * (kOD * kB),
                      kOD * kB, &full_bar[s]);
        }
        k += kOChunk;
        if (k >= d.g[g].K) { ++g; k = 0; }
      }
      if (!ok) *abort_v = 1;
      // copies in flight land before the CTA exits, also after an abort
      for (int q = max(0, it - 2); q < it; ++q) omb_wait(&full_bar[q & 1], (q >> 1) & 1, nullptr);
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    // ---- converters, then the flush of every chunk ----
    uint32_t acc[3][kPart];
#pragma unroll
    for (int j = 0; j < kPart; ++j) acc[0][j] = acc[1][j] = acc[2][j] = 0u;
    const int quarter = warp & 3, part = warp >> 2;   // 32 rows, kPart columns
    const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + part * kPart;
    bool ok = true;
    int flushed = 0;
    // A group's sums of output (m, n) are integers times 2^(ea[m] + eb[n] - kOScale);
    // with several groups they are shifted to the largest of these scales, which
    // the thread keeps for its outputs in shared memory after the stages (pairs of
    // columns, 16 bits each; only this thread reads them).  A shift common to the
    // tile would need one exponent per operand, and rows that are small as a whole
    // would lose their digits.
    const int orow = quarter * 32 + lane;             // of the tile
    uint32_t* top2 = reinterpret_cast<uint32_t*>(smem + 2 * kStage) + part * (kPart / 2) * kOBM + orow;
    auto row2 = [&](int fg) { return static_cast<uint32_t>(ea[fg][orow]) * 0x10001u; };
    auto col2 = [&](int fg, int j) { return *reinterpret_cast<const uint32_t*>(&eb[fg][part * kPart + j]); };
    if constexpr (kMulti) {
      uint32_t top[kPart / 2];
#pragma unroll
      for (int j = 0; j < kPart / 2; ++j) top[j] = 0u;
#pragma unroll 1
      for (int gi = 0; gi < d.ngroups; ++gi) {
        const uint32_t a2 = row2(gi);
#pragma unroll
        for (int j = 0; j < kPart / 2; ++j) top[j] = __vmaxu2(a2 + col2(gi, 2 * j), top[j]);
      }
#pragma unroll
      for (int j = 0; j < kPart / 2; ++j) top2[j * kOBM] = top[j];
    }
    constexpr int kF = 2;                            // columns combined together (registers)
    // add the eight accumulators of a finished chunk (of group fg) to acc
    auto flush = [&](int fg) {
      ok = __all_sync(0xffffffffu, ok && omb_wait(&done_bar, flushed & 1, abort_v, op.wait));
      ++flushed;
      if (!ok) return;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a2 = kMulti ? row2(fg) : 0u;
#pragma unroll
      for (int cb = 0; cb < kPart; cb += kF) {
        uint32_t v[kF][3];
        uint32_t r[kOD][kF];
        ld_levels(trow + cb, BN, r);
        static_assert(kF == 2, "a pair of columns per shift word");
        uint32_t sh2 = 0u;
        // (below a shift of 63, 2^-63 of the largest group's magnitudes per term)
        if constexpr (kMulti) sh2 = __vminu2(top2[cb / 2 * kOBM] - a2 - col2(fg, cb), 0x003F003Fu);
        ld_wait(r);
        combine(r, v);
        if constexpr (kMulti) {
          shift96(v[0], sh2 & 0xFFFFu);
          shift96(v[1], sh2 >> 16);
        }
#pragma unroll
        for (int j = 0; j < kF; ++j)
          asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
              : "+r"(acc[0][cb + j]), "+r"(acc[1][cb + j]), "+r"(acc[2][cb + j])
              : "r"(v[j][0]), "r"(v[j][1]), "r"(v[j][2]));
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      omb_arrive(&free_bar);
    };
    int it = 0, pend = -1;    // pend: group of the chunk that waits for its flush
    for (int c = 0; c <= nchunks && ok; ++c) {   // (one round more: the last flush)
      const int cg = g;
      const int nst = c == nchunks ? 0 : (min(d.g[g].K, k + kOChunk) - k + kOBK - 1) / kOBK;
      if (nst == 0 && nchunks == 1) break;       // a single chunk is stored from TMEM below
      // (a CTA without chunks has not entered a group: no rows)
#pragma unroll 1
      for (int st = 0; st < max(nst, 1); ++st, ++it) {
        const int s = it & 1;
        bool more = false;
        if (nst) {
          if (it >= 2) ok = __all_sync(0xffffffffu, omb_wait(&empty_bar[s], ((it >> 1) - 1) & 1, abort_v, op.wait));
          if (!ok) break;
          uint8_t* sA = smem + s * kStage;
          uint8_t* sB = sA + kOD * kA;
          more = !(c + 1 == nchunks && st + 1 == nst);
          if (b_on) store_digits(vb, cut_exponent(eb[cg][br]), sB, br, bc, kB);
          if (a_on) {
#pragma unroll
            for (int q = 0; q < kATasks; ++q) store_digits(va[q], cut_exponent(ea[cg][ar[q]]), sA, ar[q], ac[q], kA);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          omb_arrive(&full_bar[s]);
        }
        // the previous chunk is flushed once two stages of this one are staged
        if (pend >= 0 && (st == 1 || st + 1 >= nst)) {
          flush(pend);
          pend = -1;
          if (!ok) break;
        }
        // the next stage's loads: after the combination, whose registers they
        // would take (they have the time of the staged MMAs)
        if (more) {
          k += kOBK;
          if (k >= d.g[g].K) { ++g; k = 0; enter(); }
          if (b_on) load_b();
          if (a_on) {
#pragma unroll
            for (int q = 0; q < kATasks; ++q) load_a(q);
          }
        }
      }
      pend = cg;
    }
    const int m = m0 + quarter * 32 + lane;
    double* row = out_ptr(d, b, b0, b1, split, m, n0 + part * kPart);
    const long long sn = d.splits > 1 ? 1 : d.sc_n;
    const int nv = m < d.M ? min(kPart, d.N - (n0 + part * kPart)) : 0;
    const bool vec = sn == 1 && nv == kPart && (reinterpret_cast<uintptr_t>(row) & 15) == 0;
    // (split products: `row` is a partial sum, and the reduction writes the copy with C)
    float* row32 = d.c32 && d.splits <= 1 ? d.c32 + (row - static_cast<double*>(d.C)) : nullptr;
    auto put = [&](int j, double x, double y) {
      if (row32) {
        if (j < nv) row32[j * sn] = f64b::to_f32(x);
        if (j + 1 < nv) row32[(j + 1) * sn] = f64b::to_f32(y);
      }
      if (vec) {
        *reinterpret_cast<double2*>(row + j) = make_double2(x, y);
      } else {
        if (j < nv) row[j * sn] = x;
        if (j + 1 < nv) row[(j + 1) * sn] = y;
      }
    };
    if (ok && nchunks == 1) {
      // one chunk: straight from the accumulators, four columns at a time (a
      // short loop: unrolled, its instructions took longer to fetch than to run)
      ok = __all_sync(0xffffffffu, omb_wait(&done_bar, 0, abort_v, op.wait));
      if (ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // (with several groups the others' K ranges are empty here: no shift)
        const int fa = ea[g0][orow] - kOScale;
#pragma unroll 1
        for (int cb = 0; cb < kPart; cb += 4) {
          uint32_t v[4][3];
          uint32_t r[kOD][4];
          ld_levels(trow + cb, BN, r);
          ld_wait(r);
          combine(r, v);
          int e[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) e[j] = fa + eb[g0][part * kPart + cb + j];
#pragma unroll
          for (int j = 0; j < 4; j += 2)
            put(cb + j, to_double(v[j][0], v[j][1], v[j][2], e[j]),
                to_double(v[j + 1][0], v[j + 1][1], v[j + 1][2], e[j + 1]));
        }
      }
    } else if (ok) {
#pragma unroll
      for (int j = 0; j < kPart; j += 2) {
        const uint32_t t = kMulti ? top2[j / 2 * kOBM] : row2(0) + col2(0, j);
        put(j, to_double(acc[0][j], acc[1][j], acc[2][j], static_cast<int>(t & 0xFFFFu) - kOScale),
            to_double(acc[0][j + 1], acc[1][j + 1], acc[2][j + 1], static_cast<int>(t >> 16) - kOScale));
      }
    }
    if (!ok) {
      // an expired wait: reported, or where the caller has no flag to read the
      // warp's outputs are NaN
      *abort_v = 1;
      if (op.err && t == 0) atomicOr(op.err, 1);
      if (!op.err) {
        const double nan = __longlong_as_double(0x7FF8000000000000ll);
        for (int j = 0; j < kPart; j += 2) put(j, nan, nan);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kOWork)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
}


// Streamed products: one chunk of K, ready digits of A, more tiles than SMs.  A
// CTA takes an equal share of all 16-column blocks, in sub-tiles of at most 64
// columns of one row tile: every sub-tile's first two stages are staged before
// the one before it is combined, and no SM waits in a second round of tiles.
// With A ready, a converter thread has one task per stage where a tile that
// converts both operands has three.  256 tiles on 152 SMs are two rounds; 112
// columns per CTA (64 + 48) take 44 k clocks.  FP64 sweep at chi = 128: 25.57
// -> 25.29 ms, FP64 measurement of a Heisenberg chain: 3.44 -> 3.35 ms (the
// exchange of sides alone: 25.55 and 3.41); the sums are the same.
struct OzSub {
  int b, m0, n0, bn;
};

__global__ void __launch_bounds__(kOThreads, 1) gemm_oz_stream_kernel(const GemmDesc d, const OzParams op) {
  pdl_wait();
  pdl_trigger();
  constexpr int kMaxN = 64;
  constexpr int kA = kOBM * 64;                    // bytes of one digit tile of A of a stage
  constexpr int kStage = kOD * (kA + kMaxN * 64);
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  __shared__ __align__(8) uint64_t full_bar[2], empty_bar[2], done_bar, free_bar, drain_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ OzSub subs[kOBlocks];
  __shared__ short ea[kOBlocks][kOBM], eb[kOBlocks][kMaxN];   // exponents of a sub-tile's rows and columns
  __shared__ int range[4], plain_flag;               // lowest and highest of the rows', then of the columns'

  if (desc_skipped(d)) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blk_lo = static_cast<int>(static_cast<long long>(op.blocks) * blockIdx.x / gridDim.x);
  const int blk_hi = static_cast<int>(static_cast<long long>(op.blocks) * (blockIdx.x + 1) / gridDim.x);
  const int tiles_m = (d.M + kOBM - 1) / kOBM;
  auto sub_at = [&](int blk, OzSub& u) {
    const int row = blk / op.nb16, nb = blk - row * op.nb16;
    const int q = min(min(kMaxN / 16, op.nb16 - nb), blk_hi - blk);
    u.b = row / tiles_m;
    u.m0 = (row - u.b * tiles_m) * kOBM;
    u.n0 = nb * 16;
    u.bn = q * 16;
    return blk + q;
  };
  int nsub = 0;
  for (int blk = blk_lo; blk < blk_hi; ++nsub) {
    OzSub u;
    blk = sub_at(blk, u);
    if (threadIdx.x == 0) subs[nsub] = u;
  }
  if (nsub == 0) return;
  if (warp == kOWork) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(osmem(&tmem_slot)), "r"(kOD * kMaxN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  const Group& G = d.g[0];
  const OzOperand &oa = op.a[0], &ob = op.b[0];
  const int nst = (G.K + kOBK - 1) / kOBK;         // at most 4
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      omb_init(&full_bar[s], kOConv / 2 + 1);
      omb_init(&empty_bar[s], 1);
    }
    omb_init(&done_bar, 1);
    omb_init(&drain_bar, 1);
    omb_init(&free_bar, kOConv);
    abort_flag = 0;
    range[0] = range[2] = 0x7FFF;
    range[1] = range[3] = 0;
    plain_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  // converter state: half of the warps converts the even stages, the other half
  // the odd ones; each thread's cursor (cur, k) stands at its next stage, whose
  // values it has loaded
  const int hw = (threadIdx.x >> 8) & 1, t = threadIdx.x & 255;
  const bool bkf = G.b.s_k0 == 1;
  double vb[8];
  const double* pb = nullptr;
  bool bvec = false, b_on = false, fresh = true;
  int br = 0, bc = 0, k = 0, blk_next = 0;
  OzSub cur{};
  auto step = [&]() {                               // the cursor to the next stage
    k += kOBK;
    if (k < nst * kOBK) return;
    k = 0;
    fresh = true;
    if (blk_next < blk_hi) blk_next = sub_at(blk_next, cur);
    else cur.bn = 0;                                // (no stage left)
  };
  auto load_b = [&]() {
    if (fresh) {
      fresh = false;
      pb = static_cast<const double*>(G.b.p) + (cur.b % d.B0) * G.b.s_b0 + static_cast<long long>(cur.b / d.B0) * G.b.s_b1;
      bvec = bkf && ((reinterpret_cast<uintptr_t>(pb) & 15) == 0) && ((G.b.s_mn | G.b.s_k1) & 1) == 0;
      b_on = t < cur.bn * 4;
      // K contiguous: eight rows by four chunks per warp; MN contiguous: consecutive rows of one chunk
      bc = bkf ? t & 3 : t / max(cur.bn, 1);
      br = bkf ? t >> 2 : t - bc * cur.bn;
    }
    if (b_on)
      load8(G.b.s_mn, G.b.s_k0, G.b.s_k1, G.k0_log2, pb, cur.n0 + br, cur.n0 + br < d.N, k + 8 * bc, G.K, bvec, vb);
  };
  if (warp < kOWork) {
    blk_next = sub_at(blk_lo, cur);
    if (hw) step();
    load_b();
  }
  __syncthreads();
  // magnitudes: the exponents of every sub-tile's rows and columns
  constexpr int kRB = (kOBM + kMaxN) / 32;
  for (int u = warp; u < nsub * kRB; u += kOThreads / 32) {
    const int si = u / kRB, q = u % kRB;
    const bool isb = q >= kOBM / 32;
    const OzOperand& o = isb ? ob : oa;
    const OzSub w = subs[si];
    const int r = (isb ? q - kOBM / 32 : q) * 32 + lane, row = (isb ? w.n0 : w.m0) + r;
    unsigned m = 0;
    if (row < o.rows && (!isb || r < w.bn)) {
      const unsigned* p = op.words + o.off +
          static_cast<long long>((w.b % d.B0) * o.s0 + (w.b / d.B0) * o.s1) * o.parts * o.rows + row;
      for (int i = 0; i < o.parts; ++i) m = max(m, __ldcg(p + static_cast<long long>(i) * o.rows));
    }
    const int e = word_exponent(m);
    if (isb) eb[si][r] = static_cast<short>(e);
    else ea[si][r] = static_cast<short>(e);
    if (plain_row(e)) plain_flag = 1;
    add_range(&range[isb ? 2 : 0], e);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  const bool plain = plain_flag || plain_range(range);
  if (plain)
    for (int u = 0; u < nsub; ++u)
      plain_tile(d, subs[u].b, subs[u].b % d.B0, subs[u].b / d.B0, 0, subs[u].m0, subs[u].n0, subs[u].bn, 0, 1);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  volatile int* abort_v = &abort_flag;

  if (plain) {
    // (the tiles are done)
  } else if (warp == kOWork) {
    if (lane == 0) {
      // ---- MMA issuer ----
      bool ok = true;
      int it = 0;
      const uint32_t base = osmem(smem);
      for (int u = 0; u < nsub && ok; ++u) {
        const int bn = subs[u].bn;
        if (u > 0 && !omb_wait(&free_bar, (u - 1) & 1, abort_v, op.wait)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int st = 0; st < nst; ++st, ++it) {
          const int s = it & 1;
          if (!omb_wait(&full_bar[s], (it >> 1) & 1, abort_v, op.wait)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = base + s * kStage, sb = sa + kOD * kA;
#pragma unroll 1
          for (int j = 0; j < 2; ++j) {
#pragma unroll
            for (int i = 0; i < kOD; ++i) {
              const uint64_t ad = odesc(sa + i * kA + j * 32);
              const uint32_t acc = (st > 0 || j > 0 || i > 0) ? 1u : 0u;
              // digits 0 .. 7 - i of B in pieces of at most 256 columns
              const int cols = (kOD - i) * bn;
              omma(tmem + i * bn, ad, odesc(sb + j * 32), oidesc(min(256, cols)), acc);
              if (cols > 256)
                omma(tmem + i * bn + 256, ad, odesc(sb + 256 * 64 + j * 32), oidesc(cols - 256), acc);
            }
          }
          ocommit(&empty_bar[s]);
        }
        ocommit(&done_bar);
      }
      if (!ok) {
        *abort_v = 1;
        if (op.err) atomicOr(op.err, 1);
        // the MMAs issued so far must be complete before TMEM is freed
        ocommit(&drain_bar);
        omb_wait(&drain_bar, 0, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == kOWork + 1) {
    if (lane == 0) {
      // ---- A: one bulk copy of ready digits per stage ----
      bool ok = true;
      int it = 0;
      const uint32_t base = osmem(smem);
      for (int u = 0; u < nsub && ok; ++u) {
        const int b0 = subs[u].b % d.B0, b1 = subs[u].b / d.B0;
        const uint8_t* src = op.images + oa.img +
            (static_cast<long long>(b0 * oa.s0 + b1 * oa.s1) * oa.nrt + subs[u].m0 / kOBM) * oa.nks * (kOD * kA);
        for (int st = 0; st < nst; ++st, ++it) {
          const int s = it & 1;
          if (it >= 2 && !omb_wait(&empty_bar[s], ((it >> 1) - 1) & 1, abort_v, op.wait)) { ok = false; break; }
          omb_expect(&full_bar[s], kOD * kA);
          bulk_load(base + s * kStage, src + st * (kOD * kA), kOD * kA, &full_bar[s]);
        }
      }
      if (!ok) *abort_v = 1;
      // copies in flight land before the CTA exits, also after an abort
      for (int q = max(0, it - 2); q < it; ++q) omb_wait(&full_bar[q & 1], (q >> 1) & 1, nullptr);
    }
    __syncwarp();
  } else if (warp < kOWork) {
    // ---- converters; each sub-tile is combined and stored once two stages of the next are staged ----
    const int quarter = warp & 3, part = warp >> 2;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    bool ok = true;
    int stored = 0;                                   // sub-tiles
    auto flush = [&](int u) {
      ok = __all_sync(0xffffffffu, ok && omb_wait(&done_bar, u & 1, abort_v, op.wait));
      if (!ok) return;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const OzSub w = subs[u];
      const int fa = ea[u][quarter * 32 + lane] - kOScale, hc = w.bn >> 2;   // this warp's columns: 4, 8, 12 or 16
      const uint32_t tcol = trow + part * hc;
      const int m = w.m0 + quarter * 32 + lane, nf = w.n0 + part * hc;
      double* row = out_ptr(d, w.b, w.b % d.B0, w.b / d.B0, 0, m, nf);
      const long long sn = d.sc_n;
      const int nv = m < d.M ? min(hc, d.N - nf) : 0;
      const bool vec = sn == 1 && nv == hc && (reinterpret_cast<uintptr_t>(row) & 15) == 0;
      float* row32 = d.c32 ? d.c32 + (row - static_cast<double*>(d.C)) : nullptr;
      auto put = [&](int j, double x, double y) {
        if (row32) {
          if (j < nv) row32[j * sn] = f64b::to_f32(x);
          if (j + 1 < nv) row32[(j + 1) * sn] = f64b::to_f32(y);
        }
        if (vec) {
          *reinterpret_cast<double2*>(row + j) = make_double2(x, y);
        } else {
          if (j < nv) row[j * sn] = x;
          if (j + 1 < nv) row[(j + 1) * sn] = y;
        }
      };
#pragma unroll 1
      for (int cb = 0; cb < hc; cb += 4) {
        uint32_t r[kOD][4], v[4][3];
        ld_levels(tcol + cb, w.bn, r);
        ld_wait(r);
        if (cb + 4 >= hc) {                         // (all accumulators are in registers)
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          omb_arrive(&free_bar);
        }
        combine(r, v);
        int e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) e[j] = fa + eb[u][part * hc + cb + j];
#pragma unroll
        for (int j = 0; j < 4; j += 2)
          put(cb + j, to_double(v[j][0], v[j][1], v[j][2], e[j]),
              to_double(v[j + 1][0], v[j + 1][1], v[j + 1][2], e[j + 1]));
      }
      stored = u + 1;
    };
    int it = 0;
    for (int u = 0; u < nsub && ok; ++u) {
#pragma unroll 1
      for (int st = 0; st < nst; ++st, ++it) {
        if ((it & 1) == hw) {
          if (it >= 2) ok = __all_sync(0xffffffffu, omb_wait(&empty_bar[hw], ((it >> 1) - 1) & 1, abort_v, op.wait));
          if (!ok) break;
          if (b_on) store_digits(vb, cut_exponent(eb[u][br]), smem + hw * kStage + kOD * kA, br, bc, subs[u].bn * 64);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          omb_arrive(&full_bar[hw]);
          step();
          step();
          load_b();
        }
        if (u > 0 && st == min(1, nst - 1)) {
          flush(u - 1);
          if (!ok) break;
        }
      }
    }
    if (ok) flush(nsub - 1);
    if (!ok) {
      *abort_v = 1;
      if (op.err && threadIdx.x == 0) atomicOr(op.err, 1);
      // (without a flag: NaN, as above)
      for (int u = stored; u < nsub && !op.err; ++u) {
        const OzSub w = subs[u];
        const int hc = w.bn >> 2, m = w.m0 + quarter * 32 + lane, nf = w.n0 + part * hc;
        double* row = out_ptr(d, w.b, w.b % d.B0, w.b / d.B0, 0, m, nf);
        for (int j = 0; j < hc; ++j)
          if (m < d.M && nf + j < d.N) row[j * d.sc_n] = __longlong_as_double(0x7FF8000000000000ll);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kOWork)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kOD * kMaxN));
}

template <int BN>
constexpr int oz_smem() { return 2 * kOD * (kOBM + BN) * 64 + BN * kOBM * 2 + 1024; }   // stages, scales, alignment

int oz_chunks(const GemmDesc& d) {
  int t = 0;
  for (int g = 0; g < d.ngroups; ++g) t += (d.g[g].K + kOChunk - 1) / kOChunk;
  return t;
}

int oz_bn(const GemmDesc& d) { return oz_tile_n(d.N); }

bool same_operand(const AbsItem& a, const AbsItem& b) {
  return a.p == b.p && a.s_mn == b.s_mn && a.s_k0 == b.s_k0 && a.s_k1 == b.s_k1 && a.s_b0 == b.s_b0 &&
         a.s_b1 == b.s_b1 && a.mn == b.mn && a.k == b.k &&
         a.k0_log2 == b.k0_log2 && a.n0 == b.n0 && a.n1 == b.n1 && a.rt == b.rt && (a.img >= 0) == (b.img >= 0);
}

// Digits prepared in memory for an operand that at least kOzReuse CTAs read
// per row tile, while all its batches' digits stay below kOzImageMax bytes: the
// tiles' converters then have the other operand only, and the bulk copy of a
// stage costs them nothing.  (Digits take 16 bytes per value where FP64 takes
// 8, so a large operand is converted by the tiles that read it.)
constexpr int kOzReuse = 8;
constexpr long long kOzImageMax = 4 << 20;
constexpr long long kOzImageCount = 1 << 16;   // values of a batch

// The preparation of a product: items (operands, without repeats), their words
// and images; returns the blocks of oz_prepare_kernel.
struct OzPlan {
  AbsParams ap;
  OzParams op;
  int blocks;
  long long words, image_bytes;
  bool stream;
};

void plan_product(const GemmDesc& d, OzPlan& pl) {
  // (the tables are read up to ap.n and ngroups only; clearing their 9 KB for every
  // product cost a context's creation 0.2 ms)
  pl.ap.n = 0;
  pl.blocks = 0;
  pl.words = pl.image_bytes = 0;
  const int bn = oz_bn(d);
  const long long tm = (d.M + kOBM - 1) / kOBM, tn = (d.N + bn - 1) / bn, nb = static_cast<long long>(d.B0) * d.B1;
  AbsParams& ap = pl.ap;
  int chunk0 = 0;
  for (int g = 0; g < d.ngroups; ++g) {
    const int chunks = (d.g[g].K + kOChunk - 1) / kOChunk;
    for (int side = 0; side < 2; ++side) {
      const Group& G = d.g[g];
      const Operand& o = side ? G.b : G.a;
      AbsItem it;
      memset(&it, 0, sizeof(it));
      it.p = static_cast<const double*>(o.p);
      it.s_mn = o.s_mn; it.s_k0 = o.s_k0; it.s_k1 = o.s_k1; it.s_b0 = o.s_b0; it.s_b1 = o.s_b1;
      it.mn = side ? d.N : d.M;
      it.k = G.K;
      it.k0_log2 = G.k0_log2;
      it.n0 = o.s_b0 ? d.B0 : 1;
      it.n1 = o.s_b1 ? d.B1 : 1;
      it.rt = side ? bn : kOBM;
      it.nrt = (it.mn + it.rt - 1) / it.rt;
      it.nks = (G.K + kOBK - 1) / kOBK;
      const long long batches = static_cast<long long>(it.n0) * it.n1;
      const long long bytes = batches * it.nrt * it.nks * kOD * it.rt * 64;
      const long long reuse = (side ? tm : tn) * nb / batches;
      const bool image = reuse >= kOzReuse && bytes <= kOzImageMax && static_cast<long long>(it.mn) * G.K <= kOzImageCount;
      it.img = image ? 0 : -1;
      it.parts = 1;
      it.len_log2 = 30;                      // (ready digits: one part, all of K)
      if (!image) {
        // blocks of 32 rows (64 or 128 where K is short) by a part of K, a power of
        // two of at least a chunk: as many parts as make kAbsBlocks blocks
        it.rt = G.K > 64 ? 32 : (G.K > 32 ? 64 : 128);
        it.nrt = (it.mn + it.rt - 1) / it.rt;
        const long long want = std::max<long long>(1, std::min<long long>(kOzMaxParts, kAbsBlocks / (batches * it.nrt)));
        it.len_log2 = 7;
        while (((G.K - 1) >> it.len_log2) + 1 > want) ++it.len_log2;
        it.parts = ((G.K - 1) >> it.len_log2) + 1;
      }
      int at = 0;
      while (at < ap.n && !same_operand(ap.it[at], it)) ++at;
      if (at == ap.n) {
        it.off = static_cast<int>(pl.words);
        it.blocks_before = pl.blocks;
        pl.words += it.parts * batches * it.mn;
        if (image) {
          it.img = pl.image_bytes;
          pl.image_bytes += bytes;
        }
        pl.blocks += static_cast<int>(batches) * it.nrt * (image ? it.nks : it.parts);
        ap.it[ap.n++] = it;
      }
      OzOperand& w = side ? pl.op.b[g] : pl.op.a[g];
      w.off = ap.it[at].off;
      w.parts = ap.it[at].parts;
      w.len_log2 = ap.it[at].len_log2;
      w.rows = it.mn;
      w.s0 = o.s_b0 ? 1 : 0;
      w.s1 = o.s_b1 ? it.n0 : 0;
      w.nrt = it.nrt;
      w.nks = it.nks;
      w.img = ap.it[at].img;
      w.chunk0 = chunk0;
      w.chunks = chunks;
    }
    pl.op.a[g].whole = pl.op.b[g].whole = pl.op.a[g].img >= 0 || pl.op.b[g].img >= 0;
    chunk0 += chunks;
  }
  // (at most as many tiles as SMs: one round of tiles is as short)
  pl.stream = d.ngroups == 1 && d.g[0].K <= kOChunk && bn == 64 && pl.op.a[0].img >= 0 && pl.op.b[0].img < 0 &&
              tm * tn * nb > device_sm_count() && tm * tn * nb < (1LL << 28);
}

// C^T = B^T A^T: the same sums with the sides exchanged.
GemmDesc exchanged(const GemmDesc& d) {
  GemmDesc e = d;
  std::swap(e.M, e.N);
  std::swap(e.sc_m, e.sc_n);
  for (int g = 0; g < e.ngroups; ++g) std::swap(e.g[g].a, e.g[g].b);
  return e;
}

// A large operand times a small one (more tiles than SMs, one chunk of K): the
// side that is ready in memory becomes A, whatever the caller named it, so that
// every value of the large one is cut into digits once; a tile has 128 rows of
// A, so an exchange that leaves more than half of one empty is not made.
bool exchange_sides(const GemmDesc& d) {
  const int rest = d.N % kOBM;
  return d.ngroups == 1 && d.g[0].K <= kOChunk && d.splits <= 1 && d.M > d.N && (rest == 0 || rest > kOBM / 2);
}

}  // namespace

// Products the digit engine takes: FP64 in and out, K0 a whole number of
// 16-byte digit chunks, and those that it is the faster engine for (oz_rule.h).
bool gemm_oz_supported(const GemmDesc& d) {
  if (!d.digits || d.prec != 0 || d.c_f32 || d.alpha != 1.0 || d.beta != 0.0 || d.ngroups < 1 ||
      d.ngroups > kMaxGroups || d.M < 1 || d.N < 1)
    return false;
  int K[kMaxGroups];
  for (int g = 0; g < d.ngroups; ++g) {
    const Group& G = d.g[g];
    if (G.a.f32 || G.b.f32 || G.K < 1) return false;
    if (G.k0_log2 < 3 && (G.K >> G.k0_log2) > 1) return false;
    K[g] = G.K;
  }
  return d.M >= 16 && d.N >= 16 && oz_worth(d.M, d.N, static_cast<long long>(d.B0) * d.B1, K, d.ngroups);
}

int oz_pick_splits(const GemmDesc& d) {
  const int bn = oz_bn(d);
  const long long base = static_cast<long long>((d.M + kOBM - 1) / kOBM) * ((d.N + bn - 1) / bn) * d.B0 * d.B1;
  const int sms = device_sm_count();
  if (2 * base > sms) return 1;
  return static_cast<int>(std::max<long long>(1, std::min<long long>(sms / base, oz_chunks(d))));
}

// Bytes of scratch for a product: the magnitude words, then the images.
static size_t words_bytes(long long words) { return (static_cast<size_t>(words) * sizeof(unsigned) + 255) & ~size_t(255); }

size_t oz_scratch(const GemmDesc& d) {
  if (!gemm_oz_supported(d)) return 0;
  static thread_local OzPlan pl;
  plan_product(d, pl);
  size_t bytes = words_bytes(pl.words) + static_cast<size_t>(pl.image_bytes);
  if (exchange_sides(d)) {
    plan_product(exchanged(d), pl);
    bytes = std::max(bytes, words_bytes(pl.words) + static_cast<size_t>(pl.image_bytes));
  }
  return bytes;
}

// Returns the launches, or -1 when the scratch is too small (nothing launched).
int gemm_oz_launch(const GemmDesc& d0, cudaStream_t s) {
  static thread_local OzPlan pl;
  GemmDesc d = d0;
  bool planned = false;
  if (exchange_sides(d0)) {
    d = exchanged(d0);
    plan_product(d, pl);
    planned = pl.stream;
  }
  if (!planned) {
    d = d0;
    plan_product(d, pl);
  }
  if (words_bytes(pl.words) + static_cast<size_t>(pl.image_bytes) > d.words_bytes) return -1;
  pl.ap.words = d.words;
  pl.ap.images = reinterpret_cast<uint8_t*>(d.words) + words_bytes(pl.words);
  pl.ap.skip = d.skip;
  pl.ap.skip_when_zero = d.skip_when_zero;
  launch_k(oz_prepare_kernel, pl.blocks, 256, 0, s, pl.ap);
  pl.op.words = pl.ap.words;
  pl.op.images = pl.ap.images;
  pl.op.total_chunks = oz_chunks(d);
  pl.op.wait = d.no_waits ? 0 : kOWait;
  pl.op.err = d.err;
  if (pl.stream && d.splits <= 1) {
    // one CTA per SM, or more when a CTA's share would exceed kOBlocks
    pl.op.nb16 = (d.N + 15) / 16;
    const long long blocks = static_cast<long long>((d.M + kOBM - 1) / kOBM) * d.B0 * d.B1 * pl.op.nb16;
    const long long sms = device_sm_count(), waves = (blocks + sms * kOBlocks - 1) / (sms * kOBlocks);
    pl.op.blocks = static_cast<int>(blocks);
    launch_attr(true, gemm_oz_stream_kernel, dim3(static_cast<unsigned>(waves * sms)), kOThreads, oz_smem<64>(), s, d, pl.op);
    return 2;
  }
  const int bn = oz_bn(d);
  dim3 grid(((d.M + kOBM - 1) / kOBM) * ((d.N + bn - 1) / bn), d.B0 * d.B1, d.splits);
  // always with programmatic serialisation: its only predecessor is the
  // preparation, so its CTAs wait for nothing else
  const bool multi = d.ngroups > 1;
  if (bn == 64)
    launch_attr(true, multi ? gemm_oz_kernel<64, true> : gemm_oz_kernel<64, false>, grid, kOThreads, oz_smem<64>(), s, d, pl.op);
  else
    launch_attr(true, multi ? gemm_oz_kernel<32, true> : gemm_oz_kernel<32, false>, grid, kOThreads, oz_smem<32>(), s, d, pl.op);
  return 2;
}

void gemm_oz_init() {
  cudaFuncSetAttribute(gemm_oz_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz_smem<64>());
  cudaFuncSetAttribute(gemm_oz_kernel<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz_smem<64>());
  cudaFuncSetAttribute(gemm_oz_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, oz_smem<64>());
  cudaFuncSetAttribute(gemm_oz_kernel<32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz_smem<32>());
  cudaFuncSetAttribute(gemm_oz_kernel<32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz_smem<32>());
}

}  // namespace ttn
