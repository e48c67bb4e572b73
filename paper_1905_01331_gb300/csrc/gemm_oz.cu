// FP64 products on the tensor cores ("digit engine"), sm_103a.
//
// GB300 has two FP64 FMA units per SM (1.1 TFLOP/s for the whole GPU), so a
// plain FP64 product is bound by them at any shape.  Here every FP64 operand is
// cut into eight signed base-256 digits relative to the power of two above the
// operand's largest magnitude (62 bits: elements within 2^-9 of the largest
// are represented exactly) -- the error-free splitting of Ozaki, Ogita, Oishi
// and Rump, "Error-free transformations of matrix multiplication", Numer.
// Algorithms 59 (2012), with digits in place of floating-point slices (Mukunoki
// et al., "DGEMM using tensor cores", ISC 2020).  A digit is an integer in
// [-128, 127], exact in BF16; a product of two digits is below 2^14, and the
// digit products of one weight (i + j = l <= 7) over 128 values of K stay below
// 2^24, so the tensor cores' FP32 accumulation of them is exact.  The 36 digit
// products with i + j <= 7 go to eight accumulators, one per weight; what is
// dropped is below 2^-62 of max|A| max|B| per term.  Every 128 values of K the
// accumulators are combined into a 96-bit integer per output, which is rounded
// to FP64 once at the end: the result carries one rounding instead of one per
// term.
//
// One CTA owns a 128 x BN output tile (BN 64 or 32).  Warps 0-7 load FP64
// operands (any strides), cut them into digits with integer operations and
// write them to shared memory in the K-major SWIZZLE_128B layout (two stages of
// 32 K values: the two halves of the 128-byte rows); warp 8 issues the MMAs.
// The digits of B are stacked along N, so that one MMA multiplies A's digit i
// with B's digits 0 .. 7 - i and adds each product to the accumulator of its
// weight: TMEM columns (i + j) BN .. of the same instruction.  All waits are
// bounded, as in the other tensor-core kernels.
//
// Measured on a GB300 (P = n = 128): F X of 128 x 128 by 128 x 16384 takes 55
// us, the FP64 kernel 553 (its two FMA units per SM are busy throughout); the
// environment's five such products in one 186 against 2706, three close
// products over K = 16384 123 against 1976; relative error against extended
// precision 4e-17 to 2e-16 where the FP64 kernel has 2e-16 to 2e-15.  At n =
// 32 both take 15 to 30 us (latency), so kOzMinWork lies between n = 32 (2^20
// multiply-adds) and n = 64 (2^24: 24 against 62 us).
//
// An operand with an infinity or NaN, or whose range would leave the normal
// FP64 numbers, makes the CTA compute its tile with plain FP64 FMAs instead, so
// that the result is what the FP64 kernel gives.
#include <algorithm>
#include <cstdint>
#include <cstring>

#include <cuda_bf16.h>

#include "common.h"

namespace ttn {

namespace {

constexpr int kOD = 8;              // digits per operand
constexpr int kOBM = 128;
constexpr int kOChunk = 128;        // K values per exact accumulation
constexpr int kOBK = 32;            // K values per stage
constexpr int kOConv = 256;         // converter threads
constexpr int kOThreads = kOConv + 128;   // and the MMA warp's warpgroup
constexpr long kOWait = 1L << 22;

// Largest magnitude of an operand: absmax_kernel leaves `parts` words (the high
// words of |x|, at least 1 for a nonzero x) per operand and batch.
struct OzOperand {
  int off, parts, n0, s0, s1;       // word of batch (b0, b1): off + (b0 s0 + b1 s1) parts
};
struct OzParams {
  const unsigned* words;
  OzOperand a[kMaxGroups], b[kMaxGroups];
  int total_chunks;
  int* err;
};

struct AbsItem {
  const double* p;
  long long s_mn, s_k0, s_k1, s_b0, s_b1, count;
  int flat, mn, k0_log2, k, n0, n1, parts, off, blocks_before, pad;
};
constexpr int kAbsPer = 8192;       // elements per block of absmax_kernel
constexpr int kAbsMaxParts = 256;
struct AbsParams {
  AbsItem it[2 * kMaxGroups];
  int n;
  unsigned* words;
};
static_assert(sizeof(AbsParams) < 32000, "kernel parameter");

__device__ __forceinline__ unsigned mag_word(double x) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(x)) & 0x7FFFFFFFu;
  return hi | (__double2loint(x) != 0 ? 1u : 0u);
}

// words[off + batch parts + part] = the largest magnitude word of that part of
// the operand's batch.  Bound by the read of the operands (from L2 when they
// were just produced).
__global__ void __launch_bounds__(256) absmax_kernel(const AbsParams ap) {
  pdl_wait();
  pdl_trigger();
  int i = 0;
  while (i + 1 < ap.n && static_cast<int>(blockIdx.x) >= ap.it[i + 1].blocks_before) ++i;
  const AbsItem& it = ap.it[i];
  const int u = blockIdx.x - it.blocks_before;
  const int batch = u / it.parts, part = u % it.parts;
  const int b0 = batch % it.n0, b1 = batch / it.n0;
  const double* p = it.p + b0 * it.s_b0 + static_cast<long long>(b1) * it.s_b1;
  const long long lo = it.count * part / it.parts, hi = it.count * (part + 1) / it.parts;
  unsigned m = 0;
  if (it.flat) {
    long long e = lo + threadIdx.x;
    for (; e + 7 * 256 < hi; e += 8 * 256) {
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = p[e + q * 256];
#pragma unroll
      for (int q = 0; q < 8; ++q) m = max(m, mag_word(v[q]));
    }
    for (; e < hi; e += 256) m = max(m, mag_word(p[e]));
  } else {
    for (long long e = lo + threadIdx.x; e < hi; e += 256) {
      const long long k = e / it.mn, r = e - k * it.mn;
      const long long k0 = k & ((1LL << it.k0_log2) - 1), k1 = k >> it.k0_log2;
      m = max(m, mag_word(p[r * it.s_mn + k0 * it.s_k0 + k1 * it.s_k1]));
    }
  }
  m = __reduce_max_sync(0xffffffffu, m);
  __shared__ unsigned sh[8];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) m = max(m, sh[w]);
    ap.words[it.off + u] = m;
  }
}

__device__ __forceinline__ uint32_t osmem(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool omb_wait(uint64_t* bar, uint32_t parity, const volatile int* abort_flag) {
  const uint32_t a = osmem(bar);
  for (long it = 0; it < kOWait; ++it) {
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
__device__ __forceinline__ void ocommit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(osmem(bar))
      : "memory");
}
// K-major, 128-byte swizzle, 8-row atoms stacked every 1024 bytes.
__device__ __forceinline__ uint64_t odesc(uint32_t saddr) {
  return static_cast<uint64_t>((saddr >> 4) & 0x3FFF) | (1ull << 16) |
         (static_cast<uint64_t>(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void omma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}
// D = F32, A and B BF16, both K-major.
__host__ __device__ constexpr uint32_t oidesc(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(kOBM >> 4) << 24);
}

// The eight digits of x as bytes (digit + 128; the most significant digit in
// the highest byte), for |x| below 2^(emax - 1022): x / 2^(emax - 1084), cut
// to an integer, plus 128 in every byte.
__device__ __forceinline__ void digit_bytes(double x, int emax, uint32_t& lo, uint32_t& hi) {
  const uint32_t h = static_cast<uint32_t>(__double2hiint(x)), l = static_cast<uint32_t>(__double2loint(x));
  const int e = (h >> 20) & 0x7FF;
  const uint32_t mh = (h & 0xFFFFFu) | 0x100000u;
  unsigned long long v = (static_cast<unsigned long long>(__funnelshift_l(l, mh, 9)) << 32) | (l << 9);
  const int sh = emax - e;
  v = sh < 64 ? v >> sh : 0ull;                 // a subnormal x (e = 0) is far below the cut
  const long long s = static_cast<int>(h) >> 31;
  v = (v ^ s) - s + 0x8080808080808080ull;
  lo = static_cast<uint32_t>(v);
  hi = static_cast<uint32_t>(v >> 32);
}

// Two digits (bytes b of w0 and w1, each digit + 128) as a BF16 pair, by BF16
// arithmetic that is exact: 128 + (u mod 128) minus 256 (u < 128) or 128.
template <int b>
__device__ __forceinline__ uint32_t digit_pair(uint32_t w0, uint32_t w1) {
  const uint32_t t = __byte_perm(w0, w1, 0x0400 + 0x0101 * b);
  const uint32_t y = (t & 0x007F007Fu) | 0x43004300u;
  const uint32_t z = (t & 0x00800080u) ^ 0x43804380u;
  const __nv_bfloat162 r = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&y),
                                   *reinterpret_cast<const __nv_bfloat162*>(&z));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// Eight consecutive K values of one row -> a 16-byte chunk of each digit tile.
template <int ROWS>
__device__ __forceinline__ void store_digits(const double* v, int emax, uint8_t* tile, int r, int chunk) {
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) digit_bytes(v[q], emax, lo[q], hi[q]);
  uint8_t* p = tile + r * 128 + ((chunk ^ (r & 7)) << 4);
  constexpr int kTile = ROWS * 128;
#define TTN_OZ_DIGIT(d, w, b)                                                              \
  *reinterpret_cast<uint4*>(p + (d) * kTile) =                                             \
      make_uint4(digit_pair<b>(w[0], w[1]), digit_pair<b>(w[2], w[3]),                     \
                 digit_pair<b>(w[4], w[5]), digit_pair<b>(w[6], w[7]));
  TTN_OZ_DIGIT(0, hi, 3) TTN_OZ_DIGIT(1, hi, 2) TTN_OZ_DIGIT(2, hi, 1) TTN_OZ_DIGIT(3, hi, 0)
  TTN_OZ_DIGIT(4, lo, 3) TTN_OZ_DIGIT(5, lo, 2) TTN_OZ_DIGIT(6, lo, 1) TTN_OZ_DIGIT(7, lo, 0)
#undef TTN_OZ_DIGIT
}

// Position of the converters in the K range of a CTA: stage k0 .. k0 + 31 of
// group g, `left` stages in its chunk after it.
struct OzCursor {
  int g, k, chunk;     // group, first K value, chunk counted over all groups
};

// Row and 16-byte chunk of converter task `task` of a stage (4 chunks per row):
// K contiguous: eight rows by four chunks per warp, rows r and r + 4 in the
// same eight-thread store phase (their swizzled halves are disjoint); MN
// contiguous: 32 consecutive rows of one chunk per warp.
template <int ROWS>
__device__ __forceinline__ void task_pos(int task, bool kfast, int& r, int& c) {
  const int w = task >> 5, lane = task & 31;
  if (kfast) {
    r = w * 8 + ((lane >> 2) & 1) * 4 + (lane >> 3);
    c = lane & 3;
  } else {
    r = (w % (ROWS / 32)) * 32 + lane;
    c = w / (ROWS / 32);
  }
}

__device__ __forceinline__ void load8(const Operand& o, int k0_log2, const double* base, int row, bool row_ok,
                                      int k, int K, bool vec, double* v) {
  if (!row_ok || k >= K) {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = 0.0;
    return;
  }
  const int k0 = k & ((1 << k0_log2) - 1), k1 = k >> k0_log2;
  const double* p = base + row * o.s_mn + k0 * o.s_k0 + static_cast<long long>(k1) * o.s_k1;
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
      for (int q = 0; q < 8; ++q) v[q] = p[q * o.s_k0];
    }
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = k + q < K ? p[q * o.s_k0] : 0.0;
  }
}

// The 96-bit integer (a2 a1 a0, two's complement) times 2^scale, rounded to
// FP64 (the caller has checked that the result is zero or a normal number).
__device__ __forceinline__ double to_double(uint32_t a0, uint32_t a1, uint32_t a2, int scale) {
  const uint32_t neg = static_cast<uint32_t>(static_cast<int>(a2) >> 31);
  a0 ^= neg; a1 ^= neg; a2 ^= neg;
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, %2, 0;"
      : "+r"(a0), "+r"(a1), "+r"(a2)
      : "r"(neg & 1u));
  int pos = 95;
  if (a2 == 0u) { a2 = a1; a1 = a0; a0 = 0u; pos = 63; }
  if (a2 == 0u) { a2 = a1; a1 = 0u; pos = 31; }
  if (a2 == 0u) return 0.0;
  const int n = __clz(a2);
  const uint32_t t1 = __funnelshift_l(a1, a2, n), t0 = __funnelshift_l(a0, a1, n);
  const unsigned long long t = (static_cast<unsigned long long>(t1) << 32) | t0;
  const unsigned long long m = (t >> 11) + ((t >> 10) & 1ull);
  const unsigned long long bits =
      (static_cast<unsigned long long>(pos - n + scale + 1022) << 52) + m +
      (static_cast<unsigned long long>(neg & 0x80000000u) << 32);
  return __longlong_as_double(static_cast<long long>(bits));
}

// Output (or split-K partial) of one element.
__device__ __forceinline__ double* out_ptr(const GemmDesc& d, int b, int b0, int b1, int split, int m, int n) {
  if (d.splits > 1)
    return d.partial + ((static_cast<long long>(split) * d.B0 * d.B1 + b) * d.M + m) * d.N + n;
  return static_cast<double*>(d.C) + b0 * d.sc_b0 + static_cast<long long>(b1) * d.sc_b1 + m * d.sc_m + n * d.sc_n;
}

// Plain FP64 tile over the CTA's chunks (operands with infinities or NaN, or a
// range that the digits do not cover).
template <int BN>
__device__ __noinline__ void plain_tile(const GemmDesc& d, int b, int b0, int b1, int split, int m0, int n0,
                                        int c_lo, int c_hi) {
  for (int e = threadIdx.x; e < kOBM * BN; e += kOThreads) {
    const int m = m0 + e / BN, n = n0 + e % BN;
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
    *out_ptr(d, b, b0, b1, split, m, n) = acc;
  }
}

template <int BN>
__global__ void __launch_bounds__(kOThreads, 1) gemm_oz_kernel(const GemmDesc d, const OzParams op) {
  pdl_wait();
  pdl_trigger();
  constexpr int kA = kOBM * 128;                   // bytes of one digit tile of A
  constexpr int kHalf = BN / 2;                    // columns per flush warp
  constexpr int kCols = kOD * BN;                  // TMEM columns
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sA = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sB = sA + kOD * kA;
  __shared__ __align__(8) uint64_t full_bar[2], empty_bar[2], done_bar, free_bar, drain_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ unsigned ex[2 * kMaxGroups];

  if (desc_skipped(d)) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_n = (d.N + BN - 1) / BN;
  const int tm = blockIdx.x / tiles_n, tn = blockIdx.x % tiles_n;
  const int b = blockIdx.y, b0 = b % d.B0, b1 = b / d.B0;
  const int split = blockIdx.z;
  const int m0 = tm * kOBM, n0 = tn * BN;
  const int c_lo = static_cast<int>(static_cast<long long>(op.total_chunks) * split / d.splits);
  const int c_hi = static_cast<int>(static_cast<long long>(op.total_chunks) * (split + 1) / d.splits);

  // largest magnitude of every operand
  for (int i = warp; i < 2 * d.ngroups; i += kOThreads / 32) {
    const OzOperand& o = (i & 1) ? op.b[i >> 1] : op.a[i >> 1];
    const unsigned* w = op.words + o.off + static_cast<long long>(b0 * o.s0 + b1 * o.s1) * o.parts;
    unsigned m = 0;
    for (int q = lane; q < o.parts; q += 32) m = max(m, __ldcg(w + q));
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) ex[i] = m;
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      omb_init(&full_bar[s], kOConv);
      omb_init(&empty_bar[s], 1);
    }
    omb_init(&done_bar, 1);
    omb_init(&drain_bar, 1);
    omb_init(&free_bar, kOConv);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // the scale of a group's digit products is 2^(ea + eb - 68); all groups are
  // added relative to the largest one
  int sref = -100000;
  bool plain = false;
  for (int g = 0; g < d.ngroups; ++g) {
    const unsigned wa = ex[2 * g], wb = ex[2 * g + 1];
    if (wa >= 0x7FF00000u || wb >= 0x7FF00000u) plain = true;
    if (wa == 0u || wb == 0u) continue;      // an all-zero operand
    const int s = static_cast<int>(wa >> 20) + static_cast<int>(wb >> 20) - 2 * 1022 - 68;
    if (wa < (80u << 20) || wb < (80u << 20)) plain = true;
    sref = max(sref, s);
  }
  if (sref != -100000 && (sref < -1000 || sref > 900)) plain = true;
  if (plain) {
    plain_tile<BN>(d, b, b0, b1, split, m0, n0, c_lo, c_hi);
    return;
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(osmem(&tmem_slot)), "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  volatile int* abort_v = &abort_flag;

  // first chunk of the CTA: group g, K offset k
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

  // registers: three warpgroups of 168 at launch -> 72 for the MMA warp's, 216
  // for the two of the converters (2 x 216 + 72 = 3 x 168)
  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp == 8 && lane == 0) {
      // ---- MMA issuer ----
      bool ok = true;
      int g = g0, k = kfirst, it = 0;
      const uint32_t a0 = osmem(sA), b0s = osmem(sB);
      for (int c = 0; c < nchunks && ok; ++c) {
        if (c > 0 && !omb_wait(&free_bar, (c - 1) & 1, abort_v)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int kend = min(d.g[g].K, k + kOChunk);
        const int nst = (kend - k + kOBK - 1) / kOBK;
        for (int st = 0; st < nst; ++st, ++it) {
          const int s = it & 1;
          if (!omb_wait(&full_bar[s], (it >> 1) & 1, abort_v)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const uint32_t off = s * 64 + j * 32;
#pragma unroll
            for (int i = 0; i < kOD; ++i) {
              const uint64_t ad = odesc(a0 + i * kA + off);
              const uint32_t acc = (st > 0 || j > 0 || i > 0) ? 1u : 0u;
              // digits 0 .. 7 - i of B in pieces of at most 256 columns
#pragma unroll
              for (int n = 0; n < (kOD - i) * BN; n += 256) {
                constexpr int kMaxN = 256;
                const int nn = (kOD - i) * BN - n < kMaxN ? (kOD - i) * BN - n : kMaxN;
                omma(tmem + i * BN + n, ad, odesc(b0s + n * 128 + off), oidesc(nn), acc);
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
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    // ---- converters, then the flush of every chunk ----
    const int t = threadIdx.x;
    constexpr int kATasks = kOBM * 4 / kOConv;                     // 2
    const bool b_on = t < BN * 4;
    double va[kATasks][8], vb[8];
    int g = g0, k = kfirst;                               // next stage to load
    const double *pa = nullptr, *pb = nullptr;
    bool akf = false, bkf = false, avec = false, bvec = false;
    int ar[kATasks], ac[kATasks], br = 0, bc = 0;
    auto enter = [&]() {
      const Group& G = d.g[g];
      pa = static_cast<const double*>(G.a.p) + b0 * G.a.s_b0 + static_cast<long long>(b1) * G.a.s_b1;
      pb = static_cast<const double*>(G.b.p) + b0 * G.b.s_b0 + static_cast<long long>(b1) * G.b.s_b1;
      akf = G.a.s_k0 == 1;
      bkf = G.b.s_k0 == 1;
      avec = akf && ((reinterpret_cast<uintptr_t>(pa) & 15) == 0) && ((G.a.s_mn | G.a.s_k1) & 1) == 0;
      bvec = bkf && ((reinterpret_cast<uintptr_t>(pb) & 15) == 0) && ((G.b.s_mn | G.b.s_k1) & 1) == 0;
#pragma unroll
      for (int q = 0; q < kATasks; ++q) task_pos<kOBM>(t + q * kOConv, akf, ar[q], ac[q]);
      task_pos<BN>(t, bkf, br, bc);
    };
    auto load_a = [&](int q) {
      const Group& G = d.g[g];
      load8(G.a, G.k0_log2, pa, m0 + ar[q], m0 + ar[q] < d.M, k + 8 * ac[q], G.K, avec, va[q]);
    };
    auto load_b = [&]() {
      const Group& G = d.g[g];
      if (b_on) load8(G.b, G.k0_log2, pb, n0 + br, n0 + br < d.N, k + 8 * bc, G.K, bvec, vb);
    };
    uint32_t acc[3][kHalf];
#pragma unroll
    for (int j = 0; j < kHalf; ++j) acc[0][j] = acc[1][j] = acc[2][j] = 0u;
    const int quarter = warp & 3, half = warp >> 2;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + half * kHalf;
    bool ok = true;
    int flushed = 0;
    // add the eight accumulators of a finished chunk (of group fg) to acc
    auto flush = [&](int fg) {
      ok = __all_sync(0xffffffffu, ok && omb_wait(&done_bar, flushed & 1, abort_v));
      ++flushed;
      if (!ok) return;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned wa = ex[2 * fg], wb = ex[2 * fg + 1];
      const int sh = (wa == 0u || wb == 0u) ? 0 : sref - (static_cast<int>(wa >> 20) + static_cast<int>(wb >> 20) - 2 * 1022 - 68);
#pragma unroll
      for (int cb = 0; cb < kHalf; cb += 4) {
        uint32_t r[kOD][4];
#pragma unroll
        for (int l = 0; l < kOD; ++l)
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
              : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3])
              : "r"(trow + l * BN + cb));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          int L[kOD];
#pragma unroll
          for (int l = 0; l < kOD; ++l) L[l] = __float2int_rn(__uint_as_float(r[l][j]));
          const long long H = static_cast<long long>(L[0]) * (1 << 24) + static_cast<long long>(L[1]) * (1 << 16) +
                              static_cast<long long>(L[2]) * 256 + L[3];
          const long long Q = static_cast<long long>(L[4]) * (1 << 24) + static_cast<long long>(L[5]) * (1 << 16) +
                              static_cast<long long>(L[6]) * 256 + L[7];
          uint32_t v0 = static_cast<uint32_t>(Q), v1 = static_cast<uint32_t>(Q >> 32);
          uint32_t v2 = static_cast<uint32_t>(static_cast<int>(v1) >> 31);
          asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;"
              : "+r"(v1), "+r"(v2)
              : "r"(static_cast<uint32_t>(H)), "r"(static_cast<uint32_t>(H >> 32)));
          if (sh) {   // (the same in all threads of the CTA)
            const uint32_t sg = static_cast<uint32_t>(static_cast<int>(v2) >> 31);
            int s2 = sh;
            if (s2 >= 32) { v0 = v1; v1 = v2; v2 = sg; s2 -= 32; }
            if (s2 >= 32) { v0 = v1; v1 = v2; s2 -= 32; }
            if (s2 >= 32) { v0 = sg; v1 = sg; s2 = 0; }
            v0 = __funnelshift_r(v0, v1, s2);
            v1 = __funnelshift_r(v1, v2, s2);
            v2 = static_cast<uint32_t>(static_cast<int>(v2) >> s2);
          }
          asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
              : "+r"(acc[0][cb + j]), "+r"(acc[1][cb + j]), "+r"(acc[2][cb + j])
              : "r"(v0), "r"(v1), "r"(v2));
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      omb_arrive(&free_bar);
    };
    if (nchunks > 0) {
      enter();
      load_b();
#pragma unroll
      for (int q = 0; q < kATasks; ++q) load_a(q);
    }
    int it = 0, pend = -1;    // pend: group of the chunk that waits for its flush
    for (int c = 0; c <= nchunks && ok; ++c) {   // (one round more: the last flush)
      const int cg = g;
      const int nst = c == nchunks ? 0 : (min(d.g[g].K, k + kOChunk) - k + kOBK - 1) / kOBK;
      const unsigned wa = ex[2 * cg], wb = ex[2 * cg + 1];
      // (an all-zero operand: any exponent gives zero digits)
      const int ea = wa ? static_cast<int>(wa >> 20) : 1023, eb = wb ? static_cast<int>(wb >> 20) : 1023;
      for (int st = 0; st < max(nst, 1); ++st, ++it) {
        const int s = it & 1;
        if (nst) {
        if (it >= 2) ok = __all_sync(0xffffffffu, omb_wait(&empty_bar[s], ((it >> 1) - 1) & 1, abort_v));
        if (!ok) break;
        // the positions of this stage's tasks; the next stage's loads follow each conversion
        int car[kATasks], cac[kATasks];
#pragma unroll
        for (int q = 0; q < kATasks; ++q) { car[q] = ar[q]; cac[q] = ac[q]; }
        const int cbr = br, cbc = bc;
        const bool last = c + 1 == nchunks && st + 1 == nst;
        if (!last) {
          k += kOBK;
          if (k >= d.g[g].K) { ++g; k = 0; enter(); }
        }
        if (b_on) store_digits<BN>(vb, eb, sB, cbr, s * 4 + cbc);
        if (!last) load_b();
#pragma unroll
        for (int q = 0; q < kATasks; ++q) {
          store_digits<kOBM>(va[q], ea, sA, car[q], s * 4 + cac[q]);
          if (!last) load_a(q);
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
      }
      pend = cg;
    }
    if (!ok) {
      *abort_v = 1;
      if (op.err && t == 0) atomicOr(op.err, 1);
    } else {
      const int m = m0 + quarter * 32 + lane;
      if (m < d.M) {
        double* row = out_ptr(d, b, b0, b1, split, m, n0 + half * kHalf);
        const long long sn = d.splits > 1 ? 1 : d.sc_n;
        const int nv = min(kHalf, d.N - (n0 + half * kHalf));
        const bool vec = sn == 1 && nv == kHalf && (reinterpret_cast<uintptr_t>(row) & 15) == 0;
#pragma unroll
        for (int j = 0; j < kHalf; j += 2) {
          const double x = to_double(acc[0][j], acc[1][j], acc[2][j], sref);
          const double y = to_double(acc[0][j + 1], acc[1][j + 1], acc[2][j + 1], sref);
          if (vec) {
            *reinterpret_cast<double2*>(row + j) = make_double2(x, y);
          } else {
            if (j < nv) row[j * sn] = x;
            if (j + 1 < nv) row[(j + 1) * sn] = y;
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 8)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
}

template <int BN>
constexpr int oz_smem() { return kOD * (kOBM + BN) * 128 + 1024; }

int oz_chunks(const GemmDesc& d) {
  int t = 0;
  for (int g = 0; g < d.ngroups; ++g) t += (d.g[g].K + kOChunk - 1) / kOChunk;
  return t;
}

int oz_bn(const GemmDesc& d) { return d.N > 32 ? 64 : 32; }

// The elements of one batch of an operand cover a dense range: count and true,
// else the strided walk.
bool flat_operand(const Operand& o, int k0_log2, int K, int mn, long long* count) {
  const long long K0 = std::min<long long>(1LL << k0_log2, K), K1 = K0 < K ? K >> k0_log2 : 1;
  long long ext[3] = {mn, K0, K1}, str[3] = {o.s_mn, o.s_k0, o.s_k1};
  *count = static_cast<long long>(mn) * K;
  long long need = 1;
  for (int step = 0; step < 3; ++step) {
    int f = -1;
    for (int i = 0; i < 3; ++i)
      if (ext[i] > 1 && str[i] == need) f = i;
    if (f < 0) break;
    need *= ext[f];
    ext[f] = 1;
  }
  return ext[0] == 1 && ext[1] == 1 && ext[2] == 1;
}

bool same_operand(const AbsItem& a, const AbsItem& b) {
  return a.p == b.p && a.s_mn == b.s_mn && a.s_k0 == b.s_k0 && a.s_k1 == b.s_k1 && a.s_b0 == b.s_b0 &&
         a.s_b1 == b.s_b1 && a.count == b.count && a.flat == b.flat && a.mn == b.mn && a.k == b.k &&
         a.k0_log2 == b.k0_log2 && a.n0 == b.n0 && a.n1 == b.n1;
}

}  // namespace

// Products the digit engine takes: FP64 in and out, K0 a whole number of
// 16-byte digit chunks, and enough work that the launch of absmax_kernel pays.
bool gemm_oz_supported(const GemmDesc& d) {
  if (!d.digits || d.prec != 0 || d.c_f32 || d.alpha != 1.0 || d.beta != 0.0 || d.ngroups < 1 ||
      d.ngroups > kMaxGroups || d.M < 1 || d.N < 1)
    return false;
  double work = 0.0;
  for (int g = 0; g < d.ngroups; ++g) {
    const Group& G = d.g[g];
    if (G.a.f32 || G.b.f32 || G.K < 1) return false;
    if (G.k0_log2 < 3 && (G.K >> G.k0_log2) > 1) return false;
    work += static_cast<double>(d.M) * d.N * G.K * d.B0 * d.B1;
  }
  return d.M >= 16 && d.N >= 16 && work >= kOzMinWork;
}

int oz_pick_splits(const GemmDesc& d) {
  const int bn = oz_bn(d);
  const long long base = static_cast<long long>((d.M + kOBM - 1) / kOBM) * ((d.N + bn - 1) / bn) * d.B0 * d.B1;
  const int sms = device_sm_count();
  if (2 * base > sms) return 1;
  return static_cast<int>(std::max<long long>(1, std::min<long long>(sms / base, oz_chunks(d))));
}

// Words of magnitude scratch for a product.
size_t oz_words(const GemmDesc& d) {
  if (!gemm_oz_supported(d)) return 0;
  size_t n = 0;
  for (int g = 0; g < d.ngroups; ++g)
    for (int s = 0; s < 2; ++s) {
      const Operand& o = s ? d.g[g].b : d.g[g].a;
      const long long count = static_cast<long long>(s ? d.N : d.M) * d.g[g].K;
      const long long parts = std::max<long long>(1, std::min<long long>((count + kAbsPer - 1) / kAbsPer, kAbsMaxParts));
      n += static_cast<size_t>(parts) * (o.s_b0 ? d.B0 : 1) * (o.s_b1 ? d.B1 : 1);
    }
  return n;
}

int gemm_oz_launch(const GemmDesc& d, cudaStream_t s) {
  AbsParams ap;
  OzParams op;
  memset(&op, 0, sizeof(op));
  ap.n = 0;
  ap.words = d.words;
  int off = 0, blocks = 0;
  for (int g = 0; g < d.ngroups; ++g)
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
      it.flat = flat_operand(o, G.k0_log2, G.K, it.mn, &it.count) ? 1 : 0;
      it.parts = static_cast<int>(std::max<long long>(1, std::min<long long>((it.count + kAbsPer - 1) / kAbsPer, kAbsMaxParts)));
      int at = 0;
      while (at < ap.n && !same_operand(ap.it[at], it)) ++at;
      if (at == ap.n) {
        it.off = off;
        it.blocks_before = blocks;
        off += it.parts * it.n0 * it.n1;
        blocks += it.parts * it.n0 * it.n1;
        ap.it[ap.n++] = it;
      }
      OzOperand& w = side ? op.b[g] : op.a[g];
      w.off = ap.it[at].off;
      w.parts = ap.it[at].parts;
      w.s0 = o.s_b0 ? 1 : 0;
      w.s1 = o.s_b1 ? it.n0 : 0;
    }
  launch_k(absmax_kernel, blocks, 256, 0, s, ap);
  op.words = d.words;
  op.total_chunks = oz_chunks(d);
  op.err = d.err;
  const int bn = oz_bn(d);
  dim3 grid(((d.M + kOBM - 1) / kOBM) * ((d.N + bn - 1) / bn), d.B0 * d.B1, d.splits);
  if (bn == 64) launch_k(gemm_oz_kernel<64>, grid, kOThreads, oz_smem<64>(), s, d, op);
  else launch_k(gemm_oz_kernel<32>, grid, kOThreads, oz_smem<32>(), s, d, op);
  return 2;
}

void gemm_oz_init() {
  cudaFuncSetAttribute(gemm_oz_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz_smem<64>());
  cudaFuncSetAttribute(gemm_oz_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, oz_smem<32>());
}

}  // namespace ttn
