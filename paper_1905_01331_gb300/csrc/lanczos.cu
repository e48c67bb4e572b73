// Top-tensor update (Sec. III.B: the top tensor is "updated similarly"; read
// as the lowest eigenvector of the top Hamiltonian) as one persistent
// cooperative launch: restarted Lanczos with full reorthogonalisation,
// warm-started from the previous V.  Vectors, projections and the
// tridiagonal are FP64; in the mixed modes the matrix-vector products run in
// double-float pair arithmetic on pair copies of the operators and the basis.
//
// H_top acts on the c x c top tensor V as
//     H V = o_0 V + V o_1^T + sum_k (A_k0 V B_k1^T + B_k0 V A_k1^T),
// with (o, A_k, B_k) the identity-free operators of the two top sites (the
// two bonds of the periodic ring at the top).  One Lanczos step is
//     phase A   Y_k = A_k0 x, Y_{K+k} = B_k0 x               (2K products)
//     phase B   w = o_0 x + x o_1^T + sum_k Y_k B_k1^T + Y_{K+k} A_k1^T
//               (minus sigma x after the first step: the recurrence runs on
//               H - sigma I, sigma the Rayleigh quotient of the start vector)
//     projections on the basis and |w|^2, one classical Gram-Schmidt pass,
//     a second one ("twice is enough") when the first removed more than 3/4
//     of |w|^2, then alpha_j, beta_j and the next basis vector
// with every phase shared by all CTAs and a grid barrier between phases
// (bounded spin, error flag).  Each CTA owns the vector entries of the 8 x 8
// output tiles it computes (and keeps them, of w and of every basis vector, in
// shared memory); every reduction adds its per-CTA partial sums in a fixed
// order, so the result does not depend on timing.  Every kLCheck steps the
// tridiagonal so far is tested for convergence in pair arithmetic by an extra
// CTA, which has the next kLLag steps for it, and a passed test ends the cycle;
// at the end of a cycle CTA 0 finds the eigenpair of the tridiagonal.
//
// What bounds it: latency, and the FP64 units.  An FP64 warp instruction takes
// 16 clocks of an SM and about 100 of latency, so scalars are computed by one
// warp, the butterflies of four sums share their additions, and the Sturm
// sequences run in pairs.  Measured per sweep from a random start (clocks of
// one step, then the solve): c = 8, one CTA: 48 k -> 23 k, 2.37 -> 1.2 ms; c =
// 128, mixed: 45 -> 29 us a step, 4.4 -> 2.8 ms; the FP64 products of c = 128
// alone take 25 us of a step.  Then c = 8 without memory round trips (LzTiny) 1.2 ->
// 0.6 ms, and the mixed products unrolled (wide_fma).
#include <algorithm>
#include <mutex>

#include "common.h"
#include "pair_arith.cuh"
#include "tridiag_df.cuh"

namespace ttn {

namespace {

constexpr int kLT = 8;                   // output tile edge of the matrix products
constexpr int kLThreads = 256;
constexpr int kLWarps = kLThreads / 32;
constexpr int kLMaxC = 256;
constexpr int kLMaxSpin = 1 << 21;       // ~1 s of polling, then the error flag
constexpr int kLCheck = 8;               // steps between convergence checks within a cycle
constexpr int kLLag = 4;                 // steps that a check may take (less than kLCheck)

// Static shared memory; the operand tiles and the cached basis entries are
// dynamic (lz_dyn): first the tiles (LzTiles), then the cache (LzOwn).
struct __align__(16) LzSmem {
  double red[kLWarps][kLT * kLT];
  double tri[1][kLMaxM + 2];             // eigenvector of the tridiagonal
  float fa[kLMaxM + 2], fb2[kLMaxM + 2];
  double cf[kLMaxM + 2];                 // coefficients of the current combination
  double al[kLMaxM + 2], be[kLMaxM + 2]; // the tridiagonal's entries (CTA 0 and the checks)
  double bcast[4];
  unsigned ball[kLWarps];
  float bnd[2 * kLWarps];
  // scalars of the recurrence, kept by warp 0: Rayleigh shift, beta_{j-1},
  // alpha_{j-1} of H, 1 / beta_j; whether one Gram-Schmidt pass was enough, and
  // whether beta_j vanished
  double sigma, beta_prev, alpha_prev_h, inv;
  int one_pass, brk;
  int ok;
};

// Operand tiles of a matrix product: L (left rows) and R (right rows or
// columns), pitch c + 1.
struct LzTiles {
  double* L;
  double* R;
  int ld;
};

// The CTA's own entries (own_index) of basis vectors 0 .. n - 1 in shared
// memory, and of w at row `wrow` (or -1): the projections and combinations of
// every step read them here instead of from L2 (about 700 clocks per round of
// loads).  Rows have a pitch of nown + 8 doubles, so that the threads that
// share an entry read distinct banks.
struct LzOwn {
  double* p;
  int pitch, n, wrow;
  __device__ __forceinline__ void set(int i, int q, double v) const {
    if (n) p[i * pitch + q] = v;
  }
};

__device__ bool lz_barrier(LzSmem& sm, unsigned* bar, unsigned& target, int G, int* err, int max_spin) {
  __syncthreads();
  if (G == 1) return true;   // one CTA: its own barrier orders its accesses
  target += G;
  if (threadIdx.x == 0) {
    // arrive with release semantics (this CTA's writes before it), poll with
    // acquire semantics (the other CTAs' writes after it)
    int ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    int spins = 0;
    while (true) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= target) break;
      if (*reinterpret_cast<volatile int*>(err)) { ok = 0; break; }
      if (++spins > max_spin) { atomicOr(err, 4); ok = 0; break; }
      __nanosleep(32);
    }
    sm.ok = ok;
  }
  __syncthreads();
  return sm.ok != 0;
}

// Sum of x[0..count) in a fixed order (lane-strided partial sums, then a fixed
// butterfly), by warp 0; the result is returned to every thread of the CTA.
__device__ double cta_ordered_sum(LzSmem& sm, const double* x, int count, long long stride) {
  __syncthreads();
  if (threadIdx.x < 32) {
    double s = 0.0;
    for (int i = threadIdx.x; i < count; i += 32) s += __ldcg(x + i * stride);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) sm.bcast[0] = s;
  }
  __syncthreads();
  const double v = sm.bcast[0];
  __syncthreads();
  return v;
}

// Elements staged per thread: a tile edge of 8 rows or columns of length
// c <= kLMaxC.  The staging functions issue all their loads before the first
// shared-memory store, so that a staged tile costs one load latency.
constexpr int kLStage = kLT * kLMaxC / kLThreads;

// Stage rows [r0, r0+8) of the row-major c x c matrix M into dst.
__device__ void stage_rows(double* dst, const double* M, int c, int r0) {
  double v[kLStage];
#pragma unroll
  for (int u = 0; u < kLStage; ++u) {
    const int e = threadIdx.x + u * kLThreads, r = e / c, k = e - r * c;
    v[u] = (e < kLT * c && r0 + r < c) ? __ldcg(M + (long long)(r0 + r) * c + k) : 0.0;
  }
#pragma unroll
  for (int u = 0; u < kLStage; ++u) {
    const int e = threadIdx.x + u * kLThreads, r = e / c, k = e - r * c;
    if (e < kLT * c) dst[r * (c + 1) + k] = v[u];
  }
}
// Stage columns [c0, c0+8) of M as rows of dst: dst[j][k] = M[k][c0 + j].
__device__ void stage_cols(double* dst, const double* M, int c, int c0) {
  double v[kLStage];
#pragma unroll
  for (int u = 0; u < kLStage; ++u) {
    const int e = threadIdx.x + u * kLThreads, k = e / kLT, j = e - k * kLT;
    v[u] = (e < kLT * c && c0 + j < c) ? __ldcg(M + (long long)k * c + c0 + j) : 0.0;
  }
#pragma unroll
  for (int u = 0; u < kLStage; ++u) {
    const int e = threadIdx.x + u * kLThreads, k = e / kLT, j = e - k * kLT;
    if (e < kLT * c) dst[j * (c + 1) + k] = v[u];
  }
}

// acc[0..1] += sum_k L[i][k] R[j][k] over this warp's K slice (i = lane/4,
// j = 2 (lane % 4) + {0, 1}).
__device__ __forceinline__ void tile_fma(const LzTiles& ts, int c, double& a0, double& a1) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = lane >> 2, j = (lane & 3) * 2;
  for (int k = warp; k < c; k += kLWarps) {
    const double x = ts.L[i * ts.ld + k];
    a0 = fma(x, ts.R[j * ts.ld + k], a0);
    a1 = fma(x, ts.R[(j + 1) * ts.ld + k], a1);
  }
}

// Reduce the per-warp partial sums of a tile in warp order and store it,
// minus sigma X when sigma != 0 (the shifted operator H - sigma I).
__device__ void tile_store(LzSmem& sm, double a0, double a1, double* C, int c, int i0, int j0,
                           const double* X = nullptr, double sigma = 0.0,
                           const double* Xprev = nullptr, double beta = 0.0,
                           double* own_w = nullptr) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = lane >> 2, j = (lane & 3) * 2;
  sm.red[warp][i * kLT + j] = a0;
  sm.red[warp][i * kLT + j + 1] = a1;
  __syncthreads();
  if (threadIdx.x < kLT * kLT) {
    double v = 0.0;
    for (int w = 0; w < kLWarps; ++w) v += sm.red[w][threadIdx.x];
    const int r = threadIdx.x / kLT, cc = threadIdx.x % kLT;
    if (i0 + r < c && j0 + cc < c) {
      const long long e = (long long)(i0 + r) * c + j0 + cc;
      if (sigma != 0.0) v = fma(-sigma, __ldcg(X + e), v);
      if (beta != 0.0) v = fma(-beta, __ldcg(Xprev + e), v);
      __stcg(C + e, v);
      if (own_w) own_w[threadIdx.x] = v;
    }
  }
  __syncthreads();
}

// Number of eigenvalues of the symmetric tridiagonal below x (diagonal a,
// squared off-diagonal b2), by the signs of the LDL^T pivots, in FP32.
__device__ int sturm_below_f32(const float* a, const float* b2, int m, float x) {
  int cnt = 0;
  float q = a[0] - x;
  if (q < 0.f) ++cnt;
  for (int i = 1; i < m; ++i) {
    if (q == 0.f) q = 1e-30f;
    q = a[i] - x - b2[i - 1] / q;
    if (q < 0.f) ++cnt;
  }
  return cnt;
}

// The same count in FP64 without divisions (FP64 division is a long
// instruction sequence on this GPU's two FP64 units per SM): the signs of the
// leading principal minors d_i of T - x I, d_{i+1} = (a_i - x) d_i -
// b2_{i-1} d_{i-1}, whose ratios are the pivots above (a zero pivot is
// replaced by a tiny positive one, as above); the minors are rescaled by a
// power of two (exactly) every eight steps.
__device__ int sturm_below_f64(const double* a, const double* b2, int m, double x) {
  int cnt = 0;
  double dm = 1.0, d = a[0] - x;
  if (d == 0.0) d = 1e-30;
  if (d < 0.0) ++cnt;
  for (int i = 1; i < m; ++i) {
    double dn = fma(a[i] - x, d, -b2[i - 1] * dm);
    if (dn == 0.0) dn = 1e-30 * d;
    if ((dn < 0.0) != (d < 0.0)) ++cnt;
    dm = d;
    d = dn;
    if ((i & 7) == 0) {
      const int ex = (int)((__double_as_longlong(d) >> 52) & 0x7FF) - 1023;
      if (ex > -1000 && ex < 1000) {
        const double sc = __longlong_as_double((long long)(1023 - ex) << 52);
        d *= sc;
        dm *= sc;
      }
    }
  }
  return cnt;
}

// Index of the first thread of the CTA whose flag is set, else kLThreads.
__device__ int first_thread(LzSmem& sm, bool flag) {
  const unsigned bal = __ballot_sync(0xffffffffu, flag);
  if ((threadIdx.x & 31) == 0) sm.ball[threadIdx.x >> 5] = bal;
  __syncthreads();
  int f = kLThreads;
  for (int w = kLWarps - 1; w >= 0; --w)
    if (sm.ball[w]) f = w * 32 + __ffs(sm.ball[w]) - 1;
  __syncthreads();
  return f;
}

// Eigenvector of the m x m tridiagonal (al, be) for the eigenvalue th, by warp
// 0 (the twisted factorisation of tridiag_df.cuh; the two chains of pivots and
// the two of the vector on lanes 0 and 1 at the same time).  One division per
// row in each chain, where an LU with pivoting and its two substitutions need
// four.  z[0 .. m) unnormalised (FP64); scratch: 4 m values of T.
template <typename A>
__device__ void twisted_vector(const double* al, const double* be, int m, double th, typename A::T* scratch,
                               double* z) {
  typedef typename A::T T;
  const int lane = threadIdx.x;
  T* ms = scratch;           // al - th
  T* b2 = scratch + m;       // squared off-diagonal, then the multipliers
  T* dp = scratch + 2 * m;   // pivots from the top, then the vector
  T* dm = scratch + 3 * m;   // pivots from the bottom
  for (int i = lane; i < m; i += 32) tdf::twist_row<A>(al, be, m, th, i, ms, b2);
  __syncwarp();
  if (lane < 2) tdf::twist_pivots<A>(ms, b2, m, lane == 0, lane == 0 ? dp : dm);
  __syncwarp();
  // twist row: the smallest gap, the first of equals
  double best = 1e300;
  int r = 0;
  for (int i = lane; i < m; i += 32) {
    const double g = tdf::twist_gap<A>(ms, dp, dm, i);
    if (g < best) { best = g; r = i; }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int orr = __shfl_xor_sync(0xffffffffu, r, o);
    if (ob < best || (ob == best && orr < r)) { best = ob; r = orr; }
  }
  for (int i = lane; i + 1 < m; i += 32) b2[i] = tdf::twist_multiplier<A>(be, dp, dm, r, i);
  __syncwarp();
  if (lane == 0) z[r] = 1.0;
  if (lane < 2) tdf::twist_outwards<A>(b2, m, r, lane == 0, dp);
  __syncwarp();
  for (int i = lane; i < m; i += 32)
    if (i != r) z[i] = A::to(dp[i]);
  __syncwarp();
}

__device__ __forceinline__ double warp_sum(double s) {
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Lowest eigenvalue of the tridiagonal in sm.al and sm.be (m entries) by the
// whole CTA, to pair accuracy: 257-way multisection in FP32, then in pair
// arithmetic (tridiag_df.cuh).  FP64 runs at one warp instruction per 16
// clocks of an SM and about 100 clocks of latency here: one Sturm count of 48
// rows takes 26 k clocks in FP64 and 8 k in pairs.  The tridiagonal is scaled
// by a power of two to unit size first (sm.al and sm.be hold the scaled one on
// return; the result is in the same scale).  scratch: 2 m pairs.
__device__ double lowest_value(LzSmem& sm, double* scratch, int m, double& unscale) {
  using namespace tdf;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  // largest entry -> scale
  unsigned hw = 0;
  for (int i = t; i < m; i += kLThreads) {
    hw = max(hw, (unsigned)__double2hiint(sm.al[i]) & 0x7FFFFFFFu);
    if (i + 1 < m) hw = max(hw, (unsigned)__double2hiint(sm.be[i]) & 0x7FFFFFFFu);
  }
  hw = __reduce_max_sync(0xffffffffu, hw);
  if (lane == 0) sm.ball[warp] = hw;
  __syncthreads();
  for (int w = 0; w < kLWarps; ++w) hw = max(hw, sm.ball[w]);
  __syncthreads();
  const int e = min(max((int)(hw >> 20), 30), 2000);
  const double sc = __hiloint2double((2046 - e) << 20, 0);     // 2^(1023 - e)
  unscale = __hiloint2double(e << 20, 0);                       // 2^(e - 1023)
  DF* A = reinterpret_cast<DF*>(scratch);
  DF* B2 = A + m;
  for (int i = t; i < m; i += kLThreads) {
    const double al = sm.al[i] * sc, be = i + 1 < m ? sm.be[i] * sc : 0.0;
    sm.al[i] = al;
    sm.be[i] = be;
    A[i] = make(al);
    const DF b = make(be);
    B2[i] = mul(b, b);
    sm.fa[i] = (float)al;
    sm.fb2[i] = (float)be;
  }
  __syncthreads();
  // Gershgorin bounds in FP32 (entries of size <= 2, margins far above rounding)
  float glo = 3.4e38f, ghi = -3.4e38f;
  for (int i = t; i < m; i += kLThreads) {
    const float r = (i > 0 ? fabsf(sm.fb2[i - 1]) : 0.f) + fabsf(sm.fb2[i]);
    glo = fminf(glo, sm.fa[i] - r);
    ghi = fmaxf(ghi, sm.fa[i] + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    glo = fminf(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmaxf(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
  }
  if (lane == 0) { sm.bnd[warp] = glo; sm.bnd[kLWarps + warp] = ghi; }
  __syncthreads();
  for (int w = 0; w < kLWarps; ++w) {
    glo = fminf(glo, sm.bnd[w]);
    ghi = fmaxf(ghi, sm.bnd[kLWarps + w]);
  }
  const float tn = fmaxf(fabsf(glo), fabsf(ghi));
  glo -= 1e-5f * tn;
  ghi += 1e-5f * tn;
  __syncthreads();
  for (int i = t; i < m; i += kLThreads) sm.fb2[i] = sm.fb2[i] * sm.fb2[i];
  __syncthreads();
  float flo = glo, fhi = ghi;
  constexpr float kR = 1.f / (kLThreads + 1);
  for (int it = 0; it < 4; ++it) {
    if (!(fhi - flo > 2e-6f * fmaxf(fabsf(flo), fabsf(fhi)))) break;
    const float pt = flo + (fhi - flo) * ((float)(t + 1) * kR);
    const int f = first_thread(sm, sturm_below_f32(sm.fa, sm.fb2, m, pt) >= 1);
    const float nlo = f == 0 ? flo : flo + (fhi - flo) * ((float)f * kR);
    const float nhi = f == kLThreads ? fhi : flo + (fhi - flo) * ((float)(f + 1) * kR);
    flo = nlo;
    fhi = nhi;
  }
  // widen by the FP32 rounding of T, confirm in pairs (half of the CTA each)
  DF lo = {flo - 1e-5f * tn, 0.f}, hi = {fhi + 1e-5f * tn, 0.f};
  const int cnt = sturm_below(A, B2, m, t < kLThreads / 2 ? lo : hi);
  if (!__syncthreads_and(t < kLThreads / 2 ? cnt == 0 : cnt >= 1)) {
    lo = {glo, 0.f};
    hi = {ghi, 0.f};
  }
  for (int it = 0; it < 8; ++it) {
    const float w = sub(hi, lo).h;
    if (!(w > 1e-14f * fmaxf(fabsf(lo.h), fabsf(hi.h)))) break;
    const DF pt = add(lo, {w * ((float)(t + 1) * kR), 0.f});
    const int f = first_thread(sm, sturm_below(A, B2, m, pt) >= 1);
    const DF nlo = f == 0 ? lo : add(lo, {w * ((float)f * kR), 0.f});
    const DF nhi = f == kLThreads ? hi : add(lo, {w * ((float)(f + 1) * kR), 0.f});
    lo = nlo;
    hi = nhi;
  }
  return to_double(add(lo, {0.5f * sub(hi, lo).h, 0.f}));
}

// The first m entries of the tridiagonal into sm.al and sm.be (whole CTA).
__device__ __forceinline__ void load_tridiagonal(const LanczosArgs& a, LzSmem& sm, int m) {
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += kLThreads) {
    sm.al[i] = __ldcg(a.alpha + i);
    sm.be[i] = __ldcg(a.beta + i);
  }
  __syncthreads();
}

// Convergence test of the tridiagonal of the steps so far (sm.al, sm.be: m
// entries, shifted by -sigma; both are scaled on return): |beta_{m-1} y_{m-1}|
// <= tol |theta + sigma| for its lowest eigenpair (theta, y) in pair
// arithmetic.  (The end of a cycle recomputes the pair; a wrong early answer
// costs a restart, not accuracy.)  scratch: 6 m doubles of shared memory.
// Valid in thread 0.
__device__ bool ritz_check_df(LzSmem& sm, double* scratch, int m, double sigma, double tol) {
  const double blast = sm.be[m - 1];
  double unscale;
  const double th = lowest_value(sm, scratch, m, unscale);
  if (threadIdx.x >= 32) return false;
  double* z = sm.tri[0];
  twisted_vector<tdf::ArithDF>(sm.al, sm.be, m, th, reinterpret_cast<tdf::DF*>(scratch), z);
  double s = 0.0;
  for (int i = threadIdx.x; i < m; i += 32) s = fma(z[i], z[i], s);
  s = warp_sum(s);
  return fabs(blast) * fabs(z[m - 1]) <= tol * fmax(fabs(th * unscale + sigma), 1e-300) * sqrt(s);
}

// Lowest eigenpair of the m x m tridiagonal (sm.al, sm.be; scaled on return) by
// the calling CTA: y (m entries, unit norm), theta, residual |beta_{m-1}
// y_{m-1}|.  The eigenvalue and a first vector in pair arithmetic, the
// eigenvalue's FP64 digits as their Rayleigh quotient, and the vector again in
// FP64: 45 k clocks of FP64 chain instead of 570 k for a multisection and two
// rounds of inverse iteration in FP64 (m = 48).  For the mixed modes.
__device__ void ritz_pair(LzSmem& sm, double* scratch, int m, double* y, double* theta, double* res) {
  const double blast = sm.be[m - 1];
  double unscale;
  const double th0 = lowest_value(sm, scratch, m, unscale);
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  double* z = sm.tri[0];
  twisted_vector<tdf::ArithDF>(sm.al, sm.be, m, th0, reinterpret_cast<tdf::DF*>(scratch), z);
  // Rayleigh quotient of (T - th0) z, added to th0
  double nn = 0.0, rq = 0.0;
  for (int i = lane; i < m; i += 32) {
    nn = fma(z[i], z[i], nn);
    double tz = (sm.al[i] - th0) * z[i];
    if (i + 1 < m) tz = fma(2.0 * sm.be[i], z[i + 1], tz);
    rq = fma(z[i], tz, rq);
  }
  nn = warp_sum(nn);
  rq = warp_sum(rq);
  const double th = th0 + rq / nn;
  twisted_vector<tdf::ArithD>(sm.al, sm.be, m, th, scratch, z);
  double s = 0.0;
  for (int i = lane; i < m; i += 32) s = fma(z[i], z[i], s);
  const double inv = sqrt(warp_sum(s));
  for (int i = lane; i < m; i += 32) y[i] = z[i] / inv;
  if (lane == 0) {
    *theta = th * unscale;
    *res = fabs(blast * z[m - 1] / inv);
  }
}

// The same in FP64 mode, all of whose result is FP64: bracketing in FP32,
// 32-way FP64 multisection to 4e-16 and two rounds of inverse iteration.  A
// count whose point lies 1e-13 |T| or more from the pair-accurate eigenvalue is
// known without its Sturm sequence (26 k clocks in FP64; most rounds have no
// other), so the result is that of the full multisection.
__device__ void ritz_pair_f64(LzSmem& sm, const LanczosArgs& a, double* scratch, int m, double* y, double* theta,
                              double* res) {
  double unscale;
  const double near = lowest_value(sm, scratch, m, unscale) * unscale;
  load_tridiagonal(a, sm, m);    // (lowest_value scaled it)
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  const double *al = sm.al, *be = sm.be;
  double* db2 = scratch;
  double *x = scratch + m, *dd = x + m, *du = dd + m, *du2 = du + m, *rhs = du2 + m, *dl = rhs + m;
  double glo = al[0], ghi = al[0];
  for (int i = lane; i < m; i += 32) {
    const double r = (i > 0 ? fabs(be[i - 1]) : 0.0) + (i + 1 < m ? fabs(be[i]) : 0.0);
    glo = fmin(glo, al[i] - r);
    ghi = fmax(ghi, al[i] + r);
    const double b2 = i + 1 < m ? be[i] * be[i] : 0.0;
    db2[i] = b2;
    sm.fa[i] = (float)al[i];
    sm.fb2[i] = (float)b2;
  }
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
  }
  __syncwarp();
  const double tnorm = fmax(fabs(glo), fabs(ghi)), margin = 1e-13 * tnorm;
  // whether an eigenvalue lies below p (all lanes call it)
  auto below = [&](double p) {
    bool r = p > near;
    const bool close = !(fabs(p - near) > margin);
    if (__any_sync(0xffffffffu, close)) {
      const int cnt = sturm_below_f64(al, db2, m, p);
      if (close) r = cnt >= 1;
    }
    return r;
  };
  float flo = (float)glo, fhi = (float)ghi;
  for (int it = 0; it < 8; ++it) {
    const float mag = fabsf(flo) > fabsf(fhi) ? fabsf(flo) : fabsf(fhi);
    if (!(fhi - flo > 2e-6f * mag)) break;
    constexpr float r33 = 1.f / 33.f;
    const float pt = flo + (fhi - flo) * ((float)(lane + 1) * r33);
    const unsigned bal = __ballot_sync(0xffffffffu, sturm_below_f32(sm.fa, sm.fb2, m, pt) >= 1);
    const int f = bal ? __ffs(bal) - 1 : 32;
    const float nlo = f == 0 ? flo : flo + (fhi - flo) * ((float)f * r33);
    const float nhi = f == 32 ? fhi : flo + (fhi - flo) * ((float)(f + 1) * r33);
    flo = nlo;
    fhi = nhi;
  }
  double lo = (double)flo - 1e-5 * tnorm, hi = (double)fhi + 1e-5 * tnorm;
  const bool b_lo = below(lo), b_hi = below(hi);
  if (!__all_sync(0xffffffffu, !b_lo && b_hi)) { lo = glo; hi = ghi; }
  for (int it = 0; it < 16; ++it) {
    const double mag = fabs(lo) > fabs(hi) ? fabs(lo) : fabs(hi);
    if (!(hi - lo > 4e-16 * mag)) break;
    constexpr double r33 = 1.0 / 33.0;
    const double pt = lo + (hi - lo) * ((double)(lane + 1) * r33);
    const unsigned bal = __ballot_sync(0xffffffffu, below(pt));
    const int f = bal ? __ffs(bal) - 1 : 32;
    const double nlo = f == 0 ? lo : lo + (hi - lo) * ((double)f * r33);
    const double nhi = f == 32 ? hi : lo + (hi - lo) * ((double)(f + 1) * r33);
    lo = nlo;
    hi = nhi;
  }
  const double th = 0.5 * (lo + hi);
  // inverse iteration on (T - th I) x = x_prev: LU with partial pivoting of
  // the tridiagonal, two rounds.  The elimination is one chain (lane 0, its
  // running row in registers); rows are set up and scaled by all lanes.
  const double x0 = 1.0 / sqrt((double)m);
  for (int i = lane; i < m; i += 32) x[i] = x0;
  const double eps = fmax(fabs(th), 1.0) * 1e-15;
  for (int round = 0; round < 2; ++round) {
    for (int i = lane; i < m; i += 32) {
      dd[i] = al[i] - th;
      du[i] = i + 1 < m ? be[i] : 0.0;
      du2[i] = 0.0;
      rhs[i] = x[i];
      dl[i] = i + 1 < m ? be[i] : 0.0;
    }
    __syncwarp();
    if (lane == 0) {
      double cd = dd[0], cu = du[0], cr = rhs[0];   // row i: diagonal, first off-diagonal, right side
      for (int i = 0; i + 1 < m; ++i) {
        double nd = dd[i + 1], nu = du[i + 1], nr = rhs[i + 1];
        const double l = dl[i];
        if (fabs(cd) >= fabs(l)) {
          if (cd == 0.0) cd = eps;
          const double f = l / cd;
          nd -= f * cu;
          nr -= f * cr;
          dd[i] = cd;
          du[i] = cu;
          rhs[i] = cr;
        } else {
          const double f = cd / l;
          dd[i] = l;
          du[i] = nd;
          rhs[i] = nr;
          nd = cu - f * nd;
          if (i + 2 < m) { du2[i] = nu; nu = -f * nu; }
          nr = cr - f * nr;
        }
        cd = nd;
        cu = nu;
        cr = nr;
      }
      if (cd == 0.0) cd = eps;
      dd[m - 1] = cd;
      du[m - 1] = cu;
      rhs[m - 1] = cr;
      double x1 = 0.0, x2 = 0.0, nrm = 0.0;
      for (int i = m - 1; i >= 0; --i) {
        double s = rhs[i];
        if (i + 1 < m) s -= du[i] * x1;
        if (i + 2 < m) s -= du2[i] * x2;
        const double d = dd[i];
        x2 = x1;
        x1 = s / (fabs(d) < eps ? (d < 0 ? -eps : eps) : d);
        x[i] = x1;
      }
      for (int i = 0; i < m; ++i) nrm += x[i] * x[i];
      sm.bcast[3] = sqrt(nrm);
    }
    __syncwarp();
    const double nrm = sm.bcast[3];
    for (int i = lane; i < m; i += 32) x[i] /= nrm;
    __syncwarp();
  }
  for (int i = lane; i < m; i += 32) y[i] = x[i];
  if (lane == 0) {
    *theta = th;
    *res = fabs(be[m - 1] * x[m - 1]);
  }
}

// Double-float matrix-vector products (mixed modes): matrices and vectors as
// FP32 pairs (hi block of n floats, then lo block), tiles staged into the
// shared arrays L and R reinterpreted as hi/lo float rows.
// (pitch c + 1 floats; hi rows, then lo rows)
// rows [r0, r0+8) of the pair matrix M (hi at M, lo at M + n)
__device__ void stage_rows_p(double* dst, const float* M, long long n, int c, int r0) {
  float* h = reinterpret_cast<float*>(dst);
  float* l = h + kLT * (c + 1);
  float vh[kLStage], vl[kLStage];
#pragma unroll
  for (int u = 0; u < kLStage; ++u) {
    const int e = threadIdx.x + u * kLThreads, r = e / c, k = e - r * c;
    const bool ok = e < kLT * c && r0 + r < c;
    const long long i = (long long)(r0 + r) * c + k;
    vh[u] = ok ? __ldcg(M + i) : 0.f;
    vl[u] = ok ? __ldcg(M + n + i) : 0.f;
  }
#pragma unroll
  for (int u = 0; u < kLStage; ++u) {
    const int e = threadIdx.x + u * kLThreads, r = e / c, k = e - r * c;
    if (e < kLT * c) { h[r * (c + 1) + k] = vh[u]; l[r * (c + 1) + k] = vl[u]; }
  }
}
// columns [c0, c0+8) of M as rows: dst[j][k] = M[k][c0 + j]
__device__ void stage_cols_p(double* dst, const float* M, long long n, int c, int c0) {
  float* h = reinterpret_cast<float*>(dst);
  float* l = h + kLT * (c + 1);
  float vh[kLStage], vl[kLStage];
#pragma unroll
  for (int u = 0; u < kLStage; ++u) {
    const int e = threadIdx.x + u * kLThreads, k = e / kLT, j = e - k * kLT;
    const bool ok = e < kLT * c && c0 + j < c;
    const long long i = (long long)k * c + c0 + j;
    vh[u] = ok ? __ldcg(M + i) : 0.f;
    vl[u] = ok ? __ldcg(M + n + i) : 0.f;
  }
#pragma unroll
  for (int u = 0; u < kLStage; ++u) {
    const int e = threadIdx.x + u * kLThreads, k = e / kLT, j = e - k * kLT;
    if (e < kLT * c) { h[j * (c + 1) + k] = vh[u]; l[j * (c + 1) + k] = vl[u]; }
  }
}

__device__ __forceinline__ void tile_fma_p(const LzTiles& ts, int c, float& a0h, float& a0l,
                                           float& a1h, float& a1l) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = lane >> 2, j = (lane & 3) * 2;
  const int ld = c + 1;
  const float* Lh = reinterpret_cast<const float*>(ts.L) + i * ld;
  const float* Ll = Lh + kLT * ld;
  const float* Rh = reinterpret_cast<const float*>(ts.R) + j * ld;
  const float* Rl = Rh + kLT * ld;
  int cnt = 0;
  for (int k = warp; k < c; k += kLWarps) {
    const float xh = Lh[k], xl = Ll[k];
    pair_mac(xh, xl, Rh[k], Rl[k], a0h, a0l);
    pair_mac(xh, xl, Rh[ld + k], Rl[ld + k], a1h, a1l);
    if (++cnt == 8) {
      cnt = 0;
      pair_renorm(a0h, a0l);
      pair_renorm(a1h, a1l);
    }
  }
  pair_renorm(a0h, a0l);
  pair_renorm(a1h, a1l);
}

// Reduce the per-warp pair partial sums of a tile in warp order; store it as
// pairs (Cp) or as FP64 (Cd, minus sigma X when sigma != 0).
__device__ void tile_store_p(LzSmem& sm, float a0h, float a0l, float a1h, float a1l, float* Cp,
                             double* Cd, long long n, int c, int i0, int j0,
                             const double* X = nullptr, double sigma = 0.0,
                             const double* Xprev = nullptr, double beta = 0.0,
                             double* own_w = nullptr) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = lane >> 2, j = (lane & 3) * 2;
  float* rh = reinterpret_cast<float*>(&sm.red[0][0]);
  float* rl = rh + kLWarps * kLT * kLT;
  rh[warp * 64 + i * kLT + j] = a0h;
  rl[warp * 64 + i * kLT + j] = a0l;
  rh[warp * 64 + i * kLT + j + 1] = a1h;
  rl[warp * 64 + i * kLT + j + 1] = a1l;
  __syncthreads();
  if (threadIdx.x < kLT * kLT) {
    float vh = 0.f, vl = 0.f;
    for (int w = 0; w < kLWarps; ++w) pair_add(vh, vl, rh[w * 64 + threadIdx.x], rl[w * 64 + threadIdx.x], vh, vl);
    const int r = threadIdx.x / kLT, cc = threadIdx.x % kLT;
    if (i0 + r < c && j0 + cc < c) {
      const long long e = (long long)(i0 + r) * c + j0 + cc;
      if (Cp) { __stcg(Cp + e, vh); __stcg(Cp + n + e, vl); }
      if (Cd) {
        double v = (double)vh + (double)vl;
        if (sigma != 0.0) v = fma(-sigma, __ldcg(X + e), v);
        if (beta != 0.0) v = fma(-beta, __ldcg(Xprev + e), v);
        __stcg(Cd + e, v);
        if (own_w) own_w[threadIdx.x] = v;
      }
    }
  }
  __syncthreads();
}

// Wide staging (c <= kLWideMaxC, c a multiple of 8): every
// operand tile of a matrix-vector phase is requested at once by 16-byte
// asynchronous copies (cp.async.cg: L2 only, like the loads above) into
// lz_slots(c) slots of 16 rows of ldw = c + 4 floats, so that a phase costs
// one L2 latency instead of one per term.  A row tile holds rows [r0, r0+8)
// of a pair matrix (hi rows 0-7, lo rows 8-15); a column tile holds columns
// [c0, c0+8) untransposed (hi: c rows of 8 floats, then lo).  The products
// below take the same operands in the same order as tile_fma_p and tile_fma, so
// both stagings give the same bits.  In FP64 mode a slot holds 8 rows of c + 2
// doubles (or a column tile of c rows of 8).
// (eight slots up to c = 128; five at c = 256, where two CTAs per SM have no
// room for more)
constexpr int kLWideMaxC = kLMaxC;
__host__ __device__ __forceinline__ int lz_slots(int c) { return c <= 128 ? 8 : 5; }

__host__ __device__ __forceinline__ int lz_wide_ld(int c) { return c + 4; }
__host__ __device__ __forceinline__ int lz_slot_floats(int c) { return 2 * kLT * (c + 4); }

// Doubles of the operand tiles: the wide slots, or L and R.
__host__ __device__ __forceinline__ int lz_tile_doubles(int c, int wide) {
  const int t = wide ? lz_slots(c) * lz_slot_floats(c) / 2 : 2 * kLT * (c + 1);
  return t > 8 * (kLMaxM + 2) ? t : 8 * (kLMaxM + 2);   // also the checks' scratch
}

__device__ __forceinline__ float* wide_slot(float* dyn, int s, int c) {
  return dyn + s * lz_slot_floats(c);
}

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// rows [r0, r0+8) of the pair matrix M (hi at M, lo at M + n) into a row tile
__device__ void wide_rows(float* dst, const float* M, long long n, int c, int r0, int ldw) {
  const int q4 = c >> 2, per = kLT * q4;   // 16-byte chunks per half
  for (int q = threadIdx.x; q < 2 * per; q += kLThreads) {
    const int half = q >= per ? 1 : 0, qq = q - half * per;
    const int r = qq / q4, k4 = (qq - r * q4) << 2;
    cp_async16(dst + (half * kLT + r) * ldw + k4, M + half * n + (long long)(r0 + r) * c + k4);
  }
}
// columns [c0, c0+8) of M into a column tile: dst[half][k][j] = M(half)[k][c0 + j]
__device__ void wide_cols(float* dst, const float* M, long long n, int c, int c0) {
  const int per = 2 * c;                   // two 16-byte chunks per row and half
  for (int q = threadIdx.x; q < 2 * per; q += kLThreads) {
    const int half = q >= per ? 1 : 0, qq = q - half * per;
    const int k = qq >> 1, j4 = (qq & 1) << 2;
    cp_async16(dst + half * kLT * c + k * kLT + j4, M + half * n + (long long)k * c + c0 + j4);
  }
}

// acc += sum over this warp's K slice of L(i, k) R(j, k) in pair arithmetic:
// L a row tile; R a row tile (R(j, k) = row j) or, with rcol, a column tile
// (R(j, k) = M[k][c0 + j]).  Operand order, renormalisation and the final
// renormalisation are those of tile_fma_p.  Bound by the issue of 24 FP32
// instructions and the operand loads per k: eight k at a time (the loads ahead of
// the sums, no counter), neighbouring columns in one load.  Rolled, with four
// loads for them, a BF16x3 Heisenberg sweep at chi = 256 took 89.9 ms and a TF32
// torus sweep at chi = 128 12.03; now 84.3 and 11.47 (the same bits).
template <bool kCol>
__device__ __forceinline__ void wide_mac(const float* Lh, const float* Ll, const float* R, int j, int k, int c, int ldw,
                                         float& a0h, float& a0l, float& a1h, float& a1l) {
  const float xh = Lh[k], xl = Ll[k];
  float2 h, l;
  if constexpr (kCol) {
    h = *reinterpret_cast<const float2*>(R + k * kLT + j);
    l = *reinterpret_cast<const float2*>(R + kLT * c + k * kLT + j);
  } else {
    h = make_float2(R[j * ldw + k], R[(j + 1) * ldw + k]);
    l = make_float2(R[(kLT + j) * ldw + k], R[(kLT + j + 1) * ldw + k]);
  }
  pair_mac(xh, xl, h.x, l.x, a0h, a0l);
  pair_mac(xh, xl, h.y, l.y, a1h, a1l);
}
template <bool kCol>
__device__ __forceinline__ void wide_fma_t(const float* L, const float* R, int c, int ldw,
                                           float& a0h, float& a0l, float& a1h, float& a1l) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = lane >> 2, j = (lane & 3) * 2;
  const float* Lh = L + i * ldw;
  const float* Ll = L + (kLT + i) * ldw;
  int k = warp;
  for (; k + 7 * kLWarps < c; k += 8 * kLWarps) {
#pragma unroll
    for (int u = 0; u < 8; ++u) wide_mac<kCol>(Lh, Ll, R, j, k + u * kLWarps, c, ldw, a0h, a0l, a1h, a1l);
    pair_renorm(a0h, a0l);
    pair_renorm(a1h, a1l);
  }
#pragma unroll 1
  for (; k < c; k += kLWarps) wide_mac<kCol>(Lh, Ll, R, j, k, c, ldw, a0h, a0l, a1h, a1l);
  pair_renorm(a0h, a0l);
  pair_renorm(a1h, a1l);
}
// Two row tiles times the same column tile: the columns are loaded once (0.3 to
// 0.7 % of a mixed sweep; the same bits).
__device__ __forceinline__ void wide_fma2(const float* L0, const float* L1, const float* R, int c, int ldw, float (&a)[8]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = lane >> 2, j = (lane & 3) * 2;
  const float *Lh = L0 + i * ldw, *Ll = L0 + (kLT + i) * ldw;
  const float *Mh = L1 + i * ldw, *Ml = L1 + (kLT + i) * ldw;
  auto mac = [&](int k) {
    const float2 h = *reinterpret_cast<const float2*>(R + k * kLT + j);
    const float2 l = *reinterpret_cast<const float2*>(R + kLT * c + k * kLT + j);
    const float xh = Lh[k], xl = Ll[k], yh = Mh[k], yl = Ml[k];
    pair_mac(xh, xl, h.x, l.x, a[0], a[1]);
    pair_mac(xh, xl, h.y, l.y, a[2], a[3]);
    pair_mac(yh, yl, h.x, l.x, a[4], a[5]);
    pair_mac(yh, yl, h.y, l.y, a[6], a[7]);
  };
  auto renorm = [&]() {
#pragma unroll
    for (int q = 0; q < 8; q += 2) pair_renorm(a[q], a[q + 1]);
  };
  int k = warp;
  for (; k + 7 * kLWarps < c; k += 8 * kLWarps) {
#pragma unroll
    for (int u = 0; u < 8; ++u) mac(k + u * kLWarps);
    renorm();
  }
#pragma unroll 1
  for (; k < c; k += kLWarps) mac(k);
  renorm();
}
__device__ __forceinline__ void wide_fma(const float* L, const float* R, bool rcol, int c, int ldw,
                                         float& a0h, float& a0l, float& a1h, float& a1l) {
  if (rcol) wide_fma_t<true>(L, R, c, ldw, a0h, a0l, a1h, a1l);
  else wide_fma_t<false>(L, R, c, ldw, a0h, a0l, a1h, a1l);
}

// The same three for FP64 tiles (row pitch c + 2 doubles).
__device__ void wide_rows_d(float* slot, const double* M, int c, int r0) {
  double* dst = reinterpret_cast<double*>(slot);
  const int q2 = c >> 1;
  for (int q = threadIdx.x; q < kLT * q2; q += kLThreads) {
    const int r = q / q2, k2 = (q - r * q2) << 1;
    cp_async16(reinterpret_cast<float*>(dst + r * (c + 2) + k2),
               reinterpret_cast<const float*>(M + (long long)(r0 + r) * c + k2));
  }
}
__device__ void wide_cols_d(float* slot, const double* M, int c, int c0) {
  double* dst = reinterpret_cast<double*>(slot);
  for (int q = threadIdx.x; q < 4 * c; q += kLThreads) {
    const int k = q >> 2, j2 = (q & 3) << 1;
    cp_async16(reinterpret_cast<float*>(dst + k * kLT + j2),
               reinterpret_cast<const float*>(M + (long long)k * c + c0 + j2));
  }
}
__device__ __forceinline__ void wide_fma_d(const float* Ls, const float* Rs, bool rcol, int c,
                                           double& a0, double& a1) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = lane >> 2, j = (lane & 3) * 2;
  const double* L = reinterpret_cast<const double*>(Ls) + i * (c + 2);
  const double* R = reinterpret_cast<const double*>(Rs) + (rcol ? j : j * (c + 2));
  const int rk = rcol ? kLT : 1, rj = rcol ? 1 : c + 2;
#pragma unroll 4
  for (int k = warp; k < c; k += kLWarps) {
    const double x = L[k];
    a0 = fma(x, R[k * rk], a0);
    a1 = fma(x, R[k * rk + rj], a1);
  }
}

// One CTA and one tile (c <= 8, FP64): operators, vectors and Y in shared memory,
// matrices as 8 rows of 8; one thread per output.  The sums are those of
// tile_fma and tile_store, whose warp w holds the terms k = w: a chain of fused
// multiply-adds per k over the terms, then the chains in the order of k.  A step
// of the general path is a chain of L2 round trips here (operands, Y, partial
// sums, coefficients) with a cross-warp sum per product; without them a sweep of
// a per-node tree of 16 spins at chi = 8 takes 1.43 instead of 1.67 ms, with the
// same bits.
struct LzTiny {
  const double *s0, *s1;   // 1 + 2K slabs of the left and the right top site
  double* Y;               // 2K slabs
};
__device__ __forceinline__ void tiny_y(const LzTiny& ty, const double* x, int c, int K) {
  for (int t = threadIdx.x; t < 2 * K * 64; t += kLThreads) {
    const int i = (t >> 3) & 7, j = t & 7;
    const double* L = ty.s0 + 64 + (t & ~63) + i * 8;
    double p[kLT], v = 0.0;
#pragma unroll
    for (int k = 0; k < kLT; ++k) p[k] = k < c ? fma(L[k], x[k * 8 + j], 0.0) : 0.0;
#pragma unroll
    for (int k = 0; k < kLT; ++k) v += p[k];
    ty.Y[t] = v;
  }
}
__device__ __forceinline__ double tiny_hx(const LzTiny& ty, const double* x, int c, int K) {
  const int i = threadIdx.x >> 3, j = threadIdx.x & 7;
  double p[kLT], v = 0.0;
#pragma unroll
  for (int k = 0; k < kLT; ++k) p[k] = k < c ? fma(ty.s0[i * 8 + k], x[k * 8 + j], 0.0) : 0.0;
#pragma unroll
  for (int k = 0; k < kLT; ++k)
    if (k < c) p[k] = fma(x[i * 8 + k], ty.s1[j * 8 + k], p[k]);
  for (int q = 0; q < 2 * K; ++q) {
    const double* R = ty.s1 + 64 * (q < K ? 1 + K + q : 1 + q - K) + j * 8;
    const double* L = ty.Y + 64 * q + i * 8;
#pragma unroll
    for (int k = 0; k < kLT; ++k)
      if (k < c) p[k] = fma(L[k], R[k], p[k]);
  }
#pragma unroll
  for (int k = 0; k < kLT; ++k) v += p[k];
  return v;
}

// FP64 value and its pair at index e of a vector (pair vector: hi at P, lo at P + n)
__device__ __forceinline__ void store_both(double* D, float* P, long long n, long long e, double v) {
  __stcg(D + e, v);
  if (P) {
    float h, l;
    split_d(v, h, l);
    __stcg(P + e, h);
    __stcg(P + n + e, l);
  }
}

// Vector entries owned by a CTA: the entries of the 8 x 8 tiles of H x that
// the CTA computes (tiles t = bid, bid + G, ...), so that the projections of a
// new w start without a grid barrier.  Local index q -> global index, or -1
// for the padding of a partial tile.
__device__ __forceinline__ long long own_index(int q, int bid, int G, int nt, int c) {
  const int t = bid + (q >> 6) * G, e = q & 63;
  const int row = (t / nt) * kLT + (e >> 3), col = (t % nt) * kLT + (e & 7);
  return (row < c && col < c) ? (long long)row * c + col : -1;
}

// Per-CTA sum of a[i] * b[i] over the owned entries, reduced in a fixed order.
__device__ double own_dot(LzSmem& sm, const double* a, const double* b, int nown, int bid, int G,
                          int nt, int c) {
  double s = 0.0;
  for (int q = threadIdx.x; q < nown; q += kLThreads) {
    const long long i = own_index(q, bid, G, nt, c);
    if (i >= 0) s = fma(__ldcg(a + i), __ldcg(b + i), s);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sm.red[0][threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kLWarps; ++w) t += sm.red[0][w];
    sm.bcast[1] = t;
  }
  __syncthreads();
  const double v = sm.bcast[1];
  __syncthreads();
  return v;
}

// part[bid][i] = <basis_i, w> over the owned entries for i <= j, and
// part[bid][nslot] = |w|^2 when nslot >= 0.  Warp w takes the vectors
// 4w .. 4w+3, 4w+32 .. (their loads issued together); each sum runs over the
// owned entries lane by lane, then a fixed butterfly.
__device__ void own_projections(const LanczosArgs& a, const LzOwn& own, double* part, int ldp, int j,
                                int nslot, int nown, int bid, int G, int nt, int c, long long n,
                                double* only = nullptr) {
  constexpr int U = 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nv = j + 1 + (nslot >= 0 ? 1 : 0);
  for (int i0 = warp * U; i0 < nv; i0 += kLWarps * U) {
    double s[U];
#pragma unroll
    for (int u = 0; u < U; ++u) s[u] = 0.0;
    for (int q = lane; q < nown; q += 32) {
      const long long e = own_index(q, bid, G, nt, c);
      if (e < 0) continue;
      const double wv = own.wrow >= 0 ? own.p[own.wrow * own.pitch + q] : __ldcg(a.w + e);
      double bv[U];
      if (own.n) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u;
          bv[u] = i < nv ? own.p[(i > j ? own.wrow : i) * own.pitch + q] : 0.0;
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u;
          bv[u] = i < nv ? __ldcg((i > j ? a.w : a.basis + (long long)i * n) + e) : 0.0;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) s[u] = fma(bv[u], wv, s[u]);
    }
    // the butterfly of every sum, four of them together: each exchange halves
    // the number of values a lane holds (6 additions instead of 20 -- an FP64
    // warp instruction takes 16 clocks of the SM -- in the same tree, so the
    // same bits)
    static_assert(U == 4, "four sums share a butterfly");
    const bool h16 = lane & 16, h8 = lane & 8;
    double r0 = h16 ? s[1] : s[0], r1 = h16 ? s[3] : s[2];
    r0 += __shfl_xor_sync(0xffffffffu, h16 ? s[0] : s[1], 16);
    r1 += __shfl_xor_sync(0xffffffffu, h16 ? s[2] : s[3], 16);
    double r = h8 ? r1 : r0;
    r += __shfl_xor_sync(0xffffffffu, h8 ? r0 : r1, 8);
    for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    const int i = i0 + (h8 ? 2 : 0) + (h16 ? 1 : 0);
    if ((lane & 7) == 0 && i < nv) {
      // (0 + r: what the sum over one CTA gives)
      if (only) only[i > j ? nslot : i] = 0.0 + r;
      else __stcg(part + (long long)bid * ldp + (i > j ? nslot : i), r);
    }
  }
}

// out[i] = the sum over the CTAs of their partial sums of coefficient i (i = nn:
// at *out_n instead), in the order of cta_ordered_sum; warp by warp, so that a
// small grid's CTA sums eight coefficients at a time.
__device__ void sum_coefs(const double* part, int ldp, int nn, int nslot, int G, int bid, double* out,
                          double* out_n) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = bid + G * warp; i <= nn; i += G * kLWarps) {
    const double* x = part + (i == nn ? nslot : i);
    double s = 0.0;
    for (int q = lane; q < G; q += 32) s += __ldcg(x + (long long)q * ldp);
    // (lanes without a CTA hold 0: their additions change nothing)
    for (int o = 16; o > 0; o >>= 1)
      if (o < G) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) __stcg(i == nn ? out_n : out + i, s);
  }
}

// Copy cnt coefficients to shared memory (sm.cf).
__device__ __forceinline__ void load_coefs(LzSmem& sm, const double* cf, int cnt) {
  __syncthreads();
  for (int i = threadIdx.x; i < cnt; i += kLThreads) sm.cf[i] = __ldcg(cf + i);
  __syncthreads();
}

// For every owned entry e (local index q): f(q, e, base[e] + sgn * sum_{i < cnt}
// sm.cf[i] basis_i[e]) (base: w, or null: 0).  S = 1, 2 or 4 threads share an entry, each summing
// the terms i = sub, sub + S, ... with eight loads in flight; the S partial
// sums are added in a fixed order.
template <typename Fn>
__device__ void owned_combine(const LanczosArgs& a, const LzSmem& sm, const LzOwn& own, int cnt,
                              const double* base, double sgn, int nown, int bid, int G, int nt, int c, long long n,
                              Fn f) {
  const int S = nown >= kLThreads ? 1 : (nown > kLThreads / 4 ? 2 : 4);
  const int per = kLThreads / S, sub = threadIdx.x % S;
  for (int q0 = 0; q0 < nown; q0 += per) {
    const int q = q0 + threadIdx.x / S;
    const long long e = q < nown ? own_index(q, bid, G, nt, c) : -1;
    double s = 0.0;
    if (e >= 0) {
      int i = sub;
      for (; i + 7 * S < cnt; i += 8 * S) {
        double b[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          b[u] = own.n ? own.p[(i + u * S) * own.pitch + q] : __ldcg(a.basis + (long long)(i + u * S) * n + e);
#pragma unroll
        for (int u = 0; u < 8; ++u) s = fma(sm.cf[i + u * S], b[u], s);
      }
      for (; i < cnt; i += S) s = fma(sm.cf[i], own.n ? own.p[i * own.pitch + q] : __ldcg(a.basis + (long long)i * n + e), s);
    }
    if (S >= 2) s += __shfl_down_sync(0xffffffffu, s, 1);
    if (S >= 4) s += __shfl_down_sync(0xffffffffu, s, 2);
    if (sub == 0 && e >= 0) {
      const double bv = !base ? 0.0 : (own.wrow >= 0 ? own.p[own.wrow * own.pitch + q] : __ldcg(base + e));
      f(q, e, bv + sgn * s);
    }
  }
}

// Poll a word until test(v), at most `limit` times and not after *err was
// raised, by thread 0; the word is returned to every thread (ok: whether the
// wait succeeded).
template <typename Test>
__device__ unsigned lz_wait_word(LzSmem& sm, const unsigned* w, Test test, int* err, int limit, bool raise,
                                 bool& ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned v = 0;
    int good = 0;
    for (int spins = 0; spins <= limit; ++spins) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(w) : "memory");
      if (test(v)) { good = 1; break; }
      if (*reinterpret_cast<volatile int*>(err)) break;
      __nanosleep(64);
    }
    if (!good && raise) atomicOr(err, 4);
    sm.ok = good;
    sm.bcast[1] = __longlong_as_double((long long)v);
  }
  __syncthreads();
  ok = sm.ok != 0;
  const unsigned v = (unsigned)__double_as_longlong(sm.bcast[1]);
  __syncthreads();
  return v;
}

constexpr unsigned kLQuit = 0xFFFFFFFFu;

// The extra CTA of a launch with a.extra: it runs the convergence checks of
// the tridiagonal while the others take the next step.  A job (a.job[0]) is
// number << 8 | m; its answer (a.job[1]) is number << 1 | passed.
__device__ void lz_checker(const LanczosArgs& a, LzSmem& sm, double* dyn) {
  unsigned seen = 0;
  const int limit = max(a.max_spin, 1 << 23);   // between jobs it only idles
  while (true) {
    bool ok;
    const unsigned v = lz_wait_word(sm, a.job, [&](unsigned w) { return w != seen; }, a.err, limit, false, ok);
    if (!ok || v == kLQuit) return;
    seen = v;
    const int m = (int)(v & 0xFFu);
    load_tridiagonal(a, sm, m);
    {
      const bool pass = ritz_check_df(sm, dyn, m, __ldcg(a.scal + 8), a.tol);
      if (threadIdx.x == 0)
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.job + 1), "r"((v >> 8) << 1 | (pass ? 1u : 0u)) : "memory");
    }
  }
}

__device__ __forceinline__ void lz_post(const LanczosArgs& a, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.job), "r"(v) : "memory");
}

// kTiny: one CTA, one tile (c <= 8), FP64: everything a step reads is in shared memory.
template <bool kTiny>
__device__ __forceinline__ void lanczos_body(const LanczosArgs& a, LzSmem& sm, float* lz_dyn, int G) {
  const int c = a.c, K = a.K, m = a.m;
  const long long n = (long long)c * c;
  const int bid = blockIdx.x;
  const int nt = (c + kLT - 1) / kLT;
  const int ntiles = nt * nt;
  const int nown = (bid < ntiles ? (ntiles - bid + G - 1) / G : 0) * 64;
  const int ldp = m + 2;                     // stride of the per-CTA partial sums
  const int nslot = m + 1;                   // slot of |w|^2 in a CTA's partial sums
  double* part = a.part;
  double* wn2 = a.coef + 2 * ldp - 1;        // |w|^2 of the current step
  unsigned target = 0;

  const bool df = a.df != 0;
  const bool wide = a.wide != 0;
  const int ldw = lz_wide_ld(c);
  double* dynd = reinterpret_cast<double*>(lz_dyn);
  const LzTiles ts{dynd, dynd + kLT * (c + 1), c + 1};
  LzOwn own;
  own.p = dynd + lz_tile_doubles(c, a.wide);
  own.pitch = a.own_pitch;
  own.n = a.ncache;
  own.wrow = a.ncache > 0 ? a.ncache : -1;
  unsigned jobs = 0;          // checks posted to the extra CTA
  bool ok = true;
  const int wlimit = max(a.max_spin > 0 ? a.max_spin : kLMaxSpin, 1 << 16);
  auto answer = [&](bool& good) {
    return lz_wait_word(sm, a.job + 1, [&](unsigned w) { return (w >> 1) == jobs; }, a.err, wlimit, true, good);
  };
  float* bp0 = df ? a.bp : nullptr;          // pairs of basis_0
  LzTiny ty;
  if constexpr (kTiny) {
    double* p = own.p + (own.n + 1) * own.pitch;
    const int slabs = 1 + 2 * K;
    for (int t = threadIdx.x; t < 2 * slabs * 64; t += kLThreads) {
      const int i = (t >> 3) & 7, j = t & 7, q = t >> 6;
      const double* S = q < slabs ? a.s0 + q * n : a.s1 + (q - slabs) * n;
      p[t] = i < c && j < c ? __ldcg(S + i * c + j) : 0.0;
    }
    ty.s0 = p;
    ty.s1 = p + slabs * 64;
    ty.Y = p + 2 * slabs * 64;
  }
  // start: the operators as pairs (double-float mode), Vprev = V, basis_0 = V / |V|
  if (df) {
    const long long nops = (long long)(1 + 2 * K) * n;
    const long long gt = (long long)blockIdx.x * kLThreads + threadIdx.x, gs = (long long)G * kLThreads;
    for (int side = 0; side < (a.s1 == a.s0 ? 1 : 2); ++side) {
      const double* src = side ? a.s1 : a.s0;
      float* dst = side ? a.s1p : a.s0p;
      for (long long e = gt; e < nops; e += gs) {
        const long long q = e / n, r = e % n;
        float h, l;
        split_d(__ldcg(src + e), h, l);
        __stcg(dst + 2 * q * n + r, h);
        __stcg(dst + 2 * q * n + n + r, l);
      }
    }
  }
  for (int q = threadIdx.x; q < nown; q += kLThreads) {
    const long long e = own_index(q, bid, G, nt, c);
    if (e >= 0) __stcg(a.Vprev + e, __ldcg(a.V + e));
  }
  {
    const double s = own_dot(sm, a.V, a.V, nown, bid, G, nt, c);
    if (threadIdx.x == 0) __stcg(part + (long long)bid * ldp, s);
  }
  if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
  double inv = 1.0 / sqrt(cta_ordered_sum(sm, part, G, ldp));
  for (int q = threadIdx.x; q < nown; q += kLThreads) {
    const long long e = own_index(q, bid, G, nt, c);
    if (e >= 0) {
      const double v = __ldcg(a.V + e) * inv;
      store_both(a.basis, bp0, n, e, v);
      own.set(0, q, v);
    }
  }
  if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
  const float* s0p = a.s0p;
  const float* s1p = a.s1 == a.s0 ? a.s0p : a.s1p;

  int conv = 0;
  for (int cyc = 0; cyc < a.restarts && !conv; ++cyc) {
    int tdim = 0;
    int due = -1, due_m = 0;    // step whose end reads the pending check's answer, its size
    // Steps j >= 1 run on H - sigma I with sigma = alpha_0, the Rayleigh
    // quotient of the start vector (the same Krylov space; the tridiagonal is
    // shifted by -sigma, its first entry 0).  Without the shift |w|^2 ~ E^2
    // would dwarf beta_j^2 and every step would need the second
    // Gram-Schmidt pass.
    // Step j >= 1 also subtracts, while w is stored, the two recurrence terms
    // it knows: sigma_j x_j with sigma_j = alpha_{j-1} of H (the previous
    // step's diagonal entry, close to this one's) and beta_{j-1} x_{j-1}.  The
    // projections then only remove what is left (rounding and the small
    // alpha_j - sigma_j), so the one-pass test below passes in most steps and
    // the second Gram-Schmidt pass with its two grid barriers is skipped.  The
    // tridiagonal keeps the single shift sigma: its entry j is
    // c_j + sigma_j - sigma.
    for (int j = 0; j < m; ++j) {
      const double* x = a.basis + (long long)j * n;
      const double sigma_j = j == 0 ? 0.0 : (j == 1 ? sm.sigma : sm.alpha_prev_h);
      const double* xprev = j > 0 ? x - n : nullptr;
      const double beta_j1 = j > 0 ? sm.beta_prev : 0.0;
      if constexpr (kTiny) {
        const double* xs = own.p + j * own.pitch;
        tiny_y(ty, xs, c, K);
        __syncthreads();
        if (threadIdx.x < 64) {
          const int r = threadIdx.x >> 3, cc = threadIdx.x & 7;
          double v = tiny_hx(ty, xs, c, K);
          if (r < c && cc < c) {
            if (sigma_j != 0.0) v = fma(-sigma_j, xs[threadIdx.x], v);
            if (beta_j1 != 0.0) v = fma(-beta_j1, xs[threadIdx.x - own.pitch], v);
            own.p[own.wrow * own.pitch + threadIdx.x] = v;
          }
        }
        __syncthreads();
        own_projections(a, own, part, ldp, j, nslot, nown, bid, G, nt, c, n, sm.cf);
      } else {
      // phase A: Y_b = Op_b x for the 2K operators A_k0, B_k0 (stored after o_0)
      const float* xp = df ? a.bp + 2 * (long long)j * n : nullptr;
      // wide staging: all 2K products of a tile by its CTA, the columns of x
      // staged once, the operator rows as many at a time as there are slots
      for (int t = bid; t < ntiles && wide; t += G) {
        const int i0 = (t / nt) * kLT, j0 = (t % nt) * kLT;
        const int rows = lz_slots(c) - 1;
        for (int b0 = 0; b0 < 2 * K; b0 += rows) {
          const int nb = min(rows, 2 * K - b0);
          if (df) {
            if (b0 == 0) wide_cols(wide_slot(lz_dyn, 0, c), xp, n, c, j0);
            for (int u = 0; u < nb; ++u)
              wide_rows(wide_slot(lz_dyn, 1 + u, c), s0p + 2 * (long long)(1 + b0 + u) * n, n, c,
                        i0, ldw);
          } else {
            if (b0 == 0) wide_cols_d(wide_slot(lz_dyn, 0, c), x, c, j0);
            for (int u = 0; u < nb; ++u)
              wide_rows_d(wide_slot(lz_dyn, 1 + u, c), a.s0 + (long long)(1 + b0 + u) * n, c, i0);
          }
          cp_async_wait_all();
          __syncthreads();
          for (int u = 0; u < nb; ++u) {
            if (df) {
              float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
              const bool two = u + 1 < nb;
              if (two)
                wide_fma2(wide_slot(lz_dyn, 1 + u, c), wide_slot(lz_dyn, 2 + u, c), wide_slot(lz_dyn, 0, c), c, ldw, v);
              else
                wide_fma(wide_slot(lz_dyn, 1 + u, c), wide_slot(lz_dyn, 0, c), true, c, ldw, v[0], v[1], v[2], v[3]);
              tile_store_p(sm, v[0], v[1], v[2], v[3], a.Yp + 2 * (long long)(b0 + u) * n, nullptr, n, c, i0, j0);
              if (two) {
                ++u;
                tile_store_p(sm, v[4], v[5], v[6], v[7], a.Yp + 2 * (long long)(b0 + u) * n, nullptr, n, c, i0, j0);
              }
            } else {
              double a0 = 0.0, a1 = 0.0;
              wide_fma_d(wide_slot(lz_dyn, 1 + u, c), wide_slot(lz_dyn, 0, c), true, c, a0, a1);
              tile_store(sm, a0, a1, a.Y + (long long)(b0 + u) * n, c, i0, j0);
            }
          }
        }
      }
      for (int it = bid; it < 2 * K * ntiles && !wide; it += G) {
        const int b = it / ntiles, t = it % ntiles;
        const int i0 = (t / nt) * kLT, j0 = (t % nt) * kLT;
        if (df) {
          stage_rows_p(ts.L, s0p + 2 * (long long)(1 + b) * n, n, c, i0);
          stage_cols_p(ts.R, xp, n, c, j0);
          __syncthreads();
          float a0h = 0.f, a0l = 0.f, a1h = 0.f, a1l = 0.f;
          tile_fma_p(ts, c, a0h, a0l, a1h, a1l);
          tile_store_p(sm, a0h, a0l, a1h, a1l, a.Yp + 2 * (long long)b * n, nullptr, n, c, i0, j0);
          continue;
        }
        stage_rows(ts.L, a.s0 + (long long)(1 + b) * n, c, i0);
        stage_cols(ts.R, x, c, j0);
        __syncthreads();
        double a0 = 0.0, a1 = 0.0;
        tile_fma(ts, c, a0, a1);
        tile_store(sm, a0, a1, a.Y + (long long)b * n, c, i0, j0);
      }
      if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
      // phase B: w = o_0 x + x o_1^T + sum_k Y_k B_k1^T + Y_{K+k} A_k1^T on the
      // owned tiles, then their projections on basis_0..j and |w|^2
      // wide staging: the operand tiles of several terms in one round
      for (int t = bid; t < ntiles && wide; t += G) {
        const int i0 = (t / nt) * kLT, j0 = (t % nt) * kLT;
        float a0h = 0.f, a0l = 0.f, a1h = 0.f, a1l = 0.f;
        double a0 = 0.0, a1 = 0.0;
        const int nterms = 2 + 2 * K;
        const int terms = lz_slots(c) / 2;
        for (int t0 = 0; t0 < nterms; t0 += terms) {
          const int tn = min(terms, nterms - t0);
          for (int u = 0; u < tn; ++u) {
            const int term = t0 + u;
            float* Ls = wide_slot(lz_dyn, 2 * u, c);
            float* Rs = wide_slot(lz_dyn, 2 * u + 1, c);
            const int q = term - 2;            // Y_q with q < K: B_{q,1}; else A_{q-K,1}
            const long long rop = q < K ? (long long)(1 + K + q) : (long long)(1 + q - K);
            if (df) {
              if (term == 0) {
                wide_rows(Ls, s0p, n, c, i0, ldw);
                wide_cols(Rs, xp, n, c, j0);
              } else if (term == 1) {
                wide_rows(Ls, xp, n, c, i0, ldw);
                wide_rows(Rs, s1p, n, c, j0, ldw);
              } else {
                wide_rows(Ls, a.Yp + 2 * (long long)q * n, n, c, i0, ldw);
                wide_rows(Rs, s1p + 2 * rop * n, n, c, j0, ldw);
              }
            } else {
              if (term == 0) {
                wide_rows_d(Ls, a.s0, c, i0);
                wide_cols_d(Rs, x, c, j0);
              } else if (term == 1) {
                wide_rows_d(Ls, x, c, i0);
                wide_rows_d(Rs, a.s1, c, j0);
              } else {
                wide_rows_d(Ls, a.Y + (long long)q * n, c, i0);
                wide_rows_d(Rs, a.s1 + rop * n, c, j0);
              }
            }
          }
          cp_async_wait_all();
          __syncthreads();
          for (int u = 0; u < tn; ++u) {
            if (df)
              wide_fma(wide_slot(lz_dyn, 2 * u, c), wide_slot(lz_dyn, 2 * u + 1, c), t0 + u == 0, c,
                       ldw, a0h, a0l, a1h, a1l);
            else
              wide_fma_d(wide_slot(lz_dyn, 2 * u, c), wide_slot(lz_dyn, 2 * u + 1, c), t0 + u == 0,
                         c, a0, a1);
          }
          __syncthreads();
        }
        double* ow = own.wrow >= 0 ? own.p + own.wrow * own.pitch + ((t - bid) / G) * 64 : nullptr;
        if (df)
          tile_store_p(sm, a0h, a0l, a1h, a1l, nullptr, a.w, n, c, i0, j0, x, sigma_j, xprev,
                       beta_j1, ow);
        else
          tile_store(sm, a0, a1, a.w, c, i0, j0, x, sigma_j, xprev, beta_j1, ow);
      }
      for (int t = bid; t < ntiles && df && !wide; t += G) {
        const int i0 = (t / nt) * kLT, j0 = (t % nt) * kLT;
        float a0h = 0.f, a0l = 0.f, a1h = 0.f, a1l = 0.f;
        for (int term = 0; term < 2 + 2 * K; ++term) {
          if (term == 0) {
            stage_rows_p(ts.L, s0p, n, c, i0);
            stage_cols_p(ts.R, xp, n, c, j0);
          } else if (term == 1) {
            stage_rows_p(ts.L, xp, n, c, i0);
            stage_rows_p(ts.R, s1p, n, c, j0);
          } else {
            const int q = term - 2;            // Y_q with q < K: B_{q,1}; else A_{q-K,1}
            const long long rop = q < K ? (long long)(1 + K + q) : (long long)(1 + q - K);
            stage_rows_p(ts.L, a.Yp + 2 * (long long)q * n, n, c, i0);
            stage_rows_p(ts.R, s1p + 2 * rop * n, n, c, j0);
          }
          __syncthreads();
          tile_fma_p(ts, c, a0h, a0l, a1h, a1l);
          __syncthreads();
        }
        tile_store_p(sm, a0h, a0l, a1h, a1l, nullptr, a.w, n, c, i0, j0, x, sigma_j, xprev, beta_j1,
                     own.wrow >= 0 ? own.p + own.wrow * own.pitch + ((t - bid) / G) * 64 : nullptr);
      }
      for (int t = bid; t < ntiles && !df && !wide; t += G) {
        const int i0 = (t / nt) * kLT, j0 = (t % nt) * kLT;
        double a0 = 0.0, a1 = 0.0;
        for (int term = 0; term < 2 + 2 * K; ++term) {
          if (term == 0) {
            stage_rows(ts.L, a.s0, c, i0);
            stage_cols(ts.R, x, c, j0);
          } else if (term == 1) {
            stage_rows(ts.L, x, c, i0);
            stage_rows(ts.R, a.s1, c, j0);
          } else {
            const int q = term - 2;            // Y_q with q < K: B_{q,1}; else A_{q-K,1}
            const long long rop = q < K ? (long long)(1 + K + q) * n : (long long)(1 + q - K) * n;
            stage_rows(ts.L, a.Y + (long long)q * n, c, i0);
            stage_rows(ts.R, a.s1 + rop, c, j0);
          }
          __syncthreads();
          tile_fma(ts, c, a0, a1);
          __syncthreads();
        }
        tile_store(sm, a0, a1, a.w, c, i0, j0, x, sigma_j, xprev, beta_j1,
                   own.wrow >= 0 ? own.p + own.wrow * own.pitch + ((t - bid) / G) * 64 : nullptr);
      }
      own_projections(a, own, part, ldp, j, nslot, nown, bid, G, nt, c, n);
      if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
      // coefficients of the first Gram-Schmidt pass and |w|^2 (one warp each)
      sum_coefs(part, ldp, j + 1, nslot, G, bid, a.coef, wn2);
      if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
      }
      if (j == due) {
        // the answer to the check posted kLLag steps ago, which ran meanwhile:
        // when it passed, the cycle ends with that step's tridiagonal and the
        // steps since are dropped (they only extended the basis)
        const unsigned v = answer(ok);
        if (!ok) return;
        due = -1;
        if (v & 1u) {
          tdim = due_m;
          break;
        }
      }
      // |w - sum c_i b_i|^2 = |w|^2 - sum c_i^2 for orthonormal b_i; when at
      // least a quarter of |w|^2 remains, one pass is accurate to rounding
      // (the second pass of "twice is enough" is needed only after heavy
      // cancellation), and the norm needs no further reduction
      if constexpr (kTiny) __syncthreads();
      else load_coefs(sm, a.coef, j + 1);
      // warp 0 takes the step's scalars (the FP64 square root and division are
      // long: eight warps repeating them cost 4 k clocks a step): the sum of
      // c_i^2 in a fixed order (lane-strided, then a butterfly), so the same
      // one-pass decision in every CTA, then alpha_j, beta_j, 1 / beta_j
      const bool check = (j + 1) % kLCheck == 0 && j + 1 < m;
      auto scalars = [&](double alpha_j, double beta_j) {   // lane 0
        if (j == 0) {
          sm.sigma = alpha_j;
          alpha_j = 0.0;
        } else {
          alpha_j += sigma_j - sm.sigma;
        }
        const double ah = alpha_j + sm.sigma;
        sm.alpha_prev_h = ah;
        const bool brk = !(beta_j > 1e-12 * fmax(fabs(ah) + beta_j1, 1e-300));
        sm.brk = brk;
        if (bid == 0) {
          __stcg(a.alpha + j, alpha_j);
          __stcg(a.beta + j, brk ? 0.0 : beta_j);
          if (check && a.extra && !brk) {
            __stcg(a.scal + 8, sm.sigma);
            lz_post(a, (jobs + 1) << 8 | (unsigned)(j + 1));
          }
        }
        sm.beta_prev = beta_j;
        sm.inv = 1.0 / beta_j;
      };
      if (threadIdx.x < 32) {
        const double w2 = kTiny ? sm.cf[nslot] : __ldcg(wn2);
        double t = 0.0;
        for (int i = threadIdx.x; i <= j; i += 32) t = fma(sm.cf[i], sm.cf[i], t);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        const bool one = w2 - t > 0.25 * w2;
        if (threadIdx.x == 0) {
          sm.one_pass = one;
          if (one) scalars(sm.cf[j], sqrt(w2 - t));
        }
      }
      __syncthreads();
      if (!sm.one_pass) {
        // second pass: w1 = w - sum c_i b_i, then d_i = <b_i, w1> and |w1|^2 in
        // one reduction; |w1 - sum d_i b_i|^2 = |w1|^2 - sum d_i^2 (the d_i are
        // rounding-sized), and basis_{j+1} below subtracts sum d_i b_i
        const double alpha1 = sm.cf[j];
        owned_combine(a, sm, own, j + 1, a.w, -1.0, nown, bid, G, nt, c, n,
                      [&](int q, long long e, double v) {
                        __stcg(a.w + e, v);
                        if (own.wrow >= 0) own.p[own.wrow * own.pitch + q] = v;
                      });
        __syncthreads();
        own_projections(a, own, part, ldp, j, nslot, nown, bid, G, nt, c, n, kTiny ? sm.cf : nullptr);
        if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
        if constexpr (!kTiny) {
          sum_coefs(part, ldp, j + 1, nslot, G, bid, a.coef + ldp, a.coef + ldp + j + 1);
          if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
          load_coefs(sm, a.coef + ldp, j + 2);
        }
        if (threadIdx.x < 32) {
          double t = 0.0;
          for (int i = threadIdx.x; i <= j; i += 32) t = fma(sm.cf[i], sm.cf[i], t);
          for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          if (threadIdx.x == 0) scalars(alpha1 + sm.cf[j], sqrt(fmax(sm.cf[kTiny ? nslot : j + 1] - t, 0.0)));
        }
        __syncthreads();
      }
      // every kLCheck steps the tridiagonal so far is tested for convergence
      // (pair arithmetic): by the extra CTA during the next kLLag steps, or by
      // CTA 0 while the others wait
      const bool breakdown = sm.brk != 0;
      tdim = j + 1;
      if (breakdown) {
        if (due >= 0) {
          const unsigned v = answer(ok);
          if (!ok) return;
          if (v & 1u) tdim = due_m;
        }
        break;
      }
      if (check && a.extra) {
        ++jobs;
        due = min(j + kLLag, m - 1);
        due_m = j + 1;
      }
      // basis_{j+1} = (w - sum c_i b_i) / beta_j, or (w1 - sum d_i b_i) / beta_j
      const double binv = sm.inv;
      double* nb = a.basis + (long long)(j + 1) * n;
      float* nbp = df ? a.bp + 2 * (long long)(j + 1) * n : nullptr;
      // (sm.cf holds the c_i of the one-pass path or the d_i of the second pass)
      owned_combine(a, sm, own, j + 1, a.w, -1.0, nown, bid, G, nt, c, n,
                    [&](int q, long long e, double v) {
                      const double x1 = v * binv;
                      store_both(nb, nbp, n, e, x1);
                      own.set(j + 1, q, x1);
                    });
      // (without the extra CTA: CTA 0's check, while the others wait)
      const bool inline_check = check && !a.extra;
      if (inline_check && bid == 0) {
        load_tridiagonal(a, sm, j + 1);
        const bool pass = ritz_check_df(sm, dynd, j + 1, sm.sigma, a.tol);
        if (threadIdx.x == 0) __stcg(a.scal + 3, pass ? 1.0 : 0.0);
        __syncthreads();
      }
      if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
      if (inline_check && __ldcg(a.scal + 3) != 0.0) break;
    }
    // Ritz pair of the tridiagonal (CTA 0), then V = sum_i y_i basis_i
    if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
    if (bid == 0) {
      load_tridiagonal(a, sm, tdim);
      if (df) ritz_pair(sm, dynd, tdim, a.y, a.scal + 1, a.scal + 2);
      else ritz_pair_f64(sm, a, dynd, tdim, a.y, a.scal + 1, a.scal + 2);
      __syncthreads();
      if (threadIdx.x == 0) {
        // Ritz value of H: the tridiagonal's plus the shift
        const double theta = *(volatile double*)(a.scal + 1) + sm.sigma;
        a.scal[1] = theta;
        a.flags[1] = tdim;
        a.flags[0] = *(volatile double*)(a.scal + 2) <= a.tol * fmax(fabs(theta), 1e-300);
        __threadfence();
      }
    }
    if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
    conv = __ldcg(a.flags);
    load_coefs(sm, a.y, tdim);
    owned_combine(a, sm, own, tdim, nullptr, 1.0, nown, bid, G, nt, c, n,
                  [&](int, long long e, double v) { __stcg(a.V + e, v); });
    __syncthreads();
    {
      const double s = own_dot(sm, a.V, a.V, nown, bid, G, nt, c);
      if (threadIdx.x == 0) __stcg(part + (long long)bid * ldp, s);
    }
    if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
    inv = 1.0 / sqrt(cta_ordered_sum(sm, part, G, ldp));
    for (int q = threadIdx.x; q < nown; q += kLThreads) {
      const long long e = own_index(q, bid, G, nt, c);
      if (e < 0) continue;
      const double t = __ldcg(a.V + e) * inv;
      __stcg(a.V + e, t);
      store_both(a.basis, bp0, n, e, t);
      own.set(0, q, t);
    }
    if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
  }
  // sign: <V, Vprev> >= 0
  {
    const double s = own_dot(sm, a.V, a.Vprev, nown, bid, G, nt, c);
    if (threadIdx.x == 0) __stcg(part + (long long)bid * ldp + 1, s);
  }
  if (!lz_barrier(sm, a.bar, target, G, a.err, a.max_spin > 0 ? a.max_spin : kLMaxSpin)) return;
  if (cta_ordered_sum(sm, part + 1, G, ldp) < 0.0)
    for (int q = threadIdx.x; q < nown; q += kLThreads) {
      const long long e = own_index(q, bid, G, nt, c);
      if (e >= 0) __stcg(a.V + e, -__ldcg(a.V + e));
    }
}

template <bool kTiny>
__global__ void __launch_bounds__(kLThreads, 2) lanczos_kernel(const LanczosArgs a) {
  __shared__ LzSmem sm;
  extern __shared__ __align__(16) float lz_dyn[];
  const int G = (int)gridDim.x - (a.extra ? 1 : 0);
  if ((int)blockIdx.x == G) {
    lz_checker(a, sm, reinterpret_cast<double*>(lz_dyn));
    return;
  }
  lanczos_body<kTiny>(a, sm, lz_dyn, kTiny ? 1 : G);
  if (a.extra && blockIdx.x == 0 && threadIdx.x == 0) lz_post(a, kLQuit);
}

// Dynamic shared memory of a CTA at most (two CTAs per SM).
constexpr int kLMaxDyn = 96 * 1024;

struct LzGrid {
  int sms = 0, per_sm = 0;
};
std::mutex g_lz_mutex;
LzGrid g_lz_grid[64];

int lanczos_grid_cap() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lock(g_lz_mutex);
  LzGrid& g = g_lz_grid[dev];
  if (!g.sms) {
    int sms = 0, occ = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    const int dyn = kLMaxDyn;
    if (cudaFuncSetAttribute(lanczos_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) !=
            cudaSuccess ||
        cudaFuncSetAttribute(lanczos_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) !=
            cudaSuccess)
      return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, lanczos_kernel<false>, kLThreads, dyn) !=
        cudaSuccess)
      return 0;
    g.sms = sms;
    g.per_sm = std::min(occ, 2);
  }
  return g.sms * g.per_sm;
}

}  // namespace

bool lanczos_supported(int c, int m) { return c >= 1 && c <= kLMaxC && m >= 2 && m <= kLMaxM; }

int lanczos_grid(int c, int grid_share) {
  int cap = lanczos_grid_cap();
  if (cap <= 0) return 0;
  if (grid_share > 1) cap = std::max(1, cap / grid_share);
  const long long n = (long long)c * c;
  // no more CTAs than 64-entry slices of the vectors, at least one
  return (int)std::max<long long>(1, std::min<long long>(std::min(cap, kLMaxGrid), n / 64));
}

int lanczos_launch(const LanczosArgs& a0, int grid, int grid_share, cudaStream_t s) {
  if (!lanczos_supported(a0.c, a0.m) || grid < 1 || grid > kLMaxGrid) return -1;
  // the grid cap also sets the kernel's dynamic shared-memory limit
  if (lanczos_grid_cap() <= 0) return -1;
  LanczosArgs a = a0;
  a.wide = a.c <= kLWideMaxC && a.c % 8 == 0 ? 1 : 0;
  // shared-memory copies of the CTA's entries of the basis vectors, if all fit
  const int nt = (a.c + kLT - 1) / kLT;
  const int tiles = lz_tile_doubles(a.c, a.wide);
  a.own_pitch = (nt * nt + grid - 1) / grid * 64 + 8;
  a.ncache = a.m + 1 <= (kLMaxDyn / 8 - tiles) / a.own_pitch - 1 ? a.m + 1 : 0;
  // the checks run in a CTA of their own when one more is co-resident
  a.extra = grid + 1 <= lanczos_grid_cap() / std::max(1, grid_share) ? 1 : 0;
  size_t dyn = 8 * ((size_t)tiles + (a.ncache > 0 ? (size_t)(a.ncache + 1) * a.own_pitch : 0));
  // one CTA and one tile: the operators and Y stay in shared memory too (larger
  // grids exchange the vectors through L2 anyway)
  const size_t ops = 8 * 64 * (2 * (size_t)(1 + 2 * a.K) + 2 * (size_t)a.K);
  const bool tiny = !a.df && grid == 1 && a.c <= kLT && a.ncache > 0 && dyn + ops <= kLMaxDyn;
  if (tiny) dyn += ops;
  a.job = a.bar + 1;
  cudaMemsetAsync(a.bar, 0, 3 * sizeof(unsigned), s);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid + a.extra);
  cfg.blockDim = dim3(kLThreads);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, tiny ? lanczos_kernel<true> : lanczos_kernel<false>, a) != cudaSuccess) return -1;
  return 1;
}

}  // namespace ttn
