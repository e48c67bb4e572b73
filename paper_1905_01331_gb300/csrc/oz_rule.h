// When an FP64 product goes to the digit engine (gemm_oz.cu) instead of the FP64
// kernel: host-only, so that a host test can hold the rule against the times it
// was drawn from.
#pragma once

namespace ttn {

// Tiles of the digit engine: 128 x 64 outputs (128 x 32 for N <= 32), chunks of
// 128 values of K in stages of 32.
constexpr int kOBM = 128;
constexpr int kOChunk = 128;
constexpr int kOBK = 32;
constexpr int oz_tile_n(int N) { return N > 32 ? 64 : 32; }

// Below this many multiply-adds both kernels take 6 to 15 us of latency.
constexpr double kOzMinWork = 1 << 23;

// A tile costs the same however much of it is padding: about 4 us, 2.6 a stage
// and 2 (128 x 32) or 4 (128 x 64) a chunk, while an SM of the FP64 kernel does 2500
// multiply-adds in a microsecond.  Both engines keep every SM busy with a batch of
// products, so the digit engine takes a product whose tiles do more useful
// multiply-adds than the FP64 kernel would in a tile's time.  Measured (digits
// against FP64, us): 4096 products of 16 x 16 x 16 227 and 44, 192 of 16 x 16 x
// 256 56 and 41, 64 sums of five 16 x 256 x 16 80 and 47: FP64; 256 of 256 x 16 x
// 16 39 and 44, 512 of 32 x 32 x 32 35 and 43, 192 of 32 x 32 x 256 57 and 127, one
// of 16 x 16 x 32768 43 and 55: digits.  K: one value per group.
inline bool oz_worth(int M, int N, long long batches, const int* K, int groups) {
  const int bn = oz_tile_n(N);
  const double tiles = static_cast<double>((M + kOBM - 1) / kOBM) * ((N + bn - 1) / bn) * batches;
  double sum = 0.0, cost = 4.0;
  for (int g = 0; g < groups; ++g) {
    sum += K[g];
    cost += 2.6 * ((K[g] + kOBK - 1) / kOBK) + bn / 16.0 * ((K[g] + kOChunk - 1) / kOChunk);
  }
  const double work = static_cast<double>(M) * N * batches * sum;
  return work >= kOzMinWork && work >= 2500.0 * cost * tiles;
}

}  // namespace ttn
