// Columns per tile of the dense GEMM (csrc/dense.cu), on their own so that a test can ask for them.
#pragma once
#include <algorithm>
#include <cstdint>

namespace cast {

// Columns per tile: 256, or 128 where 256 would leave SMs without work.  A 64-wide k-step of a
// pair takes about 660 cycles at 256 columns (32 KB per SM) and 480 at 128 (24 KB; both bound by
// the ~50 bytes per clock that an SM takes from L2, measured at the Matrix-Game-shaped FFN: 69 and
// 96 us for its second GEMM), the epilogue of a tile about 16 cycles a column.  FFN sites of other
// sizes with either width forced on both GEMMs and by the rule (rows x D x D_ff: 128, 256, rule, us):
//   1,760 x 2048 x 8192: 121, 91, 88         17,600 x 3072 x 12288: 2,055, 1,560, 1,618
//   12,480 x 1024 x 4096: 196, 159, 159       56,320 x 1024 x 2816: 542, 428, 444
//   5,280 x 1032 x 2056: 77, 74, 72           5,280 x 264 x 2056: 45, 52, 45
//   2,048 x 768 x 3072: 37, 45, 37            1,053 x 512 x 2048: 37, 44, 38        864 x 1280 x 5120: 47, 56, 47
// row_pairs: pairs of 128-row tiles; n_k: 64-wide k-steps; pairs: pairs of SMs.
inline int tile_columns(int row_pairs, int N, int n_k, int pairs) {
  auto cycles = [&](int bn, int step) -> int64_t {
    const int64_t items = (int64_t)row_pairs * ((N + bn - 1) / bn), rounds = (items + pairs - 1) / pairs;
    return rounds * std::max<int64_t>((int64_t)n_k * step, 16 * bn) + 16 * bn;
  };
  return cycles(128, 480) < cycles(256, 660) ? 128 : 256;
}

}  // namespace cast
