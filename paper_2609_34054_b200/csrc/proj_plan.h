// Which projection kernel takes a call and how its work is cut: arithmetic on sizes alone, free of CUDA, so that the rules can be
// compiled and checked without a GPU.
#pragma once
#include <algorithm>

namespace precc {

constexpr int GEMM_BM = 128;                             // rows of a tile of the tiled kernel
constexpr int GEMM_BK = 64;                              // 64 bf16 = one 128-byte swizzle row
constexpr int PT_COLS = 128;                             // output columns of a tile of the turn kernel (the M of its MMA)
constexpr int PT_MAX_TN = 256;                           // rows of X in such a tile at most

// The turn kernel over the whole K extent (up to 256 columns): rows of a tile, or 0 where 128-row tiles are as good.  With one
// round of those they are (9000 x 128: 28.0 against 28.5 us); from two rounds on this form wins by what they fetch twice or leave
// idle.  Very few columns cost the tiled kernel little beside the rows, so there it has to save a fifth of them
// (32768 x 32: 49.1 against 50.8 us for an eighth; 20000 x 32: 47.7 against 33.7 us).  The row tiles lie on a grid axis of 65535.
inline int pick_wide_rows(int M, int K, int n_out, int sm_count) {
  (void)K;
  const long long rt = ((M + GEMM_BM - 1LL) / GEMM_BM + sm_count - 1) / sm_count;
  const long long rounds = (M + (long long)sm_count * PT_MAX_TN - 1) / ((long long)sm_count * PT_MAX_TN);
  const long long tn = ((M + sm_count * rounds - 1) / (sm_count * rounds) + 15) / 16 * 16;
  if (n_out > 2 * PT_COLS || rt < 2 || (M + tn - 1) / tn > 65535) return 0;
  return n_out <= 64 && tn * rounds * 5 > rt * GEMM_BM * 4 ? 0 : (int)tn;
}

}  // namespace precc
