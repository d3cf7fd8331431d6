// Which projection kernel takes a call and how its work is cut: arithmetic on sizes alone, free of CUDA, so that the rules can be
// compiled and checked without a GPU.
#pragma once
#include <algorithm>

namespace precc {

constexpr int GEMM_BM = 128;                             // rows of a tile of the tiled kernel
constexpr int GEMM_BK = 64;                              // 64 bf16 = one 128-byte swizzle row
constexpr int PT_COLS = 128;                             // output columns of a tile of the turn kernel (the M of its MMA)
constexpr int PT_MAX_TN = 256;                           // rows of X in such a tile at most

// The turn kernel over the whole K extent (up to 256 columns of many rows): rows of a tile, or 0 where the tiled kernel is as good.
// The tiled kernel takes rt 128-row tiles a block; this form takes `rounds` tiles of up to 256 rows, cut so that every SM has the same
// number, and so loads and multiplies fewer rows per SM.  What a row saved is worth grows with K (one row less in one 64-deep
// k-block: 2.4 ns; with two 128-column halves also the second read of the rows that the tiled kernel spends on them, less
// the columns of the second half that the call does not have), what the form costs does not: its dump and stores run behind the
// last k-block of every tile, where the tiled kernel's run under the next tile.  Fitted to 655 sizes (d_model 512 .. 6144, 16 .. 256
// columns, 4000 .. 262144 rows); of those it takes none is more than 1 % slower than on the tiled kernel, and 19000 .. 25000 rows are 0.6 .. 0.98
// of it (4096, 128 columns, 25000 rows: 54.3 -> 42.1 us; 256 columns, 32768 rows: 71.0 -> 63.9).  Taken without a look at K and at the
// rounds it lost: d_model 1024, 32768 rows of 192 columns 21.9 -> 25.7 us, 150000 rows 71 -> 104; 2048, 75000 rows of 192 columns 66 -> 79.
// Up to four rounds (what was measured to win; the row tiles also lie on a grid axis of 65535).  Very few columns cost the
// tiled kernel little beside the rows, so there it has to save a fifth of them (32768 x 32: 49.1 against 50.8 us for an eighth).
inline int pick_wide_rows(int M, int K, int n_out, int sm_count) {
  const long long rt = ((M + GEMM_BM - 1LL) / GEMM_BM + sm_count - 1) / sm_count;
  const long long rounds = (M + (long long)sm_count * PT_MAX_TN - 1) / ((long long)sm_count * PT_MAX_TN);
  if (n_out > 2 * PT_COLS || rt < 2 || rounds > 4) return 0;
  const long long tn = ((M + sm_count * rounds - 1) / (sm_count * rounds) + 15) / 16 * 16;
  if (n_out <= 64 && tn * rounds * 5 > rt * GEMM_BM * 4) return 0;
  const long long second = n_out > PT_COLS ? std::max(-16, (n_out - 213) * 3 / 4) : 0;      // what the second half is worth, in rows
  const long long saved = rt * GEMM_BM - rounds * tn + rounds * second;
  const long long price = (n_out > 192 ? 1664 : 1280) + 2432 * (rounds - 1) + 16 * std::max(0, 32 - n_out);
  return K / GEMM_BK * saved >= price ? (int)tn : 0;
}

}  // namespace precc
