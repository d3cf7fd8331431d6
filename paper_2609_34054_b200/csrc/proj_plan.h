// Which projection kernel takes a call and how its work is cut: arithmetic on sizes alone, free of CUDA, so that the rules can be
// compiled and checked without a GPU.
#pragma once
#include <algorithm>

#ifdef __CUDACC__
#define PRECC_HD __host__ __device__
#else
#define PRECC_HD
#endif

namespace precc {

constexpr int GEMM_BM = 128;                             // rows of a tile of the tiled kernel
constexpr int GEMM_BK = 64;                              // 64 bf16 = one 128-byte swizzle row
constexpr int PT_COLS = 128;                             // output columns of a tile of the turn kernel (the M of its MMA)
constexpr int PT_MAX_TN = 256;                           // rows of X in such a tile at most
constexpr int GEMM_MAX_KS = 8;                           // largest K split of a turn's projection (cluster size)
constexpr int PT_W_BYTES = PT_COLS * GEMM_BK * 2;
constexpr int PT_MAX_STAGES = 8;
constexpr int PT_MIN_SMEM = 120 * 1024;                  // keeps one block per SM, so that the cluster occupancy depends on KS alone
struct PtRow { long long slot, slot2; unsigned long long mask; int pos, ok; };   // what the routing needs to know about a row

PRECC_HD constexpr int pt_stage_bytes(int tn, int ng) { return ng * PT_W_BYTES + tn * GEMM_BK * 2; }
PRECC_HD constexpr int pt_share(int rows, int ks) { return ((rows + ks - 1) / ks + 7) / 8 * 8; }     // rows finished by one block
PRECC_HD constexpr int pt_merge_bytes(int tn, int ks) { return (tn + (ks - 1) * pt_share(tn, ks)) * PT_COLS * 4; }
PRECC_HD constexpr int pt_data_bytes(int tn, int ks, int stages, int ng) {
  const int ring = stages * pt_stage_bytes(tn, ng), merge = pt_merge_bytes(tn, ks);
  return ((ring > merge ? ring : merge) + 1023) / 1024 * 1024;
}
PRECC_HD constexpr int pt_smem_bytes(int tn, int ks, int stages, int ng) {
  return pt_data_bytes(tn, ks, stages, ng) + pt_share(tn, ks) * (int)sizeof(PtRow) + (2 * PT_MAX_STAGES + 4) * 8;
}

// Rows up to which the few-row kernel takes every call of a layer (so the same for its fused, base-only and LR-only calls).  40 of any
// layer (fused Llama-3-8B projection: 6.1 us at 16 rows, 7.8 at 32, 9.8 at 40, where the turn kernel takes 9.8 too), all 64 that it can
// hold where the weights are few and every column group still has its eight K slices: 64 rows onto 1280 columns of d_model 3584 6.6 us
// against 8.7 on the turn kernel, 1152 of 2048 5.3 against 7.4, 560 of 1024 3.8 against 5.8; LR rows alone (48 columns) 3.7 against
// 5.6; rotary keys 9.2 / 7.8 / 6.3 against 9.0 / 7.7 / 6.1.  Wider layers lose: 2304 columns of 4096 10.7 against 9.9, rotary 14.7 against 10.2;
// 2560 of 1024 rotary 10.7 against 7.0.
constexpr int PS_MAX_M = 64;
inline int few_row_limit(int K, int n_fused) { return n_fused <= 1280 && K <= 4096 && K % 512 == 0 ? PS_MAX_M : 40; }

// How a turn's projection is cut: tiles of 128 columns x tn rows, the K extent of each over ks blocks.
struct TurnPlan { int tn = 0, ks = 0, stages = 0; };

// The cut with the smallest predicted time among those whose clusters are all resident at once (a cluster lives inside one GPC;
// a second wave costs more than any split gains: 512 rows of the Llama-3-8B projection
// as 36 clusters of four, of which 33 fit, 26.9 us; as 36 clusters of three 17.2).  Time in us, fitted to some 450 cuts of
// four layers (d_model 1024 .. 4096) at 41 .. 2048 rows, mean error 4 %: what a k-block costs a block, what the merge moves into
// one, what dumping and storing a tile takes, and the cluster.  The cut it picks is within 1 % of the best one measured but for
// two in 36 (4 % and 11 %).
// The K split is the one for the width of the layer's FUSED projection, whatever this call projects, so that the base-only,
// LR-only and fused calls of one M add in the same order.  The height of the tiles changes no bit: a call of fewer columns takes lower
// tiles on the SMs that this leaves (LR rows of two agents of rank 8, d_model 2048, 768 rows: 9.9 us in tiles of the fused
// call's height, 8.2 in tiles of 32 rows; of three, d_model 1024, 1800 rows 8.8 -> 7.0; base rows of d_model 3584, 512 rows 12.6 -> 11.6).
// clusters[ks]: how many clusters of ks blocks are resident at once.
inline TurnPlan plan_turn(int M, int nkb, int n_fused, int n_out, int ks_min, int ks_max, int sm_count, int max_smem, const int* clusters) {
  TurnPlan best;
  double best_cost = 1e30;
  auto ring = [&](int tn, int ks) {                    // stages that fit
    int st = std::min((nkb + ks - 1) / ks, PT_MAX_STAGES);
    while (st > 0 && pt_smem_bytes(tn, ks, st, 1) > max_smem) --st;
    return st;
  };
  const int groups = (n_fused + PT_COLS - 1) / PT_COLS;
  for (int t = (M + PT_MAX_TN - 1) / PT_MAX_TN, last = 0;; ++t) {
    const int tn = ((M + t - 1) / t + 15) / 16 * 16, tiles = (M + tn - 1) / tn;
    if (tn < 32 || (long long)groups * tiles * ks_min > sm_count) break;
    if (tn == last) continue;
    last = tn;
    for (int ks = ks_min; ks <= ks_max && nkb / ks >= 2; ++ks) {       // at least two k-blocks per slice
      if (groups * tiles > clusters[ks]) continue;
      const int kb = (nkb + ks - 1) / ks, st = ring(tn, ks);
      if (st == 0) continue;
      const double cost = kb * (0.37 + 0.00036 * tn) + 0.005 * pt_share(tn, ks) * (ks - 1) + 0.0113 * tn + 0.1 * ks;
      if (cost < best_cost) { best_cost = cost; best.tn = tn; best.ks = ks; best.stages = st; }
    }
  }
  if (best.ks > 0 && n_out < n_fused) {                // at a given ks the lowest tiles that are all resident
    const int tiles = clusters[best.ks] / ((n_out + PT_COLS - 1) / PT_COLS);
    best.tn = std::max(32, ((M + tiles - 1) / tiles + 15) / 16 * 16);
    best.stages = ring(best.tn, best.ks);
  }
  return best;
}

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
