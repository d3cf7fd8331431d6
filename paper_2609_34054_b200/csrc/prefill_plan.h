// How a turn's prefill with a workspace is shared out among the SMs: arithmetic on sizes alone, free of CUDA, so that the rule can be
// compiled and checked without a GPU.
#pragma once
#include <algorithm>

namespace precc {

constexpr int PTC_TOK = 128;      // tokens per step
constexpr int PTC_MAX_SRC = 8;    // work-list launch: pieces of one tile (its own block + helper pieces) at most
constexpr int PTC_MAX_SEG = 16;   // work-list launch: tile pieces one helper block takes at most
constexpr int PTC_MAX_XT = 160;   // work-list launch: row tiles at most

struct WorkList { int p = 0, helpers = 0, tiles = 0; };

// Steps of row tile x; the tail of a tile is what lies beyond the first `p` steps.  Tails are laid end to end, kv
// head by kv head, and cut into `helpers` equal ranges (the kernel derives the same cuts from p and helpers).
// The cost of a plan, in steps: the longer of a tile's own block (p + its record and possibly the merge) and a
// helper (its range + a drain and refill per piece).  Returns p = 0 when the classic launch is as good.
// `min_steps`: tiles shorter than that are left alone; `forced_p` > 0 takes that p (diagnostic).
inline WorkList plan_worklist(int HD, int RK, int RV, int S, int T, int tok_per_tile, int n_kv, int sm_count, int min_steps, int forced_p) {
  WorkList best;
  const int X = (S + tok_per_tile - 1) / tok_per_tile;
  const long long tiles = (long long)X * n_kv;
  const int H = sm_count - (int)tiles;
  if (X >= PTC_MAX_XT || tiles * 2 <= sm_count || tiles > (long long)H * (PTC_MAX_SEG - 2)) return best;
  auto steps_of = [&](int x) { return (int)(((long long)T + std::min(S, (x + 1) * tok_per_tile) + PTC_TOK - 1) / PTC_TOK); };
  const int n_max = steps_of(X - 1);
  if (n_max < min_steps) return best;
  // What a record + merge costs a tile's own block, and what a piece costs a helper beyond its steps (query tile,
  // fold, pipeline fill, record), in steps at head_dim 128, rank 32 (1.0 us), scaled for shorter ones; and how much longer
  // every step takes with all SMs busy instead of one per tile, beside a plain launch whose MMA sums the denominator.  At head_dim 128
  // the launch runs at the power cap; steps with few or no key coordinates or without the sum of rounded weights are short
  // (head_dim 64 rank 64: 0.78 us, head_dim 128 without adapter: 0.86 us for 64 KB of caches each), so that what L2 delivers to
  // all SMs together bounds them and more SMs only stretch them.  Fitted to turns of 80 .. 120 tiles over 14000 .. 48000 tokens, the work-list
  // launch against the plain one: of 420 none of a plan that is taken takes longer than 1.001 of it (with 112 for ranks 0 / 8 .. 32
  // and 8 / 8 and 106 for 0 / 64, fitted to an older plain launch, 14 took 1.02 .. 1.07), 0.934 on the mean of all.
  const int f100 = 100 * 160 / (HD + (RK + RV) / 2);
  const int C_OWN = 14 * f100 / 100, C_PIECE = (HD == 64 ? 12 : RK + RV > 32 ? 18 : 13) * f100 / 100;
  const int slow = HD == 64 ? (RV == 64 ? 138 : RV == 0 ? 114 : 106) : RV == 0 ? 144 : RK == 0 ? 121 : RV == 64 ? 106 : RK == 8 ? 115 : 112;
  const int must_beat = (n_max - n_max / 25) * 100 / slow;   // a plan must win 4 % on paper
  // Of the plans with the smallest cost, the one with the largest p.  From small p on: the helpers' ranges shrink and the blocks' own parts
  // grow, so the plans whose range alone costs too much are passed by without a look at their pieces and the search ends where the own part does
  // (384 tokens over 32768: 117 us of host time a call when every p had its pieces counted, now 10).
  int best_cost = must_beat - 1;
  int steps[PTC_MAX_XT];
  for (int x = 0; x < X; ++x) steps[x] = steps_of(x);
  for (int p = std::max(8, n_max / 2); p < n_max; ++p) {
    if (forced_p > 0 ? p != forced_p : p + C_OWN > best_cost) continue;
    long long tail_sum = 0;
    for (int x = 0; x < X; ++x) tail_sum += std::max(0, steps[x] - p);
    const long long per = std::max(1ll, (tail_sum * n_kv + H - 1) / H);      // steps of a helper's range
    if (forced_p <= 0 && per + C_PIECE > best_cost) continue;
    // walk the tails in the kernel's order: tiles that meet a helper's range, ranges that a tile meets
    int max_seg = 0, max_src = 0, seg = 0;
    long long used = 0;
    for (int g = 0; g < n_kv; ++g)
      for (int x = 0; x < X; ++x) {
        long long left = std::max(0, steps[x] - p);
        if (left == 0) continue;
        if (used == per) used = seg = 0;
        int ranges = 1;
        max_seg = std::max(max_seg, ++seg);
        for (; left > per - used; ++ranges) { left -= per - used; used = 0; seg = 1; }
        used += left;
        max_src = std::max(max_src, 1 + ranges);
      }
    if (max_seg > PTC_MAX_SEG || max_src > PTC_MAX_SRC) continue;
    const int cost = (int)std::max<long long>(p + C_OWN, per + (long long)C_PIECE * max_seg);
    if (cost <= best_cost || forced_p > 0) { best_cost = cost; best.p = p; best.helpers = H; best.tiles = (int)tiles; }
  }
  return best;
}

}  // namespace precc
