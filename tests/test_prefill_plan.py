"""The rule that puts helper blocks on idle SMs, compiled from the header that the library compiles (no GPU)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2609_34054_b200", "csrc")
SMS, MIN_STEPS = 148, 48


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    """(head_dim, rank_k, rank_v, row tiles x kv heads, tokens of the context) -> (p, helpers, tiles); eight kv heads of four query heads."""
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text('#include <cstdio>\n#include "prefill_plan.h"\nint main() { int a[5]; while (scanf("%d %d %d %d %d", a, a + 1, a + 2, a + 3, a + 4) == 5) { '
                                f'precc::WorkList w = precc::plan_worklist(a[0], a[1], a[2], a[3] / 8 * 32 - 5, a[4], 32, 8, {SMS}, {MIN_STEPS}, 0); '
                                'printf("%d %d %d\\n", w.p, w.helpers, w.tiles); } }\n')
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(d / "plan.cpp"), "-o", str(d / "plan")], check=True)

    def call(rows):
        out = subprocess.run([str(d / "plan")], input="\n".join(" ".join(map(str, r)) for r in rows), capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return call


# turns measured without and with helper blocks: what the latter took of the former
MEASURED = [((128, 0, 16, 104, 24000), 1.06), ((128, 0, 16, 112, 40000), 1.04), ((128, 0, 64, 96, 14000), 1.06), ((128, 0, 64, 112, 28000), 1.06),
            ((128, 0, 64, 120, 48000), 1.05), ((128, 8, 8, 104, 24000), 1.05), ((128, 8, 8, 88, 14000), 1.06),
            ((128, 32, 32, 80, 24000), 0.85), ((128, 32, 32, 96, 33000), 0.95), ((128, 16, 16, 88, 33000), 0.85), ((128, 8, 8, 96, 24000), 0.94),
            ((128, 0, 16, 80, 33000), 0.85), ((128, 0, 64, 80, 33000), 0.92), ((128, 64, 64, 104, 33000), 0.92), ((64, 32, 32, 96, 33000), 0.85), ((64, 16, 16, 80, 24000), 0.82)]


def test_helper_blocks_are_taken_where_they_are_faster(plans):
    for (turn, share), (p, helpers, tiles) in zip(MEASURED, plans([t for t, _ in MEASURED])):
        assert (p > 0) == (share < 1), turn


def test_helper_block_plans_stay_inside_what_the_kernel_holds(plans):
    rows = [(hd, rk, rv, tiles, T) for hd in (64, 128) for rk, rv in ((0, 0), (0, 8), (0, 64), (8, 8), (32, 32), (64, 64)) for tiles in range(64, 152, 8)
            for T in (1000, 6000, 14000, 33000, 120000)]
    taken = 0
    for (hd, rk, rv, tiles, T), (p, helpers, n) in zip(rows, plans(rows)):
        if p:
            taken += 1
            longest = -(-(T + tiles // 8 * 32 - 5) // 128)
            assert helpers == SMS - tiles > 0 and n == tiles and longest // 2 <= p < longest and longest >= MIN_STEPS
    assert taken > 100


def _exhaustive(hd, rk, rv, tiles, T, tok=32, n_kv=8):
    """The definition: of the p that beat the plain launch by 4 % on paper, the largest among those with the smallest cost."""
    X, H, S = tiles // n_kv, SMS - tiles, tiles // n_kv * tok - 5
    if X >= 160 or tiles * 2 <= SMS or tiles > H * 14:
        return 0
    steps = [(T + min(S, (x + 1) * tok) + 127) // 128 for x in range(X)]
    if steps[-1] < MIN_STEPS:
        return 0
    f = 100 * 160 // (hd + (rk + rv) // 2)
    own, piece = 14 * f // 100, (12 if hd == 64 else 18 if rk + rv > 32 else 13) * f // 100
    slow = (138 if rv == 64 else 114 if rv == 0 else 106) if hd == 64 else 144 if rv == 0 else 121 if rk == 0 else 106 if rv == 64 else 115 if rk == 8 else 112
    best, best_cost = 0, (steps[-1] - steps[-1] // 25) * 100 // slow
    for p in range(steps[-1] - 1, max(8, steps[-1] // 2) - 1, -1):
        tails = [max(0, s - p) for s in steps] * n_kv
        per, pos, pieces, sources = max(1, -(-sum(tails) // H)), 0, [0] * H, 0
        for t in tails:
            if t:
                first, last = pos // per, (pos + t - 1) // per
                sources = max(sources, 2 + last - first)
                for h in range(first, last + 1):
                    pieces[h] += 1
                pos += t
        cost = max(p + own, per + piece * max(pieces))
        if max(pieces) <= 16 and sources <= 8 and cost < best_cost:
            best, best_cost = p, cost
    return best


def test_the_search_for_a_plan_misses_none(plans):
    rows = [(hd, rk, rv, tiles, T) for hd, rk, rv in ((64, 32, 32), (64, 0, 64), (128, 8, 8), (128, 64, 64), (128, 0, 16)) for tiles in range(72, 144, 8)
            for T in (6100, 9000, 15000, 24000, 33000, 47000)]
    got = [p for p, _, _ in plans(rows)]
    assert got == [_exhaustive(*r) for r in rows] and sum(p > 0 for p in got) > 60
