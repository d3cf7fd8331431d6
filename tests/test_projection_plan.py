"""The rules that cut projections, compiled from the header that the library compiles (no GPU)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2609_34054_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    """Calls a function of proj_plan.h on rows of integers."""
    d = tmp_path_factory.mktemp("plan")

    def call(expr, rows):
        src, exe = d / "plan.cpp", d / f"plan_{abs(hash(expr))}"
        if not exe.exists():
            src.write_text('#include <cstdio>\n#include "proj_plan.h"\nusing namespace precc;\n'
                           f'int main() {{ int a[4]; while (scanf("%d %d %d %d", a, a + 1, a + 2, a + 3) == 4) {{ {expr} }} }}\n')
            subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
        text = "\n".join(" ".join(map(str, (list(r) + [0] * 4)[:4])) for r in rows)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        return [[int(v) for v in line.split()] for line in out.splitlines()]
    return call


def test_tall_tiles_for_many_rows_stay_inside_the_grid_and_cover_the_rows(plan):
    rows = [(M, K, n) for M in (128 * SMS + 1, 19999, 25000, 32768, 40001, 62000, 99999, 151552, 151553, 16776960, 16776961, 2 ** 31 - 1)
            for K in (64, 1024, 2048, 4096, 16384) for n in (16, 40, 80, 128, 136, 192, 256)]
    taken = 0
    for (M, K, n), (tn,) in zip(rows, plan(f'printf("%d\\n", pick_wide_rows(a[0], a[1], a[2], {SMS}));', rows)):
        if tn:
            taken += 1
            assert tn % 16 == 0 and 16 <= tn <= 256 and (M + tn - 1) // tn <= 4 * SMS, (M, K, n, tn)
    assert taken > 50


def test_sizes_compared_with_the_tiled_kernel_take_tall_tiles(plan):
    """The rows, d_model and columns of the bitwise comparison on the GPU."""
    rows = [(18945, 2048, 192), (19999, 2048, 256), (20000, 2048, 128), (21001, 2048, 32), (40001, 3072, 128)]
    assert all(tn > 0 for tn, in plan(f'printf("%d\\n", pick_wide_rows(a[0], a[1], a[2], {SMS}));', rows))


# measured on the tiled kernel and on tall tiles (us, or shares of the former): (rows, d_model, columns, tiled, tall)
MANY_ROWS = [(19000, 1024, 192, 20.8, 18.7), (25000, 1024, 128, 19.1, 17.0), (32768, 1024, 96, 18.5, 19.4), (32768, 1024, 192, 21.9, 25.7),
             (37888, 1024, 256, 25.3, 28.3), (40000, 1024, 16, 21.4, 27.0), (75000, 1024, 192, 38.4, 54.5), (150000, 1024, 192, 71.3, 103.6),
             (20000, 2048, 32, 26.8, 20.4), (32768, 2048, 192, 34.0, 37.9), (50000, 2048, 192, 48.1, 58.2), (75000, 2048, 128, 58.0, 66.1),
             (25000, 4096, 128, 54.3, 42.1), (32768, 4096, 256, 71.0, 63.9), (40000, 4096, 64, 72.8, 67.0), (62000, 4096, 256, 138.5, 123.3),
             (75000, 4096, 192, 126.8, 138.2), (50000, 4096, 96, 76.4, 81.0)]
MANY_ROWS += [(28000, 1536, 208, 1.0, 1.06), (66000, 3584, 80, 1.0, 1.04), (33000, 3584, 208, 1.0, 1.04), (18945, 6144, 80, 1.0, 0.59), (18945, 1536, 144, 1.0, 0.89)]


def test_tall_tiles_are_taken_where_they_are_faster(plan):
    got = plan(f'printf("%d\\n", pick_wide_rows(a[0], a[1], a[2], {SMS}));', [r[:3] for r in MANY_ROWS])
    for (M, K, n, tiled, tall), (tn,) in zip(MANY_ROWS, got):
        assert (tn > 0) == (tall < tiled), (M, K, n)


# blocks of a cluster -> clusters that are resident at once, as a B200 reports them
CLUSTERS = {2: 74, 3: 45, 4: 33, 5: 26, 6: 22, 7: 15, 8: 15}
SMEM = 232448
PLAN = ("static const int fit[9] = {1, 0, %s}; " % ", ".join(str(CLUSTERS[k]) for k in range(2, 9)) +
        f"TurnPlan p = plan_turn(a[0], a[1], a[2], a[3], 2, 8, {SMS}, {SMEM}, fit); "
        'printf("%d %d %d %d\\n", p.tn, p.ks, p.stages, p.ks ? pt_smem_bytes(p.tn, p.ks, p.stages, 1) : 0);')


def test_calls_of_a_layer_are_cut_alike_in_k_and_fill_the_chip_in_rows(plan):
    """LR-only and base-only calls keep the K split of the fused call (the order of their sums) and take tiles that are no higher."""
    layers = [(16, 560, 48, 512), (16, 2560, 2048, 512), (32, 1056, 32, 1024), (32, 1152, 128, 1024), (56, 1280, 256, 1024), (64, 2304, 256, 2048),
              (64, 4096, 2048, 2048), (17, 608, 96, 512)]
    Ms = [41, 48, 64, 65, 128, 200, 301, 512, 513, 640, 768, 1000, 1280, 1791, 2048]
    rows = [(M, nkb, fused, n) for nkb, fused, lr, base in layers for M in Ms for n in (fused, lr, base)]
    got = dict(zip(rows, plan(PLAN, rows)))
    lower = 0
    for (M, nkb, fused, n), (tn, ks, stages, smem) in got.items():
        whole = got[M, nkb, fused, fused]
        assert ks == whole[1] and (ks == 0 or tn <= whole[0]), (M, nkb, fused, n)
        if ks:
            assert tn % 16 == 0 and 32 <= tn <= 256 and stages >= 1 and smem <= SMEM
            assert -(-n // 128) * -(-M // tn) <= CLUSTERS[ks], (M, nkb, fused, n)
            lower += tn < whole[0]
    assert lower > 60
    # 768 rows onto 32 of 1056 columns: with the fused call's 256-row tiles, three clusters
    assert got[768, 32, 1056, 32][0] <= 48 and got[1791, 16, 560, 48][0] <= 64


def test_forced_splits_of_the_gpu_tests_are_taken(plan):
    """(blocks per cluster, rows, k-blocks, fused width) of the tests that force a split."""
    at_every_split = [(2, 100, 16), (2, 777, 32), (3, 384, 64), (3, 130, 16), (4, 512, 32), (4, 64, 64), (4, 1000, 16), (5, 200, 32), (6, 256, 64), (7, 41, 32),
                      (8, 128, 16), (8, 77, 64)]
    rotary = [(8, 128, 4, 130), (8, 64, 3, 70), (7, 128, 2, 200), (6, 64, 4, 129), (5, 128, 3, 257), (8, 128, 2, 41), (7, 64, 1, 64), (6, 128, 1, 150),
              (4, 128, 4, 300), (3, 64, 4, 200), (3, 128, 1, 128), (2, 128, 2, 513)]
    rows = [(M, nkb, 608, ks) for ks, M, nkb in at_every_split] + [(M, 17, 2 * n_kv * hd + 96, ks) for ks, hd, n_kv, M in rotary]
    forced = PLAN.replace("a[2], a[3], 2, 8,", "a[2], a[2], a[3], a[3],")
    for row, (tn, ks, _, _) in zip(rows, plan(forced, rows)):
        assert ks == row[3], row
    shares = [((min(M, tn) + ks - 1) // ks + 7) // 8 * 8 for (M, _, _, ks), (tn, _, _, _) in zip(rows, plan(forced, rows))]
    assert any(s * (ks - 1) >= min(M, 256) for s, (M, _, _, ks) in zip(shares, rows))     # blocks that finish no rows


# measured at 64 rows on the few-row and the turn kernel (us): (d_model, fused width, few-row, turn)
SIXTY_FOUR_ROWS = [(1024, 560, 3.8, 5.8), (1024, 1024, 3.9, 5.8), (2048, 1056, 5.2, 7.4), (2048, 1152, 5.3, 7.4), (3584, 1280, 6.6, 8.7),
                   (4096, 2304, 10.7, 9.9), (4096, 4096, 15.1, 11.6)]


def test_sixty_four_rows_run_on_the_faster_kernel(plan):
    got = plan('printf("%d\\n", few_row_limit(a[0], a[1]));', [r[:2] for r in SIXTY_FOUR_ROWS])
    assert [limit for limit, in got] == [64 if few < turn else 40 for _, _, few, turn in SIXTY_FOUR_ROWS]
    assert plan('printf("%d\\n", few_row_limit(a[0], a[1]));', [(1088, 608)]) == [[40]]      # 17 k-blocks: no split, a single pass of them all
