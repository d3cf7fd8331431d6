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
                           f'int main() {{ int a[8]; while (scanf("%d %d %d %d", a, a + 1, a + 2, a + 3) == 4) {{ {expr} }} }}\n')
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
