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
            assert tn % 16 == 0 and 16 <= tn <= 256 and (M + tn - 1) // tn <= 65535, (M, K, n, tn)
    assert taken > 50

