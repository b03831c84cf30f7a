"""The host rules of csrc/mg_rules.h, compiled for the host: which kernel variant
a call gets, from sizes and counts alone."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def rule(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")

    def call(*exprs):
        src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
        body = "".join(f'  printf("%g\\n", (double)({e}));\n' for e in exprs)
        src.write_text('#include <cstdio>\n#include "mg_rules.h"\nusing namespace mgk;\nint main() {\n' + body + "}\n")
        subprocess.run([gxx, "-std=c++17", f"-I{ROOT}/paper_1909_06412_gb300/csrc", "-o", str(exe), str(src)], check=True)
        return [float(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]

    return call


def test_batches_fall_back_to_one_cta_per_sm(rule):
    # two CTAs per SM from four problems per team on, where they are to be had
    assert rule("batch_ctas(304, 76, 152)", "batch_ctas(305, 76, 152)", "batch_ctas(1, 76, 152)") == [1, 2, 1]
    # a kernel that cannot run, or runs no more teams, leaves the other one
    assert rule("batch_ctas(512, 76, 0)", "batch_ctas(512, 76, 76)", "batch_ctas(512, 76, -1)") == [1, 1, 1]


def test_chunk_costs_follow_the_number_of_sms(rule):
    # 200 chunks are one wave for the 304 teams of 152 SMs, two for those of 76
    one, two, more = rule("short_pass_cost(200, 3, 144, 384, 152)", "short_pass_cost(200, 3, 144, 384, 76)",
                          "short_pass_cost(400, 3, 144, 384, 152)")
    assert one < two == more


def test_grids_of_many_short_axes_keep_the_fp64_units(rule):
    grids = {(54, 54, 54): 1, (32, 32, 32): 0, (162, 972): 1, (256, 256): 0, (24,) * 4: 1, (18, 18, 24, 24): 0,
             (12, 12, 12, 12, 18): 1, (8, 12, 8, 18, 12): 0, (12, 12, 12, 12, 12, 18): 1, (6, 8, 6, 8, 6, 12): 0,
             (6, 8, 8, 12, 8, 12): 0, (8,) * 6 + (6,): 0, (4,) * 7 + (12,): 0, (6, 6, 6, 6, 8, 8, 8, 8): 0}
    size = {N: "*".join(f"{n}ll" for n in N) for N in grids}
    assert rule(*(f"integer_passes({len(N)}, {size[N]}, 152)" for N in grids)) == list(grids.values())
