"""The memory rule of the resident class with its adjacency in global memory
(csrc/budget.h), which marks every node of the graph for every CTA: one CTA per
SM or none. Host code, compiled here."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "budget.h"
int main(int, char **v) {
    printf("%d %.0f\n", sc::global_class_ctas(strtoull(v[1], 0, 10), strtoull(v[2], 0, 10), atoi(v[3]),
                                            strtoull(v[4], 0, 10), strtoull(v[5], 0, 10)),
           sc::traversal_budget(strtoull(v[5], 0, 10)));
}
"""
GB = 1 << 30


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("budget")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2305_16086_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", str(d / "main")], check=True)
    return str(d / "main")


@pytest.mark.parametrize("nodes,sources,held,free,ctas", [
    (160_000, 160_000, 0, 270 * GB, 152),
    (10_000_000, 10_000_000, 0, 270 * GB, 152),        # 3.0 GB
    (100_000_000, 100_000_000, 0, 270 * GB, 0),        # 30 GB: past 4 GB
    (100_000_000, 10, 0, 270 * GB, 10),                # a query: ten CTAs
    (10_000_000, 10_000_000, 0, 8 * GB, 0),            # past an eighth of what is free
    (10_000_000, 10_000_000, 3_100_000_000, GB, 152),  # held already
    (3_000_000, 1, 0, GB, 1),
])
def test_one_cta_per_sm_or_none(program, nodes, sources, held, free, ctas):
    out = subprocess.run([program, str(2 * nodes), str(sources), "152", str(held), str(free)],
                         capture_output=True, text=True, check=True).stdout.split()
    assert int(out[0]) == ctas
    assert float(out[1]) == min(4 * GB, free / 8)
