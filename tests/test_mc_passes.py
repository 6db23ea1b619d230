"""How many MC passes run side by side (csrc/mc_passes.h), on the CPU: the rule is
compiled into a small program whose reserve() refuses what exceeds a given memory."""
import subprocess

import pytest

from conftest import ROOT

SRC = """
#include "%s/paper_2510_11174_gb300/csrc/mc_passes.h"
#include <cstdio>
#include <cstdlib>
int main(int, char **v) {
    const int passes = atoi(v[1]);
    const long long cells = atoll(v[2]), limit = atoll(v[3]), memory = atoll(v[4]);
    hyb_status s = HYB_OK;
    int asked = 0;
    const int n = hyb::passes_side_by_side(passes, cells, limit, [&](int g) {
        ++asked;
        return s = g * cells <= memory ? HYB_OK : HYB_ENOMEM;
    });
    printf("%%d %%d %%d", n, (int)s, asked);
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("mc_passes")
    (d / "m.cpp").write_text(SRC % ROOT)
    subprocess.run(["g++", "-std=c++17", "-o", str(d / "m"), str(d / "m.cpp")], check=True)
    return lambda *a: tuple(int(t) for t in subprocess.run([str(d / "m")] + [str(i) for i in a], check=True,
                                                           capture_output=True, text=True).stdout.split())


NO_LIMIT = 1 << 60


# passes, cells, largest volume, memory in cells -> passes side by side, status (0 HYB_OK, 2 HYB_ENOMEM)
@pytest.mark.parametrize("passes,cells,limit,memory,want", [
    (16, 65536, 262144, NO_LIMIT, (4, 0)),
    (16, 65537, 262144, NO_LIMIT, (3, 0)),
    (16, 1, 262144, NO_LIMIT, (16, 0)),
    (7, 3840, 262144, NO_LIMIT, (7, 0)),
    (16, 262144, 262144, NO_LIMIT, (1, 0)),
    (16, 262145, 262144, NO_LIMIT, (1, 0)),
    (1, 8, 262144, NO_LIMIT, (1, 0)),
    (16, 65536, 262144, 3 * 65536, (2, 0)),      # four passes do not fit, two do
    (16, 65536, 262144, 65536, (1, 0)),          # one pass fits: the call still runs
    (7, 3840, 262144, 3840, (1, 0)),
    (16, 65536, 262144, 65535, (1, 2)),          # not even one
])
def test_fewer_passes_where_memory_is_short(rule, passes, cells, limit, memory, want):
    n, status, asked = rule(passes, cells, limit, memory)
    assert (n, status) == want and asked <= 5
