"""The launch rules of the particle push (csrc/push_shape.h), on the CPU."""
import subprocess

import pytest

from conftest import ROOT

SRC = """
#include "%s/paper_2510_11174_gb300/csrc/push_shape.h"
#include <cstdio>
int main() {
    int T, order, sms;
    long long tiles;
    while (scanf("%%d %%d %%lld %%d", &T, &order, &tiles, &sms) == 4)
        printf("%%d %%d %%lld\\n", hyb::push_split(T, order, tiles, sms), hyb::push_ctas(T, order),
               hyb::push_warps(T, order, tiles, sms));
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    d = tmp_path_factory.mktemp("push_shape")
    (d / "m.cpp").write_text(SRC % ROOT)
    subprocess.run(["g++", "-std=c++17", "-o", str(d / "m"), str(d / "m.cpp")], check=True)

    def run(rows):
        out = subprocess.run([str(d / "m")], input="\n".join("%d %d %d %d" % r for r in rows), check=True,
                             capture_output=True, text=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return run


@pytest.fixture(scope="module")
def rule(table):
    return lambda rows: [r[:2] for r in table(rows)]


@pytest.fixture(scope="module")
def rule_warps(table):
    return lambda rows: [r[2] for r in table(rows)]


@pytest.mark.parametrize("T", [4, 8])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("sms", [1, 148, 152])
def test_tiles_are_split_while_all_ctas_are_resident(rule, T, order, sms):
    tiles = list(range(0, 1200)) + [4096, 1 << 20, 1 << 33]
    for n, (split, ctas) in zip(tiles, rule([(T, order, n, sms) for n in tiles])):
        room = sms * ctas
        assert 1 <= split <= 4
        assert split == 1 or split * n <= room, (n, split)
        assert n == 0 or split == 4 or (split + 1) * n > room, (n, split)


def test_quadratic_8_tiles_count_two_ctas_an_sm(rule):
    """153 to 228 tiles of the quadratic shape fill the 304 resident CTAs: they are not split."""
    assert [s for s, _ in rule([(8, 2, n, 152) for n in (76, 77, 152, 153, 228)])] == [4, 3, 2, 1, 1]


def test_batches_count_the_tiles_of_all_their_contexts(rule):
    """1, 2, 4 and 8 contexts of 64 tiles side by side: 4, 3, 1 and 1 CTAs a tile."""
    assert [s for s, _ in rule([(8, 1, 64 * n, 152) for n in (1, 2, 4, 8)])] == [4, 3, 1, 1]


def test_warps_of_a_launch(rule_warps):
    """Each warp may leave one chunk of the migration buffer unfinished: the buffer's
    margin counts the launch's own warps, 4 a CTA on 4^3 tiles and 8 on 8^3 tiles."""
    rows = [(8, 1, 64, 152), (8, 1, 456, 152), (8, 1, 16384, 152), (4, 1, 64, 152), (4, 1, 4096, 152), (4, 2, 343, 152)]
    assert rule_warps(rows) == [64 * 4 * 8, 456 * 8, 16384 * 8, 64 * 4 * 4, 4096 * 4, 343 * 2 * 4]
