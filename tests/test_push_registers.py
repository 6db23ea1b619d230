"""The particle push keeps its prefetched particle in registers: a spilled value
waits for the load that fetches it, so the compiler's report must show no spill
in the instances without stochastic events that push whole tiles (the plasma of
a large grid), linear shape, at either tile size."""
import re
import subprocess

import pytest

from paper_2510_11174_gb300 import build


@pytest.mark.slow
def test_linear_push_has_no_spills(tmp_path):
    cmd = [build._nvcc()] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-cubin", build.CSRC + "/pic.cu", "-o",
                                                        str(tmp_path / "pic.cubin")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    spills = {}
    name = None
    for line in r.stderr.splitlines():
        m = re.search(r"k_push_depositILi(\d)ELi(\d)ELb(\d)ELb(\d)E", line)
        if m and "Function properties" in line:
            name = tuple(int(v) for v in m.groups())
        m = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)
        if m and name:
            spills[name] = (int(m.group(1)), int(m.group(2)))
            name = None
    assert len(spills) == 16, spills                     # tile x shape x events x clusters
    for T in (4, 8):
        assert spills[(T, 1, 0, 0)] == (0, 0), spills
