"""Shapes the field surrogate refuses, through the C ABI on the CPU: every entry
point answers HYB_EINVAL before it touches the handle's device state (which is
storage of zeros here), in a process of its own."""
import subprocess
import sys

import pytest

from conftest import ROOT

CODE = """
import ctypes as C
from paper_2510_11174_gb300 import _abi
lib = _abi.load()
handle, array = C.create_string_buffer(1 << 16), C.create_string_buffer(256)
p = C.addressof(array)
shape = {shape}
r = dict(forward=lambda: lib.hyb_surrogate_forward(C.addressof(handle), p, *shape, 0, p),
         mc=lambda: lib.hyb_surrogate_mc(C.addressof(handle), p, *shape, p, p),
         train=lambda: lib.hyb_surrogate_train_step(C.addressof(handle), p, p, *shape, C.byref(_abi.hyb_surrogate_stats())))
print("answer", r["{call}"]())
"""


@pytest.mark.parametrize("call", ["forward", "mc", "train"])
@pytest.mark.parametrize("shape", [(0, 16, 16, 16), (1, 0, 16, 16), (1, 16, 0, 16), (1, 16, 16, 0), (-1, 16, 16, 16),
                                   (1, 16, 12, 16)])
def test_refused_shapes(call, shape):
    from paper_2510_11174_gb300 import _abi, build
    build.build()
    r = subprocess.run([sys.executable, "-c", CODE.format(shape=shape, call=call)], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr)
    assert r.stdout.split() == ["answer", str(_abi.HYB_EINVAL)]
