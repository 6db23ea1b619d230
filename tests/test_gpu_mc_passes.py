"""What the surrogate's MC passes hold on the device."""
import pytest

from _util import require_gpu

pytestmark = pytest.mark.gpu


def _surrogate(seed, mean, std, passes):
    from paper_2510_11174_gb300 import inputs
    from paper_2510_11174_gb300.model import Surrogate
    w = inputs.surrogate_weights(seed)
    m = Surrogate(dropout=0.1, mc_passes=passes, seed=seed, mean=mean, std=std)
    for l, (a, b) in enumerate(w):
        m.set_layer(l, a, b)
    return m


def test_mc_holds_only_what_a_forward_needs():
    """65 536 cells, four passes side by side: 1.2 KB a cell and pass, 64 B a cell for the
    inputs they share; the buffers of a training step (2 KB a cell) are not taken."""
    require_gpu()
    import torch
    from paper_2510_11174_gb300 import inputs
    x, mean, std = inputs.random_states(16, 16, seed=4)
    x = torch.from_numpy(x).cuda()
    m = _surrogate(3, mean, std, 16)
    m.mc(x[:1])
    keep = m.mc(x)[0]                      # torch's own blocks and the kernels are there
    m.close()
    m = _surrogate(3, mean, std, 16)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    pm, _ = m.mc(x)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    # ten buffers in blocks of 2 MB, and torch's two outputs
    assert taken <= 65536 * (4 * 1216 + 64) + 40e6, taken
    assert torch.equal(pm, keep)
    m.close()
