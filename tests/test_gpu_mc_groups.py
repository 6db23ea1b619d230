"""The surrogate's MC passes in several groups side by side: a second group, a last
group with fewer passes, and batches too large for more than one pass a group."""
import pytest

from _util import rel_l2, require_gpu

pytestmark = pytest.mark.gpu


def _surrogate(seed, mean, std, passes):
    from oracle import surrogate as S
    from paper_2510_11174_gb300 import inputs
    from paper_2510_11174_gb300.model import Surrogate
    w = inputs.surrogate_weights(seed)
    m = Surrogate(dropout=0.1, mc_passes=passes, seed=seed, mean=mean, std=std)
    for l, (a, b) in enumerate(w):
        m.set_layer(l, a, b)
    return m, S.OracleSurrogate(w, dropout=0.1, seed=seed, mean=mean, std=std)


# 65 536 cells: groups of 4 and 3 passes; 135 168 cells: three groups of one
@pytest.mark.parametrize("batch,passes", [(16, 7), (33, 3)])
def test_several_groups_match_oracle(batch, passes):
    require_gpu()
    import torch
    from paper_2510_11174_gb300 import inputs
    x, mean, std = inputs.random_states(batch, 16, seed=4)
    m, orc = _surrogate(3, mean, std, passes)
    pm, ps = m.mc(torch.from_numpy(x).cuda())
    om, os_ = orc.mc_statistics(x, passes)
    # the bounds of the single group: BF16 rounding flips between FP32 and FP64 sums
    assert rel_l2(pm.cpu().numpy() - x, om.numpy() - x) <= 2e-3
    assert rel_l2(ps.cpu().numpy(), os_.numpy()) <= 2e-2
    # sample 0 takes the same masks in a batch of its own, where all passes form one group
    m1, _ = _surrogate(3, mean, std, passes)
    p1, s1 = m1.mc(torch.from_numpy(x[:1]).cuda())
    assert torch.equal(p1[0], pm[0]) and torch.equal(s1[0], ps[0])
    m.close()
    m1.close()
