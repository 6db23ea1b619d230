"""Weight gradients at the edges of volumes and batches, with the loss concentrated
in one cell at the edge: the gradient is then almost that cell's alone, so a row,
tile or plane that a kernel loses there shows at the size of the gradient, not as
one part in thousands.  On the CPU the oracle loses the cell's block on purpose
and must miss the bound by far; on the GPU every layer must keep it.

The bound: a product of the contraction has two BF16 operands, each at most one
rounding flip (2^-8) off where FP32 and FP64 sums round apart: 8e-3, and 2e-2
with the flips of the layers between."""
import numpy as np
import pytest
import torch

from _util import rel_l2, require_gpu, seeded_classifier

BOUND = 2e-2


def _cells(shape):
    """The volume's first and last cell, and the last cell of its first block of 8 rows x 16 cells."""
    B, D, H, W = shape
    return [(0, 0, 0, 0), (B - 1, D - 1, H - 1, W - 1), (B - 1, D // 2, 7, min(15, W - 1))]


CNN = [(s, c) for s in [(1, 1, 16, 8), (3, 5, 32, 24)] for c in _cells(s)]
SUR = [(s, c) for s in [(1, 1, 16, 8), (3, 5, 16, 24)] for c in _cells(s)]
SN = [(n, c) for n in (1, 127, 129, 20011) for c in sorted({0, (n - 1) // 64 * 64, n - 1})]


def _cnn(shape, cell):
    from oracle.classifier import OracleCNN
    from paper_2510_11174_gb300 import inputs
    B, D, H, W = shape
    net = OracleCNN(inputs.classifier_weights(21), dropout=0.2, seed=21)
    rng = np.random.default_rng(5)
    x = rng.standard_normal((B, 6, D, H, W)).astype(np.float32)
    b, z, y, i = cell
    x[b, :, z, y, i] *= 30.0                                  # 900 times the energy: the cell's weight in the loss
    t = (x[:, 0] > 0).astype(np.float32)
    t[b, z, y, i] = 0.0 if float(net.forward(x, 0)[b, z, y, i]) > 0 else 1.0   # and wrong there
    return net, x, t


def _cnn_grads(net, x, t):
    import oracle.classifier as O
    return O.train_grads(net, x, t, pass_index=0, energy_weight=1e3)["grads"]


def _sur(shape, cell):
    from oracle import surrogate as S
    from paper_2510_11174_gb300 import inputs
    B, D, H, W = shape
    x, mean, std = inputs.random_states(B, 32, seed=6)
    x = np.ascontiguousarray(x[:, :, :D, :H, :W])
    sd = np.asarray(std, np.float32)
    t = x.copy()
    b, z, y, i = cell
    t[b, :, z, y, i] += 1e5 * sd                              # a residual that outweighs all others together
    net = S.OracleSurrogate(inputs.surrogate_weights(3), dropout=0.1, seed=3, mean=mean, std=std)
    return net, x, t, mean, std


def _sur_grads(net, x, t):
    from oracle import surrogate as S
    return S.loss_and_grads(net, x, t, 0, delta=1e6, energy_weight=0.0)["grads"]


def _sn(n, cell):
    from oracle import switchnet as S
    from paper_2510_11174_gb300 import inputs
    rng = np.random.default_rng(n)
    x = rng.standard_normal((10, n)).astype(np.float32)
    x[:, cell] *= 30.0
    net = S.OracleSwitchNet(inputs.switchnet_weights(5), dropout=0.2, seed=5)
    y = (np.abs(x[1]) > 1.0).astype(np.float32)
    y[cell] = 0.0 if float(net.forward(x, 0)[cell]) > 0 else 1.0
    return net, x, y


def _sn_grads(net, x, y):
    from oracle import switchnet as S
    return S.loss_and_grads(net, x, y, 0, energy_weight=1e3)["grads"]


def _lose_block(monkeypatch, module, cell):
    """The oracle's convolution gradients without the 8-row x 16-cell block of `cell` in its plane."""
    b, z, y, i = cell
    whole = module._wgrad

    def lost(a, dz):
        dz = dz.clone()
        dz[b, :, z, y // 8 * 8:y // 8 * 8 + 8, i // 16 * 16:i // 16 * 16 + 16] = 0.0
        return whole(a, dz)
    monkeypatch.setattr(module, "_wgrad", lost)


@pytest.mark.parametrize("shape,cell", CNN)
def test_bound_catches_a_lost_block_classifier(monkeypatch, shape, cell):
    import oracle.classifier as O
    case = _cnn(shape, cell)
    ref = _cnn_grads(*case)
    _lose_block(monkeypatch, O, cell)
    bad = _cnn_grads(*case)
    for l in range(4):
        assert rel_l2(bad[l][0].numpy(), ref[l][0].numpy()) >= 5 * BOUND, l


@pytest.mark.parametrize("shape,cell", SUR)
def test_bound_catches_a_lost_block_surrogate(monkeypatch, shape, cell):
    import oracle.surrogate as O
    case = _sur(shape, cell)[:3]
    ref = _sur_grads(*case)
    _lose_block(monkeypatch, O, cell)
    bad = _sur_grads(*case)
    for l in range(6):
        assert rel_l2(bad[l][0].numpy(), ref[l][0].numpy()) >= 5 * BOUND, l


@pytest.mark.parametrize("n,cell", SN)
def test_bound_catches_a_lost_cell_switchnet(n, cell):
    net, x, y = _sn(n, cell)
    ref = _sn_grads(net, x, y)
    lost = y.astype(np.float64)
    lost[cell] = 1.0 / (1.0 + np.exp(-float(net.forward(x, 0)[cell])))   # no error there: the sums without the cell
    bad = _sn_grads(net, x, lost)
    for l in range(5):
        assert rel_l2(bad[l][0].numpy(), ref[l][0].numpy()) >= 5 * BOUND, l


@pytest.mark.gpu
@pytest.mark.parametrize("shape,cell", CNN)
def test_classifier_gradient_at_an_edge(shape, cell):
    P = require_gpu()
    net, x, t = _cnn(shape, cell)
    m, _ = seeded_classifier(P, 21, dropout=0.2, mc_passes=1, energy_weight=1e3)
    m.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    ref = _cnn_grads(net, x, t)
    for l in range(4):
        gw, gb = m.get_grad(l)
        assert rel_l2(gw, ref[l][0].numpy()) <= BOUND and rel_l2(gb, ref[l][1].numpy()) <= BOUND, l
    m.close()


@pytest.mark.gpu
@pytest.mark.parametrize("shape,cell", SUR)
def test_surrogate_gradient_at_an_edge(shape, cell):
    require_gpu()
    from paper_2510_11174_gb300 import inputs
    from paper_2510_11174_gb300.model import Surrogate
    net, x, t, mean, std = _sur(shape, cell)
    m = Surrogate(dropout=0.1, mc_passes=1, seed=3, mean=mean, std=std, huber_delta=1e6, energy_weight=0.0)
    for l, (a, b) in enumerate(inputs.surrogate_weights(3)):
        m.set_layer(l, a, b)
    m.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    ref = _sur_grads(net, x, t)
    for l in range(6):
        gw, gb = m.get_grad(l)
        assert rel_l2(gw, ref[l][0].numpy()) <= BOUND and rel_l2(gb, ref[l][1].numpy()) <= BOUND, l
    m.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n,cell", SN)
def test_switchnet_gradient_at_an_edge(n, cell):
    require_gpu()
    from paper_2510_11174_gb300 import inputs
    from paper_2510_11174_gb300.model import SwitchNet
    net, x, y = _sn(n, cell)
    m = SwitchNet(dropout=0.2, mc_passes=1, seed=5, energy_weight=1e3)
    for l, (a, b) in enumerate(inputs.switchnet_weights(5)):
        m.set_layer(l, a, b)
    m.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    ref = _sn_grads(net, x, y)
    for l in range(5):
        gw, gb = m.get_grad(l)
        assert rel_l2(gw, ref[l][0].numpy()) <= BOUND and rel_l2(gb, ref[l][1].numpy()) <= BOUND, l
    m.close()
