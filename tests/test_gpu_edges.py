"""The kernels' edges against the oracle: tiles pushed by clusters of 4, 3, 2 and
1 CTAs with a few, a ragged number and thousands of particles; tiles that empty
and fill at once (migration chunks, holes, compaction), with and without a
caller's arena; convolutions whose columns, tiles and chunks end raggedly;
MC passes that do not fill a group; weight gradients over ragged cells."""
import numpy as np
import pytest

from _util import by_id, make_pair, rel_l2, require_gpu, seeded_classifier

pytestmark = pytest.mark.gpu


def _species(n, size, seed, q=-1.0, m=1.0, u=0.5, drift=0.0, box=None):
    """n particles, the first half in the first 8^3 cells (or all of them in `box` cells)."""
    rng = np.random.default_rng(seed)
    p = [rng.uniform(0, L, n) for L in size]
    for a in range(3):
        p[a][: n // 2 + 1] = rng.uniform(0, min(8, size[a]), n // 2 + 1)
        if box is not None:
            p[a] = rng.uniform(0, box, n)
        p[a] = np.minimum(p[a].astype(np.float32), np.nextafter(np.float32(size[a]), np.float32(0)))
    v = [rng.normal(0, u, n).astype(np.float32) for _ in range(3)]
    v[0] += np.float32(drift)
    return dict(q=q, m=m, x=p[0], y=p[1], z=p[2], ux=v[0], uy=v[1], uz=v[2], w=np.full(n, 1e-3, np.float32))


# 1, 64, 152, 171 and 464 tiles: clusters of 4, 4, 3 and 2 CTAs a tile, and tiles left whole
@pytest.mark.parametrize("size", [(8, 8, 8), (32, 32, 32), (152, 64, 8), (152, 72, 8), (128, 232, 8)])
@pytest.mark.parametrize("n", [1, 255, 4097])
def test_push_splits_match_oracle(size, n):
    nx, ny, nz = size
    rng = np.random.default_rng(n)
    inp = dict(grid=dict(nx=nx, ny=ny, nz=nz, dx=0.3), species=[_species(n, size, 1), _species(n // 2 + 1, size, 2, 1.0, 100.0)],
               E=rng.normal(0, 0.3, (3, nz, ny, nx)).astype(np.float32),
               B=rng.normal(0, 0.3, (3, nz, ny, nx)).astype(np.float32))
    sim, orc = make_pair(inp)
    sim.step(1)
    orc.step(1)
    for sid in range(2):
        g, o = by_id(sim.get_species(sid)), orc.species[sid]
        k = np.argsort(o.ids)
        assert np.array_equal(g["ids"], o.ids[k])
        for c in ("ux", "uy", "uz"):
            # |u| of order 1, some forty FP32 operations of 6e-8 each
            assert np.abs(g[c] - getattr(o, c)[k]).max() <= 1e-5
    J = sim.get_fields()[2]
    # a current is a displacement (0.25 cells RMS) between FP32 positions, off by at most
    # half an ulp of 256 = 7.6e-6 each: 4e-5 of it
    assert rel_l2(J, orc.J) <= 1e-4, rel_l2(J, orc.J)
    sim.close()


@pytest.mark.parametrize("arena", [False, True])
@pytest.mark.parametrize("n", [130, 3000])
def test_tiles_that_empty_and_fill(arena, n):
    """A beam that leaves its tile within a few steps beside a species at rest; u 4 -> 0.55 cells a step."""
    P = require_gpu()
    import torch
    import oracle.sim as S
    size = (32, 16, 16)
    sps = [_species(n, size, 3, u=0.3, drift=4.0, box=8), _species(777, size, 4, 1.0, 1836.0, u=0.0)]
    for sp in sps:
        sp["w"][:] = 1e-6
    kw = dict(arena=torch.empty(1 << 28, dtype=torch.uint8, device="cuda")) if arena else {}
    sim = P.Simulation(*size, 0.3, **kw)
    orc = S.OracleSim(*size, 0.3)
    for sp in sps:
        sim.load_species(**sp)
        orc.load_species(**sp)
    for _ in range(4):
        sim.step(5)
        orc.step(5)
        for sid in range(2):
            g, o = by_id(sim.get_species(sid)), orc.species[sid]
            k = np.argsort(o.ids)
            assert np.array_equal(g["ids"], o.ids[k])
            for a, c in enumerate("xyz"):
                d = np.abs(g[c] - getattr(o, c)[k])
                # 20 steps of three roundings of half an ulp of 32 (1e-6)
                assert np.minimum(d, size[a] - d).max() <= 1e-4
    sim.close()


# rows shorter than a block of 32 nodes, and ending inside one; one fluid, and two (the second one's loads run ahead)
@pytest.mark.parametrize("size", [(4, 4, 4), (36, 8, 4)])
@pytest.mark.parametrize("nf", [1, 2])
def test_fluid_blocks_match_oracle(size, nf):
    nx, ny, nz = size
    rng = np.random.default_rng(nf)
    inp = dict(grid=dict(nx=nx, ny=ny, nz=nz, dx=0.35), species=[],
               E=(0.02 * rng.standard_normal((3, nz, ny, nx))).astype(np.float32),
               B=(0.02 * rng.standard_normal((3, nz, ny, nx))).astype(np.float32))
    sim, orc = make_pair(inp, tile=4)
    for q in range(nf):
        fl = dict(q=-1.0 if q == 0 else 1.0, m=1.0 if q == 0 else 100.0,
                  n=rng.uniform(0.4, 0.6, (nz, ny, nx)).astype(np.float32),
                  **{c: (0.05 * rng.standard_normal((nz, ny, nx))).astype(np.float32) for c in ("ux", "uy", "uz")})
        sim.load_fluid(**fl)
        orc.load_fluid(**fl)
    sim.step(4)
    orc.step(4)
    for q in range(nf):
        g, o = sim.get_fluid(q), orc.fluids[q]
        # four steps of some fifty FP32 operations a node, 6e-8 each
        assert rel_l2(g["n"], o.n) <= 1e-5
        assert rel_l2(np.stack([g["ux"], g["uy"], g["uz"]]), o.u) <= 1e-4
    sim.close()


# W = 8 and 16: one tile; 24, 40: several, the last one ragged; one plane, and more planes than a column's start
@pytest.mark.parametrize("shape", [(3, 1, 32, 40), (2, 5, 16, 16), (1, 33, 16, 48)])
def test_classifier_ragged_volumes_match_oracle(shape):
    P = require_gpu()
    import torch
    from oracle.classifier import OracleCNN
    B, D, H, W = shape
    m, weights = seeded_classifier(P, 7, dropout=0.2, mc_passes=4)
    net = OracleCNN(weights, dropout=0.2, seed=7)
    x = np.random.default_rng(3).standard_normal((B, 6, D, H, W)).astype(np.float32)
    for k in (-1, 3):
        y = m.forward(torch.from_numpy(x).cuda(), k).cpu().numpy()
        ref = net.forward(x, k).numpy()
        assert rel_l2(y, ref) <= 1e-3, rel_l2(y, ref)


# BF16 rounding flips between FP32 and FP64 sums move a weight gradient by up to
# 1e-2 of its norm; a lost row, plane, tap or tile of these volumes by 5e-2 or more
GRAD = 2e-2


@pytest.mark.parametrize("shape", [(1, 1, 16, 8), (3, 5, 32, 24)])
def test_classifier_ragged_gradients_match_oracle(shape):
    P = require_gpu()
    import torch
    from oracle.classifier import OracleCNN, train_grads
    B, D, H, W = shape
    m, weights = seeded_classifier(P, 21, dropout=0.2, mc_passes=1, energy_weight=0.1)
    net = OracleCNN(weights, dropout=0.2, seed=21)
    rng = np.random.default_rng(5)
    x = rng.standard_normal((B, 6, D, H, W)).astype(np.float32)
    y = (x[:, 0] + 0.5 * x[:, 1] > 0.2).astype(np.float32)
    m.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    ref = train_grads(net, x, y, pass_index=0, energy_weight=0.1)
    for l in range(4):
        gw, gb = m.get_grad(l)
        rw, rb = ref["grads"][l]
        assert rel_l2(gw, rw.numpy()) <= GRAD and rel_l2(gb, rb.numpy()) <= GRAD, l


def _surrogate(seed, mean, std, passes):
    from oracle import surrogate as S
    from paper_2510_11174_gb300 import inputs
    from paper_2510_11174_gb300.model import Surrogate
    w = inputs.surrogate_weights(seed)
    m = Surrogate(dropout=0.1, mc_passes=passes, seed=seed, mean=mean, std=std)
    for l, (a, b) in enumerate(w):
        m.set_layer(l, a, b)
    return m, S.OracleSurrogate(w, dropout=0.1, seed=seed, mean=mean, std=std)


@pytest.mark.parametrize("passes", [1, 2, 7])
def test_surrogate_mc_groups_match_oracle(passes):
    require_gpu()
    import torch
    from paper_2510_11174_gb300 import inputs
    x, mean, std = inputs.random_states(3, 16, seed=4)
    x = np.ascontiguousarray(x[:, :, :5, :, :])
    m, orc = _surrogate(3, mean, std, passes)
    pm, ps = m.mc(torch.from_numpy(x).cuda())
    om, os_ = orc.mc_statistics(x, passes)
    assert rel_l2(pm.cpu().numpy() - x, om.numpy() - x) <= 2e-3
    if passes > 1:
        assert rel_l2(ps.cpu().numpy(), os_.numpy()) <= 2e-2
    m.close()


@pytest.mark.parametrize("shape", [(1, 1, 16, 8), (3, 5, 16, 24)])
def test_surrogate_ragged_gradients_match_oracle(shape):
    require_gpu()
    import torch
    from oracle import surrogate as S
    from paper_2510_11174_gb300 import inputs
    B, D, H, W = shape
    x, mean, std = inputs.random_states(B, 32, seed=6)
    x = np.ascontiguousarray(x[:, :, :D, :H, :W])
    sd = np.asarray(std)[None, :, None, None, None]
    t = x + (0.2 * np.random.default_rng(7).standard_normal(x.shape) * sd).astype(np.float32)
    m, orc = _surrogate(3, mean, std, 1)
    m.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    ref = S.loss_and_grads(orc, x, t, 0)
    for l in range(6):
        gw, gb = m.get_grad(l)
        ow, ob = ref["grads"][l]
        assert rel_l2(gw, ow.numpy()) <= GRAD and rel_l2(gb, ob.numpy()) <= GRAD, l
    m.close()


@pytest.mark.parametrize("n", [1, 127, 129, 20011])
def test_switchnet_ragged_gradients_match_oracle(n):
    require_gpu()
    import torch
    from oracle import switchnet as S
    from paper_2510_11174_gb300 import inputs
    from paper_2510_11174_gb300.model import SwitchNet
    rng = np.random.default_rng(n)
    x = rng.standard_normal((10, n)).astype(np.float32)
    y = (np.abs(x[1]) > 1.0).astype(np.float32)
    w = inputs.switchnet_weights(5)
    m = SwitchNet(dropout=0.2, mc_passes=1, seed=5)
    for l, (a, b) in enumerate(w):
        m.set_layer(l, a, b)
    orc = S.OracleSwitchNet(w, dropout=0.2, seed=5)
    m.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    ref = S.loss_and_grads(orc, x, y, 0)
    for l in range(5):
        gw, gb = m.get_grad(l)
        assert rel_l2(gw, ref["grads"][l][0].numpy()) <= GRAD and rel_l2(gb, ref["grads"][l][1].numpy()) <= GRAD, l
    m.close()
