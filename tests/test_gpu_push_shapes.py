"""The particle push against the oracle in every launch shape: both particle
shapes on both tiles, with tiles split over clusters of 4, 2 and left whole
(the tile counts at which 152 SMs hold that many CTAs)."""
import numpy as np
import pytest

from _util import by_id, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,tile,n", [
    (2, 4, (40, 40, 40)), (2, 4, (28, 28, 28)), (2, 4, (20, 20, 20)),       # 1000, 343, 125 tiles: 1, 2, 4 CTAs
    (2, 8, (48, 48, 48)), (2, 8, (48, 48, 32)), (2, 8, (16, 16, 16)),       # 216, 144, 8 tiles: 1, 2, 4 CTAs
    (1, 4, (40, 40, 40)), (1, 4, (28, 28, 28)),                             # 1000, 343 tiles: 1, 2 CTAs
])
def test_launch_shapes_match_oracle(order, tile, n):
    P = require_gpu()
    import oracle.sim as S
    from paper_2510_11174_gb300 import inputs
    inp = inputs.periodic_plasma(n=n[0], ny=n[1], nz=n[2], ppc=1, seed=7, a0=2.0, temperature_keV=20.0)
    g = inp["grid"]
    sim = P.Simulation(*n, g["dx"], cfl_frac=g["cfl_frac"], shape_order=order, tile=tile)
    orc = S.OracleSim(*n, g["dx"], cfl_frac=g["cfl_frac"], shape_order=order)
    for sp in inp["species"]:
        sim.load_species(**sp)
        orc.load_species(**sp)
    sim.set_fields(inp["E"], inp["B"])
    orc.set_fields(inp["E"], inp["B"])
    sim.step(1)
    orc.step(1)
    # a current is a displacement (0.1 cells RMS along an axis) between two FP32
    # positions, each off by at most half an ulp of 64 = 1.9e-6: 4e-5 of it
    assert rel_l2(sim.get_fields()[2], orc.J) <= 4e-5
    sim.step(4)
    orc.step(4)
    for sid in range(2):
        gp, o = by_id(sim.get_species(sid)), orc.species[sid]
        k = np.argsort(o.ids)
        assert np.array_equal(gp["ids"], o.ids[k])
        for a, c in enumerate("xyz"):
            d = np.abs(gp[c] - getattr(o, c)[k])
            # five steps of three roundings of half an ulp of 64, and the momenta's
            assert np.minimum(d, n[a] - d).max() <= 1e-4
    E, B, _ = sim.get_fields()
    assert rel_l2(E, orc.E) <= 1e-4 and rel_l2(B, orc.B) <= 1e-4
    sim.close()
