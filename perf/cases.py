"""Performance cases: the work a user of the library has it do, through its public entry points.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare(case, seed)`` builds what a user's
program holds before the call (contexts with particles, fluids and fields; networks with their weights; patches on the
GPU), ``run(state)`` is one pass and returns everything it computes, ``work(case)`` counts the bytes and floating-point
operations a pass cannot do without, and ``exact(case, seed)`` is the same computation in 64 bits with plain torch.

Kinds:
  pic        full PIC steps, then the node state (E, B, J, rho): the electromagnetic PIC loop of the periodic plasma
             configuration and of boxes with absorbing walls and a laser
  carbon     full PIC steps with field ionization, photon emission and pair creation (carbon slab under a strong pulse)
  hybrid     one classification cycle of the hybrid method: N steps of fluid + particles, then the regime
             classification (16 MC-dropout passes) with its conversions, then the node state
  classify   the MC-dropout classification of every node of a grid: p_mean and p_std
  train_cnn  one training step of the regime classifier, with its gradients
  mc_sur     MC-dropout forecast of the field surrogate: mean and spread
  train_sur  one training step of the field surrogate, with its gradients
  train_sn   one training step of SwitchNet, with its gradients
"""
import math

import numpy as np
import torch

import paper_2510_11174_gb300 as P
from paper_2510_11174_gb300 import inputs
from paper_2510_11174_gb300.model import Classifier, Surrogate, SwitchNet

M_P = inputs.M_P


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the plain full-PIC configuration of the tests and the smoke run: a few dozen tiles, so launches and the
        # length of one tile's particle loop decide
        dict(name="pic_32", kind="pic", nx=32, ny=32, nz=32, ppc=8, order=1, tile=8, wall=0, pusher="boris", steps=5),
        # an uneven box with absorbing, reflecting walls and a laser on every step: walls, Mur planes, source
        dict(name="pic_walls", kind="pic", nx=72, ny=40, nz=56, ppc=3, order=1, tile=8, wall=1, pusher="vay", steps=5),
        # the smooth (quadratic) particle shape on the small tile
        dict(name="pic_quadratic", kind="pic", nx=48, ny=40, nz=32, ppc=6, order=2, tile=4, wall=0,
             pusher="higuera_cary", steps=5),
        # full PIC at a production size: 15.7 M particles, every tile occupied
        dict(name="pic_large", kind="pic", nx=128, ny=96, nz=80, ppc=8, order=1, tile=8, wall=0, pusher="boris",
             steps=4),
        # the strong-field configuration: ions that ionize, electrons that radiate, photons that decay
        dict(name="carbon_64", kind="carbon", n=64, ny=32, nz=32, ppc=8, steps=5),
        # a run of a laser-parameter scan: a small hybrid box, where host and launch costs weigh
        dict(name="hybrid_64", kind="hybrid", nx=64, ny=32, nz=32, ppc=8, steps=10, passes=16),
        # the headline workload: ramp + slab 256 x 256 x 128, 16 MC passes every 10 steps
        dict(name="hybrid_256", kind="hybrid", nx=256, ny=256, nz=128, ppc=8, steps=10, passes=16),
        # the classification of every node of a mid-size grid
        dict(name="classify_128", kind="classify", nx=128, ny=128, nz=64, passes=16),
        # training batches at the sizes the networks are trained with
        dict(name="train_cnn_32x32", kind="train_cnn", batch=32, d=32, h=32, w=32),
        dict(name="mc_sur_16x16", kind="mc_sur", batch=16, d=16, h=16, w=16, passes=16),
        dict(name="train_sur_32x16", kind="train_sur", batch=32, d=16, h=16, w=16),
        dict(name="train_sn_65536", kind="train_sn", n=65536),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["pic", "pic", "pic", "carbon", "hybrid", "hybrid", "classify", "train_cnn", "mc_sur",
                       "train_sur", "train_sn"])
    if kind == "pic":
        order = rng.choice([1, 1, 2])
        nx, ny, nz = (8 * round(_log(rng, 2, 12)) for _ in range(3))
        ppc = round(_log(rng, 1, 16))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, ppc=ppc, order=order, tile=rng.choice([8, 8, 4]),
                    wall=rng.choice([0, 1]) if order == 1 else 0,
                    pusher=rng.choice(["boris", "boris", "vay", "higuera_cary"]), steps=rng.randint(1, 8))
    if kind == "carbon":
        return dict(kind=kind, n=8 * rng.randint(7, 10), ny=8 * rng.randint(2, 5), nz=8 * rng.randint(2, 5),
                    ppc=rng.randint(4, 12), steps=rng.randint(2, 6))
    if kind == "hybrid":
        nx, ny, nz = 16 * round(_log(rng, 4, 12)), 16 * round(_log(rng, 1, 10)), 16 * round(_log(rng, 1, 8))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, ppc=rng.choice([8, 8, 12]), steps=rng.choice([5, 10]),
                    passes=rng.choice([8, 16, 16]))
    if kind == "classify":
        return dict(kind=kind, nx=8 * round(_log(rng, 3, 24)), ny=16 * round(_log(rng, 1, 10)),
                    nz=8 * round(_log(rng, 1, 12)), passes=rng.choice([4, 16, 16]))
    if kind == "train_cnn":
        return dict(kind=kind, batch=rng.randint(4, 36), d=rng.randint(20, 32), h=32, w=8 * rng.randint(3, 5))
    if kind == "mc_sur":
        return dict(kind=kind, batch=round(_log(rng, 1, 40)), d=rng.randint(8, 24), h=16, w=8 * rng.randint(1, 3),
                    passes=rng.choice([4, 16, 16]))
    if kind == "train_sur":
        return dict(kind=kind, batch=round(_log(rng, 8, 48)), d=rng.randint(12, 24), h=16, w=8 * rng.randint(1, 3))
    return dict(kind="train_sn", n=round(_log(rng, 8000, 150000)))


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float32)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)


def _clear_outer_half(F, half, bc):
    """Yee values at a half-integer position do not exist past the last node of an absorbing axis."""
    for c in range(3):
        for a in range(3):
            if bc[a] and half(c, a):
                F[c].select(2 - a, F.shape[3 - a] - 1).zero_()


def _packet(g, nx, ny, nz, dx, a0, x_c, length, w0, bc, noise=0.0):
    """A linearly polarised pulse (E_y, B_z) moving along +x, with Gaussian envelopes."""
    phase = float(torch.rand(1, generator=g, device="cuda")) * 2.0 * math.pi
    a0 = a0 * (0.9 + 0.2 * float(torch.rand(1, generator=g, device="cuda")))
    x = torch.arange(nx, device="cuda", dtype=torch.float32) * dx
    y = (torch.arange(ny, device="cuda", dtype=torch.float32) - 0.5 * (ny - 1)) * dx
    z = (torch.arange(nz, device="cuda", dtype=torch.float32) - 0.5 * (nz - 1)) * dx
    tr = torch.exp(-(y[None, :, None] ** 2 + z[:, None, None] ** 2) / w0 ** 2)
    E = noise * a0 * _randn(g, 3, nz, ny, nx)
    B = noise * a0 * _randn(g, 3, nz, ny, nx)
    for F, c, s in ((E, 1, 0.0), (B, 2, 0.5 * dx)):
        xs = x + s
        F[c] += a0 * torch.exp(-((xs - x_c) / length) ** 2) * torch.cos(xs - x_c + phase) * tr
    _clear_outer_half(E, lambda c, a: c == a, bc)
    _clear_outer_half(B, lambda c, a: c != a, bc)
    return E, B


def _pic_inputs(case, seed):
    """Periodic plasma (wall = 0) or a plasma block between absorbing walls with a laser (wall = 1): electrons and
    protons at 0.1 n_c and 1 keV under a wave of amplitude 1, lambda / 16 per cell."""
    g = _gen(seed)
    nx, ny, nz, ppc = case["nx"], case["ny"], case["nz"], case["ppc"]
    dx = 2.0 * math.pi / 16
    bc = (1, 1, 1) if case["wall"] else (0, 0, 0)
    top = [n - 1 if b else n for n, b in zip((nx, ny, nz), bc)]
    n = top[0] * top[1] * top[2] * ppc
    sp = []
    for q, m in ((-1.0, 1.0), (1.0, M_P)):
        pos = [torch.clamp(_rand(g, n) * t, max=float(np.nextafter(np.float32(t), np.float32(0)))) for t in top]
        sig = math.sqrt(1.0 / (inputs.MC2_KEV * m))
        u = [sig * _randn(g, n) for _ in range(3)]
        w = torch.full((n,), 0.1 * dx ** 3 / ppc, device="cuda")
        sp.append(dict(q=q, m=m, x=pos[0], y=pos[1], z=pos[2], ux=u[0], uy=u[1], uz=u[2], w=w))
    if case["wall"]:
        E, B = _packet(g, nx, ny, nz, dx, 1.0, 0.5 * nx * dx, 6.0, 8.0, bc, noise=0.01)
        laser = dict(a0=2.0, tau_fwhm=20.0, w0_spot=6.0, t_peak=4.0, y_c=0.5 * (ny - 1), z_c=0.5 * (nz - 1), x_src=3,
                     pol=1)
    else:
        k = 2.0 * math.pi * max(1, round(nx / 16)) / (nx * dx)
        E, B = 0.01 * _randn(g, 3, nz, ny, nx), 0.01 * _randn(g, 3, nz, ny, nx)
        i = torch.arange(nx, device="cuda", dtype=torch.float32)
        E[1] += torch.cos(k * i * dx)
        B[2] += torch.cos(k * (i + 0.5) * dx)
        laser = None
    return dict(dx=dx, bc=bc, species=sp, E=E, B=B, laser=laser)


def _weights(pairs, taps, g, bias=0.05):
    """He-uniform weights and small biases as host arrays, [(W [co][ci](taps), b [co])]."""
    out = []
    for ci, co in pairs:
        fan = ci * (27 if taps else 1)
        w = (2.0 * _rand(g, co, ci, *((3, 3, 3) if taps else ())) - 1.0) * math.sqrt(6.0 / fan)
        out.append((w.cpu().numpy(), (bias * _randn(g, co)).cpu().numpy()))
    return out


def _set(model, weights):
    for layer, (w, b) in enumerate(weights):
        model.set_layer(layer, w, b)
    return model


def _classifier_weights(seed, out_bias=0.0):
    return inputs.classifier_weights(int(seed) % (1 << 31), out_bias=out_bias)


def _pulse_patches(g, batch, channels, d, h, w):
    """Patches cut from a run: a pulse at a random place on weak noise, in some channels, and its envelope."""
    ax = lambda n: torch.linspace(-1.0, 1.0, n, device="cuda")
    cx, cz = (1.2 * _rand(g, batch) - 0.6 for _ in range(2))
    env = torch.exp(-((ax(w)[None, None, None, :] - cx[:, None, None, None]) / 0.5) ** 2
                    - (ax(h)[None, None, :, None] / 0.6) ** 2
                    - ((ax(d)[None, :, None, None] - cz[:, None, None, None]) / 0.5) ** 2)
    x = 0.3 * _randn(g, batch, channels, d, h, w)
    ph = torch.cos(12.0 * ax(w) + 6.0 * float(torch.rand(1, generator=g, device="cuda")))
    x[:, 1] += 4.0 * env * ph
    x[:, 5] += 4.0 * env * ph
    return x, env


# ------------------------------------------------------------------------------------------------ prepare
def _simulation(case, inp, seed):
    sim = P.Simulation(case["nx"], case["ny"], case["nz"], inp["dx"], bc=inp["bc"], laser=inp.get("laser"),
                       seed=int(seed) % (1 << 31), tile=case.get("tile", 8), shape_order=case.get("order", 1))
    return sim


def _prepare_pic(case, seed):
    inp = _pic_inputs(case, seed)
    sim = _simulation(case, inp, seed)
    for s in inp["species"]:
        sim.load_species(pusher=case["pusher"], **s)
    sim.set_fields(inp["E"], inp["B"])
    return dict(kind="steps", sim=sim, steps=case["steps"])


def _prepare_carbon(case, seed):
    """The carbon slab when the pulse is in it: ions of mixed charge, their electrons, some photons, no positrons."""
    g = _gen(seed)
    n, ny, nz, ppc = case["n"], case["ny"], case["nz"], case["ppc"]
    dx = 2.0 * math.pi / 20
    bc = (1, 1, 1)
    sim = P.Simulation(n, ny, nz, dx, bc=bc, seed=int(seed) % (1 << 31),
                       laser=dict(a0=100.0, tau_fwhm=70.0, w0_spot=4.0 * math.pi, t_peak=105.0, y_c=0.5 * (ny - 1),
                                  z_c=0.5 * (nz - 1), x_src=4, pol=1))
    lo, hi = int(0.35 * n), int(0.9 * n)
    m = (hi - lo) * (ny - 1) * (nz - 1) * ppc

    def place(k):
        p = [lo + (hi - lo) * _rand(g, k), (ny - 1) * _rand(g, k), (nz - 1) * _rand(g, k)]
        return dict(x=torch.clamp(p[0], max=hi - 0.01), y=torch.clamp(p[1], max=ny - 1.01),
                    z=torch.clamp(p[2], max=nz - 1.01))

    w0 = (10.0 / 6.0) * dx ** 3 / ppc
    zero = torch.zeros(m, device="cuda")
    ions = dict(q=1.0, m=inputs.M_C, ux=zero, uy=zero, uz=zero, w=torch.full((m,), w0, device="cuda"),
                zq=torch.floor(3.0 + 1.5 * _rand(g, m)), **place(m))
    u = [20.0 * _randn(g, 2 * m) for _ in range(3)]
    elec = dict(q=-1.0, m=1.0, ux=u[0] + 60.0, uy=u[1], uz=u[2], w=torch.full((2 * m,), 1.6 * w0, device="cuda"),
                **place(2 * m))
    k = m // 8
    phot = dict(q=0.0, m=0.0, ux=5.0 + 100.0 * _rand(g, k), uy=_randn(g, k), uz=_randn(g, k),
                w=torch.full((k,), w0, device="cuda"), **place(k))
    empty = {c: torch.zeros(0, device="cuda") for c in ("x", "y", "z", "ux", "uy", "uz", "w")}
    cap = 512 * ppc
    sim.load_species(qed=dict(photon_species=2, eps_min=2.0), tile_capacity=8 * cap, **elec)
    sim.load_species(ionize=dict(zmax=6, ip_eV=inputs.CARBON_IP_EV, l=inputs.CARBON_L, into=0), tile_capacity=4 * cap,
                     **ions)
    sim.load_species(kind=1, pairs=dict(electron=0, positron=3), tile_capacity=4 * cap, **phot)
    sim.load_species(q=1.0, m=1.0, qed=dict(photon_species=2, eps_min=2.0), tile_capacity=2 * cap, **empty)
    sim.set_fields(*_packet(g, n, ny, nz, dx, 100.0, 0.5 * n * dx, 0.2 * n * dx, 4.0 * math.pi, bc))
    return dict(kind="steps", sim=sim, steps=case["steps"])


def _prepare_hybrid(case, seed):
    """The ramp + slab target with the pulse in the ramp: cold electron and proton fluids, kinetic cells already
    converted by the first classification."""
    g = _gen(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    inp = inputs.ramp_slab(nx=nx, ny=1, nz=1, a0=2.0, ppc=case["ppc"], slab_lambda=min(2.0, nx / 64.0),
                           vacuum_lambda=min(1.0, nx / 128.0))
    gr, bc = inp["grid"], inp["grid"]["bc"]
    laser = dict(inp["laser"], y_c=0.5 * (ny - 1), z_c=0.5 * (nz - 1))
    sim = P.Simulation(nx, ny, nz, gr["dx"], cfl_frac=gr["cfl_frac"], bc=bc, laser=laser, seed=int(seed) % (1 << 31))
    empty = {c: torch.zeros(0, device="cuda") for c in ("x", "y", "z", "ux", "uy", "uz", "w")}
    for q, m in ((-1.0, 1.0), (1.0, M_P)):
        sim.load_species(q=q, m=m, tile_capacity=2048 * case["ppc"], **empty)
    prof = torch.from_numpy(np.ascontiguousarray(inp["fluids"][0]["n"][0, 0])).cuda()
    n = (prof[None, None, :] * (1.0 + 0.02 * (_rand(g, nz, ny, nx) - 0.5))).cpu().numpy()
    for fl in inp["fluids"]:
        sim.load_fluid(fl["q"], fl["m"], n, n_floor=fl["n_floor"])
    sim.set_fields(*_packet(g, nx, ny, nz, gr["dx"], 2.0, 0.3 * nx * gr["dx"], 0.08 * nx * gr["dx"],
                            min(4.0 * math.pi, 0.2 * ny * gr["dx"]), bc))
    model = Classifier(dropout=0.2, mc_passes=case["passes"], seed=11, std=[1.0] * 6, stream=sim.desc.stream)
    _set(model, _classifier_weights(11, out_bias=-4.0))
    sim.set_regime(dilate=2, ppc=case["ppc"], to_species=[0, 1], policy="union", reach=case["steps"] + 1)
    sim.classify(model)
    return dict(kind="hybrid", sim=sim, model=model, steps=case["steps"])


def _classify_fields(case, seed):
    g = _gen(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dx = 2.0 * math.pi / 16
    return dx, _packet(g, nx, ny, nz, dx, 10.0, 0.5 * nx * dx, 0.15 * nx * dx, 0.25 * ny * dx, (1, 1, 1), noise=0.05)


def _prepare_classify(case, seed):
    dx, (E, B) = _classify_fields(case, seed)
    sim = P.Simulation(case["nx"], case["ny"], case["nz"], dx, bc=(1, 1, 1))
    sim.set_fields(E, B)
    sim.set_regime(dilate=2)
    model = Classifier(dropout=0.2, mc_passes=case["passes"], seed=11, std=[2.0] * 6, stream=sim.desc.stream)
    _set(model, _classifier_weights(3))
    pm = torch.empty((case["nz"], case["ny"], case["nx"]), device="cuda")
    return dict(kind="classify", sim=sim, model=model, pm=pm, ps=torch.empty_like(pm))


def _cnn_batch(case, seed):
    g = _gen(seed)
    x, env = _pulse_patches(g, case["batch"], 6, case["d"], case["h"], case["w"])
    return x, (env > 0.3).float()


def _sur_batch(case, seed):
    g = _gen(seed)
    x, env = _pulse_patches(g, case["batch"], 10, case["d"], case["h"], case["w"])
    t = x + 0.2 * torch.roll(x, 1, dims=4) * env[:, None]
    return x, t


SUR_STD, SUR_DSTD = [1.0] * 10, [0.3] * 10


def _sn_batch(case, seed):
    g = _gen(seed)
    x = _randn(g, 10, case["n"])
    y = (x[1] + 0.5 * x[5] * x[9] > 0.2).float()
    return x, y


def _sur_weights(seed):
    return inputs.surrogate_weights(int(seed) % (1 << 31))


def _sn_weights(seed):
    return inputs.switchnet_weights(int(seed) % (1 << 31))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pic":
        return _prepare_pic(case, seed)
    if kind == "carbon":
        return _prepare_carbon(case, seed)
    if kind == "hybrid":
        return _prepare_hybrid(case, seed)
    if kind == "classify":
        return _prepare_classify(case, seed)
    if kind == "train_cnn":
        x, y = _cnn_batch(case, seed)
        return dict(kind="train", layers=4, model=_set(Classifier(seed=7), _classifier_weights(5)), x=x, y=y)
    if kind == "mc_sur":
        m = Surrogate(seed=11, mc_passes=case["passes"], std=SUR_STD, dstd=SUR_DSTD)
        return dict(kind="mc", model=_set(m, _sur_weights(4)), x=_sur_batch(case, seed)[0])
    if kind == "train_sur":
        x, t = _sur_batch(case, seed)
        m = Surrogate(seed=11, lr=3e-4, std=SUR_STD, dstd=SUR_DSTD)
        return dict(kind="train", layers=6, model=_set(m, _sur_weights(4)), x=x, y=t)
    x, y = _sn_batch(case, seed)
    return dict(kind="train", layers=5, model=_set(SwitchNet(seed=13), _sn_weights(6)), x=x, y=y)


# ------------------------------------------------------------------------------------------------ run
def run(state):
    kind = state["kind"]
    if kind == "steps":
        state["sim"].step(state["steps"])
        return {"node_state": state["sim"].node_state()}
    if kind == "hybrid":
        state["sim"].step(state["steps"])
        state["sim"].classify(state["model"])
        return {"node_state": state["sim"].node_state()}
    if kind == "classify":
        state["sim"].classify(state["model"], state["pm"], state["ps"])
        return {"p_mean": state["pm"], "p_std": state["ps"]}
    if kind == "mc":
        mean, spread = state["model"].mc(state["x"])
        return {"mean": mean, "spread": spread}
    st = state["model"].train_step(state["x"], state["y"])
    out = {"loss": st["loss"]}
    for layer in range(state["layers"]):
        out["w%d" % layer], out["b%d" % layer] = state["model"].get_grad(layer)
    return out


# ------------------------------------------------------------------------------------------------ work
CNN_FLOP, SUR_FLOP, SN_FLOP = 94176.0, 820908.0, 332288.0     # forward, per cell and pass
CNN_TRAIN, SUR_TRAIN, SN_TRAIN = 272160.0, 2455704.0, 992256.0  # a training step, per cell


def work(case):
    """Particles: x, u and w read, x and u written (52 B) per step; cells: E, B, J (60 B) per step and the ten node
    channels written once; fluids: n and u read and written (32 B); networks: inputs and outputs once."""
    kind = case["kind"]
    if kind == "pic":
        cells = case["nx"] * case["ny"] * case["nz"]
        parts = 2 * cells * case["ppc"]
        return {"bytes": case["steps"] * (52.0 * parts + 60.0 * cells) + 40.0 * cells, "flops": 400.0 * parts * case["steps"]}
    if kind == "carbon":
        cells = case["n"] * case["ny"] * case["nz"]
        ions = 0.55 * cells * case["ppc"]
        return {"bytes": case["steps"] * (ions * (56.0 + 2.125 * 60.0) + 60.0 * cells) + 40.0 * cells,
                "flops": 1250.0 * ions * case["steps"]}
    if kind == "hybrid":
        cells = case["nx"] * case["ny"] * case["nz"]
        parts = 2 * 0.2 * cells * case["ppc"]
        return {"bytes": case["steps"] * (52.0 * parts + 60.0 * cells + 64.0 * 0.5 * cells) + 40.0 * cells,
                "flops": CNN_FLOP * case["passes"] * 0.7 * cells + 400.0 * parts * case["steps"]}
    if kind == "classify":
        cells = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 32.0 * cells, "flops": CNN_FLOP * case["passes"] * cells}
    if kind == "train_sn":
        return {"bytes": 44.0 * case["n"], "flops": SN_TRAIN * case["n"]}
    cells = case["batch"] * case["d"] * case["h"] * case["w"]
    if kind == "train_cnn":
        return {"bytes": 28.0 * cells, "flops": CNN_TRAIN * cells}
    if kind == "mc_sur":
        return {"bytes": 120.0 * cells, "flops": SUR_FLOP * case["passes"] * cells}
    return {"bytes": 80.0 * cells, "flops": SUR_TRAIN * cells}


# ------------------------------------------------------------------------------------------------ exact: PIC
def _stag(field, c):
    """Half-integer axes (x, y, z) of component c."""
    return [0.5 if (a == c) == (field == "E") else 0.0 for a in range(3)]


def _shape_nodes(p, s, order, n, wall):
    """First node and the weights of a particle's shape on one axis (positions minus the staggering s)."""
    q = p - s
    if order == 1:
        i = torch.floor(q)
        if wall and s == 0.0:
            i = torch.clamp(i, max=n - 2)
        f = q - i
        return i.long(), [1.0 - f, f]
    m = torch.floor(q + 0.5)
    d = q - m
    return m.long() - 1, [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2]


def _gather(F, pos, stag, order, n, bc):
    ax = [_shape_nodes(pos[a], stag[a], order, n[a], bc[a]) for a in range(3)]
    flat, out = F.reshape(-1), torch.zeros_like(pos[0])

    def index(a, k):
        i = ax[a][0] + k
        if bc[a]:
            ok = (i >= 0) & (i <= n[a] - 1)
            return torch.clamp(i, 0, n[a] - 1), ax[a][1][k] * ok
        return i % n[a], ax[a][1][k]

    w = order + 1
    X, Y, Z = ([index(a, k) for k in range(w)] for a in range(3))
    for iz, wz in Z:
        for iy, wy in Y:
            for ix, wx in X:
                out += wx * wy * wz * flat[(iz * n[1] + iy) * n[0] + ix]
    return out


def _push(kind, h, e, b, u):
    cross = lambda v, w: torch.linalg.cross(v, w, dim=0)
    dot = lambda v, w: (v * w).sum(0)
    if kind == "boris":
        um = u + h * e
        t = h * b / torch.sqrt(1.0 + dot(um, um))
        up = um + cross(um + cross(um, t), 2.0 * t / (1.0 + dot(t, t)))
        return up + h * e
    tau = h * b
    w = u + h * (2.0 * e + cross(u / torch.sqrt(1.0 + dot(u, u)), b)) if kind == "vay" else u + h * e
    sg, us = 1.0 + dot(w, w) - dot(tau, tau), dot(w, tau)
    t = tau / torch.sqrt(0.5 * (sg + torch.sqrt(sg * sg + 4.0 * (dot(tau, tau) + us * us))))
    r = (w + dot(w, t) * t + cross(w, t)) / (1.0 + dot(t, t))
    return r if kind == "vay" else r + h * e + cross(r, t)


def _deposit(J, x0, x1, qw, order, n, bc, dx, dt):
    """Esirkepov's charge-conserving current for one chunk of particles."""
    def shape(d):
        d = d.abs()
        if order == 1:
            return torch.clamp(1.0 - d, min=0.0)
        return torch.where(d <= 0.5, 0.75 - d * d, 0.5 * torch.clamp(1.5 - d, min=0.0) ** 2)

    off = 0.0 if order == 1 else 0.5
    win = order + 2
    base, S0, DS = [], [], []
    for a in range(3):
        b = torch.minimum(torch.floor(x0[a] + off), torch.floor(x1[a] + off)) - (order - 1)
        s0 = [shape(x0[a] - b - k) for k in range(win)]
        base.append(b.long())
        S0.append(s0)
        DS.append([shape(x1[a] - b - k) - s0[k] for k in range(win)])

    def idx(a, k):
        i = base[a] + k
        return torch.clamp(i, 0, n[a] - 1) if bc[a] else i % n[a]

    node = [[idx(a, k) for k in range(win)] for a in range(3)]
    stride = (1, n[0], n[0] * n[1])
    for c in range(3):
        p, q = (c + 1) % 3, (c + 2) % 3
        flat = J[c].reshape(-1)
        for kq in range(win):
            for kp in range(win):
                wt = (S0[p][kp] * S0[q][kq] + 0.5 * DS[p][kp] * S0[q][kq] + 0.5 * S0[p][kp] * DS[q][kq]
                      + DS[p][kp] * DS[q][kq] / 3.0)
                acc = torch.zeros_like(wt)
                for kc in range(win - 1):
                    acc = acc + DS[c][kc] * wt
                    flat.index_add_(0, node[c][kc] * stride[c] + node[p][kp] * stride[p] + node[q][kq] * stride[q],
                                    -qw * acc / (dt * dx * dx))


def _ax(a):
    return 2 - a   # tensor axis of x, y, z in [nz][ny][nx]


def _nd(t, a, lo, size):
    return t.narrow(_ax(a), lo, size)


def _keep_half(F, a, bc):
    """Zero out the values that do not exist at the half-integer end of an absorbing axis."""
    if bc[a]:
        _nd(F, a, F.shape[_ax(a)] - 1, 1).zero_()
    return F


def _b_half(E, B, n, bc, dx, dt):
    d = lambda F, a: torch.roll(F, -1, _ax(a)) - F
    for c in range(3):
        p, q = (c + 1) % 3, (c + 2) % 3
        B[c] -= 0.5 * dt * _keep_half(_keep_half((d(E[q], p) - d(E[p], q)) / dx, p, bc), q, bc)


def _e_step(E, B, J, n, bc, dx, dt):
    old = [e.clone() for e in E]
    d = lambda F, a: F - torch.roll(F, 1, _ax(a))
    for c in range(3):
        p, q = (c + 1) % 3, (c + 2) % 3
        up = _keep_half(dt * ((d(B[q], p) - d(B[p], q)) / dx - J[c]), c, bc)
        for a in (p, q):
            if bc[a]:
                _nd(up, a, 0, 1).zero_()
                _nd(up, a, n[a] - 1, 1).zero_()
        E[c] += up
    # first-order Mur on the tangential components: faces, then the edges two absorbing axes share (lower axis)
    coef = (dt - dx) / (dt + dx)
    for edges in (False, True):
        for c in range(3):
            tang = [a for a in range(3) if a != c and bc[a]]
            for a in tang:
                other = [t for t in tang if t != a]
                if edges and (not other or a > other[0]):
                    continue
                for edge, inner in ((0, 1), (n[a] - 1, n[a] - 2)):
                    new = _nd(old[c], a, inner, 1) + coef * (_nd(E[c], a, inner, 1) - _nd(old[c], a, edge, 1))
                    sel = torch.ones_like(new, dtype=torch.bool)
                    for o in other:
                        on = torch.zeros_like(sel)
                        _nd(on, o, 0, 1).fill_(True)
                        _nd(on, o, n[o] - 1, 1).fill_(True)
                        sel &= on if edges else ~on
                    if bc[c]:
                        _nd(sel, c, n[c] - 1, 1).fill_(False)
                    dst = _nd(E[c], a, edge, 1)
                    dst.copy_(torch.where(sel, new, dst))


def _to_nodes(F, axes, bc):
    for a in axes:
        r = torch.roll(F, 1, _ax(a))
        if bc[a]:
            _nd(r, a, 0, 1).zero_()
        F = 0.5 * (F + r)
    return F


def _exact_pic(case, seed):
    inp = _pic_inputs(case, seed)
    n, bc, dx, order = (case["nx"], case["ny"], case["nz"]), inp["bc"], inp["dx"], case["order"]
    dt = 0.95 * dx / math.sqrt(3.0)
    E, B = [list(inp[k].double().unbind(0)) for k in ("E", "B")]
    E, B = [e.clone() for e in E], [b.clone() for b in B]
    sp = []
    for s in inp["species"]:
        sp.append(dict(q=s["q"], m=s["m"], w=s["w"].double(), x=torch.stack([s[k].double() for k in ("x", "y", "z")]),
                       u=torch.stack([s[k].double() for k in ("ux", "uy", "uz")])))
    las = inp["laser"]
    J = None
    for step in range(case["steps"]):
        J = [torch.zeros_like(E[0]) for _ in range(3)]
        for s in sp:
            for lo in range(0, s["x"].shape[1], 1 << 20):
                sl = slice(lo, lo + (1 << 20))
                x0, u = s["x"][:, sl], s["u"][:, sl]
                e = torch.stack([_gather(E[c], x0, _stag("E", c), order, n, bc) for c in range(3)])
                b = torch.stack([_gather(B[c], x0, _stag("B", c), order, n, bc) for c in range(3)])
                u = _push(case["pusher"], 0.5 * s["q"] * dt / s["m"], e, b, u)
                x1 = x0 + u * (dt / dx) / torch.sqrt(1.0 + (u * u).sum(0))
                for a in range(3):
                    if bc[a]:
                        top = n[a] - 1.0
                        out = (x1[a] < 0.0) | (x1[a] > top)
                        u[a] = torch.where(out, -u[a], u[a])
                        x1[a] = torch.where(x1[a] < 0.0, -x1[a], torch.where(x1[a] > top, 2.0 * top - x1[a], x1[a]))
                _deposit(J, x0, x1, s["q"] * s["w"][sl], order, n, bc, dx, dt)
                for a in range(3):
                    if not bc[a]:
                        x1[a] = x1[a] % n[a]
                s["x"][:, sl], s["u"][:, sl] = x1, u
        if las:
            c = las["pol"]
            y = (torch.arange(n[1], device="cuda").double() + (0.5 if c == 1 else 0.0) - las["y_c"]) * dx
            z = (torch.arange(n[2], device="cuda").double() + (0.5 if c == 2 else 0.0) - las["z_c"]) * dx
            prof = torch.exp(-(y[None, :] ** 2 + z[:, None] ** 2) / las["w0_spot"] ** 2)
            if bc[c]:
                prof.narrow(2 - c, n[c] - 1, 1).zero_()
            tt = (step + 0.5) * dt - las["t_peak"]
            amp = las["a0"] * math.exp(-2.0 * math.log(2.0) * tt * tt / las["tau_fwhm"] ** 2) * math.sin(tt)
            J[c][:, :, las["x_src"]] += -2.0 * amp / dx * prof
        _b_half(E, B, n, bc, dx, dt)
        _e_step(E, B, J, n, bc, dx, dt)
        _b_half(E, B, n, bc, dx, dt)
    rho = torch.zeros(n[0] * n[1] * n[2], device="cuda", dtype=torch.float64)
    for s in sp:
        ax = [_shape_nodes(s["x"][a], 0.0, 1, n[a], bc[a]) for a in range(3)]
        for kz in range(2):
            for ky in range(2):
                for kx in range(2):
                    i, j, k = ((ax[a][0] + o) % n[a] for a, o in ((0, kx), (1, ky), (2, kz)))
                    rho.index_add_(0, (k * n[1] + j) * n[0] + i,
                                   s["q"] * s["w"] / dx ** 3 * ax[0][1][kx] * ax[1][1][ky] * ax[2][1][kz])
    out = [_to_nodes(E[c], [c], bc) for c in range(3)]
    out += [_to_nodes(B[c], [a for a in range(3) if a != c], bc) for c in range(3)]
    out += [_to_nodes(J[c], [c], bc) for c in range(3)]
    return {"node_state": torch.stack(out + [rho.reshape(n[2], n[1], n[0])])}


# ------------------------------------------------------------------------------------------------ exact: networks
def _philox(ctr, key):
    """Philox4x32-10 (Salmon et al., SC 2011) on int64 tensors that hold 32-bit words."""
    M32 = 0xFFFFFFFF
    c = [torch.as_tensor(v, dtype=torch.int64, device="cuda") for v in ctr]
    k0, k1 = int(key[0]) & M32, int(key[1]) & M32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _keep(batch, channels, cells, seed, pass_index, layer, p):
    """Dropout factors [batch, channels, cells] (0 or 1 / (1 - p)) of the documented stream."""
    thr = round(p * 65536.0)
    lin = torch.arange(cells, device="cuda")[None, :]
    b = torch.arange(batch, device="cuda")[:, None]
    out = torch.empty(batch, channels, cells, device="cuda", dtype=torch.float64)
    for grp in range((channels + 7) // 8):
        r = _philox((lin + 0 * b, b + 0 * lin, torch.full_like(lin + b, (layer << 16) | grp),
                     torch.full_like(lin + b, pass_index)), (seed, 0xD0))
        for j in range(min(8, channels - 8 * grp)):
            out[:, 8 * grp + j] = ((r[j >> 1] >> (16 * (j & 1))) & 0xFFFF) >= thr
    return out / (1.0 - thr / 65536.0)


def _params(weights):
    return [tuple(torch.from_numpy(np.asarray(t)).double().cuda().requires_grad_(True) for t in wb) for wb in weights]


def _conv(x, w, b):
    return torch.nn.functional.conv3d(x, w, b, padding=1)


def _pad_to(a, c):
    return torch.cat([a, a.new_zeros((a.shape[0], c - a.shape[1]) + tuple(a.shape[2:]))], 1) if a.shape[1] < c else a


def _cnn(x, prm, seed, pass_index, drop=0.2):
    a = x
    for layer in range(3):
        a = torch.relu(_conv(a, *prm[layer]))
        k = _keep(a.shape[0], a.shape[1], a[0, 0].numel(), seed, pass_index, layer, drop)
        a = a * k.reshape(a.shape)
    return _conv(a, *prm[3])[:, 0]


def _bce(logit, y, energy, weight=0.1):
    w = 1.0 + weight * energy / energy.mean()
    bce = torch.clamp(logit, min=0.0) - logit * y + torch.log1p(torch.exp(-logit.abs()))
    return (w * bce).mean()


def _with_grads(loss, prm):
    loss.backward()
    out = {"loss": float(loss)}
    for layer, (w, b) in enumerate(prm):
        out["w%d" % layer], out["b%d" % layer] = w.grad, b.grad
    return out


def _sur(x, prm, seed, pass_index, drop=0.1):
    a = x
    for layer in range(6):
        h = _conv(a, *prm[layer])
        if layer < 5:
            h = torch.relu(h)
        if layer == 1:
            h = h * _keep(h.shape[0], h.shape[1], h[0, 0].numel(), seed, pass_index, 1, drop).reshape(h.shape)
        a = h + _pad_to(a, h.shape[1]) if layer < 3 else h
    return a


def _exact_classify(case, seed):
    if case["nx"] * case["ny"] * case["nz"] * case["passes"] > (1 << 24):
        return None
    dx, (E, B) = _classify_fields(case, seed)
    bc = (1, 1, 1)
    f = [_to_nodes(E[c].double(), [c], bc) for c in range(3)]
    f += [_to_nodes(B[c].double(), [a for a in range(3) if a != c], bc) for c in range(3)]
    x = torch.stack(f)[None] / 2.0
    prm = _params(_classifier_weights(3))
    with torch.no_grad():
        p = torch.stack([torch.sigmoid(_cnn(x, prm, 11, k)[0]) for k in range(case["passes"])])
    return {"p_mean": p.mean(0), "p_std": p.std(0, unbiased=False)}


def _exact_train_cnn(case, seed):
    x, y = (t.double() for t in _cnn_batch(case, seed))
    prm = _params(_classifier_weights(5))
    n, total = x.shape[0], 0.0
    energy = 0.5 * (x * x).sum(1)
    w = 1.0 + 0.1 * energy / energy.mean()
    # the batch in parts (the dropout stream counts samples from the start of the batch)
    for lo in range(0, n, 4):
        xs, ys, ws = x[lo:lo + 4], y[lo:lo + 4], w[lo:lo + 4]
        a = xs
        for layer in range(3):
            a = torch.relu(_conv(a, *prm[layer]))
            k = _keep(lo + a.shape[0], a.shape[1], a[0, 0].numel(), 7, 0, layer, 0.2)[lo:]
            a = a * k.reshape(a.shape)
        logit = _conv(a, *prm[3])[:, 0]
        bce = torch.clamp(logit, min=0.0) - logit * ys + torch.log1p(torch.exp(-logit.abs()))
        loss = (ws * bce).sum() / y.numel()
        loss.backward()
        total += float(loss)
    out = {"loss": total}
    for layer, (wt, b) in enumerate(prm):
        out["w%d" % layer], out["b%d" % layer] = wt.grad, b.grad
    return out


def _exact_mc_sur(case, seed):
    x = _sur_batch(case, seed)[0].double()
    prm = _params(_sur_weights(4))
    with torch.no_grad():
        y = torch.stack([x + 0.3 * _sur(x, prm, 11, k) for k in range(case["passes"])])
    return {"mean": y.mean(0), "spread": y.std(0, unbiased=False)}


def _exact_train_sur(case, seed):
    x, t = (v.double() for v in _sur_batch(case, seed))
    prm = _params(_sur_weights(4))
    y = _sur(x, prm, 11, 0)
    r = (y - (t - x) / 0.3).abs()
    hub = torch.where(r <= 0.01, 0.5 * r * r, 0.01 * (r - 0.005)).mean()
    wp, wt = (0.5 * (v[:, :6] ** 2).sum() for v in (x + 0.3 * y, t))
    return _with_grads(hub + 0.1 * ((wp - wt) / wt) ** 2, prm)


def _exact_train_sn(case, seed):
    x, y = (v.double() for v in _sn_batch(case, seed))
    prm = _params(_sn_weights(6))
    a = x.T
    for layer in range(4):
        w, b = prm[layer]
        h = a @ w.T + b
        if layer < 2:
            h = torch.relu(h)
        if layer == 1:
            h = h * _keep(1, h.shape[1], h.shape[0], 13, 0, 1, 0.2)[0].T
        a = h + _pad_to(a, h.shape[1]) if layer < 2 else h
    logit = (a @ prm[4][0].T)[:, 0] + prm[4][1]
    return _with_grads(_bce(logit, y, 0.5 * (x[:6] ** 2).sum(0)), prm)


def exact(case, seed):
    """None for the stochastic and threshold-driven runs: an event or a cell's regime that flips with the last bit of
    a rate or a probability selects another, equally valid trajectory."""
    f = {"pic": _exact_pic, "classify": _exact_classify, "train_cnn": _exact_train_cnn, "mc_sur": _exact_mc_sur,
         "train_sur": _exact_train_sur, "train_sn": _exact_train_sn}.get(case["kind"])
    return None if f is None else f(case, seed)
