"""Performance cases: what programs of this framework run, through its public
entry points (Simulation, Ensemble and Net).

A simulation is stepped a stretch at a time and read between stretches, so a
pass over most cases is one such stretch on a running simulation together with
the reading that follows it.  What is read is whole: the fixed-point node
charge and the number density (which fix every particle's cell and offset),
the particles themselves where they are few, the (x, t) pair of the latest
Poisson solve (density and potential on every node), and the event counters.

The potential is solved to 1e-10, as in the precision runs: two solutions at
1e-8 differ by 1e-4 in the space charge's share of the potential.  Stretches
are short where the particles are many (a plasma of this density doubles any
last-bit difference within a few steps).
"""
import math

import numpy as np
import torch

import paper_2109_00214_gb300 as pd
import synthetic

QE, ME, KB = 1.602176634e-19, 9.1093837015e-31, 1.380649e-23
MCU = 63.546 * 1.66053906660e-27
GAP = 6e-6                      # the electrode gap (m)
V_HEAVY = math.sqrt(KB * 2000.0 / MCU)

# cells a side of the r-z grids (the multigrid takes m * 2^k with m <= 8)
GRIDS = (64, 80, 96, 112, 128, 160, 192, 224, 256, 320, 384, 448, 512)


def listed():
    return [
        # the smallest call: one step of the paper's small breakdown from vacuum (field
        # emission, a few hundred particles), the circuit and the populations read
        # after each step: launches and latency
        dict(name="breakdown_64", kind="breakdown", n=64, warm_steps=200, steps=1),
        # the small breakdown with its plume: 2e4 particles, 20 eager steps, every
        # particle read at the end
        dict(name="plume_64", kind="plume", nz=64, nr=64, total=2e4, subcycle=10, graph=0, warm="previous",
             steps=20, particles=True),
        # production: 512^2 cells, 2e7 particles, the residual checked on the host
        dict(name="plume_512", kind="plume", nz=512, nr=512, total=2e7, subcycle=10, graph=0, warm="extrapolate",
             steps=4, particles=False),
        # a ragged grid between the two, one heavy cycle of steps as a CUDA graph
        dict(name="plume_224x96", kind="plume", nz=224, nr=96, total=7.77e5, subcycle=10, graph=7,
             warm="extrapolate", steps=10, particles=False),
        # 64 uneven breakdown runs (grids 64^2 to 256^2, 1e5 to 2e6 particles each)
        # advanced together under a CUDA graph: the parameter study
        dict(name="ensemble_64", kind="ensemble", runs=64, n_lo=1e5, n_hi=2e6, subcycle=4, graph=8, steps=4),
        # the paper's 120 x 480 domain with every collision extension and sputtering on,
        # stepped under a CUDA graph as a long run is
        dict(name="paper_domain", kind="paper", nz=120, nr=480, total=1.5e5, subcycle=10, graph=8, steps=10),
        # the DSMC microbench at full size: 1e8 particles, 100 steps without a field
        dict(name="micro_1e8", kind="micro", nz=1024, nr=1024, total=1e8, graph=0, steps=100, coulomb=0),
        # an odd grid and a middling load, under a CUDA graph
        dict(name="micro_251x509", kind="micro", nz=251, nr=509, total=3.1e6, graph=1, steps=20, coulomb=0),
        # Coulomb and heavy-pair collisions every step
        dict(name="coulomb_256x512", kind="micro", nz=256, nr=512, total=1.25e7, graph=0, steps=4, coulomb=1),
        # a short run from its start, as a parameter sweep makes many of: create, load
        # from device arrays, a few steps with about five candidates a cell, read
        dict(name="stress_run", kind="stress", nz=256, nr=512, total=1.25e7, steps=5, coll_scale=3200.0),
        # the warm-start network on the potential of one 512^2 run
        dict(name="net_forward_513", kind="net_forward", b=1, h=513, w=513),
        # one optimiser step of that network on a batch of 128^2 runs, residual loss
        dict(name="net_train_8x129", kind="net_train", b=8, h=129, w=129, loss="rz"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["breakdown", "plume", "plume", "ensemble", "paper", "micro", "micro", "coulomb", "stress",
                       "net_forward", "net_train"])
    if kind == "breakdown":
        return dict(kind=kind, n=rng.choice(GRIDS[:7]), warm_steps=rng.randrange(100, 300), steps=rng.randrange(1, 8))
    if kind == "plume":
        nz, nr = rng.choice(GRIDS), rng.choice(GRIDS)
        total = min(_log(rng, 1e4, 1e7), 200.0 * nz * nr)
        few = total < 5e4
        return dict(kind=kind, nz=nz, nr=nr, total=float(int(total)), subcycle=10 if few else 4,
                    graph=rng.choice([0, 7, 8]), warm=rng.choice(["previous", "extrapolate"]),
                    steps=10 if few else 4, particles=few)
    if kind == "ensemble":
        lo = _log(rng, 2e4, 2e5)
        return dict(kind=kind, runs=rng.randrange(2, 33), n_lo=float(int(lo)), n_hi=float(int(lo * 8)),
                    subcycle=4, graph=rng.choice([7, 8]), steps=4)
    if kind == "paper":
        return dict(kind=kind, nz=rng.choice(GRIDS[:7]), nr=rng.choice(GRIDS), total=float(int(_log(rng, 1e4, 4e5))),
                    subcycle=4, graph=rng.choice([0, 8]), steps=4)
    if kind in ("micro", "coulomb"):
        nz, nr = int(_log(rng, 40, 700)), int(_log(rng, 40, 700))
        total = nz * nr * _log(rng, 8.0, 60.0 if kind == "micro" else 120.0)
        return dict(kind="micro", nz=nz, nr=nr, total=float(int(min(total, 3e7))), graph=rng.choice([0, 1]),
                    steps=20 if kind == "micro" else 4, coulomb=int(kind == "coulomb"))
    if kind == "stress":
        nz, nr = int(_log(rng, 40, 400)), int(_log(rng, 40, 400))
        return dict(kind=kind, nz=nz, nr=nr, total=float(int(nz * nr * _log(rng, 20.0, 95.0))), steps=5,
                    coll_scale=float(int(_log(rng, 300.0, 3200.0))))
    if kind == "net_forward":
        b = rng.randrange(1, 5)
        return dict(kind=kind, b=b, h=int(_log(rng, 17, 400)), w=int(_log(rng, 17, 400)))
    return dict(kind=kind, b=rng.randrange(1, 9), h=int(_log(rng, 33, 200)), w=int(_log(rng, 33, 200)),
                loss=rng.choice(["rz", "mse"]))


# ---- inputs ----------------------------------------------------------------
def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _maxwellians(g, nr, groups):
    """Particles as device arrays.  `groups`: (species, number in each cell,
    thermal velocity: one, or one a cell)."""
    out = {k: [] for k in ("species", "iz", "ir", "pz", "pr", "vz", "vr", "vt")}
    for sp, number, v in groups:
        cell = torch.repeat_interleave(torch.arange(number.numel(), device="cuda"), number)
        n = cell.numel()
        if torch.is_tensor(v):
            v = v[cell]
        out["species"].append(torch.full((n,), sp, dtype=torch.uint8, device="cuda"))
        out["iz"].append((cell // nr).int())
        out["ir"].append((cell % nr).int())
        for k in ("pz", "pr"):
            out[k].append(torch.rand(n, generator=g, device="cuda"))
        for k in ("vz", "vr", "vt"):
            out[k].append(torch.randn(n, generator=g, device="cuda") * v)
    return {k: torch.cat(v) for k, v in out.items()}


def _plume(seed, nz, nr, total):
    """The near-cathode copper plume of a developed breakdown: exponential in z,
    Gaussian in r (1 um each), 60 % ionized with mean charge 2, electrons at
    5 eV, heavies at 2000 K; returns the particles and their weight."""
    g = _rng(seed)
    d = GAP / nz
    z = (torch.arange(nz, device="cuda", dtype=torch.float64) + 0.5) * d
    j = torch.arange(nr, device="cuda", dtype=torch.float64)
    heavy = (1e26 * torch.exp(-z / 1e-6)[:, None] * torch.exp(-((j + 0.5) * d / 1e-6) ** 2)[None, :]
             * (math.pi * (2.0 * j + 1.0) * d ** 3)[None, :]).flatten()
    weight = float(heavy.sum()) * 2.2 / total
    mean = heavy / weight
    cu, sw, di = (torch.poisson(mean * f, generator=g).long() for f in (0.4, 0.6 * 10 / 11, 0.6 / 11))
    parts = _maxwellians(g, nr, [(0, 2 * (sw + di), math.sqrt(5.0 * QE / ME)), (1, cu, V_HEAVY), (3, sw, V_HEAVY),
                                 (4, di, V_HEAVY)])
    return parts, weight


def _gas(seed, nz, nr, total):
    """The DSMC microbench's load: lognormal copper density a cell, 10 % of it
    ionized, electrons of 5 to 50 eV a cell; returns the particles and the depth."""
    g = _rng(seed)
    d, cells, w = 50e-9, nz * nr, 100.0
    vol = total * w / (cells * 1e23 * math.exp(0.5) * 1.2)
    n = torch.exp(math.log(1e23) + torch.randn(cells, generator=g, device="cuda", dtype=torch.float64))
    cu = torch.round(n * (vol / w)).long()
    ion = torch.round(0.1 * cu).long()
    te = 5.0 + 45.0 * torch.rand(cells, generator=g, device="cuda")
    parts = _maxwellians(g, nr, [(0, ion, torch.sqrt(te * (QE / ME))), (1, cu, V_HEAVY), (2, ion, V_HEAVY)])
    return parts, vol / (d * d)


def _rz_config(seed, nz, nr, weight, total, subcycle, **kw):
    d = GAP / nz
    c = synthetic.base_config(geometry="rz", nz=nz, nr=nr, dz=d, dr=d, weight=weight, seed=seed % (1 << 31),
                              heavy_subcycle=subcycle, field_on=1, inject_on=0, poisson_tol=1e-10,
                              capacity=int(2.0 * total) + (1 << 18))
    c.update(kw)
    return c


def _gas_config(case, seed, depth, **kw):
    c = synthetic.base_config(geometry="xy_periodic", nz=case["nz"], nr=case["nr"], dz=50e-9, dr=50e-9, depth=depth,
                              heavy_subcycle=1, seed=seed % (1 << 31), field_on=0, inject_on=0,
                              capacity=int(1.05 * case["total"]) + (1 << 18) + 8 * case["nz"] * case["nr"])
    c.update(kw)
    return c


def _run_size(case, k):
    """Grid and particle count of an ensemble's run k."""
    pick = np.random.Generator(np.random.Philox(key=k))
    n = int(synthetic.ENSEMBLE_GRIDS[int(pick.integers(0, len(synthetic.ENSEMBLE_GRIDS)))])
    return n, math.exp(pick.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))


def _net_params(g):
    p = []
    for cin, cout in ((1, 32), (32, 32), (32, 32), (32, 32), (32, 32), (32, 1)):
        p.append(torch.randn(9 * cout * cin, generator=g, device="cuda") * math.sqrt(2.0 / (9 * cin)))
        p.append(torch.randn(cout, generator=g, device="cuda") * 0.05)
    return torch.cat(p)


def _net_inputs(case, seed):
    g = _rng(seed)
    shape = (case["b"], case["h"], case["w"])
    params = _net_params(g)
    x = torch.randn(shape, generator=g, device="cuda")
    x = x / x.abs().amax(dim=(1, 2), keepdim=True)      # a charge density over its largest value
    t = 0.3 * torch.randn(shape, generator=g, device="cuda")
    return params, x, t


def prepare(case, seed):
    xs = synthetic.standin_cross_sections()
    kind = case["kind"]
    if kind == "breakdown":
        cfg, _ = synthetic.rz_breakdown(n=case["n"], seed=seed % (1 << 31), capacity=1 << 17)
        cfg["poisson_tol"] = 1e-10
        sim = pd.Simulation(cfg, xs)
        sim.step(case["warm_steps"])
    elif kind in ("plume", "paper"):
        parts, weight = _plume(seed, case["nz"], case["nr"], case["total"])
        extra = dict(charge_max=4, heavy_coll=1, sputter=1) if kind == "paper" else {}
        sim = pd.Simulation(_rz_config(seed, case["nz"], case["nr"], weight, case["total"], case["subcycle"], **extra),
                            xs)
        if kind == "paper":
            sim.set_sputter_yield(*synthetic.standin_sputter_yield())
        sim.load_device(parts)
        sim.set_warm_start(case.get("warm", "extrapolate"))
        if case["graph"]:
            sim.set_graph_mode(1, case["graph"])
    elif kind == "ensemble":
        cfgs, loads = [], []
        for k in range(case["runs"]):
            n, total = _run_size(case, k)
            parts, weight = _plume(1000 * seed + k, n, n, total)
            kv = synthetic.ENSEMBLE_VOLTS_KV[k % len(synthetic.ENSEMBLE_VOLTS_KV)]
            cfgs.append(_rz_config(seed, n, n, weight, total, case["subcycle"], run=k, V0=1e3 * kv))
            loads.append(parts)
        sim = pd.Ensemble(cfgs, xs)
        for k, parts in enumerate(loads):
            sim.load_run_device(k, parts)
        sim.set_warm_start("extrapolate")
        sim.set_graph_mode(1, case["graph"])
    elif kind == "micro":
        parts, depth = _gas(seed, case["nz"], case["nr"], case["total"])
        on = case["coulomb"]
        sim = pd.Simulation(_gas_config(case, seed, depth, coulomb=on, heavy_coll=on), xs)
        sim.load_device(parts)
        if case["graph"]:
            sim.set_graph_mode(1)
        sim.step(4)
    elif kind == "stress":
        parts, depth = _gas(seed, case["nz"], case["nr"], case["total"])
        # room for the slots that the candidates reserve and for the new electrons
        cfg = _gas_config(case, seed, depth, coll_dt_scale=case["coll_scale"],
                          capacity=int(2.0 * case["total"]) + 8 * case["nz"] * case["nr"] + (1 << 18))
        return dict(case=case, cfg=cfg, xs=xs, parts=parts)
    else:
        params, x, t = _net_inputs(case, seed)
        net = pd.Net(x.numel(), params.cpu().numpy())
        return dict(case=case, net=net, x=x, t=t)
    return dict(case=case, sim=sim)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "net_forward":
        return state["net"].forward(state["x"])
    if kind == "net_train":
        net = state["net"]
        if case["loss"] == "rz":
            loss, grads = net.loss_grad_rz(state["x"], want_grads=True)
        else:
            loss, grads = net.loss_grad(state["x"], state["t"], want_grads=True)
        net.adam(lr=1e-3)
        return dict(loss=loss, grads=grads, params=net.params())
    if kind == "stress":
        sim = pd.Simulation(state["cfg"], state["xs"])
        sim.load_device(state["parts"])
    else:
        sim = state["sim"]
    sim.step(case["steps"])
    if kind == "breakdown":
        x, t = sim.warmstart_pairs()
        s = sim.scalars()
        return dict(x=x, t=t, V=s["V"], I=s["I_gap"], count=np.array(s["count"]), absorbed=np.array(s["absorbed_energy"]))
    if kind in ("plume", "paper"):
        x, t = sim.warmstart_pairs()
        out = dict(x=x, t=t, events=_events(sim.counters()))
        if case.get("particles"):
            out.update(_by_id(sim.particles(), int(2 * case["total"])))
        return out
    if kind == "ensemble":
        x, t = sim.warmstart_pairs()
        return dict(x=x, t=t, events=np.stack([_events(sim.run_counters(k)) for k in range(case["runs"])]))
    rho_e, rho_h = sim.rho()
    out = dict(rho_e=rho_e, rho_h=rho_h, cu=sim.density_map(1), events=_events(sim.counters()))
    if kind == "stress":
        out["spectrum"] = sim.energy_spectrum(0).astype(np.int64)
        sim.close()
    return out


def _events(counters):
    return np.array(list(counters.values()), dtype=np.int64)


def _by_id(p, most):
    """The particles in the places of their ids (the store's own order is by cell)."""
    out = {}
    for k in ("species", "iz", "ir", "pz", "pr", "vz", "vr", "vt"):
        out[k] = np.zeros(most, p[k].dtype)
        out[k][p["id"]] = p[k]
    return out


# ---- what a pass cannot do without ------------------------------------------
def _cartesian_step(total, coulomb):
    """Bytes and operations of one field-free step: key, offset and velocity of
    each particle read (24 B), key and offset written (12 B), a ninth of the
    particles (a tenth of the gas) electrons; with Coulomb pairs the charged
    sixth writes its velocity too (12 B)."""
    return (36.0 + (2.0 if coulomb else 0.0)) * total, (30.0 + (60.0 if coulomb else 0.0)) * total


def _rz_step(total, nodes, subcycle):
    """Bytes and operations of one r-z step: the electrons (1.2 of 2.2) read and
    written (48 B) each step, the heavies every `subcycle`-th; on the nodes both
    charge densities written and read, the potential read and written, the field
    written and read (64 B), and about six V(2,2) cycles of the solve."""
    moved = total * (1.2 + 1.0 / subcycle) / 2.2
    return 48.0 * moved + 64.0 * nodes, 120.0 * moved + 600.0 * nodes


def work(case):
    kind = case["kind"]
    if kind == "breakdown":
        b, f = _rz_step(300.0, (case["n"] + 1) ** 2, 10)
        return dict(bytes=case["steps"] * b, flops=case["steps"] * f)
    if kind in ("plume", "paper"):
        nodes = (case["nz"] + 1) * (case["nr"] + 1)
        b, f = _rz_step(case["total"], nodes, case["subcycle"])
        read = 8.0 * nodes + (37.0 * case["total"] if case.get("particles") else 0.0)
        return dict(bytes=case["steps"] * b + read, flops=case["steps"] * f)
    if kind == "ensemble":
        runs = [_run_size(case, k) for k in range(case["runs"])]
        b, f = _rz_step(sum(c for _, c in runs), sum((n + 1) ** 2 for n, _ in runs), case["subcycle"])
        return dict(bytes=case["steps"] * b, flops=case["steps"] * f)
    if kind in ("micro", "stress"):
        b, f = _cartesian_step(case["total"], case.get("coulomb"))
        cells = case["nz"] * case["nr"]
        load = 29.0 * case["total"] if kind == "stress" else 0.0
        return dict(bytes=case["steps"] * b + load + 24.0 * cells, flops=case["steps"] * f)
    nodes = case["b"] * case["h"] * case["w"]
    flops = 2.0 * 9 * (32 + 4 * 1024 + 32) * nodes
    if kind == "net_forward":
        return dict(bytes=8.0 * nodes + 4 * 37601, flops=flops)
    return dict(bytes=4.0 * nodes + 7 * 4 * 37601, flops=3.0 * flops)


# ---- the network in 64 bits --------------------------------------------------
def exact(case, seed):
    """The network's outputs from float64 convolutions and their gradients.  A
    simulation's outputs have no such value: its events, charges and counts are
    whole numbers of a float32 trajectory."""
    if case["kind"] not in ("net_forward", "net_train"):
        return None
    params, x, t = _net_inputs(case, seed)
    p = params.double().requires_grad_(case["kind"] == "net_train")
    x, t = x.double(), t.double()
    y, at = x[:, None], 0
    for k, (cin, cout) in enumerate(((1, 32), (32, 32), (32, 32), (32, 32), (32, 32), (32, 1))):
        w = p[at:at + 9 * cout * cin].view(3, 3, cout, cin).permute(2, 3, 0, 1)
        at += 9 * cout * cin
        y = torch.nn.functional.conv2d(y, w, p[at:at + cout], padding=1)
        at += cout
        if k < 5:
            y = torch.relu(y)
    y = y[:, 0]
    if case["kind"] == "net_forward":
        return y
    if case["loss"] == "rz":
        W = case["w"]
        j = torch.arange(W, device=x.device, dtype=torch.float64)
        ap, am, w = j + 0.5, j - 0.5, j.clone()
        ap[-1] = am[0] = 0.0
        w[0], w[-1] = 0.125, (W - 1) / 2 - 0.125
        z = y.clone()
        z[:, 0] = 0.0
        z[:, -1] = 0.0
        c = z[:, 1:-1]
        s = (ap + am + 2 * w) * c - w * (z[:, 2:] + z[:, :-2])
        s = s - ap * torch.nn.functional.pad(c[..., 1:], (0, 1)) - am * torch.nn.functional.pad(c[..., :-1], (1, 0))
        loss = (w * x[:, 1:-1] - s).square().mean()
    else:
        loss = (y - t).square().mean()
    loss.backward()
    # the first step of Adam from zero moments
    g = p.grad
    return dict(loss=float(loss), grads=g, params=(p - 1e-3 * g / (g.abs() + 1e-8)).detach())
