"""Simulations that are alive together: each goes on as it does alone."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2109_00214_gb300 as m
    m.load_library()
    return m


def _plume(pd, xs, nz, nr, graph):
    cfg, parts = synthetic.rz_plume(n=nz, total=2e4, seed=nz + nr)
    keep = parts["ir"] < nr
    cfg.update(nr=nr, field_on=1, inject_on=0)
    sim = pd.Simulation(cfg, xs)
    sim.load({k: v[keep] for k, v in parts.items()})
    if graph:
        sim.set_graph_mode(1, 8)
    return sim


def _state(sim):
    p = sim.particles()
    order = np.argsort(p["id"], kind="stable")
    return [sim.phi(), *sim.rho()] + [p[k][order] for k in ("id", "species", "iz", "ir", "pz", "pr", "vz", "vr", "vt")]


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("first,second", [
    ((224, 96), (160, 112)),       # 55 KB of shared memory for the coarse levels, then 40 KB
    ((96, 64), (36, 36)),          # 65 KB, then 47 KB
    ((160, 768), (32, 40)),        # the most of any grid, 74 KB, then 46 KB
])
def test_solves_of_two_grids_in_turn(pd, xs, first, second, graph):
    """A solver's coarse levels keep the shared memory they need whatever other
    solver is set up after it, eagerly and in a graph captured later."""
    alone = []
    for g in (first, second):
        sim = _plume(pd, xs, *g, graph)
        sim.step(3)
        alone.append(_state(sim))
        sim.close()
    sims = [_plume(pd, xs, *g, graph) for g in (first, second)]
    for _ in range(3):
        for sim in sims:
            sim.step(1)
    for sim, want in zip(sims, alone):
        for a, b in zip(_state(sim), want):
            assert np.array_equal(a, b)
        sim.close()
