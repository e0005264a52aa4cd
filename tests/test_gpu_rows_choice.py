"""On meshes that 8^3 tiles do not divide, the automatic deposit takes the row
kernel (one launch for all species, a sort in every pass) where the particles
pay for the sort and the windows, and the global kernel (a launch per species,
a sort every sort_interval steps) for the others.  Which of the two ran is told
by the launches of the particle phase; what they give is compared with the
global kernel's mode.

Tolerances, per step, as in the other mixed parity tests: fields 3e-5 of the
largest value, positions and momenta 2e-6.
"""
import numpy as np
import pytest

import pp_synth
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu


def _sim(pp, n, shape, mode=0, capacity=200000, graphs=False):
    import torch
    stream = torch.cuda.Stream()
    sim = pp.Simulation(n, (0.5,) * 3, 0.25, shape_order=shape, precision=pp.PP_MIXED32, deposit_mode=mode,
                        relax_tol=1e-6, stream=stream.cuda_stream)
    sim._keep_stream = stream
    for q in (-1.0, 1.0):
        sim.add_species(q, 1.0, 0.02, capacity)
    if graphs:
        sim.set_graphs(True)
    return sim


def _load(sim, n, count, seed, part=(1.0, 1.0, 1.0)):
    for s in (0, 1):
        rng = np.random.default_rng([seed, s])
        x = rng.random((3, count)) * (np.array(n) * 0.5 * np.array(part))[:, None]
        sim.load_particles(s, *x, *(0.3 * rng.standard_normal((3, count))))


def _takes_rows(sim, steps=3):
    sim.profile_enable(True)
    sim.step(steps)
    launches = sim.profile_read()["particle_launches"]
    sim.profile_enable(False)
    assert launches in (steps, 2 * steps)
    return launches == steps


# particles per species; part of the box that holds them
@pytest.mark.parametrize("n,shape,count,part,rows", [
    ((60, 45, 37), 3, 400, (1, 1, 1), False),            # test particles
    ((60, 45, 37), 3, 30000, (1, 1, 1), False),
    ((60, 45, 37), 3, 200000, (1, 1, 1), True),
    ((60, 45, 37), 3, 60000, (1, 0.15, 0.2), True),      # the same particles in a beam
    ((60, 45, 37), 2, 100000, (1, 1, 1), False),
    ((60, 45, 37), 2, 300000, (1, 1, 1), True),
    ((60, 45, 37), 1, 300000, (1, 1, 1), False),
    ((60, 45, 37), 1, 900000, (1, 1, 1), True),
    ((9, 10, 11), 3, 2000, (1, 1, 1), False),
    ((9, 10, 11), 3, 5000, (1, 1, 1), True),             # more than eight per cell: the more exact kernel
    ((9, 10, 11), 2, 5000, (1, 1, 1), True),
    ((9, 10, 11), 1, 20000, (1, 1, 1), False),
    ((9, 10, 11), 1, 30000, (1, 1, 1), True),
    ((60, 45, 7), 3, 200000, (1, 1, 1), False),          # an axis below a tile
])
def test_choice_follows_the_load(n, shape, count, part, rows):
    import paper_1211_4575_gb300 as pp
    sim = _sim(pp, n, shape, capacity=count)
    _load(sim, n, count, 1, part)
    assert _takes_rows(sim) == rows


@pytest.mark.parametrize("graphs", [False, True], ids=["eager", "graphs"])
@pytest.mark.parametrize("shape", [1, 2, 3])
def test_a_run_that_crosses_the_line(shape, graphs):
    """Sparse, then loaded past the line: the particles go from the global kernel
    (unsorted by then) to the row kernel between two steps."""
    import paper_1211_4575_gb300 as pp
    n = (13, 9, 18)
    sims = []
    for mode in (0, pp.PP_DEPOSIT_GLOBAL):
        sim = _sim(pp, n, shape, mode, graphs=graphs and mode == 0)
        sim.load_fields(*pp_synth.random_fields(n, 4, 0.05))
        _load(sim, n, 300, 2)
        sim.step(4)
        if mode == 0 and not graphs:
            assert not _takes_rows(sim, 1)
        else:
            sim.step(1)
        _load(sim, n, 60000, 3)
        sim.step(4)
        if mode == 0 and not graphs:
            assert _takes_rows(sim, 1)
        else:
            sim.step(1)
        assert sim.diagnostics()["status"] == 0
        sims.append(sim)
    a, b = sims
    for F, G in zip(a.fields(), b.fields()):
        scale = max(np.abs(v).max() for v in G)
        assert max(np.abs(u - v).max() for u, v in zip(F, G)) <= 10 * 3e-5 * scale
    for s in (0, 1):
        dpos, du = H.particle_errors(a.particles(s), b.particles(s), tuple(0.5 * e for e in n))
        assert dpos <= 10 * 2e-6 and du <= 10 * 2e-6, (s, dpos, du)
