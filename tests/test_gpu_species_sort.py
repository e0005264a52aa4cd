"""The per-step sort takes all species of a run in its launches.  Against the
oracle with species of unequal size, one of them empty, one of a single
particle, one past a sort block's 8,192 keys, in any order; one species and the
most the library takes (eight); a mesh of a single tile, one that tiles do not
divide and one whose keys end inside a scan block.

Tolerances, per step, as in the other mixed parity tests: fields 3e-5 of the
largest value, positions and momenta 2e-6.
"""
import numpy as np
import pytest

import pp_synth
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

COUNTS = [(700,), (0, 8193, 1), (8193, 0, 700), (33, 64, 1, 0, 900, 2, 8192, 5)]


@pytest.mark.parametrize("n", [(8, 8, 8), (13, 9, 10), (24, 16, 8)], ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("counts", COUNTS, ids=lambda c: "-".join(map(str, c)))
def test_species_sorted_together(counts, n):
    import paper_1211_4575_gb300 as pp
    import oracle
    L = pp_synth.random_particles(n, (0.5, 0.5, 0.5), 0.3, max(counts), seed=5, w=0.02)
    base = L.species[0]
    L.species = []
    for k, c in enumerate(counts):
        part = {a: np.roll(v, 17 * k)[:c].copy() if isinstance(v, np.ndarray) else v for a, v in base.items()}
        part["q"] = base["q"] * (1 - 2 * (k % 2))
        L.species.append(part)
    E, B = pp_synth.random_fields(n, 3, 0.05)
    sim = H.gpu_sim(pp, L, pp.PP_MIXED32, 3)
    orc = H.oracle_sim(oracle, L, 3)
    sim.load_fields(E, B)
    orc.load_fields(E, B)
    steps = 3
    sim.step(steps)
    orc.step(steps)
    for name, err in H.field_errors(sim, orc).items():
        assert err <= steps * 3e-5, (name, err)
    for s in range(len(counts)):
        dpos, du = H.particle_errors(sim.particles(s), orc.species[s], H.box(L))
        assert dpos <= steps * 2e-6 and du <= steps * 2e-6, (s, dpos, du)
    assert sim.diagnostics()["status"] == 0
