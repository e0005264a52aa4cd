"""The per-step sorted kernel (mixed form, automatic deposit) against the FP64
oracle where its blocks change shape: meshes that 8^3 tiles divide and meshes
they do not (the last tiles partly empty, plain window loads), few tiles (blocks
one and two cells deep) and many (four deep), every shape order.  The particles
are fast and a step is 0.9 cells long at the speed of light, so that most of
them change their support on one, two or three axes at once: the rows beside a
cell's nodes and their corners carry current.

Tolerances, per step, are those of the other mixed parity tests: fields 3e-5 of
the largest value, positions 2e-6 (physical units), momenta 2e-6 relative.
"""
import pytest

import pp_synth
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

SIZES = [(8, 8, 8), (9, 10, 11), (17, 8, 33), (32, 32, 24), (40, 32, 32), (43, 37, 26)]


@pytest.mark.parametrize("shape", [1, 2, 3])
@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_blocks_match_oracle(n, shape):
    import paper_1211_4575_gb300 as pp
    import oracle
    steps = 2
    L = pp_synth.random_particles(n, (0.5, 0.5, 0.5), 0.45, 6 * n[0] * n[1], seed=17 + shape, u_scale=2.0, w=0.02)
    E, B = pp_synth.random_fields(n, 3, 0.05)
    sim = H.gpu_sim(pp, L, pp.PP_MIXED32, shape)
    orc = H.oracle_sim(oracle, L, shape)
    sim.load_fields(E, B)
    orc.load_fields(E, B)
    sim.step(steps)
    orc.step(steps)
    for name, err in H.field_errors(sim, orc).items():
        assert err <= steps * 3e-5, (name, err)
    dpos, du = H.particle_errors(sim.particles(0), orc.species[0], H.box(L))
    assert dpos <= steps * 2e-6 and du <= steps * 2e-6
    assert sim.diagnostics()["status"] == 0
