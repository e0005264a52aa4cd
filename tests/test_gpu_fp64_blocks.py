"""The FP64 particle kernel sorts the particles of each 256-thread block into
those that cross no support boundary in the step and the others.  Against the
oracle at particle counts around the block's and the warp's size, with no, few
and most particles crossing, every shape order.

Tolerance 1e-12 per step as in the other FP64 parity tests: both sides do the
same FP64 arithmetic up to the order of sums over at most some thousand terms.
"""
import pytest

import pp_synth
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [1, 2, 3])
@pytest.mark.parametrize("u_scale", [1e-4, 0.1, 3.0])
@pytest.mark.parametrize("count", [1, 33, 255, 256, 257, 1024 + 31])
def test_fp64_blocks_match_oracle(count, u_scale, shape):
    import paper_1211_4575_gb300 as pp
    import oracle
    L = pp_synth.random_particles((13, 9, 10), (0.5, 0.5, 0.5), 0.4, count, seed=count + shape, u_scale=u_scale)
    E, B = pp_synth.random_fields(L.n, 3, 0.05)
    sim = H.gpu_sim(pp, L, pp.PP_FP64, shape)
    orc = H.oracle_sim(oracle, L, shape)
    sim.load_fields(E, B)
    orc.load_fields(E, B)
    steps = 2
    sim.step(steps)
    orc.step(steps)
    for name, err in H.field_errors(sim, orc).items():
        assert err <= steps * 1e-12, (name, err)
    dpos, du = H.particle_errors(sim.particles(0), orc.species[0], H.box(L))
    assert dpos <= steps * 1e-12 and du <= steps * 1e-12
    assert sim.diagnostics()["status"] == 0
