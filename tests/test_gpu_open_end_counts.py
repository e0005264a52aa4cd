"""Particles that left through the open end in the last step of a pp_step call
are gone from everything read afterwards: the counts, the particle arrays and a
checkpoint, whichever particle kernel ran (with the kernels that sort at the
start of every pass the sort comes before they leave).  Against the oracle with
several steps in one call.

Tolerances, per step, as in the other mixed parity tests: fields 3e-5 of the
largest value, positions and momenta 2e-6.
"""
import pytest

from tests import test_gpu_walls as walls_tests

pytestmark = pytest.mark.gpu

# mesh of 20 x 9 x 12 (the row kernel; sparse: the global one), 24 x 16 x 16 (the tile kernel; by mode: global, tiled)
CASES = [((10, 9, 12), 40000, 0), ((10, 9, 12), 900, 0), ((12, 16, 16), 6000, 0), ((12, 16, 16), 6000, 1),
         ((12, 16, 16), 6000, 2)]


@pytest.mark.parametrize("steps", [1, 6])
@pytest.mark.parametrize("n,count,mode", CASES)
def test_escaped_particles_are_gone(orc, n, count, mode, steps, tmp_path):
    import paper_1211_4575_gb300 as pp
    L = walls_tests._load(n, count, seed=231)
    L.species[0]["w"] = 0.002
    gpu, osim = walls_tests._boundary_pair(pp, orc, L, pp.PP_MIXED32, mode=mode, steps=steps)
    left = [len(osim.particles(s)["x"]) for s in (0, 1)]
    assert left[0] < count + left[1]   # both species take the same inflow
    assert [gpu.count(s) for s in (0, 1)] == left
    path = str(tmp_path / "open.ckpt")
    gpu.step(2)
    osim.step(2)
    gpu.save(path)
    back = pp.Simulation.restore(path)
    assert [back.count(s) for s in (0, 1)] == [len(osim.particles(s)["x"]) for s in (0, 1)]
    k = steps + 2
    walls_tests._compare_all(gpu, osim, L, 2, k * 3e-5, k * 2e-6, k * 2e-6)
