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


@pytest.mark.parametrize("n,count,mode", CASES)
def test_graphs_after_the_open_end_closes(n, count, mode):
    """Graphs asked for before, the open end closed after eager steps: the steps
    that follow are captured and replayed (the particles that left are dropped
    before the capture), and the run equals one that never uses graphs."""
    import numpy as np
    import torch
    import paper_1211_4575_gb300 as pp
    from tests import gpu_helpers as H
    L = walls_tests._load(n, count, seed=233)
    L.species[0]["w"] = 0.002
    sims = []
    for graphs in (False, True):
        stream = torch.cuda.Stream()
        sim = H.gpu_sim(pp, L, pp.PP_MIXED32, 3, deposit_mode=mode, sort_interval=2, stream=stream.cuda_stream,
                        boundary_x=pp.PP_BOUNDARY_WALLS)
        sim._keep_stream = stream
        sim.set_graphs(graphs)
        sim.set_open_boundary(4, 0.2, 2.0)
        sim.step(5)
        sim.set_open_boundary(0, 0.0, 0.0)
        sim.step(12)
        sims.append(sim)
    cap, rep = sims[1].graph_stats()
    assert cap + rep == 12 and rep >= 3, (cap, rep)
    assert sims[0].count(0) == sims[1].count(0) < count
    for F, G in zip(sims[1].fields(), sims[0].fields()):
        scale = max(np.abs(v).max() for v in G)
        assert max(np.abs(u - v).max() for u, v in zip(F, G)) <= 17 * 3e-5 * scale
