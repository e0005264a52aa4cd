"""Step graphs and the tiled kernel's count of particles left to the global
mesh (pp_diag.n_slow, "last step"): after every step a replayed run reports what
the eager run reports, whichever of its captures ran.

The particles carry a weight so small that their fields (1e-12 of the momenta)
cannot change an FP32 momentum: both runs follow the same trajectories, and the
counts are equal exactly.
"""
import pytest

import pp_synth

pytestmark = pytest.mark.gpu

N = (16, 16, 16)


def _counts(pp, graphs, steps, sort_interval, current, solver):
    import torch
    L = pp_synth.random_particles(N, (0.5, 0.5, 0.5), 0.2, 4000, seed=77, u_scale=3.0, w=1e-12)
    stream = torch.cuda.Stream()
    sim = pp.Simulation(L.n, L.d, L.dt, shape_order=3, precision=pp.PP_MIXED32, sort_interval=sort_interval,
                        deposit_mode=pp.PP_DEPOSIT_TILED, relax_tol=1e-6, stream=stream.cuda_stream)
    for s in L.species:
        sid = sim.add_species(s["q"], s["m"], s["w"], len(s["x"]))
        sim.load_particles(sid, s["x"], s["y"], s["z"], s["ux"], s["uy"], s["uz"])
    sim.set_current_deposit(current)
    sim.set_field_solver(solver)
    sim.set_graphs(graphs)
    out = []
    for _ in range(steps):
        sim.step(1)
        d = sim.diagnostics()
        assert d["status"] == 0
        out.append(d["n_slow"])
    return out, sim.graph_stats()


@pytest.mark.parametrize("method", ["direct-explicit", "conserving-implicit"])
def test_slow_count_of_replayed_steps_is_the_eager_one(method):
    """No sort after the load, so that ever more particles leave their tiles."""
    import paper_1211_4575_gb300 as pp
    cur, sol = ((pp.PP_CURRENT_DIRECT, pp.PP_FIELD_EXPLICIT) if method == "direct-explicit"
                else (pp.PP_CURRENT_CONSERVING, pp.PP_FIELD_IMPLICIT))
    eager, _ = _counts(pp, False, 16, 0, cur, sol)
    graph, (cap, rep) = _counts(pp, True, 16, 0, cur, sol)
    assert cap >= 1 and rep >= 12, (cap, rep)
    assert eager[-1] > 100
    assert graph == eager


def test_slow_count_is_zero_after_passes_of_another_kernel():
    """A pass of the global kernel counts nothing, whatever a tiled pass left."""
    import torch
    import paper_1211_4575_gb300 as pp
    L = pp_synth.random_particles(N, (0.5, 0.5, 0.5), 0.2, 4000, seed=77, u_scale=3.0, w=1e-12)
    for graphs in (False, True):
        stream = torch.cuda.Stream()
        sim = pp.Simulation(L.n, L.d, L.dt, shape_order=3, precision=pp.PP_MIXED32, sort_interval=0,
                            deposit_mode=pp.PP_DEPOSIT_TILED,
                            relax_tol=1e-6, stream=stream.cuda_stream)
        for s in L.species:
            sid = sim.add_species(s["q"], s["m"], s["w"], len(s["x"]))
            sim.load_particles(sid, s["x"], s["y"], s["z"], s["ux"], s["uy"], s["uz"])
        sim.set_graphs(graphs)
        sim.step(14)
        assert sim.diagnostics()["n_slow"] > 100
        sim.set_tuning(0, pp.PP_DEPOSIT_GLOBAL)
        for _ in range(4):
            sim.step(1)
            assert sim.diagnostics()["n_slow"] == 0
