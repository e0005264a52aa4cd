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


def _counts(pp, graphs, steps, sort_interval, current, solver, filter_interval=0):
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
    if filter_interval:
        sim.set_divergence_filter(1, filter_interval)
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


def test_periodic_sorts_go_on_in_replayed_steps():
    """A sort every 4 steps for 24 steps: a replay of a step without a sort
    does not set the count of steps since the last sort back, so the sorts keep
    their interval and the particles outside their tiles stay as few as in the
    eager run."""
    import paper_1211_4575_gb300 as pp
    cur, sol = pp.PP_CURRENT_DIRECT, pp.PP_FIELD_EXPLICIT
    eager, _ = _counts(pp, False, 24, 4, cur, sol)
    graph, (cap, rep) = _counts(pp, True, 24, 4, cur, sol)
    unsorted, _ = _counts(pp, False, 24, 0, cur, sol)
    assert rep >= 8, (cap, rep)
    assert unsorted[-1] > 10 * max(1, eager[-1])   # the counts tell the sorts apart
    assert graph == eager


def test_captures_of_a_long_cycle_are_kept():
    """Tiled, a sort every 4 and a filter every 3 steps: the run cycles through
    12 states (current array, particle buffer, sort, filter), and once all are
    captured every step is a replay."""
    import paper_1211_4575_gb300 as pp
    cur, sol = pp.PP_CURRENT_CONSERVING, pp.PP_FIELD_IMPLICIT
    eager, _ = _counts(pp, False, 48, 4, cur, sol, filter_interval=3)
    graph, (cap, rep) = _counts(pp, True, 48, 4, cur, sol, filter_interval=3)
    assert cap <= 16 and rep >= 32, (cap, rep)
    assert graph == eager
