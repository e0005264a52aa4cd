"""The row kernel (mixed form, automatic deposit on meshes that 8^3 tiles do not
divide) against the FP64 oracle in every form it has: blocks of one, two and
four planes of cells for every shape order, with warps that take several
batches of 32 particles and cells that hold long runs; two species; the Boris
push, radiative cooling, the 4th-order step (whose first substep only drifts)
and a species without charge; walls on one and on all axes, the open end with
injectors, and the sliding window.  Each case asserts that this kernel ran.

The particles are fast and a step is up to 0.9 cells long at the speed of
light, so that most of them change their support on one, two or three axes.

Tolerances, per step (a 4th-order step has four), are those of the other mixed
parity tests: fields 3e-5 of the largest value, positions 2e-6 (physical
units), momenta 2e-6 relative, twice that with cooling.
"""
import numpy as np
import pytest

import pp_synth
from tests import gpu_helpers as H
from tests import test_gpu_walls as walls_tests

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pp():
    import paper_1211_4575_gb300 as m
    return m


def _assert_rows(sim):
    """Two species (or one) in one launch, after a sort in the same step."""
    sim.profile_enable(True)
    sim.step(2)
    p = sim.profile_read()
    sim.profile_enable(False)
    assert p["particle_launches"] == p["steps"] and p["sort_ms"] > 0.0, p


def _load(n, count, seed, dt=0.45, u_scale=2.0, w=0.002, second=True):
    L = pp_synth.random_particles(n, (0.5, 0.5, 0.5), dt, count, seed=seed, u_scale=u_scale, w=w)
    if second:   # a second, smaller species of the opposite charge
        s = L.species[0]
        k = count // 3
        L.species = [{a: v[k:].copy() if isinstance(v, np.ndarray) else v for a, v in s.items()},
                     {a: v[:k].copy() if isinstance(v, np.ndarray) else v for a, v in s.items()}]
        L.species[1]["q"] = -s["q"]
    return L


def _compare(sim, orc, L, steps, tol_p=2e-6):
    for name, err in H.field_errors(sim, orc).items():
        assert err <= steps * 3e-5, (name, err)
    for s in range(len(L.species)):
        dpos, du = H.particle_errors(sim.particles(s), orc.species[s], H.box(L))
        assert dpos <= steps * tol_p and du <= steps * tol_p, (s, dpos, du)
    assert sim.diagnostics()["status"] == 0


# 8, 60 and 120 tiles: blocks of one, two and four planes; particles past the line of the choice
@pytest.mark.parametrize("n,shape,count", [((9, 10, 11), 1, 60000), ((9, 10, 11), 2, 40000), ((9, 10, 11), 3, 40000),
                                           ((33, 17, 31), 1, 560000), ((33, 17, 31), 2, 145000),
                                           ((33, 17, 31), 3, 80000), ((43, 37, 26), 1, 850000),
                                           ((43, 37, 26), 2, 245000), ((43, 37, 26), 3, 120000)])
def test_blocks_match_oracle(pp, orc, n, shape, count):
    steps = 1 if count > 300000 else 2
    L = _load(n, count, 17 + shape)
    E, B = pp_synth.random_fields(n, 3, 0.05)
    sim = H.gpu_sim(pp, L, pp.PP_MIXED32, shape)
    osim = H.oracle_sim(orc, L, shape)
    sim.load_fields(E, B)
    osim.load_fields(E, B)
    sim.step(steps)
    osim.step(steps)
    _compare(sim, osim, L, steps)
    _assert_rows(sim)


@pytest.mark.parametrize("shape", [1, 2, 3])
@pytest.mark.parametrize("form", ["boris", "cooling", "step4", "neutral"])
def test_forms_match_oracle(pp, orc, form, shape):
    n, dt = (9, 10, 11), (0.2 if form in ("cooling", "step4") else 0.45)
    L = _load(n, 50000, 40 + shape, dt=dt)
    if form == "neutral":
        L.species[1]["q"] = 0.0
    E, B = pp_synth.random_fields(n, 5, 0.05)
    if form == "cooling":
        B[2] = B[2] + 2.0
    K = 0.005 if form == "cooling" else 0.0
    pusher = 1 if form == "boris" else 0
    sim = H.gpu_sim(pp, L, pp.PP_MIXED32, shape, pusher=pusher)
    osim = orc.Simulation(L.n, L.d, L.dt, shape_order=shape, pusher=pusher, relax_tol=1e-14, relax_max_iter=2000,
                          integrator=4 if form == "step4" else 2)
    for sid, s in enumerate(L.species):
        osim.add_species(s["q"], s["m"], s["w"], s["x"], s["y"], s["z"], s["ux"], s["uy"], s["uz"], rad=K)
        sim.set_radiative_cooling(sid, K)
    if form == "step4":
        sim.set_integrator(4)
    sim.load_fields(E, B)
    osim.load_fields(E, B)
    sim.step(2)
    osim.step(2)
    _compare(sim, osim, L, 8 if form == "step4" else 2, 4e-6 if form == "cooling" else 2e-6)
    _assert_rows(sim)


@pytest.mark.parametrize("walls", [(True, False, False), (False, False, True), (True, True, True)])
@pytest.mark.parametrize("shape", [1, 2, 3])
def test_walls_match_oracle(pp, orc, shape, walls):
    n = (10, 9, 12) if walls[0] else (9, 10, 11)
    cells = int(np.prod([2 * n[a] if walls[a] else n[a] for a in range(3)]))
    count = {1: 48, 2: 8, 3: 8}[shape] * min(cells, 4096) + 1000
    L = walls_tests._load(n, count, seed=200 + shape)
    L.species[0]["w"] = 0.002
    gpu, osim = walls_tests._pair(pp, orc, L, pp.PP_MIXED32, shape, walls=walls)
    gpu.step(3)
    osim.step(3)
    walls_tests._compare(gpu, osim, L, 9e-5, 6e-6, 6e-6, walls)
    _assert_rows(gpu)


@pytest.mark.parametrize("window", [0.0, 0.6], ids=["open-end", "window"])
def test_open_end_injectors_and_window_match_oracle(pp, orc, window):
    """The injected particles join the sort; those that leave through the open
    end take the key after every cell's and are dropped."""
    steps = 10
    L = walls_tests._load((10, 9, 12), 40000, seed=220)
    L.species[0]["w"] = 0.002
    gpu, osim = walls_tests._boundary_pair(pp, orc, L, pp.PP_MIXED32, window=window, steps=steps)
    assert osim.counts[1] > 0 and osim.counts[0] != 40000
    if window:
        assert osim.shifts >= 2
    walls_tests._compare_all(gpu, osim, L, 2, steps * 3e-5, steps * 2e-6, steps * 2e-6)
    _assert_rows(gpu)
