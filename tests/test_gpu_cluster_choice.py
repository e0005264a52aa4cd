"""Which form the Chebyshev sweeps of the field update take, told by the kernels
a step launches, and the meshes near the line against the FP64 oracle.

The line lies where both forms take the same time, decided by the heaviest
CTA of the cluster: meshes of equal node count fall on both sides of it.
Tolerances as in test_gpu_mesh_solve.py: per step 1e-12 (FP64) and 3e-5 (mixed)
of the largest value.
"""
import pytest

import pp_synth
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

# (precision, mesh, one cluster per component)
CASES = [
    ("fp64", (16, 16, 16), True), ("fp64", (24, 16, 16), True), ("fp64", (24, 24, 16), True),
    ("fp64", (9, 9, 64), True), ("fp64", (17, 17, 17), True),
    ("fp64", (8, 8, 64), False), ("fp64", (12, 12, 48), False), ("fp64", (16, 20, 17), False), ("fp64", (28, 24, 16), False),
    ("fp64", (23, 23, 16), False), ("fp64", (16, 16, 15), False),
    ("mixed", (32, 32, 32), True), ("mixed", (41, 41, 41), True), ("mixed", (48, 48, 48), True),
    ("mixed", (24, 24, 200), True), ("mixed", (48, 48, 16), True),
    ("mixed", (64, 64, 16), False), ("mixed", (64, 64, 17), False), ("mixed", (52, 54, 17), False),
    ("mixed", (61, 61, 16), False), ("mixed", (63, 47, 33), False), ("mixed", (7, 32, 32), False),
]


@pytest.mark.parametrize("prec,n,cluster", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_form_and_result(prec, n, cluster):
    import paper_1211_4575_gb300 as pp
    import oracle
    L = pp_synth.random_particles(n, (0.5, 0.4, 0.45), 0.25, 300, seed=n[0], w=0.02)
    E, B = pp_synth.random_fields(n, 3, 0.05)
    sim = H.gpu_sim(pp, L, pp.PP_FP64 if prec == "fp64" else pp.PP_MIXED32, 3)
    orc = H.oracle_sim(oracle, L, 3)
    sim.load_fields(E, B)
    orc.load_fields(E, B)
    sim.step(1)
    orc.step(1)
    tol = 1e-12 if prec == "fp64" else 3e-5
    for name, err in H.field_errors(sim, orc).items():
        assert err <= tol, (name, err)
    sweeps = sim.diagnostics()["relax_iters"]
    assert sweeps > 8
    sim.profile_enable(True)
    sim.deposit()
    sim.sync()
    before = sim.profile_read()["kernel_launches"]
    sim.field_update()
    launches = sim.profile_read()["kernel_launches"] - before
    # right-hand side, E update, and the sweeps: one launch or one each
    assert launches == (3 if cluster else 2 + sweeps), (launches, sweeps)
