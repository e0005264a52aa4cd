"""The field update at the sizes where its kernels change form, against the FP64
oracle: all sweeps of a component in one thread-block cluster on small meshes
(its z slabs uneven, a slab of one plane, the largest mesh it takes and the
next), a launch per sweep above them and for fewer planes than the cluster has
CTAs, one and two nodes per thread (odd and even x).

Tolerances: both solve (1 - kappa lap) B = R to tol |R|; the operator's
eigenvalues lie in [1, 1 + kappa 12 sum 1/h^2 (1.2)], so a relative residual tol is an
error of at most tol |R|_2 / |B|_inf: 1e-12 of the largest value at tol 1e-14 in
FP64.  FP32: 1e-6 is the tolerance asked for, and the rounding of the
sweeps and stencils adds some 6e-8 times the operator's condition (below 10
here): the 3e-5 of the mixed parity tests has room for both.
"""
import pytest

import pp_synth
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

CASES = [("fp64", (8, 8, 16)), ("fp64", (17, 16, 18)), ("fp64", (18, 18, 18)), ("fp64", (20, 20, 20)),
         ("fp64", (16, 16, 15)), ("mixed", (8, 9, 16)), ("mixed", (33, 17, 31)), ("mixed", (40, 41, 42)),
         ("mixed", (42, 41, 41)), ("mixed", (64, 64, 15))]


@pytest.mark.parametrize("prec,n", CASES, ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
def test_field_update_matches_oracle(prec, n):
    import paper_1211_4575_gb300 as pp
    import oracle
    L = pp_synth.random_particles(n, (0.5, 0.4, 0.45), 0.25, 500, seed=n[0], w=0.02)
    E, B = pp_synth.random_fields(n, 3, 0.05)
    sim = H.gpu_sim(pp, L, pp.PP_FP64 if prec == "fp64" else pp.PP_MIXED32, 3)
    orc = H.oracle_sim(oracle, L, 3)
    sim.load_fields(E, B)
    orc.load_fields(E, B)
    steps = 2
    sim.step(steps)
    orc.step(steps)
    tol = 1e-12 if prec == "fp64" else 3e-5
    for name, err in H.field_errors(sim, orc).items():
        assert err <= steps * tol, (name, err)
    assert sim.diagnostics()["status"] == 0
