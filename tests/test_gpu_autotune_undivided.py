"""The autotuner on a mesh that 8^3 tiles do not divide: the automatic mode,
the only one that reaches the row kernel there, is among its candidates, and a
tuned run is as fast as an untuned one."""
import types

import pytest

import pp_synth
from tests import gpu_helpers as H


class _Sim:
    def __init__(self, n, precision, sort_interval=7):
        self.g = types.SimpleNamespace(nx=n[0], ny=n[1], nz=n[2], precision=precision, sort_interval=sort_interval)

    def grid(self):
        return self.g, 2


def test_candidates_hold_the_automatic_mode():
    import paper_1211_4575_gb300 as pp
    from paper_1211_4575_gb300 import autotune
    divided = autotune.candidates(_Sim((16, 24, 32), pp.PP_MIXED32))
    assert (1, pp.PP_DEPOSIT_CELLS) in divided and pp.PP_DEPOSIT_AUTO not in [m for _, m in divided]
    for n in ((60, 45, 37), (16, 24, 12), (4, 64, 64)):
        assert (7, pp.PP_DEPOSIT_AUTO) in autotune.candidates(_Sim(n, pp.PP_MIXED32))
    assert all(m == pp.PP_DEPOSIT_GLOBAL for _, m in autotune.candidates(_Sim((60, 45, 37), pp.PP_FP64)))


@pytest.mark.gpu
def test_tuned_run_is_as_fast_as_the_default():
    """36 x 45 x 37 cells x 32 PCS particles: the global kernel takes about six times as
    long as the row kernel with its sort, so a factor of 1.5 tells them apart."""
    import paper_1211_4575_gb300 as pp
    from paper_1211_4575_gb300 import autotune

    def ms_per_step(sim, steps=20):
        sim.step(2)
        sim.profile_enable(True)
        sim.step(steps)
        p = sim.profile_read()
        sim.profile_enable(False)
        return (p["particle_ms"] + p["sort_ms"]) / steps

    L = pp_synth.thermal(n=(36, 45, 37), ppc=16, u_th=0.1, dx=0.1, dt=0.05, seed=3)
    default = ms_per_step(H.gpu_sim(pp, L, pp.PP_MIXED32, 3))
    sim = H.gpu_sim(pp, L, pp.PP_MIXED32, 3)
    choice, timings = autotune.autotune(sim, use_cache=False)
    assert choice == (20, pp.PP_DEPOSIT_AUTO), timings
    assert ms_per_step(sim) <= 1.5 * default
