"""Cases of the two particle kernels that sort in every step, run through the
library twice by tests/test_gpu_checked_sorted.py: once with the normal build
and once, in a child process with PP_GB300_CHECKED=1, with the bounds-checked
build.  Prints one JSON line: per case the status of the last diagnostics, the
particle launches of a step and the fields (E and B flattened)."""
import json
import sys

import numpy as np

import pp_synth

# name -> mesh, shape order, particles, walls
CASES = {
    "rows_9x10x11_cic": ((9, 10, 11), 1, 60000, ""),
    "rows_9x10x11_tsc": ((9, 10, 11), 2, 40000, ""),
    "rows_9x10x11_pcs": ((9, 10, 11), 3, 40000, ""),
    "rows_33x17x31_tsc": ((33, 17, 31), 2, 145000, ""),
    "rows_33x17x31_pcs": ((33, 17, 31), 3, 80000, ""),
    "rows_43x37x26_pcs": ((43, 37, 26), 3, 120000, ""),
    "rows_walls_x": ((10, 9, 12), 3, 40000, "x"),
    "rows_walls_xyz": ((5, 6, 9), 3, 40000, "xyz"),
    "tiles_16_cic": ((16, 16, 16), 1, 30000, ""),
    "tiles_16_tsc": ((16, 16, 16), 2, 30000, ""),
    "tiles_16_pcs": ((16, 16, 16), 3, 30000, ""),
    "tiles_walls_xyz": ((8, 4, 8), 3, 20000, "xyz"),
    "tiles_dense": ((8, 8, 8), 2, 30000, ""),      # more than one chunk of 4096
}


def run_cases():
    import paper_1211_4575_gb300 as pp
    from tests import gpu_helpers as H
    out = {}
    for name, (n, shape, count, walls) in CASES.items():
        L = pp_synth.random_particles(n, (0.5, 0.5, 0.5), 0.45, count, seed=91, u_scale=2.0, w=0.002)
        s = L.species[0]
        k = count // 3
        L.species = [{a: v[k:].copy() if isinstance(v, np.ndarray) else v for a, v in s.items()},
                     {a: v[:k].copy() if isinstance(v, np.ndarray) else v for a, v in s.items()}]
        sim = H.gpu_sim(pp, L, pp.PP_MIXED32, shape, capacity_extra=2000,
                        **{f"boundary_{a}": pp.PP_BOUNDARY_WALLS for a in walls})
        mesh = tuple(2 * n[a] if "xyz"[a] in walls else n[a] for a in range(3))
        sim.load_fields(*pp_synth.random_fields(mesh, 4, 0.05))
        if walls == "x":
            sim.set_open_boundary(4, 0.2, 1.5)
            sim.set_injector(0, 1.0, (0.8, 0.0, 0.0), 0.1, 5)
            sim.set_sliding_window(0.5)
        sim.step(3)
        E, B, _ = sim.fields()
        fields = np.concatenate([a.ravel() for a in E + B]).tolist()
        status = sim.diagnostics()["status"]
        sim.profile_enable(True)
        sim.step(1)
        launches = sim.profile_read()["particle_launches"]
        out[name] = (status, launches, fields)
    return out


if __name__ == "__main__":
    sys.path.insert(0, sys.argv[1])
    print(json.dumps(run_cases()))
