"""The FP32 push over the whole range of a float: the three helpers that stand
for 1/sqrt, sqrt and 1/x against FP64, and a step of particles in uniform B
against the oracle's push, at momenta whose squares reach the largest float
(Vay) and at rotation vectors whose squares do (Boris).

Tolerances.  Helpers: one ulp of the exact value, the error they claim.  Push:
about 30 dependent FP32 operations of at most one ulp each (2^-23), 3.6e-6, and
a gather whose weights sum to 1 to a few 1e-7: 1e-5 of |u|.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pp_internal.cuh"
__global__ void k_eval(int which, const float *in, float *out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float x = in[i];
    out[i] = which == 0 ? pp::inv_sqrt(x) : (which == 1 ? pp::fast_sqrt(x) : pp::inv(x));
}
extern "C" int eval(int which, const float *in, float *out, int n) {
    float *a = nullptr, *b = nullptr;
    int e = cudaMalloc(&a, sizeof(float) * n);
    if (!e) e = cudaMalloc(&b, sizeof(float) * n);
    if (!e) e = cudaMemcpy(a, in, sizeof(float) * n, cudaMemcpyHostToDevice);
    if (!e) {
        k_eval<<<(n + 255) / 256, 256>>>(which, a, b, n);
        e = cudaGetLastError();
    }
    if (!e) e = cudaMemcpy(out, b, sizeof(float) * n, cudaMemcpyDeviceToHost);
    cudaFree(a);
    cudaFree(b);
    return e;
}
"""


@pytest.fixture(scope="module")
def helpers(tmp_path_factory):
    from paper_1211_4575_gb300 import build
    d = tmp_path_factory.mktemp("helpers")
    src, so = str(d / "helpers.cu"), str(d / "helpers.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    inc = os.path.join(os.path.dirname(build.HERE), "include")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-I", inc, "-shared", "-o", so, src],
                   check=True, capture_output=True, text=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("which,exact", [(0, lambda x: 1 / np.sqrt(x)), (1, np.sqrt), (2, lambda x: 1 / x)],
                         ids=["inv_sqrt", "fast_sqrt", "inv"])
def test_helpers_within_an_ulp_over_the_whole_range(helpers, which, exact):
    big = np.float32(np.finfo(np.float32).max)
    rng = np.random.default_rng(3)
    x = np.concatenate([2.0 ** rng.uniform(0, 128, 200000), rng.uniform(1, 4, 50000), rng.uniform(2.9e38, 3.4028e38, 2000),
                        rng.uniform(7.9e37, 1.1e38, 2000), 2.0 ** np.arange(128), [1.0, big]]).astype(np.float32)
    x = np.minimum(x, big)
    out = np.zeros_like(x)
    p = ctypes.POINTER(ctypes.c_float)
    assert helpers.eval(which, x.ctypes.data_as(p), out.ctypes.data_as(p), len(x)) == 0
    ref = exact(x.astype(np.float64))
    ulp = np.spacing(ref.astype(np.float32)).astype(np.float64)   # 2^-149 among the subnormals
    err = np.abs(out.astype(np.float64) - ref) / ulp
    assert err.max() < 1.0, (x[err.argmax()], out[err.argmax()], ref[err.argmax()])
    inf = np.array([np.inf], dtype=np.float32)
    out = np.zeros(1, dtype=np.float32)
    assert helpers.eval(which, inf.ctypes.data_as(p), out.ctypes.data_as(p), 1) == 0
    assert out[0] == (np.inf if which == 1 else 0.0)


def _step(pp, n, mode, pusher, Bz, u):
    """One step of particles with u along x in B along z; their z never changes and tells them apart."""
    h, dt = 0.5, 0.25
    k = len(u)
    sim = pp.Simulation(n, (h, h, h), dt, shape_order=3, pusher=pusher, precision=pp.PP_MIXED32, deposit_mode=mode,
                        relax_tol=1e-6)
    rng = np.random.default_rng(11)
    sid = sim.add_species(-1.0, 1.0, 1e-30, k)
    z = (np.arange(k) + 0.5) / k * n[2] * h
    sim.load_particles(sid, rng.random(k) * n[0] * h, rng.random(k) * n[1] * h, z, u, np.zeros(k), np.zeros(k))
    # particles at rest without charge, so that the mesh is loaded as a plasma's
    m = 12 * n[0] * n[1] * n[2]
    rest = sim.add_species(0.0, 1.0, 1e-30, m)
    x = rng.random((3, m)) * np.array(n)[:, None] * h
    sim.load_particles(rest, *x, np.zeros(m), np.zeros(m), np.zeros(m))
    shape = n[::-1]
    sim.load_fields([np.zeros(shape)] * 3, [np.zeros(shape), np.zeros(shape), np.full(shape, Bz)])
    sim.step(1)
    sim.sync()
    p = sim.particles(sid)
    order = np.argsort(p["z"])
    return np.stack([p[a][order] for a in ("ux", "uy", "uz")], 1), dt


@pytest.mark.parametrize("n,mode", [((16, 16, 16), 0), ((9, 10, 11), 0), ((9, 10, 11), 1)],
                         ids=["tiles", "rows", "global"])
@pytest.mark.parametrize("pusher,tau,u", [
    ("vay", 0.3, 10.0 ** np.linspace(-2, 2, 40)),
    ("vay", 1e9, np.concatenate([10.0 ** np.linspace(9, 9.6, 20), np.linspace(4.1e9, 4.28e9, 60)])),
    ("boris", 0.3, 10.0 ** np.linspace(-2, 2, 40)),
    ("boris", 1e9, 10.0 ** np.linspace(7, 9.6, 20)),
    ("boris", 1.0e19, np.linspace(0.1, 0.9, 16)),
    ("boris", 1.7e19, np.linspace(0.01, 0.2, 16)),
], ids=["vay", "vay-large", "boris", "boris-large", "boris-fast", "boris-fastest"])
def test_push_matches_oracle_up_to_the_largest_float(n, mode, pusher, tau, u):
    import oracle
    import paper_1211_4575_gb300 as pp
    Bz = -tau / 0.125                 # tau = q dt B / (2 m)
    got, dt = _step(pp, n, mode, pp.PP_VAY if pusher == "vay" else pp.PP_BORIS, Bz, u)
    for k, uk in enumerate(u):
        ref = np.array([float(np.float32(uk)), 0.0, 0.0])
        ref = oracle.push(-dt, (0.0, 0.0, 0.0), (0.0, 0.0, float(np.float32(Bz))), ref,
                          oracle.VAY if pusher == "vay" else oracle.BORIS)
        assert np.abs(got[k] - ref).max() <= 1e-5 * np.linalg.norm(ref), (uk, got[k], ref)
