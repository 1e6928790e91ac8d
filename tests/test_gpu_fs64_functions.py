"""The FP64 kernels' functions as compiled for the GPU (reciprocal, 1 - e^-u, e^-u,
interval functions) and the float-float reciprocal, on arrays against mpmath, to
their stated bounds."""
import ctypes
import os
import subprocess

import mpmath
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROBE = r"""
#include "fs64_step.cuh"
#include "ff.cuh"
using namespace rt3d;
__global__ void probe(int n, const double *x, double *out) {
    __shared__ unsigned long long tab[64];
    exp_table(tab);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double u = x[i];
    const bool in = u >= 0.5 && u < 37.5;
    out[i] = recip64(u);
    out[n + i] = in ? one_minus_exp64(u, tab) : 0.0;
    out[2 * n + i] = in ? exp_neg64(u, tab) : 0.0;
    const IntervalDE f = interval64<false>(u, 0.0, tab);
    out[3 * n + i] = f.e0;
    out[4 * n + i] = f.a;
    out[5 * n + i] = f.d;
    const IntervalD w = interval64_w(u, tab);
    out[6 * n + i] = w.E;
    out[7 * n + i] = w.a0;
    out[8 * n + i] = w.a;
    out[9 * n + i] = w.d;
    out[10 * n + i] = ff_to_double(ff_recip(ff_split(u)));
}
extern "C" int run(int n, const double *x, double *out) {
    probe<<<(n + 127) / 128, 128>>>(n, x, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2102_01734_gb300 import build

    d = tmp_path_factory.mktemp("probe")
    cu, so = str(d / "probe.cu"), str(d / "probe.so")
    with open(cu, "w") as f:
        f.write(PROBE)
    subprocess.run([build.nvcc(), *build._flags(["-I", build.SRC_DIR]), "-shared", "-o", so, cu], check=True)
    lib = ctypes.CDLL(so)

    def call(x):
        t = torch.from_numpy(x).to("cuda")
        out = torch.empty((11, len(x)), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.run(len(x), ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(out.data_ptr())) == 0
        return out.cpu().numpy()

    return call


def _err(got, exact, scale=None):
    """Largest error in units of 2^-53 of scale (or of the value)."""
    scale = exact if scale is None else scale
    with mpmath.workdps(60):
        return max(float(abs(mpmath.mpf(float(g)) - e) / abs(s)) for g, e, s in zip(got, exact, scale)) * 2.0 ** 53


def test_reciprocal(run):
    rng = np.random.default_rng(5)
    x = np.concatenate([rng.uniform(1, 2, 3000), 2.0 ** rng.uniform(-1021, 1020, 3000), 2.0 ** np.arange(-1021, 1021),
                        np.nextafter(2.0 ** np.arange(-1020, 1021), 0), [2.0 ** 1021, 1e308, 2.0 ** -1022, 1e-310]])
    out = run(x)
    with mpmath.workdps(60):
        exact = [1 / mpmath.mpf(float(v)) for v in x]
        ulp = np.array([float(abs(mpmath.mpf(float(g)) - e)) for g, e in zip(out[0][:-4], exact)])
    # units in the last place of the result, a normal number
    assert np.max(ulp / np.spacing(1.0 / x[:-4])) < 0.52
    with np.errstate(all="ignore"):
        edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 2.0 ** 1021, 1.7e308])
        assert np.array_equal(run(edge)[0], 1.0 / edge, equal_nan=True)
    f32 = (x > 2.0 ** -100) & (x < 2.0 ** 100)
    assert _err(out[10][f32], [e for e, k in zip(exact, f32) if k]) < 8 * 2.0 ** 5  # 2^-48 units


def test_exponentials(run):
    rng = np.random.default_rng(6)
    ties = (np.arange(47, 3462) + 0.5) * np.log(2) / 64
    u = np.concatenate([[0.5, np.nextafter(37.5, 0)], rng.uniform(0.5, 37.5, 4000), rng.uniform(0.5, 1.0, 1000), ties])
    u = u[(u >= 0.5) & (u < 37.5)]
    out = run(u)
    with mpmath.workdps(60):
        E = [mpmath.exp(-mpmath.mpf(float(v))) for v in u]
    # the table's rounding (2^-54), the series' cut (r^6/720 < 0.31 2^-53, times
    # e^-u <= 0.607) and the last rounding (2^-55 below 1/2), over 1 - e^-u >= 0.393
    assert _err(out[1], [1 - e for e in E]) < 2.4
    # the table's rounding and the last one, each up to 2^-53 of the value, and the cut
    assert _err(out[2], E) < 2.4


def test_intervals(run):
    rng = np.random.default_rng(7)
    u = np.concatenate([10.0 ** rng.uniform(-17, 0, 3000), 10.0 ** rng.uniform(-290, -17, 200), rng.uniform(0.4, 0.6, 1000),
                        [0.5, np.nextafter(0.5, 0), 37.5, np.nextafter(37.5, 0), 1.0, 40.0, 700.0, 800.0, 1e5],
                        10.0 ** rng.uniform(0, 3, 1000)])
    out = run(u)
    with mpmath.workdps(700):  # 1 - (1 - e^-u)/u cancels to u/2
        U = [mpmath.mpf(float(v)) for v in u]
        e0 = [-mpmath.expm1(-v) for v in U]
        a = [1 - e / v for e, v in zip(e0, U)]
        d = [(2 * p - e) / v for p, e, v in zip(a, e0, U)]
        E = [mpmath.exp(-v) for v in U]
        a0 = [e - p for e, p in zip(e0, a)]
    # in 2^-53, where they are largest, at u = 1/2: e0 = 0.393 is good to 0.94 (2.4 of
    # itself), 1/u to 1.04; a = 1 - e0/u = 0.213 to 0.94 2 + 0.41 and its rounding 0.13;
    # d = (2a - e0)/u to (2 2.4 + 0.94) 2. With e^-u (good to 1.2 there) in place of e0:
    # a 2.9, d (2 2.9 + 1.2) 2, a0 = (1 - (1 + u) e^-u)/u = 0.18 (0.6 + 1.5 1.2) 2
    bounds = {3: (e0, e0, 2.4), 4: (a, a, 11.4), 5: (d, a, 54.0), 8: (a, a, 13.7), 9: (d, a, 66.0),
              7: (a0, a0, 27.0)}
    for k, (exact, scale, bound) in bounds.items():
        err = _err(out[k], exact, scale)
        assert err < bound, (k, err)
    assert _err(out[6][u < 700], [e for e, v in zip(E, u) if v < 700]) < 2.4
    zero = run(np.array([0.0]))[:, 0]
    assert np.all(zero[[3, 4, 5, 7, 8, 9]] == 0.0) and zero[6] == 1.0


def test_smallest(run):
    """Down to the subnormals e0 = u and a = u/2, to the last unit."""
    u = np.concatenate([2.0 ** -np.arange(1015.0, 1075.0), np.random.default_rng(8).uniform(0, 1e-307, 500),
                        [2.2250738585072014e-308, 2.225073858507201e-308, 4.45e-308]])
    out = run(u)
    assert np.array_equal(out[3], u)
    for k in (4, 8):
        assert np.all(np.abs(out[k] - 0.5 * u) <= 5e-324)
