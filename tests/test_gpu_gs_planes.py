"""The OS sweeps where their split changes: solves whose coefficients stay in
shared memory (from one block on, the last ones that fit and the first that do
not), and above them the Gauss-Seidel plane kernel with one block to eight per
plane, or the Jacobi sweep with less than one block a warp to many, odd and even
axes, flat and tall boxes; Jacobi and Gauss-Seidel, both precisions."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(4, 4, 1), (5, 4, 2), (6, 37, 3), (33, 70, 9), (4, 6, 130), (64, 64, 38),
                               (65, 65, 65), (68, 65, 71), (130, 5, 600), (65, 80, 70), (70, 300, 18),
                               (300, 70, 18), (512, 513, 2), (5, 5, 521)])
@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("gs", [True, False])
def test_against_oracle(n, fp64, gs):
    from paper_2102_01734_gb300 import rt3d

    nx, ny, nz = n
    rng = np.random.default_rng(nx + ny + nz)
    N = nx * ny * nz
    L = rng.uniform(0.0, 1.0, (N, 27))
    L *= 0.9 / L.sum(1, keepdims=True)
    z = np.arange(N) // (nx * ny)
    L[z == 0, :9] = 0.0
    L[z == nz - 1, 18:] = 0.0
    eps = 10.0 ** rng.uniform(-4, -1, (nz, ny, nx))
    r = rng.standard_normal((nz, ny, nx))
    g = rt3d.Grid(n, 2, 4, rt3d.LINEAR, rt3d.FP64 if fp64 else rt3d.FP32_FS_FP64_ALI)
    g.set_os_solver(rt3d.OS_GAUSS_SEIDEL if gs else rt3d.OS_JACOBI)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    for sweeps in (1, 6):
        if gs:
            ref, m = oracle.os_gauss_seidel(L, eps, r, sweeps, 1e-14, colored=True)
        else:
            ref, m = oracle.os_jacobi(L, eps, r, sweeps, 1e-14)
        x, k = g.os_solve(d(L.T), d(eps), d(r), max_sweeps=sweeps, tol=1e-14)
        x = x.cpu().numpy()
        assert k == m == sweeps
        assert np.all(np.isfinite(x))
        # FP32 mode: coefficients and neighbours rounded to 2^-24; the rows sum
        # to at most 0.9, so sweeps damp the errors they inherit
        tol = 1e-13 if fp64 else 2 * 27 * 2.0 ** -24 / (1 - 0.9)
        assert np.max(np.abs(x - ref.reshape(x.shape))) <= tol * np.max(np.abs(ref))
    # a stop test that is met on the way
    ref, m = (oracle.os_gauss_seidel(L, eps, r, 50, 0.05, colored=True) if gs
              else oracle.os_jacobi(L, eps, r, 50, 0.05))
    x, k = g.os_solve(d(L.T), d(eps), d(r), max_sweeps=50, tol=0.05)
    assert k == m < 50
    g.close()
