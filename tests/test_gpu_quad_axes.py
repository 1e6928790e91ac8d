"""The four-characteristic formal solution on faces whose sides leave every
remainder modulo its four rows, longer along x or along y, single and several
layers: angles that step along x run with x and y exchanged."""
import numpy as np
import pytest

import oracle
from paper_2102_01734_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(4, 4, 1), (5, 9, 2), (9, 5, 2), (6, 35, 3), (35, 6, 3), (7, 33, 9), (34, 7, 9),
                               (33, 36, 5)])
@pytest.mark.parametrize("parabolic", [False, True])
def test_against_oracle(n, parabolic):
    from paper_2102_01734_gb300 import rt3d

    chi, eps, B, bc = inputs.cartesian_config(n, 1e-2, seed=3)
    rng = np.random.default_rng(sum(n))
    chi = chi * 10.0 ** rng.uniform(-1, 1, chi.shape)  # both sides of u = 1 within a warp
    S = B * rng.uniform(0.1, 1.0, B.shape)
    Jo, _ = oracle.fs_cart(chi, S, 6, 10, parabolic, bc, lstar=True)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    g = rt3d.Grid(n, 6, 10, rt3d.PARABOLIC if parabolic else rt3d.LINEAR, rt3d.FP32_FS_FP64_ALI)
    tbc = {"I_top": 0.3, "I_bottom": d(bc["I_bottom"])}
    Jo, _ = oracle.fs_cart(chi, S, 6, 10, parabolic, {"I_top": 0.3, "I_bottom": bc["I_bottom"]},
                           lstar=True)
    for shape in [(64, 4, 1, 1), (128, 4, 0, 1), (256, 4, 2, 0)]:
        g.set_fs_shape(shape)
        for _ in range(2):  # the accumulation buffers are left zeroed
            J = g.formal_solution(d(chi), d(S), tbc).cpu().numpy()
            assert np.max(np.abs(J - Jo) / np.abs(Jo)) < 2e-5, shape
    # the exchanged accumulation does not leak into another shape's result
    g.set_fs_shape((128, 1, 1, 1))
    J = g.formal_solution(d(chi), d(S), tbc).cpu().numpy()
    assert np.max(np.abs(J - Jo) / np.abs(Jo)) < 2e-5
    g.close()
