"""Lambda* from the four-characteristic FP32 kernel (enough angles that the
dispatch takes it, which the memory it holds then shows) on faces whose sides leave every remainder modulo its four
rows, longer along x or along y, against the FP64 kernel. A weight is good to a
few FP32 roundings (6e-8 each) and an entry averages over angles, so the planes
agree to 1e-7 of their norm."""
import numpy as np
import pytest

from paper_2102_01734_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,angles", [((9, 5, 2), (80, 168)), ((6, 35, 3), (44, 88)), ((34, 7, 9), (44, 88)),
                                      ((7, 33, 9), (44, 88)), ((33, 36, 5), (20, 40)), ((40, 33, 1), (20, 40))])
@pytest.mark.parametrize("parabolic", [False, True])
def test_against_fp64(n, angles, parabolic):
    from paper_2102_01734_gb300 import rt3d

    chi, eps, B, bc = inputs.cartesian_config(n, 1e-2, seed=3)
    rng = np.random.default_rng(sum(n))
    chi = chi * 10.0 ** rng.uniform(-1, 1, chi.shape)  # both sides of u = 1 within a warp
    S = B * rng.uniform(0.1, 1.0, B.shape)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    tbc = {"I_top": 0.3, "I_bottom": d(bc["I_bottom"])}
    order = rt3d.PARABOLIC if parabolic else rt3d.LINEAR
    g64 = rt3d.Grid(n, *angles, order, rt3d.FP64)
    J64, L64 = g64.formal_solution(d(chi), d(S), tbc, lstar=True)
    g64.close()
    g = rt3d.Grid(n, *angles, order, rt3d.FP32_FS_FP64_ALI)
    before = g.info()["device_bytes"]
    for _ in range(2):  # the exchanged planes are left zeroed
        J, L = g.formal_solution(d(chi), d(S), tbc, lstar=True)
        # 320 bytes a voxel that no other kernel takes: this one ran
        assert g.info()["device_bytes"] - before == 320 * n[0] * n[1] * n[2]
        assert ((J - J64).abs() / J64.abs()).max() < 2e-5
        assert (L - L64).norm() < 1e-7 * L64.norm()
        assert (L[L64 == 0].abs() < 1e-30).all()
    g.close()
