"""FP32 formal solutions with the parabolic source of nearly transparent boxes
and shells, against FP64: the parabola's ratios of neighbouring optical depths
do not depend on their size, down to the smallest normal numbers. A weight is
good to a few FP32 roundings (6e-8 each), and the intensities add up positive
terms, at most 30 of them here."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEPTHS = [1e-10, 1e-16, 1e-22, 1e-28]


def _d(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _atmosphere(shape, depth):
    rng = np.random.default_rng(7)
    return depth * rng.uniform(0.3, 1.0, shape), rng.uniform(0.1, 1.0, shape)


@pytest.mark.parametrize("depth", DEPTHS)
def test_one_characteristic_a_thread(depth):
    from paper_2102_01734_gb300 import rt3d

    chi, S = _atmosphere((8, 9, 7), depth)
    Jo, _ = oracle.fs_cart(chi, S, 4, 6, True, None, lstar=True)
    g = rt3d.Grid((7, 9, 8), 4, 6, rt3d.PARABOLIC, rt3d.FP32_FS_FP64_ALI)
    g.set_fs_shape((128, 1, 1, 1))
    J = g.formal_solution(_d(chi), _d(S), None).cpu().numpy()
    g.close()
    assert np.max(np.abs(J / Jo - 1)) < 4e-6


@pytest.mark.parametrize("depth", DEPTHS)
def test_shell(depth):
    from paper_2102_01734_gb300 import rt3d

    n = (12, 9, 12)
    chi, S = _atmosphere(n[::-1], depth)
    out = {}
    for precision in (rt3d.FP64, rt3d.FP32_FS_FP64_ALI):
        g = rt3d.Grid(n, 4, 8, rt3d.PARABOLIC, precision, geometry=rt3d.SPHERICAL)
        out[precision] = g.formal_solution(_d(chi), _d(S), None)
        g.close()
    Jo, J = out[rt3d.FP64], out[rt3d.FP32_FS_FP64_ALI]
    assert ((J / Jo - 1).abs()).max() < 4e-6


@pytest.mark.parametrize("angles", [(4, 8), (64, 128)])  # the last: four characteristics a thread
@pytest.mark.parametrize("depth", DEPTHS)
def test_band(depth, angles):
    from paper_2102_01734_gb300 import rt3d

    n = (34, 7, 9)
    chi, S = _atmosphere(n[::-1], depth)
    out = {}
    for precision in (rt3d.FP64, rt3d.FP32_FS_FP64_ALI):
        g = rt3d.Grid(n, *angles, rt3d.PARABOLIC, precision)
        before = g.info()["device_bytes"]
        out[precision] = g.formal_solution(_d(chi), _d(S), None, lstar=True)
        if precision == rt3d.FP32_FS_FP64_ALI:  # the exchanged planes say which kernel ran
            N = n[0] * n[1] * n[2]
            assert g.info()["device_bytes"] - before == (320 * N if angles[0] == 64 else 0)
        g.close()
    (Jo, Lo), (J, L) = out[rt3d.FP64], out[rt3d.FP32_FS_FP64_ALI]
    assert ((J / Jo - 1).abs()).max() < 4e-6
    assert (L - Lo).norm() < 1e-6 * Lo.norm()
