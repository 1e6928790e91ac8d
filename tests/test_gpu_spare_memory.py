"""Device memory that formal solutions can do without (the four-characteristic
kernels' buffers: 96 bytes a voxel, 224 more with Lambda*): held only while the
grid's shape or its Lambda* uses them (from 16 MB on), and not taken where memory
is short."""
import numpy as np
import pytest

from paper_2102_01734_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(n, angles):
    from paper_2102_01734_gb300 import rt3d

    chi, eps, B, bc = inputs.cartesian_config(n, 1e-2, seed=3)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    g = rt3d.Grid(n, *angles, rt3d.PARABOLIC, rt3d.FP32_FS_FP64_ALI)
    return g, (d(chi), d(B), {"I_top": 0.3, "I_bottom": d(bc["I_bottom"])})


@pytest.mark.parametrize("n", [(12, 10, 9), (57, 56, 57)])  # the last: 17 MB
def test_kept_while_in_use(n):
    g, args = _problem(n, (8, 16))
    N, base = n[0] * n[1] * n[2], g.info()["device_bytes"]
    small = 96 * N < 1 << 24
    J = g.formal_solution(*args)  # tunes the shape
    info = g.info()
    assert info["device_bytes"] - base == (96 * N if small or info["fs_shape"][1] == 4 else 0)
    for shape in [(64, 4, 1, 1), (128, 1, 1, 1), (64, 4, 1, 1), (128, 2, 1, 1)]:
        g.set_fs_shape(shape)
        assert ((g.formal_solution(*args) - J).abs() / J).max() < 2e-6, shape
        assert g.info()["device_bytes"] - base == (96 * N if small or shape[1] == 4 else 0), shape
    g.close()


def test_not_taken_where_memory_is_short():
    """Less free memory than the buffers and the solvers' vectors need, 1.5 GB above
    what the calls themselves take."""
    n = (129, 129, 129)
    g, args = _problem(n, (8, 16))
    N, base = n[0] * n[1] * n[2], g.info()["device_bytes"]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    left = 1700 * N  # < 96 N + 2048 N; 3.6 GB
    fill = torch.empty(max(0, torch.cuda.mem_get_info()[0] - left), dtype=torch.uint8, device="cuda")
    try:
        J = g.formal_solution(*args)
        Jl, _ = g.formal_solution(*args, lstar=True)
        info = g.info()
        assert info["device_bytes"] == base and info["fs_shape"][1] != 4
    finally:
        del fill
        torch.cuda.empty_cache()
    g.set_fs_shape(None)
    assert ((g.formal_solution(*args) - J).abs() / J).max() < 2e-6
    Jq, _ = g.formal_solution(*args, lstar=True)
    assert g.info()["device_bytes"] - base == 320 * N
    assert ((Jq - Jl).abs() / Jl).max() < 2e-6
    g.close()
