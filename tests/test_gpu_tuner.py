"""The FP32 autotuner's first call: every candidate on a short formal solution, on
a longer one not those that have no chance any more."""
import pytest

from paper_2102_01734_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,angles,ones,fours", [
    ((20, 18, 12), (4, 8), 4, 3), ((129, 97, 65), (16, 32), 1, 3), ((16, 43, 113), (8, 16), 4, 1)])
def test_candidates(n, angles, ones, fours):
    from paper_2102_01734_gb300 import rt3d

    chi, eps, B, bc = inputs.cartesian_config(n, 1e-2, seed=3)
    d = lambda a: torch.from_numpy(a.copy()).to("cuda")
    g = rt3d.Grid(n, *angles, rt3d.PARABOLIC, rt3d.FP32_FS_FP64_ALI)
    J = g.formal_solution(d(chi), d(B), {"I_bottom": d(bc["I_bottom"])})
    info = g.info()
    shapes = [rt3d.fs_tune_shape(i) for i in range(rt3d.FS_TUNE_SHAPES)]
    timed = {s: t for s, t in zip(shapes, info["fs_tune_ms"]) if t > 0}
    assert timed[info["fs_shape"]] == min(timed.values()) and shapes[0] in timed
    # the narrow box takes some 0.27 ms, with four characteristics a thread twice as
    # long; on the wide one these are 30 % ahead
    assert [sum(s[1] == k for s in timed) for k in (1, 2, 4)] == [ones, 1, fours]
    g.set_fs_shape(shapes[1])
    other = g.formal_solution(d(chi), d(B), {"I_bottom": d(bc["I_bottom"])})
    assert ((J - other).abs() / J).max() < 2e-6
    g.close()
