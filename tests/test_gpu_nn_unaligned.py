"""Convolutions and weight gradients of BF16 arrays at any address: small whole
numbers, whose sums are exact in FP32 in every order, give the same bits from
arrays that start on a 16-byte boundary and from arrays one element past it."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _shifted(x):
    raw = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)
    raw[1:] = x.flatten()
    return raw[1:].view(x.shape)


@pytest.mark.parametrize("S,shape,ci,co", [(2, (3, 5, 9), 16, 16), (1, (4, 9, 18), 48, 32), (1, (5, 7, 6), 32, 48),
                                           (1, (65, 35, 36), 16, 16)])
def test_same_bits(S, shape, ci, co):
    from paper_2102_01734_gb300 import warmstart as ws

    lib = ws._lib()
    g = torch.Generator(device="cuda").manual_seed(ci + co)
    whole = lambda *s: torch.randint(-3, 4, s, generator=g, device="cuda").to(torch.bfloat16)
    nz, ny, nx = shape
    X, W, dY = whole(S, *shape, ci), whole(27, ci, co), whole(S, *shape, co)
    out = []
    for x, w, d in [(X, W, dY), (_shifted(X), W, dY), (X, _shifted(W), _shifted(dY)),
                    (_shifted(X), _shifted(W), _shifted(dY))]:
        Yf = torch.empty(S, *shape, co, device="cuda")
        dW, db = torch.zeros(27, ci, co, device="cuda"), torch.zeros(co, device="cuda")
        ws._ck(lib.rt3d_nn_conv3d(x.data_ptr(), w.data_ptr(), None, None, Yf.data_ptr(), S, nx, ny, nz, ci, co, 0, 0,
                                  None))
        ws._ck(lib.rt3d_nn_conv3d_wgrad(x.data_ptr(), d.data_ptr(), dW.data_ptr(), db.data_ptr(), S, nx, ny, nz, ci,
                                        co, None))
        out.append((Yf, dW, db))
    for other in out[1:]:
        assert all(torch.equal(p, q) for p, q in zip(out[0], other))
    assert out[0][0].abs().max() > 0
