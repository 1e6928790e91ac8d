"""The warm start's convolution tiles and vector kernels at the sizes where
they change: volumes below and above the large tiles' threshold, edges past a
tile on every axis, several samples, pointers that rule out 16-byte accesses."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ws():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2102_01734_gb300 import warmstart
    return warmstart


def reference(X, W, b):
    """conv in FP64 (X [S][nz][ny][nx][Ci], W [27][Ci][Co]) by 27 shifts."""
    out = torch.zeros(X.shape[:4] + (W.shape[2],), dtype=torch.float64, device=X.device) + b
    for d in range(27):
        dz, dy, dx = d // 9 - 1, (d // 3) % 3 - 1, d % 3 - 1
        Z = torch.roll(X, (-dy, -dx), (2, 3))
        Y = torch.zeros_like(Z)
        n = X.shape[1]
        Y[:, max(0, -dz):n - max(0, dz)] = Z[:, max(0, dz):n - max(0, -dz)]
        out = out + Y @ W[d]
    return out


@pytest.mark.parametrize("S,shape,ci,co", [
    (1, (1, 1, 1), 16, 16), (2, (1, 2, 3), 32, 16), (1, (9, 17, 33), 16, 16),
    (3, (5, 9, 8), 48, 32), (1, (7, 16, 65), 96, 32), (2, (4, 5, 17), 64, 64),
    (1, (3, 33, 16), 32, 96), (1, (65, 35, 36), 16, 16), (1, (66, 37, 33), 16, 48)])
def test_conv_tiles(ws, S, shape, ci, co):
    lib = ws._lib()
    g = torch.Generator(device="cuda").manual_seed(ci + co + sum(shape))
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    nz, ny, nx = shape
    X = rnd(S, *shape, ci).to(torch.bfloat16)
    W = (rnd(27, ci, co) * 0.2).to(torch.bfloat16)
    b = rnd(co)
    dY = rnd(S, *shape, co).to(torch.bfloat16)
    ref = reference(X.double(), W.double(), b.double())
    # FP32 sums of 27 ci products: each rounding 2^-24 of a partial sum, which
    # stays below the sum of the terms' magnitudes
    bound = 27 * ci * 2.0 ** -24 * reference(X.double().abs(), W.double().abs(), b.double().abs())
    Y = torch.empty(S, *shape, co, dtype=torch.bfloat16, device="cuda")
    Yf = torch.empty(S, *shape, co, device="cuda")
    ws._ck(lib.rt3d_nn_conv3d(X.data_ptr(), W.data_ptr(), b.data_ptr(), Y.data_ptr(), Yf.data_ptr(),
                              S, nx, ny, nz, ci, co, 0, 0, None))
    assert bool(((Yf - ref).abs() <= bound).all())
    assert torch.equal(Y, Yf.to(torch.bfloat16))
    # an output that no 4-byte store may touch, with ReLU
    raw = torch.empty(Y.numel() + 1, dtype=torch.bfloat16, device="cuda")
    ws._ck(lib.rt3d_nn_conv3d(X.data_ptr(), W.data_ptr(), b.data_ptr(), raw.data_ptr() + 2, None,
                              S, nx, ny, nz, ci, co, 1, 0, None))
    assert torch.equal(raw[1:].view_as(Y), Y.clamp_min(0))
    # the transposed convolution is the adjoint: <conv(X), dY> = <X, conv^T(dY)>
    WT = W.transpose(1, 2).contiguous()
    dX = torch.empty(S, *shape, ci, device="cuda")
    ws._ck(lib.rt3d_nn_conv3d(dY.data_ptr(), WT.data_ptr(), None, None, dX.data_ptr(), S, nx, ny,
                              nz, co, ci, 0, 1, None))
    flip = torch.arange(26, -1, -1, device="cuda")
    refT = reference(dY.double(), WT.double()[flip], torch.zeros(ci, dtype=torch.float64, device="cuda"))
    magT = reference(dY.double().abs(), WT.double()[flip].abs(),
                     torch.zeros(ci, dtype=torch.float64, device="cuda"))
    assert bool(((dX - refT).abs() <= 27 * co * 2.0 ** -24 * magT).all())
    # weight and bias gradients accumulate onto what is there
    if (ci // 16) * (co // 16) <= 16:
        dW, db = torch.ones(27, ci, co, device="cuda"), torch.ones(co, device="cuda")
        ws._ck(lib.rt3d_nn_conv3d_wgrad(X.data_ptr(), dY.data_ptr(), dW.data_ptr(), db.data_ptr(), S,
                                        nx, ny, nz, ci, co, None))
        Xd = X.double().requires_grad_(False)
        Wv = torch.zeros(27, ci, co, dtype=torch.float64, device="cuda", requires_grad=True)
        reference(Xd, Wv, torch.zeros(co, dtype=torch.float64, device="cuda")).backward(dY.double())
        Wa = torch.zeros(27, ci, co, dtype=torch.float64, device="cuda", requires_grad=True)
        reference(Xd.abs(), Wa, torch.zeros(co, dtype=torch.float64, device="cuda")).backward(
            dY.double().abs())
        n = S * nx * ny * nz
        assert bool(((dW - 1 - Wv.grad).abs() <= (n + 2) * 2.0 ** -24 * (Wa.grad + 1)).all())
        dys = dY.double().sum((0, 1, 2, 3))
        dya = dY.double().abs().sum((0, 1, 2, 3))
        assert bool(((db - 1 - dys).abs() <= (n + 2) * 2.0 ** -24 * (dya + 1)).all())


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 4, 5), (6, 7, 9)])
def test_elementwise_with_and_without_vectors(ws, shape):
    """The 16-byte and the one-channel forms give the same bits."""
    lib = ws._lib()
    g = torch.Generator(device="cuda").manual_seed(7)
    nz, ny, nx = shape
    V, C, S = nx * ny * nz, 16, 2
    h = ws.half(shape)
    Vp = int(np.prod(h))

    def off(t, k):
        """t's values `k` elements into an allocation."""
        raw = torch.empty(t.numel() + 8, dtype=t.dtype, device="cuda")
        v = raw[k:k + t.numel()].view(t.shape)
        v.copy_(t)
        return v

    fine = torch.randn(S, V, C, generator=g, device="cuda").to(torch.bfloat16)
    gate = torch.randn(S, V, C, generator=g, device="cuda").to(torch.bfloat16)
    coarse = torch.randn(S, Vp, C, generator=g, device="cuda").to(torch.bfloat16)
    f32 = torch.randn(S, V, C, generator=g, device="cuda")
    got = []
    for k in (0, 1):
        a, b, c, f = off(fine, k), off(gate, k), off(coarse, k), off(f32, k)
        r = []
        o = off(fine, k)
        ws._ck(lib.rt3d_nn_relu_bwd(a.data_ptr(), b.data_ptr(), o.data_ptr(), a.numel(), None))
        r.append(o.clone())
        o = off(coarse, k)
        ws._ck(lib.rt3d_nn_pool(a.data_ptr(), o.data_ptr(), S, nx, ny, nz, C, None))
        r.append(o.clone())
        o = off(f32, k)
        ws._ck(lib.rt3d_nn_pool_bwd(c.data_ptr(), o.data_ptr(), S, nx, ny, nz, C, None))
        r.append(o.clone())
        o = torch.zeros(S, V, 2 * C, dtype=torch.bfloat16, device="cuda")
        ws._ck(lib.rt3d_nn_upsample(c.data_ptr(), o.data_ptr(), S, nx, ny, nz, C, 2 * C, C if k == 0 else C - k,
                                    None))
        r.append(o[..., C - k:2 * C - k].clone())
        o = off(torch.ones(S, Vp, C, device="cuda"), k)
        ws._ck(lib.rt3d_nn_upsample_bwd(a.data_ptr(), o.data_ptr(), S, nx, ny, nz, C, C, 0, None))
        r.append(o.clone())
        o = off(fine, k)
        ws._ck(lib.rt3d_nn_add_bf16_f32(a.data_ptr(), f.data_ptr(), o.data_ptr(), a.numel(), None))
        r.append(o.clone())
        o = off(fine, k)
        ws._ck(lib.rt3d_nn_f32_to_bf16(f.data_ptr(), o.data_ptr(), f.numel(), None))
        r.append(o.clone())
        o = torch.zeros(S, V, 2 * C, dtype=torch.bfloat16, device="cuda")
        ws._ck(lib.rt3d_nn_channel_copy(a.data_ptr(), C, 0, o.data_ptr(), 2 * C, 8 + k, C, S * V, None))
        r.append(o[..., 8 + k:8 + k + C].clone())
        got.append(r)
    torch.cuda.synchronize()
    for x, y in zip(*got):
        assert torch.equal(x, y)
    assert torch.equal(got[0][0], torch.where(gate > 0, fine, torch.zeros_like(fine)))
