"""Host side of the warm-start network without a GPU: the library's calls are
recorded by a stand-in, tensors live on the CPU."""
import pytest

torch = pytest.importorskip("torch")


class _Calls:
    def __getattr__(self, name):
        return lambda *args: 0


@pytest.mark.parametrize("default", [torch.float32, torch.float64])
def test_gradients_are_fp32_whatever_the_default_type(monkeypatch, default):
    """The kernels accumulate FP32 through these pointers."""
    from paper_2102_01734_gb300 import warmstart

    monkeypatch.setattr(warmstart, "_lib", lambda: _Calls())
    net = warmstart.UNet(device="cpu")
    shape = (4, 4, 6)
    X = torch.zeros(1, 96, 16, dtype=torch.bfloat16)
    old = torch.get_default_dtype()
    torch.set_default_dtype(default)
    try:
        y = net.forward(X, shape)
        gW, gb = net.backward(torch.zeros(y.shape, dtype=torch.bfloat16))
    finally:
        torch.set_default_dtype(old)
    for layer in warmstart.LAYERS:
        assert gW[layer[0]].dtype == gb[layer[0]].dtype == torch.float32
        assert gW[layer[0]].shape == net.W32[layer[0]].shape and gb[layer[0]].shape == net.b32[layer[0]].shape
        assert gW[layer[0]].is_contiguous() and (gW[layer[0]] == 0).all()
