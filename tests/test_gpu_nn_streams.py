"""The accumulating gradients of the pooling and the upsampling, many launches on
two streams into one buffer: nothing is lost. Ones, whose sums are exact."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])  # eight channels a thread, or one
@pytest.mark.parametrize("C", [16, 64])
def test_two_streams_one_buffer(C, offset):
    from paper_2102_01734_gb300 import warmstart as ws

    lib = ws._lib()
    nx, ny, nz, S, launches = 33, 32, 48, 2, 40
    fine, coarse = nx * ny * nz, 17 * 16 * 24
    dP = torch.ones(S * coarse * C, dtype=torch.bfloat16, device="cuda")
    dU = torch.ones(S * fine * C, dtype=torch.bfloat16, device="cuda")
    raw = [torch.zeros(S * v * C + 1, device="cuda") for v in (fine, coarse)]
    dX, dS = (r[offset:offset + r.numel() - 1] for r in raw)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(launches):
        for st in streams:
            ws._ck(lib.rt3d_nn_pool_bwd(dP.data_ptr(), dX.data_ptr(), S, nx, ny, nz, C, st.cuda_stream))
    for _ in range(launches):
        for st in streams:
            ws._ck(lib.rt3d_nn_upsample_bwd(dU.data_ptr(), dS.data_ptr(), S, nx, ny, nz, C, C, 0, st.cuda_stream))
    torch.cuda.synchronize()
    x = dX.view(S, nz, ny, nx, C)
    # x = 0 is also the second child of the last parent of the odd axis
    assert (x[:, :, :, 1:] == 2 * launches / 8).all() and (x[:, :, :, 0] == 4 * launches / 8).all()
    p = dS.view(S, 24, 16, 17, C)
    assert (p[:, :, :, :16] == 2 * launches * 8).all() and (p[:, :, :, 16] == 2 * launches * 4).all()
