"""Network inference whose outputs land on its inputs."""
import pytest

from gpu_util import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [0, 2])
@pytest.mark.parametrize("n", [1000, 2 ** 17, 2 ** 17 + 1, 2 ** 18 + 777])
@pytest.mark.parametrize("n_in,n_out,x0,y0", [(3, 8, 0, 0), (8, 3, 0, 0), (8, 8, 0, 0), (8, 3, 0, 3000), (3, 8, 5000, 4)])
def test_outputs_over_inputs(n, n_in, n_out, x0, y0, bf16):
    """The layers run over pieces of 2^17 rows; X starts x0 floats into the buffer that takes Y from its float y0 on.
    The same bits as into a buffer of its own."""
    tam = need_gpu()
    net = tam.Mlp(n_in, 16, 1, n_out, seed=3)
    X = torch.randn((n, n_in), device="cuda", generator=torch.Generator(device="cuda").manual_seed(n))
    ref = net.forward(X, bf16=bf16)
    buf = torch.zeros(max(x0 + n * n_in, y0 + n * n_out), device="cuda")
    buf[x0:x0 + n * n_in] = X.reshape(-1)
    status = tam.lib.tam_mlp_forward(net.handle, n, buf.data_ptr() + 4 * x0, buf.data_ptr() + 4 * y0, bf16,
                                     torch.cuda.current_stream().cuda_stream)
    assert status == 0
    assert torch.equal(buf[y0:y0 + n * n_out].view(n, n_out), ref)


@pytest.mark.parametrize("width,extra", [(128, 1), (96, 777), (16, 1), (16, 2 ** 20 + 777)])
@pytest.mark.parametrize("n_in,n_out,x0,y0", [(3, 8, 0, 0), (8, 3, 0, 3000), (3, 8, 5000, 4)])
def test_outputs_over_inputs_of_several_pieces(width, extra, n_in, n_out, x0, y0):
    """FP32 pieces hold 2^24 values a layer: `extra` rows more than one, against the rows taken in two calls (each
    row's arithmetic does not depend on its piece)."""
    tam = need_gpu()
    net = tam.Mlp(n_in, width, 1, n_out, seed=3)
    n = 2 ** 24 // width + extra
    X = torch.randn((n, n_in), device="cuda", generator=torch.Generator(device="cuda").manual_seed(n))
    ref = torch.cat([net.forward(X[:n // 2].contiguous()), net.forward(X[n // 2:].contiguous())])
    assert torch.equal(net.forward(X), ref)
    buf = torch.zeros(max(x0 + n * n_in, y0 + n * n_out), device="cuda")
    buf[x0:x0 + n * n_in] = X.reshape(-1)
    status = tam.lib.tam_mlp_forward(net.handle, n, buf.data_ptr() + 4 * x0, buf.data_ptr() + 4 * y0, 0,
                                     torch.cuda.current_stream().cuda_stream)
    assert status == 0
    assert torch.equal(buf[y0:y0 + n * n_out].view(n, n_out), ref)
