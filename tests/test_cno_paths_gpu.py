"""Paths of the surrogate's kernels that a call's sizes choose, against the FP64
reference or a plain evaluation: bars as in test_cno_gpu.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09422_gb300 import _build
    _build.build()
    from paper_2511_09422_gb300 import cno
    cno.load()
    cno.read_status(clear=True)
    yield
    assert cno.read_status() == 0, "a tensor-core kernel gave up a wait"


def _net(seed=3):
    from paper_2511_09422_gb300 import cno, surrogate
    net = cno.Net()
    net.set_params(surrogate.init_params(seed))
    return net


@pytest.mark.parametrize("n,h,w,out_cs", [(1, 8, 8, 7), (2, 24, 64, 9), (1, 8, 1032, 8), (3, 16, 128, 12)])
def test_forward_writes_the_callers_channels_only(n, h, w, out_cs):
    net = _net()
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((n, h, w, 64), device="cuda", generator=gen).to(torch.bfloat16)
    want = net.forward(x)
    buf = torch.full((n * h * w * out_cs + 1,), -3.0, device="cuda")
    out = buf[1:].view(n, h, w, out_cs)  # 4-byte aligned only
    net.forward(x, out=out)
    assert torch.equal(out[..., :7], want)
    assert bool((out[..., 7:] == -3.0).all()) and float(buf[0]) == -3.0
    net.close()


@pytest.mark.parametrize("n,h,w,scale", [(1, 8, 8, 1.0), (2, 40, 64, 1e-3), (1, 16, 128, 1e15)])
def test_loss_is_the_mean_square_in_fp64(n, h, w, scale):
    net = _net()
    gen = torch.Generator(device="cuda").manual_seed(h)
    x = torch.randn((n, h, w, 64), device="cuda", generator=gen).to(torch.bfloat16)
    t = scale * torch.randn((n, h, w, 7), device="cuda", generator=gen)
    out = net.forward(x)
    d = (out - t).double()  # the FP32 difference, squared and summed in FP64
    loss = net.train_step(x, t, 0.0, update=False)
    assert loss == pytest.approx(float((d * d).mean()), rel=1e-12)
    net.close()
