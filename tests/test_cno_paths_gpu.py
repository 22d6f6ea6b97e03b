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


def _conv_case(n, h, w, cin, cout, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((n, h, w, cin), device="cuda", generator=gen).to(torch.bfloat16)
    w32 = torch.randn((cout, 9, cin), device="cuda", generator=gen) / (9 * cin) ** 0.5
    b = torch.randn(cout, device="cuda", generator=gen)
    return x, w32, b


def _ref(x, w, b=None):
    """FP64 convolution and the sum of its terms' magnitudes (NHWC)."""
    def conv(v, k, c):
        o, _, i = k.shape
        z = torch.nn.functional.conv2d(v.double().permute(0, 3, 1, 2), k.double().reshape(o, 3, 3, i).permute(0, 3, 1, 2), c, padding=1)
        return z.permute(0, 2, 3, 1)
    return conv(x, w, None if b is None else b.double()), conv(x.abs(), w.abs(), None if b is None else b.double().abs())


def _inside(got, ref, mag, what):
    tol = 2.0 ** -8 * ref.abs() + 2.0 ** -12 * mag + 1e-30
    bad = (got.double() - ref).abs() > tol
    assert not bool(bad.any()), "%s: %d of %d outside the bar" % (what, int(bad.sum()), bad.numel())


# 64 input channels: tiles of 8 x 16 pixels with whole, ragged and single tiles, several per block, three output blocks
@pytest.mark.parametrize("n,h,w,cout", [(1, 1, 1, 64), (1, 16, 8, 64), (2, 17, 16, 64), (1, 15, 256, 64), (1, 33, 129, 64),
                                        (3, 64, 64, 64), (2, 48, 130, 192), (5, 128, 128, 64)])
def test_64_channel_layers(n, h, w, cout):
    from paper_2511_09422_gb300 import cno
    x, w32, b = _conv_case(n, h, w, 64, cout, h + w)
    wf, wd = cno.weights_to_bf16(w32)
    ref, mag = _ref(x, wf, b)
    for act in (True, False):
        want = torch.where(ref > 0, ref, ref / 16) if act else ref
        _inside(cno.conv3x3_forward(x, wf, b, act), want, mag, "forward")
    if cout == 64:
        y = cno.conv3x3_forward(x, wf, b, False, out_f32=True, n_store=8)
        assert bool(((y.double() - ref[..., :8]).abs() <= 2.0 ** -12 * mag[..., :8] + 1e-30).all())
    # data gradient: 64 channels in, cin out
    dz, w32, _ = _conv_case(n, h, w, 64, cout, h + w + 1)  # weights [cout][9][64] read as Wd
    wd = w32.to(torch.bfloat16)
    slope = torch.randn((n, h, w, cout), device="cuda").to(torch.bfloat16)
    ref, mag = _ref(dz, wd)
    _inside(cno.conv3x3_dgrad(dz, wd), ref, mag, "dgrad")
    k = torch.where(slope > 0, 1.0, 1.0 / 16).double()
    _inside(cno.conv3x3_dgrad(dz, wd, slope), ref * k, mag * k, "dgrad with slope")


# 64 input channels: K blocks of one row, of two, four and eight rows (w 64 .. 8), ragged rows, widths the kernel leaves
# to the general one (4), one block, several pixel ranges, several output tiles
@pytest.mark.parametrize("n,h,w,cout", [(1, 1, 8, 64), (2, 5, 4, 64), (1, 8, 8, 64), (3, 9, 16, 128), (1, 33, 32, 64),
                                        (2, 40, 64, 64), (1, 7, 129, 192), (2, 31, 200, 256), (4, 128, 128, 64)])
def test_64_channel_weight_gradients(n, h, w, cout):
    from paper_2511_09422_gb300 import cno
    x, _, _ = _conv_case(n, h, w, 64, cout, 3 * h + w)
    dz = torch.randn((n, h, w, cout), device="cuda").to(torch.bfloat16)
    dw, db = cno.conv3x3_wgrad(dz, x)

    def ref(d, v):
        vp = torch.nn.functional.pad(v.double(), (0, 0, 1, 1, 1, 1))
        taps = [torch.einsum("nhwo,nhwi->oi", d.double(), vp[:, dy:dy + h, dx:dx + w]) for dy in range(3) for dx in range(3)]
        return torch.stack(taps, 1)

    assert bool(((dw.double() - ref(dz, x)).abs() <= 2.0 ** -13 * ref(dz.abs(), x.abs()) + 1e-30).all())
    s = dz.double().sum((0, 1, 2))
    assert bool(((db.double() - s).abs() <= 2.0 ** -13 * dz.double().abs().sum((0, 1, 2)) + 1e-30).all())


# streamed weights: one, two and four 64-channel blocks in, one, two and four out; whole, ragged and single tiles, several per block
@pytest.mark.parametrize("cin,cout", [(64, 128), (64, 256), (128, 64), (128, 128), (128, 192), (128, 256), (256, 64), (256, 128), (256, 256)])
@pytest.mark.parametrize("n,h,w", [(1, 1, 8), (2, 17, 16), (1, 33, 130), (3, 64, 128)])
def test_wide_layers(n, h, w, cin, cout):
    from paper_2511_09422_gb300 import cno
    x, w32, b = _conv_case(n, h, w, cin, cout, h + w + cin)
    wf, _ = cno.weights_to_bf16(w32)
    ref, mag = _ref(x, wf, b)
    for act in (True, False):
        want = torch.where(ref > 0, ref, ref / 16) if act else ref
        _inside(cno.conv3x3_forward(x, wf, b, act), want, mag, "forward")
    ref, mag = _ref(x, wf)  # the weights read as Wd: a data gradient from cin to cout channels
    _inside(cno.conv3x3_dgrad(x, wf), ref, mag, "dgrad")
    slope = torch.randn((n, h, w, cout), device="cuda").to(torch.bfloat16)
    k = torch.where(slope > 0, 1.0, 1.0 / 16).double()
    _inside(cno.conv3x3_dgrad(x, wf, slope), ref * k, mag * k, "dgrad with slope")
