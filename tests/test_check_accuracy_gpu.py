"""The acceptance checks and the training loss to FP64's accuracy: exact
references (rationals), cell by cell, over the whole range of the values.

Bars: an FP64 sum of N terms rounds N times, each by 2^-53 of the terms'
magnitudes; the terms themselves are within a few 2^-53."""
import math
from fractions import Fraction as F

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53
HC = tuple(float(np.float32(v)) for v in (1.0, 0.9, 0.37, 11.3))


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09422_gb300 import _build
    _build.build()
    from paper_2511_09422_gb300 import cno
    cno.load()


def _root(q):
    """Square root of a rational, to 90 bits."""
    if q == 0:
        return F(0)
    k = max(0, 200 + q.denominator.bit_length() - q.numerator.bit_length())
    k += k & 1
    return F(math.isqrt((q.numerator << k) // q.denominator), 1 << (k // 2))


def _exact(phi, fs, T, hc):
    """The six sums as rationals, and the sums of their terms' magnitudes."""
    ny, nx = phi.shape
    p, s, t = ([[F(float(v)) for v in row] for row in a] for a in (phi, fs, T))
    cl, cs, cg, lat = (F(v) for v in hc)
    out, mag = [F(0)] * 6, [F(0)] * 6
    for y in range(ny):
        for x in range(nx):
            f = p[y][x]
            gx = (p[y][(x + 1) % nx] - p[y][x - 1]) / 2
            up, dn = min(y + 1, ny - 1), max(y - 1, 0)
            gy = (p[up][x] - p[dn][x]) / (2 if up - dn == 2 else 1)
            chi = min(max((1 + f) / 2, F(0)), F(1))
            so = min(max(s[y][x], F(0)), chi)
            cap = so * cs + (chi - so) * cl + (1 - chi) * cg
            terms = (f, chi, s[y][x], 1 - f * f, _root(gx * gx + gy * gy), t[y][x] * cap + lat * (chi - so))
            mags = (abs(f), chi, abs(s[y][x]), 1 + f * f, terms[4], abs(t[y][x]) * cap + lat * chi)
            out = [a + b for a, b in zip(out, terms)]
            mag = [a + b for a, b in zip(mag, mags)]
    return out, mag


def _compare(phi, fs, T, hc, roundings):
    from paper_2511_09422_gb300 import cno
    got = cno.field_checks(*(torch.as_tensor(a).cuda() for a in (phi, fs, T)), hc)
    want, mag = _exact(phi, fs, T, hc)
    for k, g in enumerate(got[:5] + got[7:]):
        assert abs(F(g) - want[k]) <= roundings * F(U) * mag[k], (k, g, float(want[k]))


# few cells, so that a cell's own error shows: each block's sum, its FP64 value and the blocks' total are 8 roundings
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 1), (1, 2), (3, 3)])
@pytest.mark.parametrize("seed", range(6))
def test_terms_of_a_few_cells(nx, ny, seed):
    rng = np.random.default_rng(seed)
    phi = np.tanh(rng.standard_normal((ny, nx)) * 3).astype(np.float32)
    fs = rng.uniform(-0.1, 1.1, (ny, nx)).astype(np.float32)
    T = rng.standard_normal((ny, nx)).astype(np.float32)
    _compare(phi, fs, T, HC, 8)


# one pattern repeated: the errors of equal terms add up.  Warps, blocks and their total: 64 roundings
def test_repeated_terms():
    rng = np.random.default_rng(7)
    phi = np.tile(np.tanh(rng.standard_normal(4)).astype(np.float32), (24, 75))
    fs = np.full_like(phi, 0.3)
    T = np.full_like(phi, -0.7)
    _compare(phi, fs, T, HC, 64)


# all of a field so small or so large that FP32 products of it leave the range, down to subnormal values
@pytest.mark.parametrize("scale", [1e-40, 1e-30, 1e-20, 1e-13, 1e-12, 1e-9, 1e10, 1e15])
def test_fields_of_any_scale(scale):
    nx, ny = 37, 9
    rng = np.random.default_rng(3)
    phi = (scale * rng.standard_normal((ny, nx))).astype(np.float32)
    fs = rng.uniform(-0.1, 1.1, (ny, nx)).astype(np.float32)
    T = (scale * rng.standard_normal((ny, nx))).astype(np.float32)
    _compare(phi, fs, T, HC[:3] + (0.0,), nx * ny)
    small = tuple(float(np.float32(scale * v)) for v in HC)  # and the coefficients
    if scale < 1e10:
        _compare(phi, fs, np.ones_like(T), small, nx * ny)


# the loss: squares of FP32 differences, exact in FP64.  One block: its sum and the division are 4 roundings
@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1e-14, 1e-6, 1.0, 1e15])
def test_loss_at_any_scale(scale):
    from paper_2511_09422_gb300 import cno, surrogate
    net = cno.Net()
    net.set_params(np.zeros_like(surrogate.init_params(1)))  # the network's output is 0
    gen = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((1, 8, 16, 64), device="cuda", generator=gen).to(torch.bfloat16)
    t = scale * torch.randn((1, 8, 16, 7), device="cuda", generator=gen)
    assert not bool(net.forward(x).any())
    loss = net.train_step(x, t, 0.0, update=False)
    net.close()
    d = t.cpu().double().numpy().ravel()
    want = math.fsum(d * d) / d.size
    # beyond 1e12 and below 2^-48 the squares are added in FP64 one by one
    assert abs(loss - want) <= (4 if 1e-12 < scale < 1e10 else d.size) * U * want
