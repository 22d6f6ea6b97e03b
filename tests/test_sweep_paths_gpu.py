"""Paths of the strip sweep that a lattice's width, height and storage choose:
windows wrapped at the x ends against windows inside the row, segment heights
from one row up, and field read-out straight into the caller's arrays.

x is periodic and nothing here varies along the walls, so a lattice whose
inputs are shifted by some columns must give the shifted outputs, and every
cell's arithmetic is the same whichever strip, lane or segment it falls into:
the comparisons are bitwise."""
import numpy as np
import pytest

from paper_2511_09422_gb300 import lbfreeze
from paper_2511_09422_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FIELDS = lbfreeze.FIELD_NAMES


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2511_09422_gb300 import _build
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _build.build()
    lbfreeze.load()


def _run(w, fields, storage, steps=6):
    p = dict(w["params"], pop_storage=storage[0], lattice_fl=storage[1])
    s = lbfreeze.Solver(w["grid"], p, fields)
    s.step(steps)
    out, red = s.fields(), s.reduce()
    s.close()
    return out, red


# widths around the strips (30 columns), the chunks (4 FP32, 8 half columns) and rows of whole chunks or not
@pytest.mark.parametrize("nx", [4, 8, 28, 30, 32, 36, 37, 60, 64, 88, 90, 93, 96, 120, 124])
@pytest.mark.parametrize("storage", [(0, 0), (1, 0), (2, 0), (0, 1)], ids=["f32", "f16", "f16h32", "d2q5"])
def test_shifted_lattice_gives_shifted_fields(nx, storage):
    w = W.parity_droplet(nx=nx, ny=33, steps=6)
    f = {k: np.asarray(v, np.float32) for k, v in w["fields"].items()}
    a, ra = _run(w, f, storage)
    k = nx // 3 + 1
    b, rb = _run(w, {n: np.roll(v, k, axis=1) for n, v in f.items()}, storage)
    for n in FIELDS:
        assert np.isfinite(a[n]).all()
        assert np.array_equal(np.roll(a[n], k, axis=1), b[n]), n
    # sums over other strips: the order of the additions differs
    assert np.allclose(ra[:5], rb[:5], rtol=1e-12, atol=1e-12)


# heights whose inner rows are none, one, and not a whole number of segments, against a batch (other segment heights)
@pytest.mark.parametrize("ny", [1, 2, 3, 4, 5, 6, 7, 9, 17, 30, 64])
def test_segment_heights_do_not_change_the_step(ny):
    w = W.parity_droplet(nx=70, ny=ny, steps=5)
    f = {k: np.asarray(v, np.float32) for k, v in w["fields"].items()}
    a, _ = _run(w, f, (0, 0), 5)
    b = lbfreeze.Batch([dict(w, fields=f)] * 40)
    b.step(5)
    got = b.instance(39).fields()
    b.close()
    for n in FIELDS:
        assert np.array_equal(a[n], got[n]), n


@pytest.mark.parametrize("nx,ny", [(5, 4), (30, 7), (64, 33), (101, 40)])
def test_device_read_out_matches_host(nx, ny):
    w = W.parity_droplet(nx=nx, ny=ny, steps=3)
    s = lbfreeze.Solver(w["grid"], w["params"], {k: np.asarray(v, np.float32) for k, v in w["fields"].items()})
    s.step(3)
    host = s.fields()
    dev = s.fields(device=True)
    for n in FIELDS:
        assert np.array_equal(host[n], dev[n].cpu().numpy()), n
    # some of the fields, into views that start anywhere in a larger buffer, which keeps its other values
    buf = torch.full((3 * nx * ny + 8,), 7.5, device="cuda")
    out = {n: buf[1 + i * (nx * ny + 1):1 + i * (nx * ny + 1) + nx * ny] for i, n in enumerate(("fs", "p", "T"))}
    s.fields(out=out)
    s.close()
    for n, v in out.items():
        assert np.array_equal(host[n].reshape(-1), v.cpu().numpy()), n
    rest = torch.ones_like(buf, dtype=torch.bool)
    for i in range(3):
        rest[1 + i * (nx * ny + 1):1 + i * (nx * ny + 1) + nx * ny] = False
    assert bool((buf[rest] == 7.5).all())
