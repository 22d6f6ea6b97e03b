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


# a lattice repeated in x: above 8 waves the fields, above 16 also the diagnostics are read in taller
# segments than the narrow lattice's, the last of them not whole; half storage keeps the step's
@pytest.mark.parametrize("ny", [1001, 1711])
@pytest.mark.parametrize("storage", [(0, 0), (1, 0), (2, 0), (0, 1)], ids=["f32", "f16", "f16h32", "d2q5"])
def test_repeated_lattice_reads_out_repeated_fields(ny, storage):
    w = W.parity_droplet(nx=512, ny=ny, steps=2)
    f = {k: np.asarray(v, np.float32) for k, v in w["fields"].items()}
    a, ra = _run(w, f, storage, 2)
    big = W.parity_droplet(nx=4096, ny=ny, steps=2)
    big["params"] = w["params"]
    b, rb = _run(big, {n: np.tile(v, (1, 8)) for n, v in f.items()}, storage, 2)
    for n in FIELDS:
        assert np.array_equal(np.tile(a[n], (1, 8)), b[n]), n
    # compensated sums over other segments, terms of both signs: 1e-12 of the sum and of one a cell
    assert np.allclose(8 * ra[:5], rb[:5], rtol=1e-12, atol=1e-12 * 4096 * ny)


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


def _checks(phi, fs, T, hc):
    """The acceptance checks in FP64 numpy, as long sums."""
    p, f, t = (a.astype(np.longdouble) for a in (phi, fs, T))
    gx = 0.5 * (np.roll(p, -1, 1) - np.roll(p, 1, 1))
    gy = np.zeros_like(p)
    if len(p) > 1:
        gy[1:-1], gy[0], gy[-1] = 0.5 * (p[2:] - p[:-2]), p[1] - p[0], p[-1] - p[-2]
    chi = np.clip(0.5 * (1 + p), 0, 1)
    sol = np.minimum(np.maximum(f, 0), chi)
    H = t * (sol * hc[1] + (chi - sol) * hc[0] + (1 - chi) * hc[2]) + hc[3] * (chi - sol)
    return [v.sum() for v in (p, chi, f, 1 - p * p, np.sqrt(gx * gx + gy * gy))] + [t.min(), t.max(), H.sum()]


# one row, two rows, more columns than threads, more rows than blocks; values up to and beyond the FP32 form's range
@pytest.mark.parametrize("nx,ny", [(1, 1), (5, 2), (33, 3), (300, 7), (17, 1300), (512, 96)])
@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e14])
def test_field_checks_keep_fp64_accuracy(nx, ny, scale):
    from paper_2511_09422_gb300 import cno
    rng = np.random.default_rng(nx + ny)
    phi = np.tanh(rng.standard_normal((ny, nx)) * 3).astype(np.float32)
    phi[rng.random((ny, nx)) < 0.05] *= np.float32(1.1 * scale)
    fs = (rng.uniform(-0.1, 1.1, (ny, nx))).astype(np.float32)
    T = (scale * rng.standard_normal((ny, nx))).astype(np.float32)
    hc = tuple(float(np.float32(v)) for v in (1.0, 0.9, 0.37, 11.3))
    got = cno.field_checks(*(torch.as_tensor(a).cuda() for a in (phi, fs, T)), hc)
    want = _checks(phi, fs, T, hc)
    mags = _checks(np.abs(phi), np.abs(fs), np.abs(T), hc)
    for k in range(8):  # FP64 sums of N terms: N 2^-53 of the terms' magnitudes; 1 - phi^2 of 1 + phi^2
        mag = abs(mags[k]) + (2 * nx * ny + 2 * float((phi.astype(np.float64) ** 2).sum()) if k == 3 else 0)
        mag += (2 * nx * ny * 12 if k == 7 else 0)
        assert abs(got[k] - want[k]) <= 1e-12 * float(mag) + 1e-300, (k, got[k], want[k])


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_field_checks_with_non_finite_values(bad):
    from paper_2511_09422_gb300 import cno
    rng = np.random.default_rng(1)
    phi, fs, T = (rng.uniform(0.1, 0.9, (40, 50)).astype(np.float32) for _ in range(3))
    hc = (1.0, 0.9, 0.4, 11.0)
    clean = cno.field_checks(*(torch.as_tensor(a).cuda() for a in (phi, fs, T)), hc)
    T[20, 30] = bad
    got = cno.field_checks(*(torch.as_tensor(a).cuda() for a in (phi, fs, T)), hc)
    assert got[:5] == pytest.approx(clean[:5], rel=1e-14)
    assert np.isnan(got[7]) if np.isnan(bad) else got[7] == bad
    phi[3, 3] = bad
    got = cno.field_checks(*(torch.as_tensor(a).cuda() for a in (phi, fs, T)), hc)
    assert not np.isfinite(got[0]) and not np.isfinite(got[3]) and not np.isfinite(got[4]) and np.isfinite(got[1])


@pytest.mark.parametrize("nx,ny,cin,nfield", [(1, 1, 8, 1), (31, 3, 64, 7), (32, 1, 64, 8), (100, 33, 24, 5), (64, 64, 256, 7)])
def test_pack_fields_rounds_and_pads(nx, ny, cin, nfield):
    from paper_2511_09422_gb300 import cno
    gen = torch.Generator(device="cuda").manual_seed(nx)
    f = [torch.randn((ny, nx), device="cuda", generator=gen) for _ in range(nfield)]
    off, sc = np.linspace(-1, 1, nfield).astype(np.float32), np.linspace(0.5, 3, nfield).astype(np.float32)
    buf = torch.full((ny * nx * cin + 8,), 3.0, dtype=torch.bfloat16, device="cuda")
    x = buf[:ny * nx * cin].view(1, ny, nx, cin)
    cno.pack_fields(f, off, sc, cin=cin, out=x)
    want = torch.zeros((1, ny, nx, cin), dtype=torch.bfloat16, device="cuda")
    for k in range(nfield):
        want[0, ..., k] = ((f[k] - float(off[k])) * float(sc[k])).to(torch.bfloat16)
    assert torch.equal(x, want)
    assert bool((buf[ny * nx * cin:] == 3.0).all())


def test_field_checks_from_several_threads_and_streams():
    """The checks keep scratch memory between calls: calls on other threads and streams give the same sums."""
    import threading

    from paper_2511_09422_gb300 import cno
    rng = np.random.default_rng(2)
    fields = [tuple(torch.as_tensor(rng.uniform(0, 1, (200 + 10 * i, 300)).astype(np.float32)).cuda() for _ in range(3)) for i in range(4)]
    hc = (1.0, 0.9, 0.4, 11.0)
    want = [cno.field_checks(*f, hc) for f in fields]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(50):
                if cno.field_checks(*fields[i], hc) != want[i]:
                    bad.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
