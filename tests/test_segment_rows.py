"""The height of the step's segments: the estimate of csrc/segment_rows.hpp, compiled
for the host, against measured step times."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09422_gb300", "csrc")

# storage, nx, ny, the first height, us per step at that height and the ones after it (up to the greatest that is allowed)
MEASURED = [
    ("f32", 64, 256, 1, "8.7 8.7 9.9 11.4 13.0 14.6 16.2 17.9 19.5 21.1 22.6 24.5"),
    ("f32", 512, 256, 1, "24.0 18.4 22.0 15.5 17.8 20.0 22.2 23.9 20.1 21.6 23.2 25.0"),
    ("f32", 300, 300, 1, "19.2 18.3 13.8 16.2 18.6 16.0 17.7 19.5 21.1 22.7 23.6 25.1"),
    ("f32", 512, 512, 1, "45.4 34.7 33.4 29.1 33.0 36.8 39.4 26.1 28.5 30.9 33.2 35.6"),
    ("f32", 700, 700, 1, "80.0 61.1 56.2 54.8 51.0 54.4 46.0 48.9 52.7 56.5 59.8 63.0"),
    ("f32", 1024, 1024, 1, "165 122 110 103 99.1 96.0 97.4 93.5 98.0 89.7 92.5 97.4"),
    ("f32", 1500, 1300, 6, "167 165 162 160 162 156 162"),
    ("f32_d2q5", 512, 512, 1, "41.3 31.2 29.6 26.0 29.2 32.3 33.7 23.1 25.1 27.2 29.3 31.4 33.6 35.7 37.8 38.1 32.7 34.3 36.0 37.6 39.2 40.5 42.0 43.7"),
    ("f32_d2q5", 1037, 771, 1, "116 85.1 76.9 72.5 70.8 67.4 69.3 64.4 68.2 71.8 67.0 61.5 64.5 67.8 71.2 74.6 78.0 81.2 84.3 84.9 82.7 80.1 57.2 58.6"),
    ("f32_d2q5", 1024, 1024, 1, "152 111 98.0 92.5 87.6 84.7 86.1 83.0 86.8 78.6 81.6 85.9 89.8 89.2 75.5 77.8 81.0 84.3 87.7 91.1 94.4 97.7 101 104"),
    ("f32_d2q5", 3000, 2000, 6, "432 422 414 406 402 400 398 395 392 390 389 388 389 387 388 381 390 390 379"),
    ("f16", 300, 300, 1, "17.2 14.7 18.1 17.9 20.0 20.9 23.3 25.6 28.1 30.4 32.8 35.1 37.5 39.8 41.9 44.4 46.8 49.2 50.0 52.4 54.8 58.7 61.4 64.1"),
    ("f16", 512, 512, 1, "40.0 31.0 30.0 31.0 30.6 26.6 30.0 33.1 36.4 39.6 32.4 34.8 37.1 39.4 41.6 43.8 37.9 39.8 41.5 43.4 45.5 47.4 49.2 51.4"),
    ("f16", 701, 901, 1, "95.6 74.2 66.3 62.1 62.0 58.4 61.0 61.4 63.9 65.5 70.0 54.6 57.7 61.2 64.6 68.2 71.7 75.3 78.7 82.2 85.6 89.0 92.5 96.1"),
    ("f16", 1037, 771, 1, "118 90.2 81.5 77.7 75.0 74.8 76.4 72.3 74.7 76.6 79.4 81.2 85.3 89.3 72.9 75.8 79.5 82.5 86.0 89.5 93.2 96.7 101 104"),
    ("f16", 1024, 1024, 1, "142 107 95.8 93.2 88.4 87.4 86.1 87.1 87.7 80.2 84.4 81.1 85.2 90.0 85.4 89.2 93.7 97.5 101 77.6 76.9 80.1 83.3 86.4"),
    ("f16", 3000, 2000, 6, "448 440 431 425 424 422 420 409 406 410 408 405 405 411 401 413 408 420 398"),
    ("f16h32", 512, 256, 1, "21.0 19.3 16.5 19.4 22.5 18.9 21.1 22.1 21.1 22.8 24.5 26.1 27.8 29.3 31.0 32.6 34.1 35.8 37.4 39.0 40.7 42.3 44.0 45.7"),
    ("f16h32", 700, 700, 1, "75.0 58.1 54.0 51.1 47.4 48.1 51.3 53.4 56.6 45.6 48.8 52.1 55.5 59.0 62.4 65.7 69.2 72.5 75.2 65.7 68.2 70.6 73.3 75.4"),
    ("f16h32", 1037, 771, 1, "117 90.2 81.7 77.7 75.0 74.5 76.6 72.4 74.4 76.0 79.0 81.3 84.8 87.8 79.8 80.8 84.6 87.0 89.9 92.3 95.0 98.1 101 104"),
    ("f16h32", 1500, 1300, 6, "159 155 154 153 151 152 153 154 154 159 160 165 166 159 164 166 165 170 174"),
    ("f16h32", 2048, 2048, 6, "315 311 301 298 294 296 290 294 286 286 296 283 287 287 289 295 284 291 285"),
    ("f16", 1317, 2095, 5, "228 220 215 212 210 209 206 205 206 205 210 209 210 210 211 210 216 219 220 227"),
    ("f16h32", 1063, 1980, 5, "180 174 171 169 168 166 166 168 171 168 168 172 177 179 185 178 184 184 186 188"),
    ("f16h32", 859, 1230, 5, "94.5 93.9 92.0 91.9 94.1 89.1 91.3 91.0 93.1 97.3 100 104 108 112 116 102 104 108 112 115"),
    ("f16h32", 2274, 926, 5, "172 167 164 165 161 162 161 162 161 164 163 168 170 175 179 169 174 178 180 180"),
]
WARPS = {"f32": 152 * 8, "f32_d2q5": 152 * 8, "f16": 152 * 12, "f16h32": 152 * 12}


@pytest.fixture(scope="module")
def pick(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    src, so = d / "rows.cpp", d / "rows.so"
    src.write_text('#include "segment_rows.hpp"\n'
                   'extern "C" int ragged_rows() { return lbk::RAGGED_ROWS; }\n'
                   'extern "C" int rows(long long W, int half, int most, int n, const long long *strips, const int *ny)\n'
                   '{ return lbk::best_segment_rows(W, half != 0, most, [&](int h) { return lbk::batch_items(h, [&](auto f) {\n'
                   '    for (int i = 0; i < n; i++) f(strips[i], ny[i]); }); }); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wall", "-Werror", "-I", CSRC, "-o", str(so), str(src)], check=True)
    lib = C.CDLL(str(so))

    def f(storage, sizes, most=None):
        half = storage.startswith("f16")
        if most is None:  # a single lattice's
            most = 12 if storage == "f32" else (lib.ragged_rows() if half and sizes[0][0] % 8 else 24)
        n = len(sizes)
        strips, ny = (C.c_longlong * n)(*(-(-x // 30) for x, _ in sizes)), (C.c_int * n)(*(y for _, y in sizes))
        return lib.rows(C.c_longlong(WARPS[storage]), half, most, n, strips, ny)

    return f


@pytest.mark.parametrize("storage,nx,ny,first,times", MEASURED, ids=["%s-%dx%d" % m[:3] for m in MEASURED])
def test_the_height_is_near_the_best(pick, storage, nx, ny, first, times):
    us = {first + i: float(t) for i, t in enumerate(times.split())}
    assert us[pick(storage, [(nx, ny)])] <= 1.07 * min(us.values())


@pytest.mark.parametrize("storage", sorted(WARPS))
@pytest.mark.parametrize("ny", [1, 4, 5, 6, 9])
def test_low_lattices_have_a_height(pick, storage, ny):
    assert 1 <= pick(storage, [(4, ny)]) <= 24


# many small lattices of different heights: their short items fill no rounds (7 rows, by count, took 2 to 11 % longer than 12 to 16)
@pytest.mark.parametrize("storage", sorted(WARPS))
def test_small_uneven_batches_take_tall_segments(pick, storage):
    sides = [48 + (37 * i) % 53 for i in range(200)]
    assert 12 <= pick(storage, [(s, s) for s in sides], most=16) <= 16
