"""Which kernel takes a convolution, and with how many blocks: the rules of
csrc/cno_dispatch.hpp, compiled for the host."""
import ctypes as C
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09422_gb300", "csrc")
SMS = 152


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("dispatch")
    src = d / "rules.cpp"
    src.write_text('#include "cno_dispatch.hpp"\n'
                   'extern "C" int persistent_ctas(long long t, int b, int s) { return cnok::persistent_ctas(t, b, s); }\n'
                   'extern "C" int choose_conv(int n, int h, int w, int cin, int cout, int slope, int head, int s)\n'
                   '{ return cnok::choose_conv({n, h, w, cin, cout, slope != 0, head != 0}, s); }\n')
    so = d / "rules.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wall", "-Werror", "-I", CSRC, "-o", str(so), str(src)], check=True)
    lib = C.CDLL(str(so))
    lib.persistent_ctas.argtypes = [C.c_longlong, C.c_int, C.c_int]
    return lib


@pytest.mark.parametrize("nblocks", [1, 2, 3, 5, 8, 64, 200])
@pytest.mark.parametrize("tiles", [1, 32, 50, 51, 152, 153, 100000, 2 ** 31 - 1])
def test_persistent_blocks_are_resident_at_once(rules, tiles, nblocks):
    per_block = rules.persistent_ctas(tiles, nblocks, SMS)
    assert 1 <= per_block <= tiles
    assert per_block * nblocks <= max(SMS, nblocks)
    assert per_block == min(tiles, max(1, SMS // nblocks))


# Device times (us) of both kernels, conv_fprop_kernel / the one with 8 x 16 pixel tiles, per image and form: f forward,
# s data gradient with slopes, h head.  Rows that differ by less than 5 % are left out.
MEASURED = [
    ((64, 16, 256), """64>64f 30.4/26.7, 64>64s 36.2/27.6, 64>64h 23.1/24.3, 64>192f 89.2/70.6, 64>192s 115.8/70.6, 64>128f 47.4/32.2, 64>128s
        59.8/44, 64>256f 75.6/57.2, 64>256s 122.7/79.6, 128>128f 70.8/63, 128>128s 82.5/64.5, 128>256s 139.8/118.4, 128>384f
        206.7/172.4, 128>384s 250.8/176.6, 128>512s 277.4/236"""),
    ((64, 14, 256), """64>64s 31.4/27, 64>64h 21.1/24, 64>192f 79.6/69.9, 64>192s 102.2/69.9, 64>128f 40.7/31.3, 64>128s 52.4/42.7, 64>256f
        65.8/56.8, 64>256s 106.5/77.8, 128>128s 72/63.7, 128>256f 98.8/115.2, 128>384f 183.4/172, 128>384s 222.7/174.9, 128>512f
        195.7/225.3, 128>512s 242.5/229.1"""),
    ((64, 12, 256), """64>64f 23.8/25.9, 64>64s 27.8/26.3, 64>64h 18.5/23.8, 64>192s 88.1/69.6, 64>128f 36.8/30.9, 64>128s 47.5/41.8, 64>256f
        60.1/56.4, 64>256s 96.7/76.4, 128>128f 56.2/62, 128>256f 89.9/114.8, 128>256s 110/116.8, 128>384f 161.4/171.2, 128>384s
        195.6/174.1, 128>512f 171.9/224.7, 128>512s 213.7/228"""),
    ((1, 1024, 1024), """64>64f 107.9/92.1, 64>64s 130.7/91.6, 64>64h 80.6/86.4, 64>192f 326/265.3, 64>192s 424.3/264.1, 64>128f 171.7/111,
        64>128s 214.9/155.5, 64>256f 277/215.9, 64>256s 452.7/302.4, 128>128f 259.6/227.2, 128>128s 299.7/233, 128>256s
        524.6/465.3, 128>384f 787.4/673.2, 128>384s 1005/724, 128>512s 1055.1/942.9"""),
    ((1, 256, 256), """64>64f 11.5/9.6, 64>64s 13.1/9.7, 64>64h 9.9/8.6, 64>192f 28.8/20.8, 64>192s 33.6/20.9, 64>128f 15.2/11.4, 64>128s
        18.9/12.3, 64>256f 23.8/17.3, 64>256s 32.7/20.4, 128>128f 21.4/20.2, 128>128s 25/20.7, 128>256f 34.3/32.5, 128>256s
        40.1/33.4, 128>384f 59.7/48.8, 128>384s 73.7/50.7, 128>512s 79.4/63.6"""),
    ((1, 64, 64), """64>64f 5.8/4.8, 64>64s 6.6/5, 64>64h 5.4/4, 64>192f 6.4/4.9, 64>192s 7/5.1, 64>128f 6.7/5.3, 64>128s 7.9/5.6, 64>256f
        8.4/5.4, 64>256s 10.5/5.8, 128>128f 9.4/7.6, 128>128s 10.7/7.9, 128>256f 11/7.7, 128>256s 13.2/8, 128>384f 10.4/8,
        128>384s 11.5/8.2, 128>512f 11.1/8.1, 128>512s 13.5/8.4"""),
    ((8, 33, 129), """64>64f 10.9/8.1, 64>64s 12.6/8.2, 64>64h 9.4/7.2, 64>192f 25.6/17.4, 64>192s 28.8/17.4, 64>128f 15/9.4, 64>128s 18.5/10,
        64>256f 23.7/15.2, 64>256s 31.7/16.5, 128>128f 20.7/16.1, 128>128s 24.4/16.6, 128>256f 34/28.3, 128>256s 38.4/28.9,
        128>384f 52.8/40.3, 128>384s 59.9/40.9, 128>512f 59.5/48.7, 128>512s 69.8/49.7"""),
    ((1, 7, 129), """64>64f 6.1/5.0, 64>64h 5.6/4.3, 64>64s 6.4/5.1, 128>128f 9.5/7.8, 128>384f 10.3/7.7"""),
    ((3, 12, 1000), """64>64f 7.3/8, 64>64h 6.7/7.1, 64>192f 17.6/16, 64>192s 20.4/16.1, 64>128s 11.7/10, 64>256s 17.7/14.3, 128>128f 12.6/16,
        128>128s 15/16.4, 128>256f 19.5/24.2, 128>256s 22.2/24.7, 128>384s 44.4/37, 128>512f 38.1/44.5"""),
]
FPROP, CONV64, HALO = 0, 1, 2


@pytest.mark.parametrize("shape,times", MEASURED, ids=["%dx%dx%d" % m[0] for m in MEASURED])
def test_the_faster_kernel_is_taken(rules, shape, times):
    for cin, cout, form, general, other in re.findall(r"(\d+)>(\d+)([fsh])\s+([\d.]+)/([\d.]+)", times):
        got = rules.choose_conv(*shape, int(cin), int(cout), form == "s", form == "h", SMS)
        want = FPROP if float(general) < float(other) else (CONV64 if int(cout) % 128 else HALO)
        assert got == want, (shape, cin, cout, form, general, other)


# what neither of the two kernels takes, and images whose tiles would be mostly padding
@pytest.mark.parametrize("shape,cin,cout,slope,head", [((1, 256, 256), 128, 64, 0, 0), ((1, 256, 256), 256, 256, 0, 0),
                                                       ((1, 256, 256), 192, 192, 1, 0), ((1, 256, 256), 128, 128, 0, 1),
                                                       ((64, 1, 256), 64, 64, 1, 0), ((64, 1, 256), 64, 128, 0, 0)])
def test_the_general_kernel_takes_the_rest(rules, shape, cin, cout, slope, head):
    assert rules.choose_conv(*shape, cin, cout, slope, head, SMS) == FPROP
