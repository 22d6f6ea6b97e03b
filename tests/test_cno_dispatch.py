"""Which kernel takes a convolution, and with how many blocks: the rules of
csrc/cno_dispatch.hpp, compiled for the host."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09422_gb300", "csrc")
SMS = 152


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("dispatch")
    src = d / "rules.cpp"
    src.write_text('#include "cno_dispatch.hpp"\n'
                   'extern "C" int persistent_ctas(long long t, int b, int s) { return cnok::persistent_ctas(t, b, s); }\n')
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
