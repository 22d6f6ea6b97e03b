"""A block of the tensor-core kernels that gave a wait up does not end with loads or MMAs
of its own under way: read off the sources, and the bookkeeping of the last loads
compiled for the host against a plain count."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09422_gb300", "csrc")


def _source():
    with open(os.path.join(CSRC, "cno_kernels.cuh")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _braces(text, at):
    depth = 0
    for i in range(text.index("{", at), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i + 1]
    raise AssertionError("unbalanced braces")


def _kernels():
    text = _source()
    out = {}
    for m in re.finditer(r"__global__", text):
        f = _braces(text, m.start())
        name = re.search(r"(\w+_kernel)\s*\(", f).group(1)
        if "tma_load_4d(" in f:
            out[name] = f
    return out


KERNELS = _kernels()


def test_all_kernels_with_loads_are_seen():
    assert set(KERNELS) == {"conv_fprop_kernel", "conv64_kernel", "conv_halo_kernel", "conv_wgrad_kernel", "wgrad64_kernel"}


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_issued_work_is_over_before_the_block_ends(name):
    body = KERNELS[name]
    # every ring or barrier that a load signals is waited for
    signalled = set(re.findall(r"mbar_expect_tx\(&?(\w+)", body)) - {"bar"}
    drained = set(re.findall(r"(?:drain_loads<[^>]*>|mbar_drain)\((\w+)", body))
    assert signalled <= drained, signalled - drained
    if "uint64_t *bar = &sl_full" in body:  # signalled through a local name
        assert "sl_full" in drained
    assert body.count("drain_mmas(drained);") == 1 and "mbar_init(drained, 1);" in body
    # in the branch that an abort takes behind the roles, and every role that gives a wait up sets the flag
    end = body[body.rindex("if (__builtin_expect(*abort_flag, 0)) {"):]
    assert all(d in end for d in ("drain_mmas(", "drain_loads<", "__syncthreads();", "tmem_dealloc("))
    assert body.index("__syncthreads();", body.rindex("ST_TIMEOUT_EPILOGUE")) < len(body) - len(end)
    assert body.count("ST_TIMEOUT") == body.count("*abort_flag = 1;")
    # stores are waited for outside the tile loop, whichever way it was left
    if "tma_store_4d(" in body:
        assert "cp.async.bulk.wait_group 0;" in body


def test_the_last_load_of_every_slot_is_waited_for(tmp_path):
    text = _source()
    at = text.index("template <int SLOTS>\n__device__ __forceinline__ void drain_loads")
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text('''#include <cstdint>
#include <cstdio>
#include <vector>
#define __device__
#define __forceinline__ inline
static std::vector<int> seen;
static uint64_t bars[8];
static void mbar_drain(uint64_t *bar, uint32_t parity) { seen.push_back(2 * (int)(bar - bars) + (int)parity); }
''' + _braces(text, at) + '''
template <int SLOTS> static int check()
{
    int bad = 0;
    for (int fills = 0; fills < 40; fills++) {
        int last[SLOTS];  // phase of the last fill of each slot, by counting
        for (int &x : last) x = -1;
        for (int f = 0; f < fills; f++) last[f % SLOTS]++;
        std::vector<int> want;
        for (int s = 0; s < SLOTS; s++)
            if (last[s] >= 0) want.push_back(2 * s + (last[s] & 1));
        seen.clear();
        drain_loads<SLOTS>(bars, fills);
        bad += seen != want;
    }
    return bad;
}
int main() { printf("%d\\n", check<2>() + check<3>() + check<4>()); }
''')
    subprocess.run(["g++", "-std=c++17", "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["0"]
