"""The acceptance checks' scratch: kept between calls, bounded, given back, never shared."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09422_gb300", "csrc")

PROGRAM = r"""
#include "slot_pool.hpp"
#include <atomic>
#include <cstdio>
#include <thread>
static SlotPool<int, 4, 2> pool;
static std::atomic<int> made{0}, freed{0}, shared{0}, in_use[1024];
static void call(int dev)
{
    int s;
    if (!pool.take(dev, &s)) s = made++;
    if (in_use[s]++) shared++;
    std::this_thread::yield();
    in_use[s]--;
    if (!pool.keep(dev, s)) freed++;
}
int main()
{
    std::vector<std::thread> t;
    for (int i = 0; i < 12; i++) t.emplace_back([i] { for (int k = 0; k < 20; k++) call(i % 2); });
    for (auto &x : t) x.join();
    const int idle = (int)pool.drain().size(), again = (int)pool.drain().size();
    printf("%d %d %d %d\n", shared.load(), idle <= 8, made == freed + idle, again);
}
"""


def test_slots_are_owned_bounded_and_given_back(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    for _ in range(5):
        assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["0", "1", "1", "0"]


def test_the_last_network_frees_the_idle_slots():
    with open(os.path.join(CSRC, "cno_api.cu")) as f:
        text = f.read()
    destroy = text[text.index('extern "C" cno_status cno_destroy'):text.index('extern "C" cno_status cno_set_stream')]
    assert "g_check_slots.drain()" in destroy


@pytest.mark.gpu
def test_checks_in_a_capture_are_refused_and_leave_it_whole():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09422_gb300 import _build
    _build.build()
    from paper_2511_09422_gb300 import cno
    phi = torch.linspace(-1, 1, 40 * 50, device="cuda").view(40, 50)
    want = cno.field_checks(phi)
    y = torch.zeros(4, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        with pytest.raises(RuntimeError):
            cno.field_checks(phi)
        y += 1
    g.replay()
    torch.cuda.synchronize()
    assert y.tolist() == [1.0] * 4
    for _ in range(2):  # before and after the idle slots are freed
        assert cno.field_checks(phi) == want
        net = cno.Net()
        net.close()
