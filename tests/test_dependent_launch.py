"""What kernels under programmatic dependent launch may not do, read off the
sources: their blocks are resident while the kernel in front of them still
writes their inputs, so those inputs are not read-only data for as long as the
kernel lives.  They wait first, and read by coherent loads only."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09422_gb300", "csrc")
# read-only for the whole of a step: the host writes the records, and no kernel does
HOST_WRITTEN = {"const StepRec *__restrict__ inst"}


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _function(text, at):
    """The signature and body of the function whose parameter list opens at or after ``at``."""
    depth = 0
    for i in range(text.index("{", at), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i + 1]
    raise AssertionError("unbalanced braces")


def _kernels(text):
    """Kernel name -> (signature, body), helpers excluded."""
    out = {}
    for m in re.finditer(r"__global__", text):
        f = _function(text, m.start())
        sig, body = f[:f.index("{")], f[f.index("{"):]
        name = re.search(r"(\w+_kernel)\s*\(", sig)
        if name:
            out[name.group(1)] = (sig, body)
    return out


def _dependent():
    """(name, signature, body) of every kernel passed to one of the launchers."""
    cno, lb = _source("cno_kernels.cuh") + _source("cno_api.cu"), _source("lb_kernels.cuh") + _source("lb_api.cu")
    cases = []
    for text, launcher in ((cno, r"\blaunch\("), (lb, r"\blaunch_dependent\(")):
        kernels = _kernels(text)
        for name in sorted(set(re.findall(launcher + r"\s*(?:\w+::)?(\w+_kernel)\b", text))):
            cases.append((name,) + kernels[name])
    return cases


DEPENDENT = _dependent()


def test_every_dependent_kernel_is_seen():
    names = {c[0] for c in DEPENDENT}
    assert {"lb_step_kernel", "lb_strip_kernel", "conv64_kernel", "conv_halo_kernel", "wgrad64_kernel", "mse_kernel", "adam_kernel",
            "field_sums_kernel", "field_total_kernel", "sum_partials_kernel", "weights_to_bf16_kernel"} <= names


@pytest.mark.parametrize("name,sig,body", DEPENDENT, ids=[c[0] for c in DEPENDENT])
def test_dependent_kernels_wait_and_read_coherently(name, sig, body):
    begin = re.search(r"\b(grid_begin|sweep_begin)\(\)", body)
    assert begin, "no wait for the kernel in front"
    assert "return" not in body[:begin.start()], "a block may leave before it has waited"
    read_only = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s*\w+", sig + body)
    assert [r for r in read_only if re.sub(r"\s+", " ", r) not in HOST_WRITTEN] == []
    assert "__ldg(" not in body


@pytest.mark.parametrize("helper", ["stage9", "strip_rows", "phase_b"])
def test_sweep_helpers_read_coherently(helper):
    text = _source("lb_kernels.cuh")
    at = re.search(r"\bvoid %s\(" % helper, text).start()
    assert "__ldg(" not in _function(text, at)
