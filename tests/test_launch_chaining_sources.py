"""Kernels that begin while the launch before them is still running (launch chaining) read what that launch writes.  Loads
through a `const ... * __restrict__` pointer may be compiled to the non-coherent kind, whose memory must not change for the
kernel's whole lifetime -- and that begins before the writer ends.  Only the weights, which are complete before, may be
declared so."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_06063_b200", "csrc")


def _functions(text):
    """(name, parameters, body) of the device functions and kernels of a source file."""
    for m in re.finditer(r"^(?:__global__|__device__)[^;{}]*?\b(\w+)\(((?:[^()]|\([^()]*\))*)\)\s*\{\n(.*?)^\}", text, re.S | re.M):
        yield m.group(1), m.group(2), m.group(3)


def test_no_read_only_promise_on_memory_an_earlier_launch_writes():
    waiting = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        for name, params, body in _functions(open(path).read()):
            waits = "griddepcontrol.wait" in body
            waiting += waits
            if waits or name == "xprep_load":      # (inlined into kernels that wait)
                promised = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params)
                assert set(promised) <= {"W"}, f"{os.path.basename(path)}: {name}: {promised}"
    assert waiting >= 9    # xprep, GEMV, slice sum, rmsnorm, dequantisation, two tensor-core kernels and their two sums
