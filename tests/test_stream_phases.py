"""The streaming tensor-core kernel's waits test the parity of a barrier's phase.  tests/host/stream_phases.cpp enumerates, with the
kernel's own choice of barrier and phase (fdqp_plan.h), the states in which a wait can find its barrier."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_no_wait_passes_before_its_phase(tmp_path):
    exe = str(tmp_path / "stream_phases")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2602_06063_b200", "csrc"), "-o", exe,
                           os.path.join(ROOT, "tests", "host", "stream_phases.cpp")])
    run = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout
