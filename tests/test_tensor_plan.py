"""The plans of prefill-sized calls, made by the library's own functions (fdqp_tensor_plan.h, compiled for the CPU) over a grid of
sizes and launch parameters: tests/host/tensor_plan.cpp."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "tensor_plan")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                           "-I", os.path.join(ROOT, "paper_2602_06063_b200", "csrc"), "-o", exe, os.path.join(ROOT, "tests", "host", "tensor_plan.cpp")])
    return exe


def check(program, what):
    run = subprocess.run([program, what], capture_output=True, text=True, timeout=600)
    assert run.returncode == 0, run.stdout + run.stderr


def test_every_unit_once_within_the_bounds(program):
    """Streaming kernel: every unit of work in one pair's range, no slot of partial sums and no counter used twice, shared memory,
    tensor memory and workspace within their sizes."""
    check(program, "cuts")


def test_calls_keep_fp32_weights(program):
    """Which calls of nine and more rows go through the GEMV kernels, whose weights are not rounded to bf16."""
    check(program, "routes")


def test_workspace_of_a_context(program):
    check(program, "workspaces")


def test_parameters_select_the_tile_kernels(program):
    check(program, "tile_kernels")
