"""The table of kept dispatches: what a call launches and returns depends on its sizes and the parameters alone."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import paper_2602_06063_b200 as fd
import synthgen
from gpu_common import Case

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _calls(ctx, case, gamma):
    """A plain and a normalised device call: (launches, output) of each."""
    K, N, M = case.K, case.N, case.M
    got = []
    for norm in (False, True):
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        before = fd.fdqp_launch_count(ctx)
        if norm:
            fd.fdqp_run_rmsnorm_epilogue(ctx, case.x_dev, gamma, 1e-6, case.W_dev, y, fd.EPI_NONE, M, K, N)
        else:
            fd.fdqp_run(ctx, case.x_dev, case.W_dev, y, M, K, N)
        torch.cuda.synchronize()
        assert fd.fdqp_last_status(ctx) == 0
        got.append((fd.fdqp_launch_count(ctx) - before, y.cpu().numpy().view(np.uint32)))
    return got


# fused normalisation; in-kernel preparation but a normalisation launch; records written by the normalisation; K slices
@pytest.mark.parametrize("K,N,M", [(2560, 2048, 1), (2560, 512, 2), (1152, 6912, 2), (2560, 512, 4), (21504, 320, 2)])
def test_a_host_call_leaves_no_trace_in_device_calls(K, N, M):
    """fdqp_run_host with page-locked x has the preparation kernel read x whatever the plan says: only in that call."""
    case = Case(K, N, M, seed=70 + M, amp=1.0 / np.sqrt(K))
    gamma = torch.from_numpy(synthgen.activations(71, 1, K).view(np.int16)).cuda()
    x_pin = torch.from_numpy(case.x.view(np.int16)).pin_memory()
    results = []
    for host_first in (False, True):
        ctx = fd.fdqp_create(0, 8, K, N)
        try:
            if host_first:
                y_host = torch.empty((M, N), dtype=torch.float32).pin_memory()
                fd.fdqp_run_host(ctx, x_pin, case.W_dev, y_host, M, K, N)
            results.append(_calls(ctx, case, gamma))
        finally:
            fd.fdqp_destroy(ctx)
    for (launches, y), (launches_after, y_after) in zip(*results):
        assert launches_after == launches
        assert np.array_equal(y_after, y)


def test_interleaved_shapes_keep_their_launches_and_bits():
    """More shapes than the table has slots, plain, with epilogues, normalised and of other formats, called in shuffled orders
    without a parameter being touched in between: each call launches and returns what it does on a context of its own."""
    rng = np.random.default_rng(5)
    max_M, max_K, max_N = 40, 3072, 640
    calls = []
    for i in range(96):
        kind = ("run", "bf16", "norm", "fmt")[i % 4]
        M = int(rng.choice([1, 2, 3, 4, 8, 9, 40]))
        K = int(rng.integers(1, max_K // 256 + 1)) * 256 if kind == "fmt" else int(rng.integers(2, max_K // 32 + 1)) * 32
        N = int(rng.integers(1, max_N // 32 + 1)) * 32
        x = torch.from_numpy(synthgen.activations(200 + i, M, K).view(np.int16)).cuda()
        if kind == "fmt":
            w = synthgen.weights_fmt(300 + i, K, N, fd.FMT_MXFP4)
            W = torch.from_numpy(fd.q4nx_pack_fmt(fd.FMT_MXFP4, w.codes, w.scales, w.offsets)).cuda()
        else:
            w = synthgen.weights(300 + i, K, N)
            W = torch.from_numpy(fd.q4nx_pack(w.codes, w.scales, w.offsets)).cuda()
        calls.append((kind, M, K, N, x, W))

    def call(ctx, c):
        kind, M, K, N, x, W = c
        out = torch.zeros((M, N), dtype=torch.int16 if kind == "bf16" else torch.int32, device="cuda")
        before = fd.fdqp_launch_count(ctx)
        if kind == "run":
            fd.fdqp_run(ctx, x, W, out, M, K, N)
        elif kind == "bf16":
            fd.fdqp_run_epilogue(ctx, x, W, out, fd.EPI_BF16, M, K, N)
        elif kind == "norm":
            fd.fdqp_run_rmsnorm_epilogue(ctx, x, x, 1e-6, W, out, fd.EPI_NONE, M, K, N)
        else:
            fd.fdqp_run_fmt(ctx, fd.FMT_MXFP4, x, W, out, M, K, N)
        launches = fd.fdqp_launch_count(ctx) - before
        torch.cuda.synchronize()
        assert fd.fdqp_last_status(ctx) == 0
        return launches, out

    expected = []
    for c in calls:
        ctx = fd.fdqp_create(0, max_M, max_K, max_N)
        try:
            expected.append(call(ctx, c))
        finally:
            fd.fdqp_destroy(ctx)
    ctx = fd.fdqp_create(0, max_M, max_K, max_N)
    try:
        for _ in range(3):
            for i in rng.permutation(len(calls)):
                launches, out = call(ctx, calls[i])
                assert launches == expected[i][0], calls[i][:4]
                assert torch.equal(out, expected[i][1]), calls[i][:4]
    finally:
        fd.fdqp_destroy(ctx)


# One thread calls fdqp_run over and over; the other sets "prep_inline", waits until the first is between calls, and counts
# the launches of a call of its own.  (In Python the interpreter lock would keep the two apart.)
STRESS = r"""
#include <atomic>
#include <thread>
#include "fdqp.h"
extern "C" int64_t stress(fdqp_ctx* ctx, const void* x, const void* W, float* y, int64_t K, int64_t N, void* stream, int64_t rounds) {
    std::atomic<int> go{0}, busy{0}, stop{0};
    std::thread other([&] {
        while (!stop) {
            busy = 1;
            if (go) fdqp_run(ctx, x, W, y, 1, K, N, stream);
            busy = 0;
        }
    });
    int64_t stale = 0;
    for (int64_t i = 0; i < rounds; ++i) {
        go = 1;
        for (volatile int spin = 0; spin < 500 + (int)(i % 97) * 100; ++spin) {}
        fdqp_set_param(ctx, "prep_inline", i & 1);
        go = 0;
        while (busy) {}
        const int64_t before = fdqp_launch_count(ctx);
        fdqp_run(ctx, x, W, y, 1, K, N, stream);
        stale += fdqp_launch_count(ctx) - before != (i & 1 ? 1 : 2);
    }
    stop = 1;
    other.join();
    return stale;
}
"""


def test_a_parameter_takes_effect_under_a_concurrent_caller(tmp_path):
    """From fdqp_set_param's return on every call obeys the new value, whatever another thread was calling meanwhile.  (Both
    threads use one stream, so that the context's workspace has one user at a time on the device.)"""
    lib = fd.load_library()
    src, so = tmp_path / "stress.cpp", tmp_path / "libstress.so"
    src.write_text(STRESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I", os.path.join(ROOT, "include"), "-o", str(so), str(src),
                    lib._name], check=True)
    K, N = 2560, 64
    case = Case(K, N, 1, seed=77)
    y = torch.empty((1, N), dtype=torch.float32, device="cuda")
    ctx = fd.fdqp_create(0, 1, K, N)
    try:
        fn = ctypes.CDLL(str(so)).stress
        fn.restype, fn.argtypes = ctypes.c_int64, [ctypes.c_void_p] * 4 + [ctypes.c_int64] * 2 + [ctypes.c_void_p, ctypes.c_int64]
        stale = fn(ctx, case.x_dev.data_ptr(), case.W_dev.data_ptr(), y.data_ptr(), K, N, torch.cuda.current_stream().cuda_stream, 5000)
        torch.cuda.synchronize()
        assert fd.fdqp_last_status(ctx) == 0
    finally:
        fd.fdqp_destroy(ctx)
    assert stale == 0


# rings of eight warps in half an SM's shared memory; only in all of it; sixteen warps' too large for it
@pytest.mark.parametrize("K,N,M,warps,got", [(2560, 4096, 1, 8, 8), (2560, 262144, 8, 8, 8), (10240, 40960, 1, 8, 8), (2560, 4096, 1, 16, 16),
                                             (10240, 40960, 1, 16, 16), (7168, 4096, 8, 16, 8)])
def test_consumer_warps_are_what_was_asked_for_where_their_rings_fit(K, N, M, warps, got):
    ctx = fd.fdqp_create(0, 8, K, N)
    try:
        fd.fdqp_set_param(ctx, "consumer_warps", warps)
        assert f"fdqp_gemv_kernel<{got}," in fd.fdqp_describe(ctx, M, K, N)
    finally:
        fd.fdqp_destroy(ctx)
