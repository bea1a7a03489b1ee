"""Weights written on the stream just before the call that reads them.  The library reads weights ahead of the stream order: by
default right behind any kernel that does not trigger its dependents early, with "launch_ahead" = 0 behind any kernel."""
import ctypes
import subprocess

import pytest
import torch

import paper_2602_06063_b200 as fd
import synthgen

pytestmark = pytest.mark.gpu

# Lets its dependents begin at once, and writes 40 us later.
WRITER = r"""
__global__ void __launch_bounds__(128) late_writer(const uint4* src, uint4* dst, long long n) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int i = 0; i < 40; ++i) __nanosleep(1000);
    for (long long i = blockIdx.x * 128ll + threadIdx.x; i < n; i += gridDim.x * 128ll) dst[i] = src[i];
}
extern "C" int write_late(const void* src, void* dst, long long bytes, void* stream) {
    late_writer<<<32, 128, 0, (cudaStream_t)stream>>>((const uint4*)src, (uint4*)dst, bytes / 16);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def write_late(tmp_path_factory):
    d = tmp_path_factory.mktemp("writer")
    (d / "writer.cu").write_text(WRITER)
    subprocess.run(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-Xcompiler", "-fPIC", "-o",
                    str(d / "writer.so"), str(d / "writer.cu")], check=True)
    fn = ctypes.CDLL(str(d / "writer.so")).write_late
    fn.restype, fn.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p]

    def write(src, dst):
        assert fn(src.data_ptr(), dst.data_ptr(), src.numel(), torch.cuda.current_stream().cuda_stream) == 0
    return write


def _ordinary(src, dst):
    torch.bitwise_or(src, 0, out=dst)


K, N = 2560, 2048
CALLS = {
    "M = 1": lambda ctx, x, W, y: fd.fdqp_run(ctx, x, W, y, 1, K, N),
    "M = 4": lambda ctx, x, W, y: fd.fdqp_run(ctx, x, W, y, 4, K, N),
    "M = 4, K slices": lambda ctx, x, W, y: fd.fdqp_run(ctx, x, W, y, 4, K, N),
    "M = 40": lambda ctx, x, W, y: fd.fdqp_run(ctx, x, W, y, 40, K, N),
    "M = 200": lambda ctx, x, W, y: fd.fdqp_run(ctx, x, W, y, 200, K, N),
    "M = 400": lambda ctx, x, W, y: fd.fdqp_run(ctx, x, W, y, 400, K, N),
    "normalised M = 4": lambda ctx, x, W, y: fd.fdqp_run_rmsnorm_epilogue(ctx, x, x, 1e-6, W, y, fd.EPI_BF16, 4, K, N),
    "chain": lambda ctx, x, W, y: fd.fdqp_run_chain(ctx, [fd.chain_step(x, W, y[:4 * N], K, N), fd.chain_step(x[K:], W, y[4 * N:], K, N)], 2),
    "dequant": lambda ctx, x, W, y: fd.fdqp_dequant(ctx, W, y, False, K, N),
    "dequant g64": lambda ctx, x, W, y: fd.fdqp_dequant_fmt(ctx, fd.FMT_G64, W, y, True, K, N),
}


@pytest.mark.parametrize("early", [False, True])
@pytest.mark.parametrize("call", list(CALLS))
def test_weights_written_just_before_the_call(write_late, call, early):
    packed = []
    for seed in (81, 82):
        w = synthgen.weights(seed, K, N)
        packed.append(torch.from_numpy(fd.q4nx_pack(w.codes, w.scales, w.offsets)).cuda())
    x = torch.from_numpy(synthgen.activations(83, 400, K).view("int16")).cuda().view(-1)
    W = torch.zeros_like(packed[0])
    ctx = fd.fdqp_create(0, 400, K, N)
    try:
        if early:
            fd.fdqp_set_param(ctx, "launch_ahead", 0)
        if "slices" in call:
            fd.fdqp_set_param(ctx, "split_k", 2)

        def run(weights):
            y = torch.zeros(K * N, dtype=torch.float32, device="cuda")
            torch.cuda.synchronize()
            return y, lambda: CALLS[call](ctx, x, weights, y)
        expected = []
        for p in packed:
            y, go = run(p)
            go()
            torch.cuda.synchronize()
            expected.append(y)
        assert not torch.equal(*expected)
        for i in range(6):
            y, go = run(W)
            (write_late if early else _ordinary)(packed[i % 2], W)
            go()
            torch.cuda.synchronize()
            assert fd.fdqp_last_status(ctx) == 0
            assert torch.equal(y.view(torch.int32), expected[i % 2].view(torch.int32))
    finally:
        fd.fdqp_destroy(ctx)
