"""Accuracy of the GEMV kernels: at 3 to 8 tokens no larger an error against 64 bits than per-group fp32 arithmetic has; and which
calls of nine and more rows they serve."""
import math

import pytest
import torch

import paper_2602_06063_b200 as fd

pytestmark = pytest.mark.gpu


def _weights(g, K, N, mx):
    """Codes [N][K], scales and offsets [N][K/32] of a min/max quantised matrix of unit gain (MXFP4: E8M0 scales, no offsets)."""
    codes = torch.randint(0, 16, (N, K), dtype=torch.uint8, device="cuda", generator=g)
    if mx:
        middle = 127 + round(math.log2(1.0 / (2.9 * math.sqrt(K))))
        return codes, torch.randint(middle - 2, middle + 2, (N, K // 32), dtype=torch.uint8, device="cuda", generator=g), None
    d = (0.5 + torch.rand((N, K // 32), device="cuda", generator=g)) / (4.6 * math.sqrt(K))
    m = -7.5 * d * (1 + 0.1 * torch.randn((N, K // 32), device="cuda", generator=g))
    return codes, d.to(torch.bfloat16), m.to(torch.bfloat16)


def _packed(codes, d, m, K, N):
    """The container's bytes: strips of 32 rows, blocks of 256 inputs (K is a multiple of 256 here)."""
    nibbles = codes[:, 0::2] | (codes[:, 1::2] << 4)                                             # [N][K/2]
    blocks = nibbles.view(N // 32, 32, K // 256, 8, 16).permute(0, 2, 3, 1, 4).reshape(N // 32, K // 256, 4096)
    parts = [blocks]
    for s in (d, m):
        if s is not None:
            s = s.view(N // 32, 32, K // 256, 8).permute(0, 2, 3, 1).contiguous()
            parts.append(s.view(torch.uint8).reshape(N // 32, K // 256, -1))
    return torch.cat(parts, dim=2).contiguous().view(-1)


# The last column: K slices of the reference.  Strips of one to many blocks per warp, K that one CTA's shared memory does
# not hold beside 16 or beside 12 rings (M = 8: from 4608 and 5376 on), the format without offsets.
@pytest.mark.parametrize("K,N,M,mx,slices", [(768, 8192, 3, False, 1), (768, 8192, 8, False, 1), (2560, 20480, 3, False, 1),
                                             (2560, 20480, 8, False, 1), (5376, 43008, 8, False, 2), (21504, 16384, 6, True, 4)])
def test_no_less_exact_than_per_group_sums(K, N, M, mx, slices):
    """Reference: per 32-group sum_k code x exactly, then two FMAs per group (scale, offset) in fp32 into 16 sums per K slice,
    which are added in fp32 -- the arithmetic Eq. 3 and 15 suggest, a warp per 16th group-tile.  The norm of the kernel's
    error may be 2 % above that one's: it is a mean over M N >= 24576 independent errors, so its own spread is below
    1 / sqrt(2 M N) = 0.5 %, on either side."""
    g = torch.Generator(device="cuda").manual_seed(K + M)
    x = torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16)
    codes, d, m = _weights(g, K, N, mx)
    W = _packed(codes, d, m, K, N)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    ctx = fd.fdqp_create(0, M, K, N)
    try:
        if mx:
            fd.fdqp_run_fmt(ctx, fd.FMT_MXFP4, x, W, y, M, K, N)
        else:
            fd.fdqp_run(ctx, x, W, y, M, K, N)
        torch.cuda.synchronize()
        assert fd.fdqp_last_status(ctx) == 0
    finally:
        fd.fdqp_destroy(ctx)
    if mx:
        table = torch.tensor([0, .5, 1, 1.5, 2, 3, 4, 6, -0., -.5, -1, -1.5, -2, -3, -4, -6], dtype=torch.float64, device="cuda")
        d = torch.exp2(d.double() - 127)
    exact = torch.zeros((M, N), dtype=torch.float64, device="cuda")
    sums = [torch.zeros((M, N), dtype=torch.float64, device="cuda") for _ in range(16 * slices)]  # fp32 values
    per_slice = K // 32 // slices
    for t in range(K // 32):
        q = codes[:, 32 * t:32 * t + 32]
        q = table[q.long()] if mx else q.double()
        xt = x[:, 32 * t:32 * t + 32].double()
        terms = [(xt @ q.t()) * d[:, t].double()]
        if m is not None:
            terms.append(xt.sum(1, keepdim=True) * m[:, t].double())
        into = min(t // per_slice, slices - 1) * 16 + t % 16
        for term in terms:
            exact += term
            sums[into] = (sums[into] + term).float().double()
    ref = sums[0]
    for s in sums[1:]:
        ref = (ref + s).float().double()
    norm = exact.norm()
    got, allowed = float((y.double() - exact).norm() / norm), float((ref - exact).norm() / norm)
    assert got <= 1.02 * allowed, f"{got:.3e} against {allowed:.3e}"


@pytest.mark.parametrize("K,N,M", [(6912, 256, 9), (21504, 1024, 9), (15360, 1024, 10)])
def test_few_outputs_of_a_long_reduction_keep_fp32_weights(K, N, M):
    """Nine and more rows that the GEMV kernels serve: fp32 sums of unrounded weights differ from 64 bits by 1e-7 .. 2e-7 (norm of the
    difference over norm of y), weights rounded to bf16 by 1.5e-3.  The limit, 2e-6, lies ten times above the one."""
    g = torch.Generator(device="cuda").manual_seed(K + M)
    x = torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16)
    codes, d, m = _weights(g, K, N, False)
    W = _packed(codes, d, m, K, N)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    ctx = fd.fdqp_create(0, M, K, N)
    try:
        assert "fdqp_gemv_kernel" in fd.fdqp_describe(ctx, M, K, N)
        fd.fdqp_run(ctx, x, W, y, M, K, N)
        torch.cuda.synchronize()
        assert fd.fdqp_last_status(ctx) == 0
    finally:
        fd.fdqp_destroy(ctx)
    w = codes.double() * d.double().repeat_interleave(32, dim=1) + m.double().repeat_interleave(32, dim=1)
    exact = x.double() @ w.t()
    assert float((y.double() - exact).norm() / exact.norm()) <= 2e-6
