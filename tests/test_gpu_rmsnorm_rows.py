"""The normalisation kernel at the edges of what a row's threads hold in registers: rows shorter than a warp's piece, one value
group past a piece, exactly what is held and a group past it (clusters of up to eight rows, one CTA per row beyond), and the
longest rows, whose rest is read twice -- with a residual, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_06063_b200 as fd
import synthgen
from gpu_common import ABS_TOL, MAX_K, MAX_M, REL_TOL, Case

pytestmark = pytest.mark.gpu

# up to eight rows 8192 values are held (M = 1: K too long for the projection to normalise itself), beyond that 4096; up to 2048 values
# a single CTA takes a row whatever their number
ROWS = [(1152, 2), (1152, 8), (2048, 2), (2048, 3), (2048, 8), (2080, 2), (2080, 3), (2080, 8), (32, 3), (32, 9), (256, 9), (288, 4), (4096, 9), (4128, 9), (8192, 3), (8224, 8), (8224, 1), (21504, 2), (21504, 5), (21504, 9)]


@pytest.fixture(scope="module")
def ctx():
    h = fd.fdqp_create(0, MAX_M, MAX_K, 256)
    yield h
    torch.cuda.synchronize()
    fd.fdqp_destroy(h)


@pytest.mark.parametrize("K,M", ROWS)
def test_rows_match_oracle(ctx, K, M):
    N, eps = 64, 1e-6
    case = Case(K, N, M, seed=7600 + K + M, amp=2.0)
    res = synthgen.activations(7700 + K + M, M, K, 1.5)
    gamma = synthgen.bf16_bits((0.25 * synthgen.bf16_to_f32(synthgen.activations(7800 + K, 1, K))[0]).astype(np.float32))
    gamma_dev, res_dev = torch.from_numpy(gamma.view(np.int16)).cuda(), torch.from_numpy(res.view(np.int16)).cuda()
    h_dev = torch.full((M, K), 0x7FC0, dtype=torch.int16, device="cuda")
    outs = [torch.zeros((M, N), dtype=torch.float32, device="cuda") for _ in range(2)]
    for out in outs:
        fd.fdqp_run_add_rmsnorm_epilogue(ctx, case.x_dev, res_dev, h_dev, gamma_dev, eps, case.W_dev, out, fd.EPI_NONE, M, K, N)
    torch.cuda.synchronize()
    assert fd.fdqp_last_status(ctx) == 0
    h_ref = oracle.add_residual(case.x, res)
    assert np.array_equal(h_dev.cpu().numpy().view(np.uint16), h_ref)
    y_ref, a_ref = oracle.project(oracle.rmsnorm(h_ref, gamma, eps), case.w.codes, case.w.scales, case.w.offsets, nthreads=8)
    y = outs[0].cpu().numpy()
    assert np.all(np.isfinite(y)) and np.all(np.abs(y.astype(np.float64) - y_ref) <= REL_TOL * a_ref + ABS_TOL)
    assert torch.equal(outs[0], outs[1])
