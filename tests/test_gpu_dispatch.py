"""The table of kept dispatches: what a call launches and returns depends on its sizes and the parameters alone."""
import numpy as np
import pytest
import torch

import paper_2602_06063_b200 as fd
import synthgen
from gpu_common import Case

pytestmark = pytest.mark.gpu


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
