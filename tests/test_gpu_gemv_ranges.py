"""The streaming GEMV kernels where their work split has edges: strips shared by several warps of a CTA and by several CTAs,
fewer blocks than warps, one block per strip, a short last block, rings that wrap, K slices -- for every number of warps."""
import re

import numpy as np
import pytest
import torch

import paper_2602_06063_b200 as fd
import synthgen
from gpu_common import Case, exact_regime_weights, exact_regime_x

pytestmark = pytest.mark.gpu

KEYS = ("ctas_per_sm", "consumer_warps", "stages", "split_k", "strip_aligned", "prep_inline")
FORMS = [{}, {"consumer_warps": 8}, {"consumer_warps": 16}, {"ctas_per_sm": 2}, {"stages": 2}, {"strip_aligned": 0},
         {"strip_aligned": 0, "consumer_warps": 16, "stages": 2}, {"strip_aligned": 1, "prep_inline": 0}, {"split_k": 2}]
# (K, N): one block per strip; a short block alone; 1 + a short block; nb = 10, strips over several warps; one long strip
# per CTA; enough blocks that every ring wraps; 12 blocks per CTA (its own number of warps); blocks enough for 16 warps
SHAPES = [(256, 6400), (96, 64), (288, 9600), (2560, 2592), (10240, 96), (1024, 40960), (1536, 9472), (1024, 81920)]


@pytest.fixture(scope="module")
def ctx():
    h = fd.fdqp_create(0, 8, 10240, 81920)
    yield h
    torch.cuda.synchronize()
    fd.fdqp_destroy(h)


def _bound(case):
    """Every term enters within 2^-24 of itself, K / 32 group terms and K / 256 block sums are added in fp32: 2^-17 of the
    sum of magnitudes covers K up to 10240 with a factor of four to spare."""
    d = synthgen.bf16_to_f32(case.w.scales).astype(np.float64)
    m = synthgen.bf16_to_f32(case.w.offsets).astype(np.float64)
    mag = np.abs(np.repeat(d, 32, axis=1) * case.w.codes) + np.abs(np.repeat(m, 32, axis=1))
    return 2.0 ** -17 * (np.abs(synthgen.bf16_to_f32(case.x).astype(np.float64)) @ mag.T) + 1e-7


def _check_form(form, K, M, shown):
    """The form that the parameters ask for is the one that runs (K = 10240 leaves no room for the larger ones)."""
    warps, active, depth, split, aligned, smem = (int(re.search(p, shown).group(1)) for p in (
        r"fdqp_gemv_kernel<(\d+),", r"ring_blocks=(\d+)x", r"ring_blocks=\d+x(\d+)", r"split_k=(\d+)", r"strip_aligned=(\d)", r"smem=(\d+)"))
    if K < 10240:
        assert warps == form.get("consumer_warps", warps) and active == warps, shown
        if "ctas_per_sm" in form and M <= 3:
            assert warps == 8 and smem <= 115712, shown      # two CTAs fit an SM's 228 KB, of which each takes 1 KB more
    assert depth <= form.get("stages", 16), shown
    assert split == form.get("split_k", split), shown
    assert aligned == (1 if split > 1 else form.get("strip_aligned", aligned)), shown
    if "prep_inline" in form:
        assert shown.startswith("fdqp_xprep_kernel + "), shown


def test_every_number_of_warps_occurs(ctx):
    seen = {re.search(r"fdqp_gemv_kernel<(\d+),", fd.fdqp_describe(ctx, M, K, N)).group(1) for K, N in SHAPES for M in (1, 2, 3, 8)}
    assert seen == {"8", "12", "16"}


@pytest.mark.parametrize("K,N", SHAPES)
@pytest.mark.parametrize("M", [1, 2, 3, 8])
def test_every_split_gives_the_same_sums(ctx, K, N, M):
    exact = Case(K, N, M, 0, weights=exact_regime_weights(91, K, N), x=exact_regime_x(92, M, K))
    e_ref, _ = exact.reference()
    case = Case(K, N, M, seed=90 + M)
    y_ref, _ = case.reference()
    bound = _bound(case)
    try:
        for form in FORMS:
            for k in KEYS:
                fd.fdqp_set_param(ctx, k, form.get(k, -1))
            if form.get("split_k", 1) > (K + 255) // 256:
                continue
            _check_form(form, K, M, fd.fdqp_describe(ctx, M, K, N))
            assert np.array_equal(exact.run(ctx).astype(np.float64), e_ref), form
            y = case.run(ctx)
            assert np.all(np.abs(y.astype(np.float64) - y_ref) <= bound), form
            assert np.array_equal(case.run(ctx).view(np.uint32), y.view(np.uint32)), form   # fixed orders: the same bits again
    finally:
        for k in KEYS:
            fd.fdqp_set_param(ctx, k, -1)


# Where the prepared activations leave little room: rings of one block, and rings for four of the eight warps only.
@pytest.mark.parametrize("K,N,M,split_k,ring", [(40960, 64, 1, 1, "4x1"), (21504, 64, 8, 2, "4x1"), (21504, 96, 3, 1, "8x1"), (11264, 320, 8, 1, "4x1"),
                                                (61440, 64, 1, 2, "8x2")])
def test_the_tightest_layouts(K, N, M, split_k, ring):
    """Bound: as above with K / 32 <= 1920 group terms, six times those of K = 10240 in a worst case that no random case comes near."""
    exact = Case(K, N, M, 0, weights=exact_regime_weights(93, K, N), x=exact_regime_x(94, M, K))
    case = Case(K, N, M, seed=95 + M, amp=1.0 / np.sqrt(K))
    h = fd.fdqp_create(0, M, K, N)
    try:
        fd.fdqp_set_param(h, "split_k", split_k)
        shown = fd.fdqp_describe(h, M, K, N)
        assert f"ring_blocks={ring} split_k={split_k}" in shown, shown
        assert np.array_equal(exact.run(h).astype(np.float64), exact.reference()[0])
        y = case.run(h)
        assert np.all(np.abs(y.astype(np.float64) - case.reference()[0]) <= _bound(case))
        assert np.array_equal(case.run(h).view(np.uint32), y.view(np.uint32))
    finally:
        fd.fdqp_destroy(h)
