"""The streaming tensor-core kernel (pairs of SMs that stay for the call) against the CPU oracle, at the sizes where it can go
wrong: short last blocks and odd groups along K, strips missing from a tile of 256 outputs, token tiles of every accumulator
layout, ranges that cut tiles into many pieces and ranges that do not, whole x in shared memory and rings of it."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_06063_b200 as fd
import synthgen
from gpu_common import ABS_TOL, MAX_K, MAX_M, MAX_N, REL_TOL, Case, assert_close, dev_bytes, exact_regime_weights, exact_regime_x

pytestmark = pytest.mark.gpu

KEYS = ("path", "prefill_pair", "prefill_split_k", "prefill_tokens", "prefill_blocks", "prefill_cluster")


@pytest.fixture(scope="module")
def shared():
    h = fd.fdqp_create(0, MAX_M, MAX_K, MAX_N)
    yield h
    torch.cuda.synchronize()
    fd.fdqp_destroy(h)


@pytest.fixture()
def ctx(shared):
    for key in KEYS:
        fd.fdqp_set_param(shared, key, -1)
    fd.fdqp_set_param(shared, "path", 3)
    yield shared
    for key in KEYS:
        fd.fdqp_set_param(shared, key, -1)


def configure(ctx, params):
    for key, value in params.items():
        fd.fdqp_set_param(ctx, key, value)


# K: one group; one odd group; a k-step more; a whole block; a group and a k-step past a block; many blocks.  N: one strip, one
# strip of the pair's second SM, a strip short of / past a tile.  M: one and two 16-token granules, the last size with three
# stages of converted weights (64) and the next, with whole blocks of x per stage (96) and the next, with two sets of
# accumulators (128) and the next, one token tile (256) and the next, a third one.
SHAPES = [(32, 32, 9), (96, 160, 16), (64, 256, 17), (256, 288, 33), (288, 128, 48), (320, 96, 64), (1056, 320, 65), (512, 544, 96),
          (1152, 224, 97), (2592, 512, 112), (2560, 256, 128), (1024, 1120, 129), (544, 256, 208), (768, 288, 256), (1056, 320, 257),
          (512, 544, 300), (768, 160, 511), (10240, 64, 40), (21504, 32, 12)]


@pytest.mark.parametrize("K,N,M", SHAPES)
def test_matches_oracle_and_repeats(ctx, K, N, M):
    case = Case(K, N, M, seed=7000 + K + N + M, amp=1.0 / np.sqrt(K) if K > 20000 else 1.0)
    assert fd.fdqp_describe(ctx, M, K, N).startswith("fdqp_prefill_stream_kernel")
    y = case.run(ctx)
    y_ref, a_ref = case.reference()
    assert_close(y, y_ref, a_ref, f"K={K} N={N} M={M}")
    assert np.array_equal(case.run(ctx), y)          # whoever arrives last adds the pieces in the same order


# (K, N, M, parameters): a block per pair (as many pieces as blocks), two and three (ranges that begin and end inside tiles),
# whole tiles, several small token tiles, a few larger ones
CUTS = [(1056, 544, 40, {"prefill_blocks": 1}), (2560, 1024, 20, {"prefill_blocks": 3}), (2560, 768, 130, {"prefill_blocks": 4}),
        (2560, 1024, 100, {"prefill_blocks": 10}), (768, 512, 200, {"prefill_blocks": 2}), (1280, 320, 70, {"prefill_tokens": 16}),
        (1056, 544, 150, {"prefill_tokens": 64, "prefill_blocks": 2}), (544, 1056, 300, {"prefill_tokens": 128}),
        (512, 288, 512, {"prefill_tokens": 112, "prefill_blocks": 1})]


@pytest.mark.parametrize("K,N,M,params", CUTS)
def test_every_cut_is_exact_on_exact_inputs(ctx, K, N, M, params):
    """Weights that bf16 holds and small integers: any order of summation is exact, so every cut returns the oracle's numbers."""
    case = Case(K, N, M, seed=0, weights=exact_regime_weights(81, K, N), x=exact_regime_x(82, M, K))
    y_ref, _ = case.reference()
    assert np.array_equal(case.run(ctx).astype(np.float64), y_ref)
    configure(ctx, params)
    assert np.array_equal(case.run(ctx).astype(np.float64), y_ref)


# Three and more tiles to a pair of SMs, of one block of K (160 tiles) and of two (with five blocks to a pair a range ends in the
# middle of a tile): the last of them is read by warps that have read none of the others.  Both numbers of stages of converted weights.
@pytest.mark.parametrize("K,N,params", [(32, 40960, {}), (256, 40960, {}), (288, 40960, {}), (512, 47360, {"prefill_blocks": 5}), (512, 56864, {"prefill_blocks": 7})])
@pytest.mark.parametrize("M", [17, 33, 48, 64, 100, 128])
def test_short_tiles_in_a_row(ctx, K, N, params, M):
    case = Case(K, N, M, seed=0, weights=exact_regime_weights(85, K, N), x=exact_regime_x(86, M, K))
    configure(ctx, params)
    assert fd.fdqp_describe(ctx, M, K, N).startswith("fdqp_prefill_stream_kernel")
    y_ref, _ = case.reference()
    ys = [torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda") for _ in range(4)]
    for y in ys:                                       # back to back: a launch begins while the one before it ends
        fd.fdqp_run(ctx, case.x_dev, case.W_dev, y, M, K, N)
    torch.cuda.synchronize()
    assert fd.fdqp_last_status(ctx) == 0
    for y in ys:
        assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref)


@pytest.mark.parametrize("K,N,M,params", CUTS)
def test_bf16_and_gated_stores(ctx, K, N, M, params):
    case = Case(K, N, M, seed=7500 + K + N + M)
    configure(ctx, params)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    b = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    g = torch.empty((M, N // 2), dtype=torch.bfloat16, device="cuda")
    fd.fdqp_run(ctx, case.x_dev, case.W_dev, y, M, K, N)
    fd.fdqp_run_epilogue(ctx, case.x_dev, case.W_dev, b, fd.EPI_BF16, M, K, N)
    fd.fdqp_run_epilogue(ctx, case.x_dev, case.W_dev, g, fd.EPI_GEGLU_BF16, M, K, N)
    torch.cuda.synchronize()
    assert fd.fdqp_last_status(ctx) == 0
    assert torch.equal(b, y.to(torch.bfloat16))       # the same sums, one more rounding
    gate, up = y.double().view(M, N // 32, 2, 16).unbind(2)
    want = (torch.nn.functional.gelu(gate, approximate="tanh") * up).reshape(M, N // 2)
    # one rounding to bf16 (2^-8), and gelu by fp32 fast-math instructions: 2^-20 of |g u|
    bound = want.abs() * 2.0 ** -8 + (gate * up).abs().reshape(M, N // 2) * 2.0 ** -20 + 1e-30
    assert torch.all((g.double() - want).abs() <= bound)


# (K, N, M): clusters of two and of four pairs, with a remainder of K blocks, one or two 16-token granules to a part, strips missing
@pytest.mark.parametrize("K,N,M", [(512, 32, 9), (1056, 160, 37), (2592, 288, 64), (2560, 1024, 96), (2560, 4096, 128), (1280, 544, 200), (6912, 1152, 20)])
def test_pairs_of_a_cluster_add_their_sums(ctx, K, N, M):
    case = Case(K, N, M, seed=0, weights=exact_regime_weights(83, K, N), x=exact_regime_x(84, M, K))
    y_ref, _ = case.reference()
    fd.fdqp_set_param(ctx, "prefill_cluster", 1)
    assert "cut=clusters" in fd.fdqp_describe(ctx, M, K, N)
    assert np.array_equal(case.run(ctx).astype(np.float64), y_ref)
    fd.fdqp_set_param(ctx, "prefill_cluster", 0)
    assert "cut=clusters" not in fd.fdqp_describe(ctx, M, K, N)
    assert np.array_equal(case.run(ctx).astype(np.float64), y_ref)


@pytest.mark.parametrize("fmt", [fd.FMT_G64, fd.FMT_G128, fd.FMT_MXFP4])
@pytest.mark.parametrize("K,N,M,blocks", [(256, 32, 9, -1), (1280, 288, 37, 2), (2560, 544, 130, 3)])
def test_format_variants(ctx, fmt, K, N, M, blocks):
    fd.fdqp_set_param(ctx, "prefill_blocks", blocks)
    w, x = synthgen.weights_fmt(7800 + K + fmt, K, N, fmt), synthgen.activations(7801 + K, M, K)
    W = dev_bytes(fd.q4nx_pack_fmt(fmt, w.codes, w.scales, w.offsets))
    y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    fd.fdqp_run_fmt(ctx, fmt, dev_bytes(x), W, y, M, K, N)
    torch.cuda.synchronize()
    assert fd.fdqp_last_status(ctx) == 0
    y_ref, a_ref = oracle.fmt_project(fmt, x, w.codes, w.scales, w.offsets, nthreads=min(16, oracle.max_threads()))
    assert_close(y.cpu().numpy(), y_ref, a_ref, f"format {fmt}")


def test_weights_are_rounded_once_for_every_finite_scale(ctx):
    """One-hot activations read out the converted weights: Eq. 3 rounded once to bf16, for scales and offsets over the whole finite
    range (64-fold scales that overflow, subnormals).  Magnitudes stay below 2^120 d * 15 + m so that nothing overflows."""
    K, N, M = 544, 96, 32
    r = synthgen.u64(78, 0, 2 * N * (K // 32)).reshape(2, N, K // 32)
    bits = ((r >> np.uint64(48)) & np.uint64(0xFFFF)).astype(np.uint16)
    expo = (bits >> 7) & 0xFF
    bits = np.where(expo > 249, (bits & 0x807F) | (249 << 7), bits).astype(np.uint16)       # up to 2^122
    codes = (synthgen.u64(79, 0, N * K).reshape(N, K) >> np.uint64(60)).astype(np.uint8)
    w = synthgen.Q4NXWeights(codes, np.ascontiguousarray(bits[0]), np.ascontiguousarray(bits[1]))
    ks = np.linspace(0, K - 1, M).astype(np.int64)
    x = np.zeros((M, K), np.float32)
    x[np.arange(M), ks] = 1.0
    y = Case(K, N, M, 0, weights=w, x=synthgen.bf16_bits(x)).run(ctx)
    d = synthgen.bf16_to_f32(w.scales).astype(np.longdouble).repeat(32, axis=1)
    m = synthgen.bf16_to_f32(w.offsets).astype(np.longdouble).repeat(32, axis=1)
    want = (d * codes + m)[:, ks].T
    # half a unit in the last place of bf16, whose smallest is that of its subnormals (2^-133); the sum above is itself rounded
    # to 64 bits, which decides nothing but exact ties
    ulp = np.exp2(np.maximum(np.floor(np.log2(np.maximum(np.abs(want), np.longdouble(2) ** -140))), -126) - 7)
    assert np.all(np.abs(y.astype(np.longdouble) - want) <= ulp / 2 * (1 + np.longdouble(2) ** -50))
    assert np.all((y.view(np.uint32) & 0xFFFF) == 0)


def test_calls_in_a_row_share_the_workspace(ctx):
    """Shared tiles' counters and partial sums are the same memory from call to call, and a launch may begin before the one before
    it has ended."""
    cases = [Case(2560, 544, 20, 1), Case(1056, 320, 200, 2), Case(10240, 96, 40, 3), Case(768, 1120, 100, 4)]
    alone = [c.run(ctx) for c in cases]
    ys = [torch.full((c.M, c.N), float("nan"), dtype=torch.float32, device="cuda") for c in cases]
    for _ in range(8):
        for c, y in zip(cases, ys):
            fd.fdqp_run(ctx, c.x_dev, c.W_dev, y, c.M, c.K, c.N)
    torch.cuda.synchronize()
    assert fd.fdqp_last_status(ctx) == 0
    for a, y in zip(alone, ys):
        assert np.array_equal(y.cpu().numpy(), a)


def test_small_contexts_hold_their_partial_sums():
    """The workspace is sized from the maxima alone: the largest call of a small context runs."""
    for M, K, N in ((9, 2560, 64), (40, 10240, 32), (300, 1056, 288)):
        own = fd.fdqp_create(0, M, K, N)
        try:
            case = Case(K, N, M, seed=7900 + M)
            y_ref, a_ref = case.reference()
            assert_close(case.run(own), y_ref, a_ref)
        finally:
            fd.fdqp_destroy(own)


def test_parameter_values(shared):
    lib = fd.load_library()
    for key, bad in ((b"prefill_tokens", (0, 8, 24, 272)), (b"prefill_blocks", (0,))):
        for value in bad:
            assert lib.fdqp_set_param(shared, key, value) == 1
        assert lib.fdqp_set_param(shared, key, -1) == 0
