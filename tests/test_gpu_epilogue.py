"""GPU parity of the fused store-side epilogues (bf16 output, gated GELU on a fused gate|up projection) against the
CPU oracle, through the C ABI, on every kernel family the projection dispatches to."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_06063_b200 as fd
import synthgen
from gpu_common import ABS_TOL, MAX_K, MAX_M, MAX_N, REL_TOL, Case

pytestmark = pytest.mark.gpu

PARAMS = ("path", "split_k", "prefill_pair", "prefill_split_k", "strip_aligned", "blocks_per_warp")


@pytest.fixture(scope="module")
def ctx():
    h = fd.fdqp_create(0, MAX_M, MAX_K, MAX_N)
    yield h
    torch.cuda.synchronize()
    fd.fdqp_destroy(h)


@pytest.fixture()
def fresh(ctx):
    for key in PARAMS:
        fd.fdqp_set_param(ctx, key, -1)
    fd.fdqp_set_param(ctx, "prefill_a_tmem", 1)
    yield ctx
    for key in PARAMS:
        fd.fdqp_set_param(ctx, key, -1)
    fd.fdqp_set_param(ctx, "prefill_a_tmem", 1)


def bf16_rne_bits(f32: np.ndarray) -> np.ndarray:
    u = f32.astype(np.float32).view(np.uint32).astype(np.uint64)
    return ((u + 0x7FFF + ((u >> 16) & 1)) >> 16).astype(np.uint16)


def run_epilogue(ctx, case, epi, M=None):
    M = case.M if M is None else M
    n_out = case.N // 2 if epi == fd.EPI_GEGLU_BF16 else case.N
    out = torch.full((M, n_out), -1, dtype=torch.int16, device="cuda")
    fd.fdqp_run_epilogue(ctx, case.x_dev, case.W_dev, out, epi, M, case.K, case.N)
    torch.cuda.synchronize()
    assert fd.fdqp_last_status(ctx) == 0
    return out.cpu().numpy().view(np.uint16)


def geglu_bound(y_ref, a_ref):
    """Per-output bound on |out - out_ref| that follows from the projection's acceptance bound: the gate and the up
    value may each be off by tol = REL_TOL * A + ABS_TOL; |gelu'| <= 1.13; then one bf16 rounding (2^-8 relative,
    which also covers the fp32 evaluation of tanh)."""
    M, N = y_ref.shape
    tol = REL_TOL * a_ref + ABS_TOL
    yv = y_ref.reshape(M, N // 32, 2, 16)
    tv = tol.reshape(M, N // 32, 2, 16)
    g, u, tg, tu = yv[:, :, 0], yv[:, :, 1], tv[:, :, 0], tv[:, :, 1]
    gelu_g = np.vectorize(oracle.gelu_tanh)(g)
    out = gelu_g * u
    bound = 1.13 * tg * (np.abs(u) + tu) + np.abs(gelu_g) * tu + np.abs(out) * 2.0 ** -8 + 1e-6
    return bound.reshape(M, N // 2)


# (K, N, M, launch parameters): every kernel family and reduction path
CASES = [
    (1152, 288, 1, {}),                                  # GEMV, one token, tail block
    (2560, 2048, 2, {}),                                 # GEMV, two tokens
    (1024, 512, 5, {}),                                  # GEMV, plane mode
    (4096, 4736, 8, {"strip_aligned": 0}),               # strips shared between CTAs (arrival counters)
    (10240, 320, 3, {"split_k": 4}),                     # K slices + sum kernel
    (1056, 320, 20, {"path": 2}),                        # GEMV eight rows at a time
    (1056, 320, 40, {"path": 3}),                        # streaming tensor-core kernel
    (1056, 320, 40, {"path": 3, "prefill_pair": 0}),     # one-SM tile kernel
    (1056, 320, 200, {"path": 3, "prefill_pair": 0}),    # ... 256-row tiles
    (2048, 256, 64, {"path": 3, "prefill_split_k": 4}),  # ... with K slices + sum kernel
    (1056, 320, 40, {"path": 3, "prefill_pair": 0, "prefill_a_tmem": 2}),   # ... three CTAs per SM (up to 64 tokens)
    (2048, 256, 64, {"path": 3, "prefill_a_tmem": 2, "prefill_split_k": 4}),
    (544, 1056, 300, {"path": 3}),                       # streaming kernel, two token tiles
    (544, 1056, 300, {"path": 3, "prefill_pair": 1}),    # two-SM tile kernel, ragged tokens
    (4096, 288, 512, {"path": 3, "prefill_split_k": 3}),
]


@pytest.mark.parametrize("K,N,M,params", CASES)
def test_bf16_epilogue_is_the_rounded_fp32_result(fresh, K, N, M, params):
    case = Case(K, N, M, seed=4000 + K + N + M)
    for k, v in params.items():
        fd.fdqp_set_param(fresh, k, v)
    y = case.run(fresh)                                   # fp32 through the same kernels
    out = run_epilogue(fresh, case, fd.EPI_BF16)
    assert np.array_equal(out, bf16_rne_bits(y))          # same arithmetic, one extra rounding: bit for bit
    # and EPI_NONE is fdqp_run
    o32 = torch.empty((M, N), dtype=torch.float32, device="cuda")
    fd.fdqp_run_epilogue(fresh, case.x_dev, case.W_dev, o32, fd.EPI_NONE, M, K, N)
    torch.cuda.synchronize()
    assert np.array_equal(o32.cpu().numpy(), y)


@pytest.mark.parametrize("K,N,M,params", CASES)
def test_geglu_epilogue_matches_oracle(fresh, K, N, M, params):
    case = Case(K, N, M, seed=5000 + K + N + M)
    for k, v in params.items():
        fd.fdqp_set_param(fresh, k, v)
    out = synthgen.bf16_to_f32(run_epilogue(fresh, case, fd.EPI_GEGLU_BF16)).astype(np.float64)
    y_ref, a_ref = case.reference()
    out_ref, _ = oracle.geglu(y_ref)
    err = np.abs(out - out_ref)
    bound = geglu_bound(y_ref, a_ref)
    assert np.all(np.isfinite(out))
    bad = err > bound
    assert not bad.any(), f"{bad.sum()} of {bad.size} outside the bound, first {np.argwhere(bad)[0]}"


@pytest.mark.parametrize("M,params", [(1, {}), (2, {}), (6, {"strip_aligned": 0}), (8, {"split_k": 2}), (24, {"path": 3}),
                                      (300, {"path": 3}), (24, {"path": 3, "prefill_pair": 0}), (300, {"path": 3, "prefill_pair": 1})])
def test_geglu_pairing_exact(fresh, M, params):
    # d = 2^-3, m = 1, x = 1: every y is an exact dyadic >= K, where gelu(g) = g in fp32 (tanh saturates), so the
    # output is exactly the bf16 of the exact product of rows r and r + 16 of each strip, as the oracle computes it
    K, N = 128, 576
    r = synthgen.u64(77, 0, N * K).reshape(N, K)
    w = synthgen.Q4NXWeights((r >> np.uint64(60)).astype(np.uint8), np.full((N, K // 32), 0x3E00, np.uint16),
                             np.full((N, K // 32), 0x3F80, np.uint16))
    x = np.full((M, K), 0x3F80, np.uint16)
    x[:, ::3] = 0x4000                                    # some activations are 2
    case = Case(K, N, M, seed=0, weights=w, x=x)
    for k, v in params.items():
        fd.fdqp_set_param(fresh, k, v)
    y_ref, _ = case.reference()
    assert y_ref.min() >= K
    _, out16_ref = oracle.geglu(y_ref)
    assert np.array_equal(run_epilogue(fresh, case, fd.EPI_GEGLU_BF16), out16_ref)


def test_epilogue_argument_errors(fresh):
    case = Case(256, 64, 1, seed=9)
    out = torch.empty((1, 64), dtype=torch.int16, device="cuda")
    lib = fd.load_library()
    s = torch.cuda.current_stream().cuda_stream
    args = (fresh, case.x_dev.data_ptr(), case.W_dev.data_ptr(), out.data_ptr())
    assert lib.fdqp_run_epilogue(*args, 3, 1, 256, 64, s) == 1       # unknown epilogue
    assert lib.fdqp_run_epilogue(*args[:3], None, 1, 1, 256, 64, s) == 1
    fd.fdqp_set_param(fresh, "path", 1)
    assert lib.fdqp_run_epilogue(*args, 1, 1, 256, 64, s) == 1       # the plain self-check kernel is fp32-only
    assert lib.fdqp_run_epilogue(*args, 0, 1, 256, 64, s) == 0
    torch.cuda.synchronize()


def test_gemma3_12b_gate_up_gated_gelu_full_size(ctx):
    # the fused gate|up projection of the 12B model at its full size, decode batch sizes, default launch plan; the
    # fused matrix's rows are read as interleaved gate / up rows (sixteen by sixteen per strip)
    for key in PARAMS:
        fd.fdqp_set_param(ctx, key, -1)
    _, K, N, seed = synthgen.GEMMA3_12B_GATE_UP
    case = Case(K, N, 8, seed)
    y_ref, a_ref = case.reference()
    out_ref, _ = oracle.geglu(y_ref)
    bound = geglu_bound(y_ref, a_ref)
    for M in (1, 2, 4, 8):
        out = synthgen.bf16_to_f32(run_epilogue(ctx, case, fd.EPI_GEGLU_BF16, M=M)).astype(np.float64)
        assert np.all(np.isfinite(out))
        assert np.all(np.abs(out - out_ref[:M]) <= bound[:M]), f"12B gate|up gated GELU M={M}"


# ---- RMS normalisation ahead of the projection ----------------------------------------------------------------------

def run_norm(ctx, case, gamma_dev, eps, epi, M=None):
    M = case.M if M is None else M
    n_out = case.N // 2 if epi == fd.EPI_GEGLU_BF16 else case.N
    dt = torch.float32 if epi == fd.EPI_NONE else torch.int16
    out = torch.zeros((M, n_out), dtype=dt, device="cuda")
    fd.fdqp_run_rmsnorm_epilogue(ctx, case.x_dev, gamma_dev, eps, case.W_dev, out, epi, M, case.K, case.N)
    torch.cuda.synchronize()
    assert fd.fdqp_last_status(ctx) == 0
    return out.cpu().numpy()


# (K, N, M, launch parameters, launches expected for the call)
NORM_CASES = [
    (2560, 2048, 1, {}, 1),                # fused into the GEMV launch
    (1152, 288, 3, {}, 1),                 # fused, three token rows, tail block
    (2560, 512, 2, {}, 2),                 # more than one item per thread: norm kernel + GEMV (which prepares in-kernel)
    (2560, 512, 4, {}, 2),                 # three and more token rows: the norm kernel leaves the rows prepared for the GEMV launch
    (1056, 320, 8, {}, 2),                 # the same, short last block (its absent group-tiles are prepared from zeros)
    (10240, 320, 1, {}, 3),                # too many items for in-kernel preparation: norm kernel + preparation + GEMV
    (1056, 320, 20, {"path": 2}, 6),       # norm kernel, two GEMV chunks of eight rows with their preparation, one of four without
    (1056, 320, 40, {"path": 3, "prefill_split_k": 2}, 3),  # norm kernel + tensor-core kernel (K slices) + its sum kernel
    (1056, 320, 40, {"path": 3, "prefill_split_k": 1}, 2),       # norm kernel + tensor-core kernel
    (544, 1056, 300, {"path": 3, "prefill_split_k": 1}, 2),
]


@pytest.mark.parametrize("K,N,M,params,launches", NORM_CASES)
def test_rmsnorm_then_projection_matches_oracle(fresh, K, N, M, params, launches):
    case = Case(K, N, M, seed=6000 + K + N + M, amp=3.0)
    gamma = synthgen.bf16_bits((0.25 * synthgen.bf16_to_f32(synthgen.activations(6100 + K, 1, K))[0]).astype(np.float32))
    gamma_dev = torch.from_numpy(gamma.view(np.int16)).cuda()
    eps = 1e-6
    for k, v in params.items():
        fd.fdqp_set_param(fresh, k, v)
    before = fd.fdqp_launch_count(fresh)
    y = run_norm(fresh, case, gamma_dev, eps, fd.EPI_NONE)
    assert fd.fdqp_launch_count(fresh) - before == launches
    x_n = oracle.rmsnorm(case.x, gamma, eps)
    y_ref, a_ref = oracle.project(x_n, case.w.codes, case.w.scales, case.w.offsets, nthreads=8)
    err = np.abs(y.astype(np.float64) - y_ref)
    assert np.all(np.isfinite(y)) and np.all(err <= REL_TOL * a_ref + ABS_TOL)
    # together with the gated GELU epilogue
    out = synthgen.bf16_to_f32(run_norm(fresh, case, gamma_dev, eps, fd.EPI_GEGLU_BF16).view(np.uint16)).astype(np.float64)
    out_ref, _ = oracle.geglu(y_ref)
    assert np.all(np.abs(out - out_ref) <= geglu_bound(y_ref, a_ref))


@pytest.mark.parametrize("K,N,M,params", [(2560, 1024, 1, {}), (2560, 512, 2, {}), (512, 288, 40, {"path": 3})])
def test_rmsnorm_of_constant_rows_is_exact(fresh, K, N, M, params):
    # a row of constant magnitude normalises to +-1 exactly (gamma = 0), whatever the magnitude: the result must be
    # bit-equal to the plain projection of that +-1 row
    case = Case(K, N, M, seed=61)
    signs = np.where(synthgen.bf16_to_f32(case.x) >= 0, 1.0, -1.0).astype(np.float32)
    mags = np.array([0.37, 5.0, 1000.0, 0.002] * ((M + 3) // 4), np.float32)[:M, None]
    scaled = Case(K, N, M, seed=61, weights=case.w, x=synthgen.bf16_bits(signs * mags))
    unit = Case(K, N, M, seed=61, weights=case.w, x=synthgen.bf16_bits(signs))
    for k, v in params.items():
        fd.fdqp_set_param(fresh, k, v)
    gamma_dev = torch.zeros(K, dtype=torch.int16, device="cuda")
    assert np.array_equal(run_norm(fresh, scaled, gamma_dev, 0.0, fd.EPI_NONE), unit.run(fresh))


def test_rmsnorm_argument_errors(fresh):
    case = Case(256, 64, 1, seed=9)
    out = torch.empty((1, 64), dtype=torch.float32, device="cuda")
    g = torch.zeros(256 + 8, dtype=torch.int16, device="cuda")
    lib = fd.load_library()
    s = torch.cuda.current_stream().cuda_stream
    a = (fresh, case.x_dev.data_ptr())
    b = (case.W_dev.data_ptr(), out.data_ptr(), 0, 1, 256, 64, s)
    assert lib.fdqp_run_rmsnorm_epilogue(*a, None, 1e-6, *b) == 1                  # null gamma
    assert lib.fdqp_run_rmsnorm_epilogue(*a, g.data_ptr() + 2, 1e-6, *b) == 3      # misaligned gamma
    assert lib.fdqp_run_rmsnorm_epilogue(*a, g.data_ptr(), -1.0, *b) == 1          # negative eps
    assert lib.fdqp_run_rmsnorm_epilogue(*a, g.data_ptr(), 1e-6, *b) == 0
    torch.cuda.synchronize()


# ---- residual addition + RMS normalisation ahead of the projection ---------------------------------------------------

@pytest.mark.parametrize("K,N,M,params,launches", NORM_CASES)
def test_residual_add_rmsnorm_then_projection_matches_oracle(fresh, K, N, M, params, launches):
    case = Case(K, N, M, seed=6500 + K + N + M, amp=2.0)
    res = synthgen.activations(6600 + K + M, M, K, 1.5)
    res[0, :8] = case.x[0, :8] ^ 0x8000                          # exact cancellation inside a row
    gamma = synthgen.bf16_bits((0.25 * synthgen.bf16_to_f32(synthgen.activations(6700 + K, 1, K))[0]).astype(np.float32))
    gamma_dev = torch.from_numpy(gamma.view(np.int16)).cuda()
    res_dev = torch.from_numpy(res.view(np.int16)).cuda()
    h_dev = torch.full((M, K), 0x7FC0, dtype=torch.int16, device="cuda")
    out = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    eps = 1e-6
    for k, v in params.items():
        fd.fdqp_set_param(fresh, k, v)
    before = fd.fdqp_launch_count(fresh)
    fd.fdqp_run_add_rmsnorm_epilogue(fresh, case.x_dev, res_dev, h_dev, gamma_dev, eps, case.W_dev, out, fd.EPI_NONE, M, K, N)
    torch.cuda.synchronize()
    assert fd.fdqp_last_status(fresh) == 0
    assert fd.fdqp_launch_count(fresh) - before == launches      # the addition costs no launch of its own
    h_ref = oracle.add_residual(case.x, res)
    assert np.array_equal(h_dev.cpu().numpy().view(np.uint16), h_ref)          # the residual stream, bit for bit
    x_n = oracle.rmsnorm(h_ref, gamma, eps)
    y_ref, a_ref = oracle.project(x_n, case.w.codes, case.w.scales, case.w.offsets, nthreads=8)
    y = out.cpu().numpy()
    err = np.abs(y.astype(np.float64) - y_ref)
    assert np.all(np.isfinite(y)) and np.all(err <= REL_TOL * a_ref + ABS_TOL)
    # without an output for h the projection is the same, bit for bit
    out2 = torch.zeros_like(out)
    fd.fdqp_run_add_rmsnorm_epilogue(fresh, case.x_dev, res_dev, None, gamma_dev, eps, case.W_dev, out2, fd.EPI_NONE, M, K, N)
    torch.cuda.synchronize()
    assert torch.equal(out, out2)
    # a zero residual is the normalisation alone, bit for bit
    zero = torch.zeros_like(res_dev)
    fd.fdqp_run_add_rmsnorm_epilogue(fresh, case.x_dev, zero, None, gamma_dev, eps, case.W_dev, out2, fd.EPI_NONE, M, K, N)
    torch.cuda.synchronize()
    assert np.array_equal(out2.cpu().numpy(), run_norm(fresh, case, gamma_dev, eps, fd.EPI_NONE))


def test_residual_add_argument_errors(fresh):
    case = Case(256, 64, 1, seed=9)
    out = torch.empty((1, 64), dtype=torch.float32, device="cuda")
    g = torch.zeros(256, dtype=torch.int16, device="cuda")
    r = torch.zeros(256 + 8, dtype=torch.int16, device="cuda")
    h = torch.zeros(256, dtype=torch.int16, device="cuda")
    lib = fd.load_library()
    s = torch.cuda.current_stream().cuda_stream
    x = case.x_dev.data_ptr()
    tail = (case.W_dev.data_ptr(), out.data_ptr(), 0, 1, 256, 64, s)
    f = lib.fdqp_run_add_rmsnorm_epilogue
    assert f(fresh, x, None, h.data_ptr(), g.data_ptr(), 1e-6, *tail) == 1                 # null residual
    assert f(fresh, x, r.data_ptr() + 2, h.data_ptr(), g.data_ptr(), 1e-6, *tail) == 3     # misaligned residual
    assert f(fresh, x, r.data_ptr(), x, g.data_ptr(), 1e-6, *tail) == 1                    # h aliases x
    assert f(fresh, x, r.data_ptr(), r.data_ptr(), g.data_ptr(), 1e-6, *tail) == 1         # h aliases the residual
    assert f(fresh, x, r.data_ptr(), h.data_ptr(), g.data_ptr(), 1e-6, *tail) == 0
    torch.cuda.synchronize()
