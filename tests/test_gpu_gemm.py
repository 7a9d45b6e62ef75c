"""GPU parity: W8A8 linear (tcgen05 int8 GEMM + de-quantising epilogue) vs the oracle."""
import os

import numpy as np
import pytest
import torch

import synth
from oracle import dit, linear, quant
from oracle.quant import QParams

from gpu_util import bf16_steps_err, bf16_to_f64, code_mismatch_report, dev, dev_i8, host_codes, max_rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import paper_2503_02508_b200 as q
    return q


@pytest.fixture(scope="module")
def ctx(q):
    c = q.qdit_create(0, None)
    yield c
    q.qdit_destroy(c)


def _codes(seed, name, shape, lo, hi):
    return synth.uniform_int(seed, name, shape, lo, hi + 1)


def _run_i32(q, ctx, qa, qw, a_unsigned=False):
    M, K = qa.shape
    N = qw.shape[0]
    A, W = dev_i8(qa), dev_i8(qw)
    out = torch.full((M, N), -7, dtype=torch.int32, device="cuda")
    qp = q.qparams(1.0, 0, 0, 255) if a_unsigned else q.qparams(1.0)
    q.qdit_w8a8_linear(ctx, A, W, M, N, K, qp, None, q.QDIT_EPI_OUT_I32, None, out, N)
    q.qdit_sync(ctx)
    return out.cpu().numpy().astype(np.int64)


SHAPES = [(1, 8, 16), (128, 192, 128), (130, 200, 272), (256, 384, 1152), (517, 1152, 4608), (512, 1152, 384),
          (1000, 3456, 1152), (64, 6912, 1152), (2048, 64, 64), (129, 1536, 384)]


def _select_kernel(q, ctx, variant):
    """"NNN": token-major kernel with 128 x NNN tiles; "tNNN": channel-major kernel with 128 x NNN tiles; else automatic."""
    q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 0)
    q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_T, 0)
    if variant.startswith("t"):
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_T, int(variant[1:]))
    elif variant.isdigit():
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, int(variant))


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("bn", ["auto", "64", "128", "192", "t128", "t256"])
def test_accumulators_bit_exact(q, ctx, M, N, K, bn):
    _select_kernel(q, ctx, bn)
    try:
        qa = _codes(31, f"a{M}.{K}", (M, K), -128, 127)
        qw = _codes(31, f"w{N}.{K}", (N, K), -127, 127)
        got = _run_i32(q, ctx, qa, qw)
    finally:
        _select_kernel(q, ctx, "auto")
    np.testing.assert_array_equal(got, linear.gemm_i8(qa, qw))


def test_accumulators_extremes_and_structure(q, ctx):
    K = 4608
    lo = np.full((130, K), -128)
    hi = np.full((200, K), 127)
    assert (_run_i32(q, ctx, lo, hi) == -128 * 127 * K).all()
    u8 = np.full((130, K), 255)
    assert (_run_i32(q, ctx, u8, hi, a_unsigned=True) == 255 * 127 * K).all()
    # identity weights return the activations; catches any K-offset / swizzle / transposition slip
    A = _codes(32, "aid", (300, 256), -128, 127)
    np.testing.assert_array_equal(_run_i32(q, ctx, A, np.eye(256, dtype=np.int64)), A)
    # one-hot rows pick single weights
    W = _codes(32, "wsel", (200, 1152), -127, 127)
    onehot = np.zeros((128, 1152), dtype=np.int64)
    ks = synth.uniform_int(32, "ks", (128,), 0, 1152)
    onehot[np.arange(128), ks] = 1
    np.testing.assert_array_equal(_run_i32(q, ctx, onehot, W), W[:, ks].T)


def test_unsigned_activations_bit_exact(q, ctx):
    qa = _codes(33, "au", (260, 1152), 0, 255)
    qw = _codes(33, "wu", (392, 1152), -127, 127)
    np.testing.assert_array_equal(_run_i32(q, ctx, qa, qw, a_unsigned=True), linear.gemm_i8(qa, qw))


def test_repeatable(q, ctx):
    qa = _codes(34, "ar", (1024, 1152), -128, 127)
    qw = _codes(34, "wr", (1152, 1152), -127, 127)
    a = _run_i32(q, ctx, qa, qw)
    b = _run_i32(q, ctx, qa, qw)
    np.testing.assert_array_equal(a, b)


def _layer(seed, M, N, K, T, a_qp):
    x = synth.outlier_activations(seed, "x", M, K, gain=6.0)
    Wf = synth.normal(seed, "W", (N, K), 0.02)
    bias = synth.normal(seed, "b", (N,), 0.02)
    gate = synth.normal(seed, "g", (-(-M // T), N), 0.35)
    resid = synth.normal(seed, "r", (M, N), 1.0)
    qw, s_w, cs = quant.quantize_weight_per_channel(Wf)
    qa = quant.quantize(x, a_qp)
    return dict(qa=qa, qw=qw, s_w=s_w, cs=cs, bias=bias, gate=gate, resid=resid)


@pytest.mark.parametrize("M,N,K,T", [(512, 384, 384, 256), (300, 200, 1152, 100), (1024, 1152, 4608, 256)])
@pytest.mark.parametrize("a_qp", [QParams(0.05, 0, -127, 127), QParams(0.047, 131, 0, 255)])
def test_dequant_bias_f32(q, ctx, M, N, K, T, a_qp):
    L = _layer(41, M, N, K, T, a_qp)
    A, W = dev_i8(L["qa"]), dev_i8(L["qw"])
    epi = q.epilogue(w_scale=dev(L["s_w"]), w_colsum=dev(L["cs"].astype(np.int32)), bias=dev(L["bias"]))
    keep = [epi]
    ws, wc, bi = dev(L["s_w"]), dev(L["cs"].astype(np.int32)), dev(L["bias"])
    epi = q.epilogue(w_scale=ws, w_colsum=wc, bias=bi)
    out = torch.empty((M, N), dtype=torch.float32, device="cuda")
    q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale, a_qp.zero_point, a_qp.qmin, a_qp.qmax), None,
                       q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32, epi, out, N)
    q.qdit_sync(ctx)
    ref = linear.w8a8_linear(L["qa"], a_qp, L["qw"], L["s_w"], L["cs"], L["bias"])
    assert max_rel_err(out.cpu().numpy(), ref) < 1e-3      # the stated layer tolerance ...
    assert max_rel_err(out.cpu().numpy(), ref) < 1e-5      # ... and what f32 arithmetic actually gives


@pytest.fixture(params=["single", "192", "t128", "t256"])
def kernel_variant(request, q, ctx):
    _select_kernel(q, ctx, request.param)
    yield request.param
    _select_kernel(q, ctx, "auto")


def test_gate_residual_cache_epilogue(q, ctx, kernel_variant):
    M, N, K, T = 512, 1152, 1152, 256
    a_qp = QParams(0.05, 0, -127, 127)
    L = _layer(42, M, N, K, T, a_qp)
    A, W = dev_i8(L["qa"]), dev_i8(L["qw"])
    ws, bi, g = dev(L["s_w"]), dev(L["bias"]), dev(L["gate"])
    x = dev(L["resid"]).to(torch.bfloat16)
    xh = bf16_to_f64(x)
    cache = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    epi = q.epilogue(w_scale=ws, bias=bi, gate=g, ld_gate=N, tokens_per_sample=T, residual=x, cache_out=cache)
    flags = q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_CACHE_STORE | q.QDIT_EPI_OUT_BF16
    q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None, flags, epi, x, N)    # in place on x
    q.qdit_sync(ctx)
    f = linear.w8a8_linear(L["qa"], a_qp, L["qw"], L["s_w"], L["cs"], L["bias"])
    rows = np.arange(M) // T
    want_x = xh + L["gate"].astype(np.float64)[rows] * f
    # bf16 outputs: equal to the rounded oracle value up to one bf16 step where f32 and f64 straddle a tie
    got_c, got_x = bf16_to_f64(cache), bf16_to_f64(x)
    assert np.abs(got_c - dit.round_bf16(f)).max() <= 2.0 ** -8 * np.abs(f).max()
    assert (got_c != dit.round_bf16(f)).mean() < 1e-3
    assert (got_x != dit.round_bf16(want_x)).mean() < 1e-3
    assert max_rel_err(got_x, want_x) < 2.0 ** -8


def test_bias_bf16_epilogue(q, ctx, kernel_variant):
    # the QKV layer's epilogue, on ragged sizes (M, N not multiples of the tiles)
    M, N, K, T = 300, 1096, 384, 100
    a_qp = QParams(0.045, 0, -127, 127)
    L = _layer(45, M, N, K, T, a_qp)
    A, W = dev_i8(L["qa"]), dev_i8(L["qw"])
    ws, bi = dev(L["s_w"]), dev(L["bias"])
    out = torch.full((M, N), 7.0, dtype=torch.bfloat16, device="cuda")
    q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None, q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_BF16,
                       q.epilogue(w_scale=ws, bias=bi), out, N)
    q.qdit_sync(ctx)
    f = linear.w8a8_linear(L["qa"], a_qp, L["qw"], L["s_w"], L["cs"], L["bias"])
    got = bf16_to_f64(out)
    assert (got != dit.round_bf16(f)).mean() < 1e-3
    assert np.abs(got - f).max() <= 2.0 ** -8 * np.abs(f).max()


def test_gelu_requant_epilogue(q, ctx, kernel_variant):
    M, N, K, T = 384, 1536, 384, 128
    a_qp = QParams(0.04, 0, -127, 127)
    L = _layer(43, M, N, K, T, a_qp)
    A, W = dev_i8(L["qa"]), dev_i8(L["qw"])
    ws, bi = dev(L["s_w"]), dev(L["bias"])
    u = dit.gelu_tanh(linear.w8a8_linear(L["qa"], a_qp, L["qw"], L["s_w"], L["cs"], L["bias"]))
    o_qp = quant.qparams_symmetric(float(np.abs(u).max()) * 0.9)
    epi = q.epilogue(w_scale=ws, bias=bi, out_qp=q.qparams(o_qp.scale))
    out = torch.empty((M, N), dtype=torch.uint8, device="cuda")
    q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None,
                       q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT, epi, out, N)
    outf = torch.empty((M, N), dtype=torch.float32, device="cuda")
    q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None,
                       q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_OUT_F32, epi, outf, N)
    q.qdit_sync(ctx)
    assert max_rel_err(outf.cpu().numpy(), u) < 1e-3
    assert max_rel_err(outf.cpu().numpy(), u) < 2e-5
    got, want = host_codes(out), quant.quantize(u, o_qp)
    pre = u.astype(np.float32).astype(np.float64) * float(o_qp.inv_scale)
    n_bad, ok = code_mismatch_report(got, want, pre, 2e-5 * np.abs(pre).max() + 1e-6)
    assert ok and n_bad <= 1e-3 * got.size, (n_bad, got.size)
    # the fused codes are exactly the quantizer applied to the kernel's own f32 values
    np.testing.assert_array_equal(got, quant.quantize(outf.cpu().numpy(), o_qp))


@pytest.mark.parametrize("M,N,K", [(300, 384, 1152), (1024, 2304, 256)])
def test_per_token_scales(q, ctx, kernel_variant, M, N, K):
    """Per-token activation scales (QDIT_EPI_ROW_SCALE): quantizer in per-token mode, then the linear layer."""
    x = synth.outlier_activations(45, f"pt{M}", M, K) * (1.0 + (np.arange(M, dtype=np.float32)[:, None] % 5))
    W = synth.normal(45, f"ptw{N}", (N, K), 0.02)
    bias = synth.normal(45, f"ptb{N}", (N,), 0.02)
    wq, ws, wc = quant.quantize_weight_per_channel(W)
    qa, sa = quant.quantize_per_token(x)
    ref = linear.w8a8_linear_per_token(qa, sa, wq, ws, bias)
    a8 = torch.empty((M, K), dtype=torch.uint8, device="cuda")
    sc = torch.empty(M, dtype=torch.float32, device="cuda")
    q.qdit_quantize_act(ctx, dev(x), q.QDIT_F32, M, K, K, q.QDIT_QUANT_DYNAMIC_TOKEN, None, sc, a8, K)
    out = torch.empty((M, N), dtype=torch.float32, device="cuda")
    ws_d, bias_d, wq_d = dev(ws), dev(bias), dev_i8(wq)     # the epilogue struct holds raw addresses: keep the tensors alive
    epi = q.epilogue(w_scale=ws_d, bias=bias_d, a_scale_rows=sc)
    q.qdit_w8a8_linear(ctx, a8, wq_d, M, N, K, q.qparams(1.0), None,
                       q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32 | q.QDIT_EPI_ROW_SCALE, epi, out, N)
    q.qdit_sync(ctx)
    assert max_rel_err(out.cpu().numpy(), ref) < 1e-5
    # closer to the un-quantized product than one tensor-wide scale is, on rows of very different magnitude
    exact = x.astype(np.float64) @ W.astype(np.float64).T + bias
    qp = quant.qparams_symmetric(float(np.abs(x).max()))
    tens = linear.w8a8_linear(quant.quantize(x, qp), qp, wq, ws, wc, bias)
    small = np.arange(M) % 5 == 0
    assert np.abs(out.cpu().numpy()[small] - exact[small]).mean() < np.abs(tens[small] - exact[small]).mean()
    # the flag needs its scales and a symmetric quantizer
    L = q.lib
    import ctypes as C
    bad = q.epilogue(w_scale=ws_d, bias=bias_d)
    assert L.qdit_w8a8_linear(ctx, a8.data_ptr(), wq_d.data_ptr(), M, N, K, q.qparams(1.0), None,
                              q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32 | q.QDIT_EPI_ROW_SCALE, C.byref(bad), out.data_ptr(), N) == q.QDIT_ERR_INVALID_ARG


def test_device_scale_override(q, ctx):
    M, N, K = 256, 192, 256
    a_qp = QParams(0.05, 0, -127, 127)
    L = _layer(44, M, N, K, 256, a_qp)
    A, W, ws = dev_i8(L["qa"]), dev_i8(L["qw"]), dev(L["s_w"])
    sd = dev(np.array([a_qp.scale], dtype=np.float32))
    out = torch.empty((M, N), dtype=torch.float32, device="cuda")
    q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(123.0), sd, q.QDIT_EPI_OUT_F32, q.epilogue(w_scale=ws), out, N)
    q.qdit_sync(ctx)
    ref = linear.w8a8_linear(L["qa"], a_qp, L["qw"], L["s_w"], L["cs"], None)
    assert max_rel_err(out.cpu().numpy(), ref) < 1e-5


def test_rejects_bad_arguments(q, ctx):
    import ctypes as C
    A = torch.zeros((128, 64), dtype=torch.int8, device="cuda")
    W = torch.zeros((64, 64), dtype=torch.int8, device="cuda")
    o = torch.zeros((128, 64), dtype=torch.int32, device="cuda")
    L, qp = q.lib, q.qparams(1.0)
    f = L.qdit_w8a8_linear
    assert f(ctx, A.data_ptr(), W.data_ptr(), 128, 64, 24, qp, None, q.QDIT_EPI_OUT_I32, None, o.data_ptr(), 64) == q.QDIT_ERR_SHAPE
    assert f(ctx, A.data_ptr(), W.data_ptr(), 128, 60, 64, qp, None, q.QDIT_EPI_OUT_I32, None, o.data_ptr(), 64) == q.QDIT_ERR_SHAPE
    assert f(ctx, None, W.data_ptr(), 128, 64, 64, qp, None, q.QDIT_EPI_OUT_I32, None, o.data_ptr(), 64) == q.QDIT_ERR_INVALID_ARG
    assert f(ctx, A.data_ptr() + 1, W.data_ptr(), 128, 64, 64, qp, None, q.QDIT_EPI_OUT_I32, None, o.data_ptr(), 64) == q.QDIT_ERR_ALIGN
    assert f(ctx, A.data_ptr(), W.data_ptr(), 128, 64, 64, qp, None, 0, None, o.data_ptr(), 64) == q.QDIT_ERR_INVALID_ARG
    assert f(ctx, A.data_ptr(), W.data_ptr(), 128, 64, 64, qp, None, q.QDIT_EPI_OUT_F32 | q.QDIT_EPI_OUT_BF16, None, o.data_ptr(), 64) == q.QDIT_ERR_INVALID_ARG
    assert f(ctx, A.data_ptr(), W.data_ptr(), 128, 64, 64, qp, None, q.QDIT_EPI_OUT_F32, None, o.data_ptr(), 64) == q.QDIT_ERR_INVALID_ARG
    assert f(ctx, A.data_ptr(), W.data_ptr(), 0, 64, 64, qp, None, q.QDIT_EPI_OUT_I32, None, o.data_ptr(), 64) == q.QDIT_OK
    q.qdit_sync(ctx)


@pytest.mark.parametrize("M,T", [(192, 64), (300, 100), (1184, 32)])
def test_gated_epilogue_on_ragged_rows_with_an_exactly_sized_gate(q, ctx, kernel_variant, M, T):
    """The last tile is ragged (M % 128 != 0) and the gate tensor has exactly ceil(M / T) rows: no row past it may
    be read (the warps of a tile whose rows lie wholly past M have no sample)."""
    N, K = 1152, 384
    a_qp = QParams(0.05, 0, -127, 127)
    L = _layer(46, M, N, K, T, a_qp)
    B = -(-M // T)
    gate_h = synth.normal(46, "g2", (B, N), 0.35)
    A, W = dev_i8(L["qa"]), dev_i8(L["qw"])
    ws, bi = dev(L["s_w"]), dev(L["bias"])
    # the gate sits at the very end of its allocation, followed by a canary region that must stay untouched (reads
    # past the end cannot be seen directly; the exact size is what the kernels are given)
    g = dev(gate_h)
    x = dev(L["resid"]).to(torch.bfloat16)
    xh = bf16_to_f64(x)
    cache = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    epi = q.epilogue(w_scale=ws, bias=bi, gate=g, ld_gate=N, tokens_per_sample=T, residual=x, cache_out=cache)
    flags = q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_CACHE_STORE | q.QDIT_EPI_OUT_BF16
    q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None, flags, epi, x, N)
    q.qdit_sync(ctx)
    f = linear.w8a8_linear(L["qa"], a_qp, L["qw"], L["s_w"], L["cs"], L["bias"])
    rows = np.arange(M) // T
    want_x = xh + gate_h.astype(np.float64)[rows] * f
    got_c, got_x = bf16_to_f64(cache), bf16_to_f64(x)
    assert (got_c != dit.round_bf16(f)).mean() < 1e-3
    assert (got_x != dit.round_bf16(want_x)).mean() < 1e-3
    assert max_rel_err(got_x, want_x) < 2.0 ** -8


FULL_M = 8192   # tokens of the 50-step workload: network batch 32 x 256 tokens


@pytest.mark.parametrize("K,N,name", [(1152, 3456, "qkv"), (1152, 1152, "proj"), (1152, 4608, "fc1"), (4608, 1152, "fc2")])
def test_full_size_layers_element_by_element(q, ctx, K, N, name):
    """The four block-level layers at the full workload's size, in the kernels the model path selects: raw int32
    accumulators bit-exact, f32 outputs within 1e-3 (measured 1e-5), and each layer's own fused epilogue against the
    oracle on every element."""
    M, T = FULL_M, 256
    a_qp = QParams(0.05, 0, -127, 127)
    L = _layer(47, M, N, K, T, a_qp)
    A, W = dev_i8(L["qa"]), dev_i8(L["qw"])
    ws, bi, g = dev(L["s_w"]), dev(L["bias"]), dev(L["gate"])
    acc = linear.gemm_i8(L["qa"], L["qw"])
    f = linear.w8a8_linear(L["qa"], a_qp, L["qw"], L["s_w"], L["cs"], L["bias"])
    for variant in ("auto", "t256"):
        _select_kernel(q, ctx, variant)
        try:
            np.testing.assert_array_equal(_run_i32(q, ctx, L["qa"], L["qw"]), acc)
            outf = torch.empty((M, N), dtype=torch.float32, device="cuda")
            q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None, q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32,
                               q.epilogue(w_scale=ws, bias=bi), outf, N)
            q.qdit_sync(ctx)
            assert max_rel_err(outf.cpu().numpy(), f) < 1e-5
        finally:
            _select_kernel(q, ctx, "auto")
    if name == "qkv":
        out = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
        q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None, q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_BF16,
                           q.epilogue(w_scale=ws, bias=bi), out, N)
        q.qdit_sync(ctx)
        got = bf16_to_f64(out)
        assert (got != dit.round_bf16(f)).mean() < 1e-4 and bf16_steps_err(got, f) <= 1.0
    elif name == "fc1":
        u = dit.gelu_tanh(f)
        o_qp = quant.qparams_symmetric(float(np.abs(u).max()) * 0.9)
        out = torch.empty((M, N), dtype=torch.uint8, device="cuda")
        q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None,
                           q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT,
                           q.epilogue(w_scale=ws, bias=bi, out_qp=q.qparams(o_qp.scale)), out, N)
        q.qdit_sync(ctx)
        got, want = host_codes(out), quant.quantize(u, o_qp)
        pre = u.astype(np.float32).astype(np.float64) * float(o_qp.inv_scale)
        n_bad, ok = code_mismatch_report(got, want, pre, 2e-5 * np.abs(pre).max() + 1e-6)
        assert ok and n_bad <= 1e-3 * got.size, (n_bad, got.size)
    else:
        x = dev(L["resid"]).to(torch.bfloat16)
        xh = bf16_to_f64(x)
        cache = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
        epi = q.epilogue(w_scale=ws, bias=bi, gate=g, ld_gate=N, tokens_per_sample=T, residual=x, cache_out=cache)
        flags = q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_CACHE_STORE | q.QDIT_EPI_OUT_BF16
        q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None, flags, epi, x, N)
        q.qdit_sync(ctx)
        want_x = xh + L["gate"].astype(np.float64)[np.arange(M) // T] * f
        got_c, got_x = bf16_to_f64(cache), bf16_to_f64(x)
        assert (got_c != dit.round_bf16(f)).mean() < 1e-4 and bf16_steps_err(got_c, f) <= 1.0
        assert (got_x != dit.round_bf16(want_x)).mean() < 1e-3 and bf16_steps_err(got_x, want_x) <= 1.0


def test_options_select_kernels_and_reject_bad_values(q, ctx):
    assert q.qdit_get_option(ctx, q.QDIT_OPT_PDL) == 1
    for opt, bad in ((q.QDIT_OPT_GEMM_BN, 96), (q.QDIT_OPT_GEMM_T, 64), (q.QDIT_OPT_ATTN, 3), (q.QDIT_OPT_PDL, 2), (99, 0)):
        assert q.lib.qdit_set_option(ctx, opt, bad) == q.QDIT_ERR_INVALID_ARG
    q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_T, 128)
    assert q.qdit_get_option(ctx, q.QDIT_OPT_GEMM_T) == 128
    q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_T, 0)
    # with and without programmatic dependent launch: same bits
    qa = _codes(35, "ap", (600, 384), -128, 127)
    qw = _codes(35, "wp", (384, 384), -127, 127)
    a = _run_i32(q, ctx, qa, qw)
    q.qdit_set_option(ctx, q.QDIT_OPT_PDL, 0)
    try:
        b = _run_i32(q, ctx, qa, qw)
    finally:
        q.qdit_set_option(ctx, q.QDIT_OPT_PDL, 1)
    np.testing.assert_array_equal(a, b)


# ----------------------------------------------------------------------------- packed 4-bit weights (W4A8, Table 2)
def _w4_codes(seed, name, N, K):
    return synth.uniform_int(seed, name, (N, K), -8, 8).astype(np.int64)


def test_w4_pack_unpack_match_the_oracle_bytes(q, ctx):
    N, K = 200, 1152
    codes = _w4_codes(51, "w4", N, K)
    codes[0, :4] = [-8, 7, -1, 0]
    w8 = dev_i8(codes)
    packed = torch.zeros((N, K // 2), dtype=torch.uint8, device="cuda")
    q.qdit_pack_weight_int4(ctx, w8, N, K, packed)
    q.qdit_sync(ctx)
    np.testing.assert_array_equal(packed.cpu().numpy(), quant.pack_int4(codes))
    back = torch.zeros((N, K), dtype=torch.uint8, device="cuda")
    q.qdit_unpack_weight_int4(ctx, packed, N, K, back)
    q.qdit_sync(ctx)
    np.testing.assert_array_equal(host_codes(back), codes)
    np.testing.assert_array_equal(host_codes(back), quant.unpack_int4(quant.pack_int4(codes)))
    # a code outside [-8, 7] cannot be stored
    bad = codes.copy()
    bad[3, 5] = 9
    assert q.lib.qdit_pack_weight_int4(ctx, dev_i8(bad).data_ptr(), N, K, packed.data_ptr()) == q.QDIT_ERR_INVALID_ARG
    assert q.lib.qdit_pack_weight_int4(ctx, w8.data_ptr(), N, 24, packed.data_ptr()) == q.QDIT_ERR_SHAPE


@pytest.mark.parametrize("M,N,K", [(64, 392, 1152), (1152, 1152, 1152), (300, 6912, 384), (2048, 256, 4608)])
@pytest.mark.parametrize("scratch", [False, True])
def test_w4a8_accumulators_bit_exact_and_stage_equals_the_codes(q, ctx, M, N, K, scratch):
    """The weight tile the tensor core reads must be the oracle's codes exactly: raw int32 accumulators on random
    activations equal the oracle's integer product, and one-hot activations (row m selects column m of W) return the
    widened codes themselves.  Both forms: widened inside the GEMM kernel, and widened into a scratch matrix first."""
    codes = _w4_codes(52, f"w4.{N}.{K}", N, K)
    packed = torch.from_numpy(quant.pack_int4(codes)).cuda()
    w8s = torch.empty((N, K), dtype=torch.uint8, device="cuda") if scratch else None
    qa = _codes(52, f"a4.{M}.{K}", (M, K), -128, 127)
    out = torch.empty((M, N), dtype=torch.int32, device="cuda")
    q.qdit_w4a8_linear(ctx, dev_i8(qa), packed, M, N, K, q.qparams(1.0), None, q.QDIT_EPI_OUT_I32, None, out, N, w8s)
    q.qdit_sync(ctx)
    np.testing.assert_array_equal(out.cpu().numpy().astype(np.int64), linear.gemm_i8(qa, codes))
    Ms = min(M, K)
    onehot = np.zeros((Ms, K), dtype=np.int64)
    ks = synth.uniform_int(52, f"ks{K}", (Ms,), 0, K)
    onehot[np.arange(Ms), ks] = 1
    out1 = torch.empty((Ms, N), dtype=torch.int32, device="cuda")
    q.qdit_w4a8_linear(ctx, dev_i8(onehot), packed, Ms, N, K, q.qparams(1.0), None, q.QDIT_EPI_OUT_I32, None, out1, N, w8s)
    q.qdit_sync(ctx)
    np.testing.assert_array_equal(out1.cpu().numpy(), quant.unpack_int4(quant.pack_int4(codes))[:, ks].T)


@pytest.mark.parametrize("M,T", [(512, 256), (96, 32)])
def test_w4a8_epilogues_equal_w8a8_on_the_same_codes(q, ctx, M, T):
    """Same codes, same arithmetic after the accumulator: the packed layer and the one-code-per-byte layer give the
    same bits for the f32, the GELU + re-quantised and the gated epilogue; and the f32 output matches the oracle."""
    N, K = 1152, 1152
    a_qp = QParams(0.05, 0, -127, 127)
    L = _layer(53, M, N, K, T, a_qp)
    Wf = synth.normal(53, "W", (N, K), 0.02)
    codes, s_w, cs = quant.quantize_weight_per_channel(Wf, bits=4)
    A = dev_i8(L["qa"])
    W8, W4 = dev_i8(codes), torch.from_numpy(quant.pack_int4(codes)).cuda()
    ws, bi, g = dev(s_w), dev(L["bias"]), dev(L["gate"])
    ref = linear.w8a8_linear(L["qa"], a_qp, codes, s_w, cs, L["bias"])
    outs = {}
    for name, fn, W in (("w8", q.qdit_w8a8_linear, W8), ("w4", q.qdit_w4a8_linear, W4)):
        of = torch.empty((M, N), dtype=torch.float32, device="cuda")
        fn(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None, q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32, q.epilogue(w_scale=ws, bias=bi), of, N)
        oq = torch.empty((M, N), dtype=torch.uint8, device="cuda")
        fn(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None, q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT,
           q.epilogue(w_scale=ws, bias=bi, out_qp=q.qparams(0.01)), oq, N)
        x = dev(L["resid"]).to(torch.bfloat16)
        cache = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
        fn(ctx, A, W, M, N, K, q.qparams(a_qp.scale), None,
           q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_CACHE_STORE | q.QDIT_EPI_OUT_BF16,
           q.epilogue(w_scale=ws, bias=bi, gate=g, ld_gate=N, tokens_per_sample=T, residual=x, cache_out=cache), x, N)
        q.qdit_sync(ctx)
        outs[name] = (of.cpu().numpy(), oq.cpu().numpy(), x.float().cpu().numpy(), cache.float().cpu().numpy())
    assert max_rel_err(outs["w4"][0], ref) < 1e-5
    for a, b in zip(outs["w4"], outs["w8"]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("N,ldo", [(2312, 2336), (2312, 2312), (2304, 2312)])
def test_code_output_leaves_the_padding_of_its_rows_alone(q, ctx, N, ldo):
    """8-bit output whose width or row pitch is not a multiple of 16: accepted at every row count, and nothing beyond column N
    is written."""
    M, K = 1040, 256
    A, W = dev_i8(_codes(92, "a", (M, K), -127, 127)), dev_i8(_codes(92, "w", (N, K), -127, 127))
    ws, bi = dev(np.full(N, 1e-4, dtype=np.float32)), dev(synth.normal(92, "b", (N,), 0.5))
    epi = q.epilogue(w_scale=ws, bias=bi, out_qp=q.qparams(0.02))

    def run(rows):
        out = torch.full((M, ldo), 3, dtype=torch.int8, device="cuda")
        for m0 in range(0, M, rows):
            m = min(rows, M - m0)
            q.qdit_w8a8_linear(ctx, A[m0:], W, m, N, K, q.qparams(0.03), None, q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT,
                               epi, out[m0:], ldo)
        q.qdit_sync(ctx)
        return out

    got = run(M)
    assert (got[:, N:] == 3).all()
    assert torch.equal(got, run(520))


@pytest.mark.parametrize("M,N,K", [
    (1, 8, 512),         # one small tile, four k-blocks: not split
    (8, 8, 1024),        # f32, per-token, raw: shortest split reduction, one tile, four CTAs with two k-blocks each
    (8, 8, 3072),        # the others: 24 k-blocks over six CTAs
    (64, 392, 4608),     # six CTAs per tile, ragged columns (392 = 6 * 64 + 8)
    (100, 1152, 1040),   # 9 k-blocks, the last one short: four CTAs per tile with those outputs, else whole
    (200, 832, 3440),    # four CTAs per tile: ragged rows, 27 k-blocks, the last one short
    (256, 1152, 4608),   # three CTAs per tile: row groups 6, 5, 5
    (300, 1152, 800),    # seven k-blocks: not split
    (300, 1152, 5120),   # two CTAs per tile: ragged rows
    (1040, 2312, 256),   # bf16, f32, per-token: channel-major, ragged rows and columns
    (1025, 2304, 1152),
    (4000, 1160, 1152),  # gated layer by pairs: 32 x 7 token-major tiles of 192 exceed one wave; ragged rows and columns
    (8000, 1152, 4608),  # gated layer of a long reduction, channel-major: two waves of 128 x 256 tiles, ragged rows
])
@pytest.mark.parametrize("kind", ["i32", "f32", "bf16", "row", "gelu", "gated", "gated_nocache"])
def test_automatic_kernel_gives_the_bits_of_the_token_major_kernel(q, ctx, M, N, K, kind):
    """Every kernel computes exact integer sums and the same f32 epilogue: whatever the automatic choice runs (reduction split
    over a cluster, channel-major with staged stores) equals the plain token-major kernel with run-time epilogue flags."""
    T = 32
    qa, qw = _codes(91, f"a{M}.{K}", (M, K), -127, 127), _codes(91, f"w{N}.{K}", (N, K), -127, 127)
    A, W = dev_i8(qa), dev_i8(qw)
    ws, bi = dev(np.abs(synth.normal(91, "s", (N,), 1e-4)) + 1e-5), dev(synth.normal(91, "b", (N,), 0.5))
    gate, resid = dev(synth.normal(91, "g", (-(-M // T), N), 0.5)), dev(synth.normal(91, "r", (M, N), 1.0)).to(torch.bfloat16)
    rows = dev(np.abs(synth.normal(91, "rs", (M,), 1.0)) + 0.1)
    flags = {"i32": q.QDIT_EPI_OUT_I32, "f32": q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32, "bf16": q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_BF16,
             "row": q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_BF16 | q.QDIT_EPI_ROW_SCALE,
             "gelu": q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT,
             "gated": q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16 | q.QDIT_EPI_CACHE_STORE,
             "gated_nocache": q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16}[kind]
    dtype = {"i32": torch.int32, "f32": torch.float32, "gelu": torch.int8}.get(kind, torch.bfloat16)
    ldo = -(-N // 16) * 16 + 16     # rows of the output are wider than the layer

    def run():
        out = torch.full((M, ldo), 3, dtype=dtype, device="cuda")
        res = torch.zeros((M, ldo), dtype=torch.bfloat16, device="cuda")
        res[:, :N] = resid
        cache = torch.full((M, N), 3, dtype=torch.bfloat16, device="cuda")
        epi = q.epilogue(w_scale=ws, bias=bi, gate=gate, ld_gate=N, tokens_per_sample=T, residual=res,
                         cache_out=cache if kind == "gated" else None, out_qp=q.qparams(0.02), a_scale_rows=rows)
        q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(0.03), None, flags, epi, out, ldo)
        q.qdit_sync(ctx)
        return out, cache

    got = run()
    try:
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 64)
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, 1)
        ref = run()
    finally:
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 0)
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, 0)
    assert torch.equal(got[0], ref[0])
    assert torch.equal(got[1], ref[1])


@pytest.mark.parametrize("M,N,K", [(1, 8, 1024), (64, 392, 4608), (100, 1152, 1056), (256, 1152, 4608), (300, 1152, 1536),
                                   (512, 1152, 4608)])
@pytest.mark.parametrize("kind", ["i32", "gated", "gelu"])
def test_packed_weights_with_a_split_reduction(q, ctx, M, N, K, kind):
    """Packed 4-bit weights widened inside the split-reduction kernel: the bits of the one-code-per-byte layer, whole reductions."""
    T = 32
    codes = _w4_codes(93, f"w4s.{N}.{K}", N, K)
    A, W8, W4 = dev_i8(_codes(93, f"a{M}.{K}", (M, K), -127, 127)), dev_i8(codes), torch.from_numpy(quant.pack_int4(codes)).cuda()
    ws, bi = dev(np.abs(synth.normal(93, "s", (N,), 1e-3)) + 1e-4), dev(synth.normal(93, "b", (N,), 0.5))
    gate, resid = dev(synth.normal(93, "g", (-(-M // T), N), 0.5)), dev(synth.normal(93, "r", (M, N), 1.0)).to(torch.bfloat16)
    flags = {"i32": q.QDIT_EPI_OUT_I32, "gelu": q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT,
             "gated": q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16 | q.QDIT_EPI_CACHE_STORE}[kind]
    cache = [torch.zeros((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    out = [torch.zeros((M, N), dtype={"i32": torch.int32, "gelu": torch.int8}.get(kind, torch.bfloat16), device="cuda") for _ in range(2)]
    for i in range(2):
        epi = q.epilogue(w_scale=ws, bias=bi, gate=gate, ld_gate=N, tokens_per_sample=T, residual=resid, cache_out=cache[i], out_qp=q.qparams(0.02))
        if i == 0:
            q.qdit_w4a8_linear(ctx, A, W4, M, N, K, q.qparams(0.03), None, flags, epi, out[0], N)
        else:
            try:
                q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 64)   # unsplit
                q.qdit_w8a8_linear(ctx, A, W8, M, N, K, q.qparams(0.03), None, flags, epi, out[1], N)
            finally:
                q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 0)
        q.qdit_sync(ctx)
    assert torch.equal(out[0], out[1]) and torch.equal(cache[0], cache[1])


@pytest.mark.parametrize("M,N,K,T", [
    (129, 392, 400, 32),        # f32 and per-token scales: one pair, its second CTA one row, ragged channels, a short last k-block
    (4801, 1160, 1152, 64),     # second wave of gated tiles: a last row of tiles with one token, a last column with 8 channels
    (5000, 1152, 2304, 1000),   # gated by the long-reduction form, samples longer than a tile; 1000 % 32 != 0: not by pairs
    (5120, 1152, 2304, 256),
    (1300, 4624, 128, 32),      # one k-block: the ring is longer than the reduction
    (19200, 384, 384, 256),     # narrow layer, many tiles per pair
    (300, 44000, 1152, 32),     # weights of more than 48 MB: tiles along the tokens first
])
@pytest.mark.parametrize("kind,zp", [("f32", 0), ("bf16", 0), ("bf16", 131), ("row", 0), ("gelu", 0), ("gelu", 131), ("gelu_f32", 0),
                                     ("gated", 0), ("gated_nocache", 131)])
def test_pair_kernel_gives_the_bits_of_the_token_major_kernel(q, ctx, M, N, K, T, kind, zp):
    """Pairs of CTAs: whatever tile width the rule takes, exact integer sums and the same f32 epilogue as the plain token-major
    kernel with run-time epilogue flags; the padding of the rows stays untouched."""
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    lo, hi = (0, 256) if zp else (-127, 128)
    A = torch.randint(lo, hi, (M, K), generator=g, device="cuda").to(torch.uint8 if zp else torch.int8)
    W = torch.randint(-127, 128, (N, K), generator=g, device="cuda", dtype=torch.int8)
    ws, bi = torch.rand(N, generator=g, device="cuda") * 2e-4 + 1e-5, torch.randn(N, generator=g, device="cuda") * 0.5
    colsum = W.sum(dim=1, dtype=torch.int32)
    gate, resid = torch.randn(-(-M // T), N, generator=g, device="cuda") * 0.5, torch.randn(M, N, generator=g, device="cuda").bfloat16()
    rows = torch.rand(M, generator=g, device="cuda") + 0.1
    flags = {"f32": q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32, "bf16": q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_BF16,
             "row": q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_BF16 | q.QDIT_EPI_ROW_SCALE,
             "gelu": q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT, "gelu_f32": q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_OUT_F32,
             "gated": q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16 | q.QDIT_EPI_CACHE_STORE,
             "gated_nocache": q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16}[kind]
    dtype = {"f32": torch.float32, "gelu_f32": torch.float32, "gelu": torch.int8}.get(kind, torch.bfloat16)
    ldo = -(-N // 16) * 16 + 16
    qp = q.qparams(0.03, zp, 0, 255) if zp else q.qparams(0.03)

    def run():
        out = torch.full((M, ldo), 3, dtype=dtype, device="cuda")
        if kind.startswith("gated"):
            out[:, :N] = resid                 # in place, as in a block
        cache = torch.full((M, N), 3, dtype=torch.bfloat16, device="cuda")
        epi = q.epilogue(w_scale=ws, w_colsum=colsum, bias=bi, gate=gate, ld_gate=N, tokens_per_sample=T, residual=out,
                         cache_out=cache if kind == "gated" else None, out_qp=q.qparams(0.02, 5, -100, 90), a_scale_rows=rows)
        torch.cuda.synchronize()
        q.qdit_w8a8_linear(ctx, A, W, M, N, K, qp, None, flags, epi, out, ldo)
        q.qdit_sync(ctx)
        return out, cache

    got = run()
    try:
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 64)
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, 1)
        ref = run()
    finally:
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 0)
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, 0)
    assert torch.equal(got[0], ref[0])
    assert torch.equal(got[1], ref[1])


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("M,N,K,zp", [(1, 8, 32, 0), (2, 40, 1152, 7), (3, 4608, 1152, 0), (4, 1160, 1184, 0), (1, 19208, 1152, 11), (4, 24, 4608, 3),
                                      (4, 24, 4640, 0), (5, 1152, 384, 0)])   # (the last two are served by the tensor-core kernels)
def test_few_rows_kernel_gives_the_bits_of_the_tensor_core_kernels(q, ctx, bits, M, N, K, zp):
    """One to four rows with f32 output: exact integer sums and the same f32 epilogue; the padding of the rows stays untouched."""
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    lo, hi = (0, 256) if zp else (-127, 128)
    A = torch.randint(lo, hi, (M, K), generator=g, device="cuda").to(torch.uint8 if zp else torch.int8)
    top = 127 if bits == 8 else 7
    W = torch.randint(-top - 1, top + 1, (N, K), generator=g, device="cuda", dtype=torch.int8)
    ws, bi = torch.rand(N, generator=g, device="cuda") * 2e-4 + 1e-5, torch.randn(N, generator=g, device="cuda") * 0.5
    colsum = W.sum(dim=1, dtype=torch.int32)
    epi = q.epilogue(w_scale=ws, w_colsum=colsum, bias=bi)
    qp = q.qparams(0.03, zp, 0, 255) if zp else q.qparams(0.03)
    packed = None
    if bits == 4:
        packed = torch.empty((N, K // 2), dtype=torch.uint8, device="cuda")
        q.qdit_pack_weight_int4(ctx, W, N, K, packed)

    def run(option):
        out = torch.full((M, N + 8), 3.0, device="cuda")
        torch.cuda.synchronize()
        try:
            q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, option)
            if bits == 4:
                q.qdit_w4a8_linear(ctx, A, packed, M, N, K, qp, None, q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32, epi, out, N + 8, None)
            else:
                q.qdit_w8a8_linear(ctx, A, W, M, N, K, qp, None, q.QDIT_EPI_BIAS | q.QDIT_EPI_OUT_F32, epi, out, N + 8)
            q.qdit_sync(ctx)
        finally:
            q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 0)
        return out

    assert torch.equal(run(0), run(64))


@pytest.mark.parametrize("step", [4e-39, 2.0 ** -125, 1e-30, 0.01])
def test_codes_of_tiny_steps(q, ctx, step):
    """GELU codes by pairs of CTAs equal those of the run-time-flag epilogue down to steps at which subnormal activations count."""
    M, N, K = 1200, 4608, 64
    A, W = dev_i8(_codes(101, "a", (M, K), -127, 127)), dev_i8(_codes(101, "w", (N, K), -127, 127))
    # products of +-50000 or so: the activations are some ten steps
    ws = torch.full((N,), step / 4096.0 * 1e10, dtype=torch.float32, device="cuda")
    bi = torch.zeros(N, dtype=torch.float32, device="cuda")
    scale = torch.tensor([step], dtype=torch.float32, device="cuda")
    got = []
    for generic in (0, 1):
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, generic)
        try:
            for dev_scale in (None, scale):
                out = torch.zeros((M, N), dtype=torch.int8, device="cuda")
                q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(1e-10), None, q.QDIT_EPI_BIAS | q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT,
                                   q.epilogue(w_scale=ws, bias=bi, out_qp=q.qparams(step), out_scale_dev=dev_scale), out, N)
                q.qdit_sync(ctx)
                got.append(out)
        finally:
            q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, 0)
    assert (got[2].int().abs() > 0).float().mean() > 0.1
    for g in (got[0], got[1], got[3]):
        assert torch.equal(g, got[2])


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("M,tiles", [(128, 148), (128, 149), (90, 148), (300, 149), (300, 444), (300, 447)])
@pytest.mark.parametrize("T", [100, 128])
def test_gated_layer_with_as_many_tiles_as_ctas_and_more(q, ctx, bits, M, tiles, T):
    """One tile per CTA (what the epilogue reads comes before the accumulator is complete) and more give the bits of tiles of 64 channels with
    run-time flags; `tiles` of 192 channels, with packed weights of 128, samples that end inside a tile."""
    width, K = (192, 256) if bits == 8 else (128, 256)
    N = tiles // -(-M // 128) * width - 8
    g = torch.Generator(device="cuda").manual_seed(M + tiles)
    top = 127 if bits == 8 else 7
    A = torch.randint(-127, 128, (M, K), generator=g, device="cuda", dtype=torch.int8)
    W = torch.randint(-top, top + 1, (N, K), generator=g, device="cuda", dtype=torch.int8)
    ws, bi = torch.rand(N, generator=g, device="cuda") * 2e-4 + 1e-5, torch.randn(N, generator=g, device="cuda") * 0.5
    gate, resid = torch.randn((-(-M // T), N), generator=g, device="cuda"), torch.randn((M, N), generator=g, device="cuda").bfloat16()
    packed = torch.empty((N, K // 2), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    if bits == 4:
        q.qdit_pack_weight_int4(ctx, W, N, K, packed)
    flags = q.QDIT_EPI_BIAS | q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16 | q.QDIT_EPI_CACHE_STORE

    def run(plain):
        out, cache = (torch.full((M, N), 3.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        epi = q.epilogue(w_scale=ws, bias=bi, gate=gate, ld_gate=N, tokens_per_sample=T, residual=resid, cache_out=cache)
        torch.cuda.synchronize()
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 64 if plain else 192)
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, int(plain))
        try:
            if bits == 4 and not plain:
                q.qdit_w4a8_linear(ctx, A, packed, M, N, K, q.qparams(0.03), None, flags, epi, out, N, None)
            else:
                q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(0.03), None, flags, epi, out, N)
            q.qdit_sync(ctx)
        finally:
            q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 0)
            q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, 0)
        return out, cache

    got, ref = run(False), run(True)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])


@pytest.mark.parametrize("kind", ["codes", "f32", "gelu_f32", "bf16", "gated"])
@pytest.mark.parametrize("M,N,K,zp", [(2304, 3472, 320, 7), (1300, 4624, 784, 255), (600, 12304, 128, 128), (1300, 4624, 784, 0)])
def test_many_rows_with_a_zero_point(q, ctx, kind, M, N, K, zp):
    """Unsigned activations with a zero point through the automatic choice (pairs of CTAs, channel-major tiles; ragged in both directions): the bits of
    tiles of 64 channels with run-time flags.  The weights' sums are distinct, so that a channel with another one's term shows."""
    T = 32
    g = torch.Generator(device="cuda").manual_seed(M + N + zp)
    A = torch.randint(0, 256, (M, K), generator=g, device="cuda").to(torch.uint8)
    W = torch.randint(-127, 128, (N, K), generator=g, device="cuda", dtype=torch.int8)
    colsum = W.sum(dim=1, dtype=torch.int32)
    ws, bi = torch.rand(N, generator=g, device="cuda") * 2e-4 + 1e-5, torch.randn(N, generator=g, device="cuda") * 0.5
    gate, resid = torch.randn((-(-M // T), N), generator=g, device="cuda"), torch.randn((M, N), generator=g, device="cuda").bfloat16()
    flags = q.QDIT_EPI_BIAS | {"codes": q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT, "f32": q.QDIT_EPI_OUT_F32, "gelu_f32": q.QDIT_EPI_GELU | q.QDIT_EPI_OUT_F32,
                               "bf16": q.QDIT_EPI_OUT_BF16, "gated": q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16}[kind]
    dtype = {"codes": torch.int8, "f32": torch.float32, "gelu_f32": torch.float32}.get(kind, torch.bfloat16)

    def run(plain):
        out = torch.full((M, N), 3, dtype=dtype, device="cuda")
        epi = q.epilogue(w_scale=ws, w_colsum=colsum, bias=bi, gate=gate, ld_gate=N, tokens_per_sample=T, residual=resid, out_qp=q.qparams(0.02))
        torch.cuda.synchronize()
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 64 * plain)
        q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, plain)
        try:
            q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(0.03, zp, 0, 255), None, flags, epi, out, N)
            q.qdit_sync(ctx)
        finally:
            q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_BN, 0)
            q.qdit_set_option(ctx, q.QDIT_OPT_GEMM_GENERIC_EPILOGUE, 0)
        return out

    assert torch.equal(run(0), run(1))
