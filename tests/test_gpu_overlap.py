"""Kernels that start beside their predecessor and read constants early give the bits of launches that wait for one another."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("B", [1, 5])
def test_overlapped_evaluations_equal_plain_ones(bits, B):
    """Back-to-back evaluations of one sampler on changing inputs and timesteps (so a modulation, a gate or a scale read too early would
    be the previous evaluation's), also right after the scales change; with overlapped launches and without."""
    import paper_2503_02508_b200 as q
    cfg, rounds = synth.DIT_S2_BLOCK, 6
    w = synth.model_weights(7, cfg)
    g = torch.Generator(device="cuda").manual_seed(B)
    latent = torch.randn(rounds, B, cfg.channels, cfg.latent_side, cfg.latent_side, generator=g, device="cuda")
    t = torch.randint(0, 1000, (rounds, B), generator=g, device="cuda").float()
    y = torch.randint(0, cfg.num_classes, (rounds, B), generator=g, device="cuda", dtype=torch.int32)
    torch.cuda.synchronize()
    got = []
    for overlapped in (1, 0):
        ctx = q.qdit_create(0, None)
        q.qdit_set_option(ctx, q.QDIT_OPT_PDL, overlapped)
        model = q.qdit_model_create(ctx, cfg, w, bits)
        s = q.qdit_sampler_create(ctx, model, batch=B, num_steps=10, cache_interval=2)
        out = torch.empty(rounds, B, 2 * cfg.channels, cfg.latent_side, cfg.latent_side, device="cuda")
        q.qdit_model_begin_calibration(ctx, model)
        q.qdit_forward(ctx, s, latent[0], t[0], y[0], B, out[0], q.QDIT_FWD_CALIBRATE)
        q.qdit_model_finish_calibration(ctx, model)
        for i in range(1, rounds):
            q.qdit_forward(ctx, s, latent[i], t[i], y[i], B, out[i], q.QDIT_FWD_STORE_CACHE if i % 2 else 0)
            if i == 3:
                ada, blocks = q.qdit_model_get_act_scales(ctx, model, cfg.depth)
                q.qdit_model_set_act_scales(ctx, model, ada * 1.5, np.asarray(blocks) * 0.75)
        q.qdit_sync(ctx)
        got.append(out.clone())
        q.qdit_sampler_destroy(s)
        q.qdit_model_destroy(model)
        q.qdit_destroy(ctx)
    assert torch.isfinite(got[0]).all() and torch.equal(got[0], got[1])


@pytest.mark.parametrize("bits,B", [(8, 1), (8, 5), (4, 2)])
def test_ranges_found_by_the_writing_kernels(bits, B):
    """Calibration ranges are folded together by the kernels that write the quantizers' inputs (LayerNorm, attention on tcgen05, GELU layer
    token-major, by pairs and with packed weights): against the same pass of the oracle; a second pass starts from zero."""
    import paper_2503_02508_b200 as q
    from oracle import calib, dit
    cfg = synth.DIT_S2_BLOCK
    w = synth.model_weights(11, cfg)
    latent = synth.normal(11, "latent", (B, cfg.channels, cfg.latent_side, cfg.latent_side))
    t, y = np.full(B, 500.0), synth.uniform_int(11, "y", (B,), 0, cfg.num_classes)
    ref = calib.calibrate_model(dit.make_qmodel(cfg, w, bits), [(latent, t, y)])
    ctx = q.qdit_create(0, None)
    model = q.qdit_model_create(ctx, cfg, w, bits)
    s = q.qdit_sampler_create(ctx, model, batch=B, num_steps=10)
    out = torch.empty(B, 2 * cfg.channels, cfg.latent_side, cfg.latent_side, device="cuda")
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (latent, t.astype(np.float32), y.astype(np.int32))]
    torch.cuda.synchronize()
    got = []
    for scale in (8.0, 1.0):     # the larger inputs first: their ranges must not stay
        x = (dev[0] * scale).contiguous()
        torch.cuda.synchronize()
        q.qdit_model_begin_calibration(ctx, model)
        q.qdit_forward(ctx, s, x, dev[1], dev[2], B, out, q.QDIT_FWD_CALIBRATE)
        q.qdit_model_finish_calibration(ctx, model)
        got.append(q.qdit_model_get_act_scales(ctx, model, cfg.depth))
    q.qdit_sync(ctx)
    ada, blocks = got[1]
    want = np.array([[ref.blocks[i][n].scale for n in ("qkv", "proj", "fc1", "fc2")] for i in range(cfg.depth)])
    # a flipped code in front moves a later maximum by a quantization step of its inputs, not by rounding: 1 % (f32 alone gives 1e-5)
    assert abs(ada / ref.ada.scale - 1.0) < 1e-5 and np.abs(blocks / want - 1.0).max() < 1e-2
    assert not np.allclose(got[0][1], blocks, rtol=1e-3)
    q.qdit_sampler_destroy(s)
    q.qdit_model_destroy(model)
    q.qdit_destroy(ctx)


# More than one block, so that a block's modulation is read beside the previous block's last layer.  A network batch of 4 with 384 columns stays
# token-major and split; with 1152 columns 2 images stay so too, 8 run QKV and fc1 by pairs, 32 all four layers by pairs or channel-major
CHAINS = [(synth.DiTConfig(hidden=384, heads=6, mlp=1536, depth=3, grid=16), 8, 2), (synth.DiTConfig(hidden=1152, heads=16, mlp=4608, depth=2, grid=16), 8, 4),
          (synth.DiTConfig(hidden=1152, heads=16, mlp=4608, depth=2, grid=16), 4, 1), (synth.DiTConfig(hidden=1152, heads=16, mlp=4608, depth=2, grid=16), 8, 16)]


@pytest.mark.parametrize("cfg,bits,B", CHAINS, ids=["narrow", "wide8", "wide4", "many"])
def test_overlapped_trajectories_equal_plain_ones(cfg, bits, B):
    """Evaluations, refreshed and reused steps, and steps that serve one branch from the cache, one behind the other without a wait on
    inputs, labels and scales that change: a modulation, gate or scale read too early would be the one before."""
    import paper_2503_02508_b200 as q
    steps, N = 6, 2 * B   # network batch with guidance
    w = synth.model_weights(13, cfg)
    g = torch.Generator(device="cuda").manual_seed(B)
    latent = torch.randn(4, B, cfg.channels, cfg.latent_side, cfg.latent_side, generator=g, device="cuda")
    x = torch.randn(3, N, cfg.channels, cfg.latent_side, cfg.latent_side, generator=g, device="cuda")
    t = torch.randint(0, 1000, (3, N), generator=g, device="cuda").float()
    y = torch.randint(0, cfg.num_classes, (4, N), generator=g, device="cuda", dtype=torch.int32)
    noise = torch.randn(steps, B, cfg.channels, cfg.latent_side ** 2, generator=g, device="cuda")
    # every mixture: the attention branch served, the other one served, first block and last block; step 0 fills the cache
    mask = np.random.default_rng(3).integers(0, 2, (steps, cfg.depth, 2)).astype(np.uint8)
    mask[0], mask[1, 0], mask[2, 0], mask[3] = 0, (1, 0), (0, 1), 1
    torch.cuda.synchronize()
    got = []
    for overlapped in (1, 0):
        ctx = q.qdit_create(0, None)
        q.qdit_set_option(ctx, q.QDIT_OPT_PDL, overlapped)
        model = q.qdit_model_create(ctx, cfg, w, bits)
        samplers = []
        outs = [torch.empty(3, N, 2 * cfg.channels, cfg.latent_side, cfg.latent_side, device="cuda")]
        for chunk in (0, -1, 2):     # the conditioning of the whole trajectory at once, of each step by itself, in chunks
            q.qdit_set_option(ctx, q.QDIT_OPT_CONDITIONING_CHUNK, chunk)
            samplers.append(q.qdit_sampler_create(ctx, model, batch=B, num_steps=steps, cache_interval=2, use_cfg=True, guidance=1.5))
        s = samplers[0]
        q.qdit_model_begin_calibration(ctx, model)
        q.qdit_forward(ctx, s, x[0], t[0], y[0], N, outs[0][0], q.QDIT_FWD_CALIBRATE)
        q.qdit_forward(ctx, s, x[1], t[1], y[1], N, outs[0][1], q.QDIT_FWD_CALIBRATE)
        q.qdit_model_finish_calibration(ctx, model)
        q.qdit_forward(ctx, s, x[2], t[2], y[2], N, outs[0][2])

        def trajectory(s, k):
            q.qdit_sampler_reset(ctx, s, latent[k], y[k, :B].contiguous())
            for i in range(steps):
                q.qdit_sample_step(ctx, s, i)
            q.qdit_sync(ctx)
            view = torch.empty(B, cfg.channels, cfg.latent_side, cfg.latent_side, device="cuda")
            view.copy_(_latent(q, s, view.shape))
            torch.cuda.synchronize()
            outs.append(view)

        for k, s in enumerate(samplers):
            trajectory(s, k)
        q.qdit_sampler_set_schedule(ctx, samplers[0], mask)
        trajectory(samplers[0], 3)
        q.qdit_sampler_set_schedule(ctx, samplers[0], None)
        q.qdit_sampler_set_ddpm(ctx, samplers[0], noise)
        trajectory(samplers[0], 0)
        q.qdit_sync(ctx)
        got.append(outs)
        for s in samplers:
            q.qdit_sampler_destroy(s)
        q.qdit_model_destroy(model)
        q.qdit_destroy(ctx)
    for a, b in zip(*got):
        assert torch.isfinite(a).all() and torch.equal(a, b)


def _latent(q, s, shape):
    from gpu_util import view
    return view(q.qdit_sampler_latent(s), shape, "<f4")


def _block(hidden, heads, grid):
    return synth.DiTConfig(hidden=hidden, heads=heads, mlp=4 * hidden, depth=1, grid=grid)


@pytest.mark.parametrize("cfg,B,bits,options", [
    (_block(144, 2, 24), 1, 8, {}),                                  # 576 tokens of head dim 72: half of the last query tile must not count
    (_block(144, 2, 24), 3, 4, {}),                                  # 1728 rows, weights widened into the scratch matrix
    (_block(144, 2, 24), 3, 8, {"ATTN": 1}),                         # mma.sync attention
    (_block(384, 6, 8), 1, 8, {}),                                   # 64 rows: token-major or split layers, mma.sync attention
    (_block(384, 6, 8), 3, 4, {}),                                   # packed weights widened in the kernel
    (_block(384, 6, 24), 1, 8, {"GEMM_T": 256}),                     # channel-major GELU layer, ragged token tile
    (_block(384, 6, 24), 2, 8, {"GEMM_T": 128}),
    (_block(384, 6, 16), 2, 8, {"GEMM_GENERIC_EPILOGUE": 1}),
    (_block(1152, 16, 24), 2, 8, {}),                                # 1152 rows by pairs
    (_block(1152, 16, 16), 1, 4, {}),
])
def test_ranges_are_those_of_the_written_tensors(cfg, B, bits, options):
    """The range that a kernel publishes is the largest magnitude of the very tensor that it writes: each tensor is written again by the
    public call from what the pass has left in the sampler's buffers."""
    import paper_2503_02508_b200 as q
    from gpu_util import view
    ctx = q.qdit_create(0, None)
    for name, value in options.items():
        q.qdit_set_option(ctx, getattr(q, "QDIT_OPT_" + name), value)
    model = q.qdit_model_create(ctx, cfg, synth.model_weights(17, cfg), bits)
    s = q.qdit_sampler_create(ctx, model, batch=B, num_steps=10)
    g = torch.Generator(device="cuda").manual_seed(B)
    latent = torch.randn(B, cfg.channels, cfg.latent_side, cfg.latent_side, generator=g, device="cuda")
    t, y = torch.full((B,), 500.0, device="cuda"), torch.randint(0, 1000, (B,), generator=g, device="cuda", dtype=torch.int32)
    out = torch.empty(B, 2 * cfg.channels, cfg.latent_side, cfg.latent_side, device="cuda")
    q.qdit_model_begin_calibration(ctx, model)
    q.qdit_forward(ctx, s, latent, t, y, B, out, q.QDIT_FWD_CALIBRATE)
    q.qdit_model_finish_calibration(ctx, model)
    _, (got,) = q.qdit_model_get_act_scales(ctx, model, 1)

    T, D, F = cfg.tokens, cfg.hidden, cfg.mlp
    M = B * T
    mod = view(q.qdit_sampler_buffer(s, "mod"), (B, 6 * D), "<f4")
    qkv = q.qdit_sampler_buffer(s, "qkv")
    x = torch.empty(M, D, dtype=torch.bfloat16, device="cuda")
    y32 = torch.empty(M, D, device="cuda")
    u32 = torch.empty(M, F, device="cuda")
    at = lambda k: mod.data_ptr() + 4 * k * D

    def layer(A, which, scale, flags, out, **epi):
        L = q.qdit_model_linear(model, 0, which)
        e = q.epilogue(w_scale=L["w_scale"], w_colsum=L["w_colsum"], bias=L["bias"], **epi)
        if q.qdit_model_weights_packed(model):
            q.qdit_w4a8_linear(ctx, A, L["w_q"], M, L["N"], L["K"], q.qparams(float(scale)), None, flags | q.QDIT_EPI_BIAS, e, out, L["N"], None)
        else:
            q.qdit_w8a8_linear(ctx, A, L["w_q"], M, L["N"], L["K"], q.qparams(float(scale)), None, flags | q.QDIT_EPI_BIAS, e, out, L["N"])

    want = []
    q.qdit_patch_embed(ctx, model, latent, B, x)
    q.qdit_adaln_modulate(ctx, x, M, D, T, 1e-6, at(0), at(1), 6 * D, y32, q.QDIT_F32)
    q.qdit_sync(ctx)
    want.append(y32.abs().max())
    q.qdit_attention(ctx, qkv, qkv + 2 * D, qkv + 4 * D, 3 * D, B, cfg.heads, T, cfg.head_dim, cfg.head_dim ** -0.5, y32, q.QDIT_F32)
    q.qdit_sync(ctx)
    want.append(y32.abs().max())
    layer(q.qdit_sampler_buffer(s, "a"), 2, got[1], q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16, x, gate=at(2), ld_gate=6 * D,
          tokens_per_sample=T, residual=x)
    q.qdit_adaln_modulate(ctx, x, M, D, T, 1e-6, at(3), at(4), 6 * D, y32, q.QDIT_F32)
    q.qdit_sync(ctx)
    want.append(y32.abs().max())
    layer(q.qdit_sampler_buffer(s, "h"), 3, got[2], q.QDIT_EPI_GELU | q.QDIT_EPI_OUT_F32, u32)
    q.qdit_sync(ctx)
    want.append(u32.abs().max())
    np.testing.assert_array_equal(got, torch.stack(want).cpu().numpy() / np.float32(127.0))
    q.qdit_sampler_destroy(s)
    q.qdit_model_destroy(model)
    q.qdit_destroy(ctx)
