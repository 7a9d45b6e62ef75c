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
