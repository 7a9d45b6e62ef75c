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
