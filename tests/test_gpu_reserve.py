"""wm_ctx_reserve allocates what later compute calls of that batch need, the
whole-rollout kernel's weights and workspace for narrow latents included: the
first step, rollout and uneven batch after it take no device memory."""
import dataclasses

import pytest
import torch

import paper_2503_22235_gb300 as wm
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [wm.WM_PREC_BF16, wm.WM_PREC_FP32])
def test_first_calls_after_reserve_allocate_nothing(precision):
    s = dataclasses.replace(synth.SMALL, blocks_p6=8, blocks_p1=8)
    p6, p1 = synth.processor_weights(s, seed=2)
    blob = synth.pack_weights(p6, p1)
    x = [torch.from_numpy(synth.latent(s, 1, seed=i)).cuda() for i in range(4)]
    ens = torch.cat(x)

    def calls(ctx):
        wm.wm_processor_step(ctx, ens, wm.WM_P6)
        wm.wm_processor_step(ctx, x[0], wm.WM_P1)
        if precision == wm.WM_PREC_BF16:
            wm.wm_latent_rollout(ctx, x[0], 8)
            wm.wm_rollout_batch(ctx, x, [3, 1, 8, 2])
        torch.cuda.synchronize()

    ctx = wm.wm_create_from_host(wm.make_config(s, precision, 4), blob)   # loads the kernels
    calls(ctx)
    wm.wm_destroy(ctx)
    ctx = wm.wm_create_from_host(wm.make_config(s, precision, 1), blob)
    try:
        wm.wm_ctx_reserve(ctx, 4)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        calls(ctx)
        assert torch.cuda.mem_get_info()[0] == free
        wm.wm_device_status()
    finally:
        wm.wm_destroy(ctx)
