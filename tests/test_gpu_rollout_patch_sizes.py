"""Every patch size of the whole-rollout kernel, forced and confirmed, gives the
same bits: steps, rollouts of one to four latents where the patches fit on the
device, windows of 1, 3 and 5. And the size that the library chooses follows
from the latents of a launch."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm
import synth

pytestmark = pytest.mark.gpu

BASE = dataclasses.replace(synth.SMALL, blocks_p6=2, blocks_p1=1)
SMS = 152


@pytest.fixture(autouse=True)
def restore():
    yield
    wm.wm_rollout_patch_override(0)


def _ctx(s):
    p6, p1 = synth.processor_weights(s, seed=3, stress=True)
    return wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16, 4), synth.pack_weights(p6, p1))


@pytest.mark.parametrize("D,H,W,kd,kh,kw", [(4, 24, 48, 3, 5, 5), (4, 24, 48, 1, 3, 5), (4, 32, 64, 3, 5, 5),
                                            (2, 8, 32, 1, 5, 3), (3, 16, 48, 3, 1, 1), (2, 40, 32, 1, 3, 3)])
def test_sizes_agree(D, H, W, kd, kh, kw):
    s = dataclasses.replace(BASE, D=D, H=H, W=W, kd=kd, kh=kh, kw=kw)
    ctx = _ctx(s)
    try:
        x = np.concatenate([synth.latent(s, 1, seed=30 + i) for i in range(4)])
        ran = set()
        for G in (1, 2, 4):
            outs = {}
            for tokens in (128, 64, 32):
                if G * D * (H // 8) * (W // (tokens // 8)) > SMS:
                    continue
                wm.wm_rollout_patch_override(tokens)
                t = torch.from_numpy(x[:G]).cuda()
                wm.wm_latent_rollout(ctx, t, 8)
                torch.cuda.synchronize()
                assert wm.wm_rollout_patch_tokens(ctx) == tokens
                outs[tokens] = t
                ran.add(tokens)
            for o in outs.values():
                assert torch.equal(o, outs[128])
        assert {128, 64} <= ran
        wm.wm_device_status()
    finally:
        wm.wm_destroy(ctx)


def test_chosen_and_refused():
    ctx = _ctx(BASE)   # 4 x 24 x 48: 36, 72 or 144 patches a latent
    try:
        wm.wm_rollout_patch_override(32)
        two = torch.from_numpy(np.concatenate([synth.latent(BASE, 1, seed=i) for i in range(2)])).cuda()
        with pytest.raises(Exception):
            wm.wm_latent_rollout(ctx, two, 6)   # 288 patches
        wm.wm_rollout_patch_override(0)
        for _ in range(8):   # launches of this stream alone
            wm.wm_latent_rollout(ctx, two, 6)
            torch.cuda.synchronize()
        assert wm.wm_rollout_patch_tokens(ctx) == 64
        wm.wm_latent_rollout(ctx, two[:1], 6)
        assert wm.wm_rollout_patch_tokens(ctx) == 32
        torch.cuda.synchronize()
        with pytest.raises(Exception):
            wm.wm_rollout_patch_override(16)
    finally:
        wm.wm_destroy(ctx)
