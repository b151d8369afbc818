"""The patch sizes of the whole-rollout kernel (128, 64 or 32 tokens a CTA, by
how many latents share the launch) give the same bits: a latent alone (the
smallest patch whose CTAs are resident at once) equals the same latent among
others, where the launch takes larger patches, and stays within the oracle's
tolerance. Windows of 3 and 5, one to three key levels, grids whose single
latent takes 32-token patches and grids that take 64."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm
import synth
from oracle import wm_oracle as orc
from parity_util import assert_close

pytestmark = pytest.mark.gpu

CUDA = torch.device("cuda")
BASE = dataclasses.replace(synth.SMALL, blocks_p6=2, blocks_p1=1)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_22235_gb300 import build as wm_build
    wm_build.build()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"


@pytest.mark.parametrize("D,H,W,kd,kh,kw", [
    (4, 24, 48, 3, 5, 5),    # 32 tokens alone, 64 in pairs, 128 from three on
    (4, 24, 48, 1, 3, 5),
    (4, 32, 64, 3, 5, 5),    # 64 alone, 128 in pairs
    (8, 24, 48, 3, 5, 3),
    (2, 8, 32, 1, 5, 3),     # 32 whatever the number
])
def test_patch_sizes_agree_bit_for_bit(D, H, W, kd, kh, kw):
    s = dataclasses.replace(BASE, D=D, H=H, W=W, kd=kd, kh=kh, kw=kw)
    p6, p1 = synth.processor_weights(s, seed=3, stress=True)
    ctx = wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16, 4), synth.pack_weights(p6, p1))
    try:
        x = [synth.latent(s, 1, seed=30 + i) for i in range(4)]
        alone = []
        for xi in x:
            t = torch.from_numpy(xi).to(CUDA)
            wm.wm_latent_rollout(ctx, t, 8)
            alone.append(t)
        for G in (2, 3, 4):
            ens = torch.from_numpy(np.concatenate(x[:G])).to(CUDA)
            wm.wm_latent_rollout(ctx, ens, 8)
            torch.cuda.synchronize()
            for i in range(G):
                assert torch.equal(ens[i:i + 1], alone[i]), (G, i)
        wm.wm_device_status()   # raises on a recorded timeout
        n6, n1 = orc.greedy_schedule(8)
        ref = orc.rollout(x[0], 8, p6, p1, s)
        assert_close(alone[0].detach().to("cpu", torch.float64).numpy(), ref,
                     2e-2 * (n6 * s.blocks_p6 + n1 * s.blocks_p1), s.C, (D, H, W))
    finally:
        wm.wm_destroy(ctx)
