"""Uneven batches of narrow latents (wm_rollout_batch): the launches cut
rollouts at steps so that their places stay filled. Every latent equals its
own rollout bit for bit, whatever the cuts: fewer latents than a launch takes,
as many, and more; leads equal, spread, and with one far longer than the rest;
six-hour processors deeper and shallower than the one-hour one."""
import dataclasses

import pytest
import torch

import paper_2503_22235_gb300 as wm
import synth

pytestmark = pytest.mark.gpu

CUDA = torch.device("cuda")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_22235_gb300 import build as wm_build
    wm_build.build()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"


@pytest.mark.parametrize("L6,L1", [(2, 1), (1, 3)])
@pytest.mark.parametrize("leads", [
    [9, 2],
    [48, 6, 5],
    [24, 24, 24, 24, 24],
    [11, 0, 30, 1, 17, 4, 29, 23],
    [100, 1, 2, 3, 4, 5, 6, 7, 8],
], ids=lambda v: "-".join(map(str, v)) if isinstance(v, list) else str(v))
def test_uneven_batch_equals_alone(L6, L1, leads):
    s = dataclasses.replace(synth.SMALL, blocks_p6=L6, blocks_p1=L1)
    p6, p1 = synth.processor_weights(s, seed=4)
    ctx = wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16, 4), synth.pack_weights(p6, p1))
    try:
        xs = [torch.from_numpy(synth.latent(s, 1, seed=50 + i)).to(CUDA) for i in range(len(leads))]
        batch = [x.clone() for x in xs]
        wm.wm_rollout_batch(ctx, batch, leads)
        for x, b, t in zip(xs, batch, leads):
            wm.wm_latent_rollout(ctx, x, t)
            torch.cuda.synchronize()
            assert torch.equal(b, x), t
        wm.wm_device_status()   # raises on a recorded timeout
    finally:
        wm.wm_destroy(ctx)
