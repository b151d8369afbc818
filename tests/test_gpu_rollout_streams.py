"""Hourly outputs of narrow latents on several streams at once: the library's
captured launches take patches that leave room for one another, as launches made
directly do, and the results are those of a context alone, bit for bit."""
import dataclasses

import pytest
import torch

import paper_2503_22235_gb300 as wm
import synth

pytestmark = pytest.mark.gpu


def test_hourly_graphs_share_the_device():
    s = dataclasses.replace(synth.SMALL, blocks_p6=8, blocks_p1=4)   # 4 x 24 x 48: 36, 72 or 144 patches a latent
    p6, p1 = synth.processor_weights(s, seed=5)
    blob = synth.pack_weights(p6, p1)
    lead = 40
    n = s.D * s.H * s.W
    ctxs = [wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16, 1), blob) for _ in range(4)]
    try:
        xs = [torch.from_numpy(synth.latent(s, 1, seed=i)).cuda() for i in range(4)]
        outs = [torch.zeros(lead + 1, n, s.C, device="cuda") for _ in range(4)]
        streams = [torch.cuda.Stream() for _ in range(4)]
        alone = []
        for _ in range(3):   # alone, often enough that no earlier launch of the process counts
            alone = []
            for c, x, o, st in zip(ctxs, xs, outs, streams):
                wm.wm_rollout_hourly(c, x, lead, o, 1, st.cuda_stream)
                torch.cuda.synchronize()
                alone.append(o.clone())
        assert [wm.wm_rollout_patch_tokens(c) for c in ctxs] == [32] * 4
        for _ in range(6):   # the first rounds capture, which leaves gaps between the streams
            for o in outs:
                o.zero_()
            torch.cuda.synchronize()
            for c, x, o, st in zip(ctxs, xs, outs, streams):
                wm.wm_rollout_hourly(c, x, lead, o, 1, st.cuda_stream)
            torch.cuda.synchronize()
            assert all(torch.equal(a, o) for a, o in zip(alone, outs))
            if [wm.wm_rollout_patch_tokens(c) for c in ctxs] == [128] * 4:
                break
        assert [wm.wm_rollout_patch_tokens(c) for c in ctxs] == [128] * 4
        wm.wm_device_status()
    finally:
        for c in ctxs:
            wm.wm_destroy(c)


def test_a_callers_graph_leaves_room_for_every_context():
    """A captured step keeps its patches: they are sized for all contexts that there are."""
    s = dataclasses.replace(synth.SMALL, blocks_p6=2, blocks_p1=1)
    p6, p1 = synth.processor_weights(s, seed=5)
    blob = synth.pack_weights(p6, p1)
    ctxs = []
    try:
        for alive, tokens in ((1, 32), (2, 64), (4, 128)):
            while len(ctxs) < alive:
                ctxs.append(wm.wm_create_from_host(wm.make_config(s, wm.WM_PREC_BF16, 1), blob))
                wm.wm_ctx_reserve(ctxs[-1], 1)
            x = torch.from_numpy(synth.latent(s, 1, seed=1)).cuda()
            ref = x.clone()
            wm.wm_processor_step(ctxs[0], ref, wm.WM_P6)
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                wm.wm_processor_step(ctxs[0], x, wm.WM_P6)
            assert wm.wm_rollout_patch_tokens(ctxs[0]) == tokens
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(x, ref)
        wm.wm_device_status()
    finally:
        for c in ctxs:
            wm.wm_destroy(c)
