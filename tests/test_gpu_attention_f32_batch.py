"""FP32 attention of a latent is the same function of it whatever batch it is in,
bit for bit, also where the batch size changes the kernel's tile (on 152 SMs:
3 x 68 x 130 takes tiles of 4 x 8 query blocks for one or two latents and 4 x 4
from three on; 10 x 36 x 66 takes 4 x 4 and 4 x 2). Scores that spread by far
more than 8, and ordinary ones."""
import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 6.0])
@pytest.mark.parametrize("grid,window,heads,dh", [
    ((3, 68, 130), (3, 5, 5), 8, 32),
    ((10, 36, 66), (5, 5, 5), 8, 64),
    ((4, 24, 48), (3, 5, 5), 4, 32),
    ((5, 33, 51), (3, 7, 7), 8, 48),
    ((3, 30, 61), (1, 3, 3), 4, 16),
])
def test_batch_does_not_change_a_latent(grid, window, heads, dh, scale):
    B, n, C = 6, int(np.prod(grid)), heads * dh
    g = torch.Generator(device="cuda").manual_seed(5)
    qkv = torch.randn(B, n, 3 * C, generator=g, device="cuda")
    qkv[..., :C] *= scale

    def run(x):
        out = torch.full((x.shape[0], n, C), float("nan"), device="cuda")
        wm.wm_op_neighborhood_attention(x, out, x.shape[0], *grid, C, heads, *window, True, wm.WM_PREC_FP32)
        torch.cuda.synchronize()
        return out

    alone = torch.cat([run(qkv[i:i + 1].contiguous()) for i in range(B)])
    for b in (2, 3, 4, 6):
        assert torch.equal(run(qkv[:b].contiguous()), alone[:b]), b
    wm.wm_device_status()
