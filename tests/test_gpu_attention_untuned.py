"""BF16 attention of shapes that no context has tuned: whatever plan the launcher
picks, the arithmetic is the eight-group chunks', so the bits equal those of
that variant and of every batch size. Shapes on which the plan with the
smallest modelled time belongs to another family."""
import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,C,heads,window", [
    ((9, 90, 178), 768, 16, (5, 7, 7)),
    ((5, 33, 70), 128, 4, (3, 5, 5)),
    ((4, 37, 67), 384, 8, (3, 7, 7)),
    ((3, 29, 41), 256, 4, (3, 5, 5)),
    ((2, 19, 40), 256, 16, (1, 3, 3)),
])
def test_untuned_arithmetic(grid, C, heads, window):
    n = int(np.prod(grid))
    g = torch.Generator(device="cuda").manual_seed(3)
    qkv = (2.0 * torch.randn(2, n, 3 * C, generator=g, device="cuda")).bfloat16()

    def run(x, variant):
        out = torch.full((x.shape[0], n, C), float("nan"), device="cuda", dtype=torch.bfloat16)
        wm.wm_op_neighborhood_attention(x, out, x.shape[0], *grid, C, heads, *window, True, wm.WM_PREC_BF16, variant)
        torch.cuda.synchronize()
        return out

    both = run(qkv, wm.WM_NA_AUTO)
    assert torch.equal(both, run(qkv, wm.WM_NA_QK_CHUNK8))
    assert torch.equal(both[1:], run(qkv[1:].contiguous(), wm.WM_NA_AUTO))
    wm.wm_device_status()
