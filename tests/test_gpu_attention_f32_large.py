"""FP32 attention with V near the largest float: probabilities are held up to e^8
above their final scale while a query's keys are walked, which must not reach
the result. The output is an average of V: with V = v everywhere it is v, to
the rounding of the sums (245 keys, a few 1e-6)."""
import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v", [1e37, 1e36, -3e37])
@pytest.mark.parametrize("dh,window", [(16, (1, 3, 3)), (32, (3, 5, 5)), (48, (5, 7, 7)), (64, (3, 7, 5))])
def test_average_of_large_values(dh, window, v):
    grid, heads, C = (5, 14, 22), 2, 2 * dh
    n = int(np.prod(grid))
    qkv = torch.zeros(1, n, 3 * C, device="cuda")
    qkv[..., :C] = 1.0
    # scores that grow by less than 8 from one latitude to the next
    lat = torch.arange(n, device="cuda") // grid[2] % grid[1]
    qkv[..., C:2 * C] = (lat * 2.0 / dh ** 0.5)[None, :, None]
    qkv[..., 2 * C:] = v
    out = torch.empty(1, n, C, device="cuda")
    wm.wm_op_neighborhood_attention(qkv, out, 1, *grid, C, heads, *window, True, wm.WM_PREC_FP32)
    torch.cuda.synchronize()
    assert float((out.double() / v - 1.0).abs().max()) <= 1e-5
