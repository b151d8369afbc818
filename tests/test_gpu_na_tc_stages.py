"""The tcgen05 attention kernel where only two slab stages fit (head dimension
64): more key levels per CTA than stages, within the bound of its waits."""
import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm
from oracle import wm_oracle as orc
from parity_util import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,kd", [((3, 9, 12), 3), ((5, 17, 24), 5)])
def test_two_stages(grid, kd):
    C, heads, window = 128, 2, (kd, 5, 5)
    x = np.random.default_rng(7).standard_normal((1, int(np.prod(grid)), 3 * C)).astype(np.float32)
    q = torch.from_numpy(x).cuda().bfloat16()
    out = torch.empty(1, x.shape[1], C, device="cuda", dtype=torch.bfloat16)
    wm.wm_op_neighborhood_attention(q, out, 1, *grid, C, heads, *window, True, wm.WM_PREC_BF16, wm.WM_NA_TCGEN05)
    torch.cuda.synchronize()
    wm.wm_device_status()   # no wait ran out
    x = q.float().cpu().numpy()
    nbr = orc.neighbor_index(*grid, *window, True)
    ref = orc.neighborhood_attention(x[..., :C], x[..., C:2 * C], x[..., 2 * C:], heads, nbr)
    assert_close(out.float().cpu().numpy(), ref, 1e-2, C // heads)
