"""FP32 attention on latents that are partly or wholly NaN: the NaN reach exactly
the queries whose windows hold them, every other query keeps its accuracy, and
the call takes at most eight times its time on finite values (twice what the
kernel with one query per four threads took, which treated every value alike)."""
import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm
from oracle import wm_oracle as orc

pytestmark = pytest.mark.gpu


def _attend(qkv, out, grid, C, heads, window, periodic=True):
    wm.wm_op_neighborhood_attention(qkv, out, qkv.shape[0], *grid, C, heads, *window, periodic, wm.WM_PREC_FP32)


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("dh", [16, 32, 48, 64])
@pytest.mark.parametrize("window", [(1, 3, 3), (3, 5, 5), (3, 3, 7)])
def test_nan_values_stay_in_their_windows(window, dh, periodic):
    grid, heads, C = (3, 13, 21), 2, 2 * dh
    n = int(np.prod(grid))
    rng = np.random.default_rng(dh)
    qkv = rng.standard_normal((1, n, 3 * C)).astype(np.float32) * 1.5
    nbr = orc.neighbor_index(*grid, *window, periodic)
    ref = orc.neighborhood_attention(qkv[..., :C], qkv[..., C:2 * C], qkv[..., 2 * C:], heads, nbr)[0]
    bad = rng.choice(n, 9, replace=False)
    ch = rng.choice(C, 9)
    qkv[0, bad, 2 * C + ch] = np.nan
    out = torch.full((1, n, C), 7.0, device="cuda")
    _attend(torch.from_numpy(qkv).cuda(), out, grid, C, heads, window, periodic)
    torch.cuda.synchronize()
    got = out.cpu().numpy()[0]
    hit = np.zeros((n, C), bool)
    for t, c in zip(bad, ch):
        hit[(nbr == t).any(1), c] = True
    assert np.array_equal(np.isnan(got), hit)
    # FP32 sums of at most 245 keys of values near 1, probabilities within a few 1e-7
    assert np.abs(got[~hit] - ref[~hit]).max() <= 2e-5


@pytest.mark.parametrize("every", [1, 2, 50, 1000])
def test_time(every):
    grid, window, heads, C = (9, 60, 120), (5, 7, 7), 16, 768
    n = int(np.prod(grid))
    g = torch.Generator(device="cuda").manual_seed(1)
    qkv = torch.randn(1, n, 3 * C, generator=g, device="cuda")
    out = torch.empty(1, n, C, device="cuda")

    def ms():
        _attend(qkv, out, grid, C, heads, window)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        for _ in range(3):
            _attend(qkv, out, grid, C, heads, window)
        e[1].record()
        torch.cuda.synchronize()
        return e[0].elapsed_time(e[1]) / 3

    finite = ms()
    qkv[:, ::every] = float("nan")
    assert ms() <= 8.0 * finite
