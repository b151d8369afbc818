"""FP32 neighborhood attention on 2 x 2 query blocks against the FP64 oracle.

Shapes at the edges of its tiles (8, 12 or 16 latitudes and longitudes, two
queries a block): odd grids, grids smaller than a tile or as small as the
window, every head dimension and longitude window it takes, both longitude
modes. Tolerance 1e-6 relative L2 (FP32 sums over at most 64 channels and 245
keys, random signs: a few 1e-7).
"""
import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm
from oracle import wm_oracle as orc
from parity_util import assert_close

pytestmark = pytest.mark.gpu


def _run(qkv, grid, C, heads, window, periodic):
    B = qkv.shape[0]
    out = torch.full((B, int(np.prod(grid)), C), float("nan"), device="cuda")
    wm.wm_op_neighborhood_attention(torch.from_numpy(qkv).cuda(), out, B, *grid, C, heads, *window, periodic,
                                    wm.WM_PREC_FP32)
    torch.cuda.synchronize()
    wm.wm_device_status()
    return out.cpu().numpy()


def _qkv(B, grid, C, seed):
    return np.random.default_rng(seed).standard_normal((B, int(np.prod(grid)), 3 * C)).astype(np.float32) * 1.5


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("dh", [16, 32, 48, 64])
@pytest.mark.parametrize("grid,window", [((2, 7, 7), (1, 7, 7)), ((3, 9, 10), (3, 5, 7)), ((2, 17, 25), (1, 3, 5)),
                                         ((3, 13, 33), (3, 7, 5)), ((1, 31, 16), (1, 9, 3)), ((4, 24, 48), (3, 5, 5)),
                                         ((2, 11, 40), (1, 1, 7))])
def test_matches_oracle(grid, window, dh, periodic):
    heads, C = 2, 2 * dh
    qkv = _qkv(2, grid, C, 1)
    got = _run(qkv, grid, C, heads, window, periodic)
    nbr = orc.neighbor_index(*grid, *window, periodic)
    ref = orc.neighborhood_attention(qkv[..., :C], qkv[..., C:2 * C], qkv[..., 2 * C:], heads, nbr)
    assert_close(got, ref, 1e-6, dh, (grid, window, dh, periodic))


@pytest.mark.parametrize("scale", [30.0, 1e-3])
def test_wide_and_flat_scores(scale):
    """Scores over a range of hundreds (the reference moves often, most probabilities underflow), and nearly equal."""
    grid, window, heads, C = (3, 12, 24), (3, 7, 7), 2, 96
    qkv = _qkv(1, grid, C, 2)
    qkv[..., :C] *= scale
    got = _run(qkv, grid, C, heads, window, True)
    nbr = orc.neighbor_index(*grid, *window, True)
    ref = orc.neighborhood_attention(qkv[..., :C], qkv[..., C:2 * C], qkv[..., 2 * C:], heads, nbr)
    # a score s carries an error of a few 2^-24 |s|, its probability as much relative to itself
    smax = 16.0 * max(scale, 1.0)
    assert_close(got, ref, 1e-6 + 4 * 2.0 ** -24 * smax, C // heads, scale)


@pytest.mark.parametrize("part", [1, 2])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_nonfinite_stays_in_its_windows(part, value):
    """A K (part 1) or V (part 2) value that is not finite reaches the queries whose windows hold it and no other."""
    grid, window, heads, C = (3, 10, 20), (3, 5, 7), 2, 64
    qkv = _qkv(1, grid, C, 3)
    nbr = orc.neighbor_index(*grid, *window, True)
    clean = orc.neighborhood_attention(qkv[..., :C], qkv[..., C:2 * C], qkv[..., 2 * C:], heads, nbr)
    tok, ch = (1 * 10 + 4) * 20 + 19, 5           # next to the longitude wrap, first head
    qkv[0, tok, part * C + ch] = value
    got = _run(qkv, grid, C, heads, window, True)[0]
    sees = (nbr == tok).any(1)
    hit = np.zeros((len(sees), C), bool)
    if part == 2:
        hit[:, ch] = sees                          # that channel of the queries that weigh it
    else:
        # +-inf * q gives a score of +inf (NaN after the softmax), -inf (probability 0) or NaN
        score = qkv[0, :, ch] * value
        hit[:, :C // heads] = (sees & ~(score == -np.inf))[:, None]
    assert not np.isfinite(got[hit]).any()
    assert np.isfinite(got[~hit]).all()
    same = ~hit & ~sees[:, None]
    assert np.abs(got[same] - clean[0][same]).max() <= 1e-5
