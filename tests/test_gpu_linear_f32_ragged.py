"""FP32 linear layers whose last column tile is ragged, over many tiles a CTA: a
warp may stage one 32-column chunk of such a tile and two of the next, and
every copy must have left its staging tile before that is written again. Every
row is compared with float64.

Elementwise bound as for the FP32 linear layers at large: with S = sum_k |a_k
w_k|, 2^-25 S for the products left out, 24 additions of 2^-23 S in a 64-wide
group, (K / 64 + 1) of 2^-24 S between groups, 2^-23 of the result for the
bias and 2^-23 for the residual."""
import pytest
import torch

import paper_2503_22235_gb300 as wm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("epilogue", [wm.EPI_STORE_F32, wm.EPI_RESID_F32])
@pytest.mark.parametrize("K", [32, 64, 128, 320])
@pytest.mark.parametrize("N", [32, 68, 96, 132, 160, 272])
def test_every_row(N, K, epilogue):
    M = 60011
    g = torch.Generator(device="cuda").manual_seed(N + K)
    A, W = torch.randn(M, K, generator=g, device="cuda"), torch.randn(N, K, generator=g, device="cuda")
    b, x = torch.randn(N, generator=g, device="cuda"), torch.randn(M, N, generator=g, device="cuda")
    ref = A.double() @ W.double().T + b.double()
    bound = (2.0 ** -25 + 24 * 2.0 ** -23 + (K / 64 + 1) * 2.0 ** -24) * (A.abs().double() @ W.abs().double().T)
    bound += 2.0 ** -23 * ref.abs()
    if epilogue == wm.EPI_RESID_F32:
        ref += x.double()
        bound += 2.0 ** -23 * ref.abs()
    for _ in range(3):
        out = x.clone()
        wm.wm_op_linear(A, W, b, out, wm.WM_PREC_FP32, epilogue)
        err = (out.double() - ref).abs()
        assert bool((err <= bound).all()), float((err - bound).max())
