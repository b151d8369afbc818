"""Linear layers whose bias does not start on a 16-byte boundary (a view into a
packed weight vector) give the bits of the same bias aligned: BF16 plain store
and GELU over tile widths and CTA pairs, e4m3 GELU; whole and ragged 32-column
chunks."""
import pytest
import torch

import paper_2503_22235_gb300 as wm

pytestmark = pytest.mark.gpu


def _inputs(M, N, K, offset):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.randn(M, K, generator=g, device="cuda")
    W = torch.randn(N, K, generator=g, device="cuda") / K ** 0.5
    bias = torch.randn(N, generator=g, device="cuda")
    packed = torch.zeros(N + 8, device="cuda")
    packed[offset:offset + N] = bias
    return A, W, bias, packed[offset:offset + N]


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("mode", [wm.GEMM_TILES_128, wm.GEMM_TILES_256, wm.GEMM_TILES_PAIR, wm.GEMM_TILES_64])
@pytest.mark.parametrize("epi", [wm.EPI_STORE, wm.EPI_GELU, wm.EPI_STORE_F32])
@pytest.mark.parametrize("M,N,K", [(130, 256, 64), (70, 72, 72)])
def test_bf16(M, N, K, epi, mode, offset):
    A, W, bias, view = _inputs(M, N, K, offset)
    outs = []
    try:
        wm.wm_gemm_tile_override(mode)
        for b in (bias, view):
            out = torch.zeros(M, N, device="cuda", dtype=torch.float32 if epi == wm.EPI_STORE_F32 else torch.bfloat16)
            wm.wm_op_linear(A.bfloat16(), W.bfloat16(), b, out, wm.WM_PREC_BF16, epi)
            torch.cuda.synchronize()
            outs.append(out)
    finally:
        wm.wm_gemm_tile_override(wm.GEMM_TILES_TUNED)
    assert torch.equal(*outs)


@pytest.mark.parametrize("offset", [1, 2])
def test_e4m3_gelu(offset):
    M, N, K = 130, 272, 64
    A, W, bias, view = _inputs(M, N, K, offset)
    A8, W8 = (t.to(torch.float8_e4m3fn).view(torch.uint8) for t in (A, W))
    outs = []
    for b in (bias, view):
        out = torch.zeros(M, N, device="cuda", dtype=torch.uint8)
        wm.wm_op_linear_e4m3(A8, W8, 1.0, b, out, 0.5, wm.EPI_GELU_F8)
        torch.cuda.synchronize()
        outs.append(out)
    assert torch.equal(*outs)
