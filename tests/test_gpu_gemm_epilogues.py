"""The BF16 linear layer's bf16 epilogues (plain store; GELU on sixteen epilogue
warps) over tile widths: 64, 128 and 256 columns, CTA pairs, and the default
choice (pairs for large products with K >= 768) give the same bits, within the
bf16 rounding of the float64 reference. Ragged M, N inside a 32-column chunk, K
of a partial slice, with and without a bias."""
import numpy as np
import pytest
import torch
from scipy.special import erf

import paper_2503_22235_gb300 as wm

pytestmark = pytest.mark.gpu

CUDA = torch.device("cuda")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_22235_gb300 import build as wm_build
    wm_build.build()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    yield
    wm.wm_gemm_tile_override(wm.GEMM_TILES_TUNED)


@pytest.mark.parametrize("epi", [0, 1])
@pytest.mark.parametrize("M,N,K,bias", [(1, 8, 8, True), (129, 136, 72, True), (300, 264, 200, False),
                                        (1000, 512, 768, True), (20001, 768, 768, True), (19900, 512, 776, False)])
def test_tile_widths_agree(M, N, K, bias, epi):
    rng = np.random.default_rng(M + N + K)
    A = torch.from_numpy(rng.standard_normal((M, K)).astype(np.float32)).to(CUDA, torch.bfloat16)
    W = torch.from_numpy((rng.standard_normal((N, K)) / np.sqrt(K)).astype(np.float32)).to(CUDA, torch.bfloat16)
    b = torch.from_numpy((0.1 * rng.standard_normal(N)).astype(np.float32)).to(CUDA) if bias else None
    outs = []
    try:
        for mode in range(5):
            wm.wm_gemm_tile_override(mode)
            o = torch.full((M, N), float("nan"), device=CUDA, dtype=torch.bfloat16)
            wm.wm_op_linear(A, W, b, o, wm.WM_PREC_BF16, epi)
            torch.cuda.synchronize()
            outs.append(o)
    finally:
        wm.wm_gemm_tile_override(wm.GEMM_TILES_TUNED)
    for mode in range(1, 5):
        assert torch.equal(outs[0], outs[mode]), mode
    rows = rng.choice(M, size=min(M, 300), replace=False)
    ref = A[rows].double().cpu().numpy() @ W.double().cpu().numpy().T
    if bias:
        ref = ref + b.double().cpu().numpy()
    if epi:
        ref = 0.5 * ref * (1 + erf(ref / np.sqrt(2)))
    got = outs[0][rows].double().cpu().numpy()
    # bf16 rounding (2^-9 relative), FP32 sums of K terms of size 1 / sqrt(K), and the erf formula's 1.5e-7
    np.testing.assert_array_less(np.abs(got - ref), 2.0 ** -8 * np.abs(ref) + 2e-5)
    wm.wm_device_status()
