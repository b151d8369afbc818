"""FP32 linear layers (wm_op_linear, WM_PREC_FP32) against float64.

The kernel splits every operand exactly into three bf16 parts and adds six
products per pair. Elementwise bound on the error, with S = sum_k |a_k w_k|:
the products left out are below 2^-25 |a w| each; the 24 tensor-core additions
of a 64-wide group of k round the group's sum by at most 2^-23 each; the
K / 64 groups are added in FP32 (2^-24 each), then bias and residual (2^-23 of
the result's parts). Random signs leave a small part of that bound, so the
relative L2 error is also held to 1e-6, a tenth of the FP32 path's 1e-5.
"""
import numpy as np
import pytest
import torch

import paper_2503_22235_gb300 as wm

pytestmark = pytest.mark.gpu


def _inputs(M, N, K, seed, offset=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn(M * K + offset, generator=g, device="cuda")[offset:].view(M, K)
    W = torch.randn(N * K + offset, generator=g, device="cuda")[offset:].view(N, K)
    return A, W, torch.randn(N, generator=g, device="cuda")


def _check(A, W, b, epilogue, out0=None):
    M, K = A.shape
    N = W.shape[0]
    out = torch.zeros(M, N, device="cuda") if out0 is None else out0.clone()
    wm.wm_op_linear(A, W, b, out, wm.WM_PREC_FP32, epilogue)
    ref = A.double() @ W.double().T
    bound = (2.0 ** -25 + 24 * 2.0 ** -23 + (K / 64 + 1) * 2.0 ** -24) * (A.abs().double() @ W.abs().double().T)
    if b is not None:
        ref = ref + b.double()
    bound = bound + 2.0 ** -23 * ref.abs()
    if epilogue == wm.EPI_GELU:   # slope at most 1.13, erff within 2 ulp
        ref = 0.5 * ref * (1 + torch.erf(ref / 2 ** 0.5))
        bound = 1.13 * bound + 2.0 ** -22 * ref.abs() + 1e-6 * 2.0 ** -2
    if out0 is not None and epilogue == wm.EPI_RESID_F32:
        ref = ref + out0.double()
        bound = bound + 2.0 ** -23 * ref.abs()
    err = (out.double() - ref).abs()
    assert bool((err <= bound).all()), float((err - bound).max())
    assert float((out.double() - ref).norm() / ref.norm()) <= 1e-6


@pytest.mark.parametrize("M", [1, 127, 129, 300])
@pytest.mark.parametrize("N", [1, 7, 64, 65, 132, 200])
@pytest.mark.parametrize("K", [1, 4, 31, 32, 33, 64, 68, 129])
def test_tile_edges(M, N, K):
    """Rows, columns and k around the tiles' edges; K and N that tensor copies cannot address."""
    A, W, b = _inputs(M, N, K, 1)
    _check(A, W, b, wm.EPI_STORE_F32)


@pytest.mark.parametrize("M,N,K", [(20475, 192, 96), (4609, 384, 1000), (2500, 3072, 768), (5000, 512, 38)])
@pytest.mark.parametrize("epilogue", [wm.EPI_STORE, wm.EPI_GELU, wm.EPI_RESID_F32])
def test_many_tiles(M, N, K, epilogue):
    """More tiles than SMs (a CTA walks several), weights split beforehand; every epilogue."""
    A, W, b = _inputs(M, N, K, 2)
    _check(A, W, b, epilogue, torch.randn(M, N, device="cuda"))


def test_unaligned_and_no_bias():
    """Operands 4 bytes off a 16-byte boundary take the plain loads; bias may be absent."""
    A, W, b = _inputs(700, 256, 128, 3, offset=1)
    _check(A, W, b, wm.EPI_STORE_F32)
    _check(A, W, None, wm.EPI_STORE_F32)


@pytest.mark.parametrize("scale", [1e-38, 1e-34, 1e-25, 1e25])
def test_scales(scale):
    """The split is exact far from 1 too; sums of the smallest operands are recomputed."""
    A, W, _ = _inputs(300, 128, 96, 4)
    out = torch.zeros(300, 128, device="cuda")
    wm.wm_op_linear(A * scale, W, None, out, wm.WM_PREC_FP32, wm.EPI_STORE_F32)
    ref = (A * scale).double() @ W.double().T
    assert float((out.double() - ref).norm() / ref.norm()) <= 1e-6


@pytest.mark.parametrize("M", [260, 40000])
def test_nonfinite(M):
    """Infinities, NaN and values that round up to infinity give what a chain of FP32 FMAs gives, in their rows and
    columns only."""
    N, K = 96, 64
    A, W, _ = _inputs(M, N, K, 5)
    A[3, 5], A[130, 7], A[200, 1] = float("inf"), float("nan"), 3.4028e38
    W[9, 2] = float("-inf")
    W[11] *= 0.25
    out = torch.zeros(M, N, device="cuda")
    wm.wm_op_linear(A, W, None, out, wm.WM_PREC_FP32, wm.EPI_STORE_F32)
    out = out[:260].cpu().numpy()
    a, w = A[:260].double().cpu().numpy(), W.double().cpu().numpy()
    ref = np.zeros((260, N), np.float32)
    with np.errstate(all="ignore"):
        for k in range(K):
            ref = (a[:, k:k + 1] * w[None, :, k] + ref.astype(np.float64)).astype(np.float32)
    assert np.array_equal(np.isnan(out), np.isnan(ref))
    assert np.array_equal(np.isinf(out), np.isinf(ref))
    inf = np.isinf(ref)
    assert np.array_equal(out[inf], ref[inf])
    fin = np.isfinite(ref)
    scale = np.abs(a).clip(0, 3e38) @ np.abs(w).clip(0, 3e38).T
    assert np.all(np.abs(out[fin].astype(np.float64) - ref[fin]) <= 1e-5 * scale[fin])


def test_capture():
    """A captured call allocates nothing and its replay computes the same function."""
    A, W, b = _inputs(6000, 512, 256, 6)
    out = torch.zeros(6000, 512, device="cuda")
    wm.wm_op_linear(A, W, b, out, wm.WM_PREC_FP32, wm.EPI_STORE_F32)
    eager = out.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        wm.wm_op_linear(A, W, b, out, wm.WM_PREC_FP32, wm.EPI_STORE_F32)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert float((out - eager).abs().max()) <= 1e-5
