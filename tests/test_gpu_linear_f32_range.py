"""FP32 linear layers on operands far from 1 on either side: small operands lose
parts of their bf16 split in the tensor core, and sums may overflow on the way.
The results must be what FP32 multiply-adds give.

Elementwise bound against float64, with S = sum_k |a_k w_k|: a chain of K FMAs is
off by at most K 2^-24 S (its roundings) plus K 2^-149 (subnormal results).
Where S passes the largest float, or an operand is infinite, partial sums may
overflow in one order and not in another: nothing is asked there, except that
the result is not finite where the sum itself is not."""
import pytest
import torch

import paper_2503_22235_gb300 as wm

pytestmark = pytest.mark.gpu


def _run(A, W, out=None, epilogue=wm.EPI_STORE_F32):
    out = torch.full((A.shape[0], W.shape[0]), float("nan"), device="cuda") if out is None else out
    wm.wm_op_linear(A, W, None, out, wm.WM_PREC_FP32, epilogue)
    torch.cuda.synchronize()
    wm.wm_device_status()
    return out


def _check(A, W):
    K = A.shape[1]
    out = _run(A, W).double()
    ref, S = A.double() @ W.double().T, A.abs().double() @ W.abs().double().T
    err = (out - ref).abs()
    bound = K * 2.0 ** -24 * S + K * 2.0 ** -149
    sound = S * (1 + K * 2.0 ** -24) < 3.4028234e38
    assert bool((err <= bound)[sound].all()), float((err / bound)[sound].max())
    over = ~(ref.abs() < 3.4028236e38 * (1 + K * 2.0 ** -24))
    assert not bool(out[over].isfinite().any())


def _randn(M, K, seed):
    return torch.randn(M, K, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")


# (300, 128, 96): W split in the kernel; (20000, 272, 160): split beforehand, several tiles a CTA;
# (130, 70, 37): operands that no tensor copy addresses
@pytest.mark.parametrize("M,N,K", [(300, 128, 96), (20000, 272, 160), (130, 70, 37)])
@pytest.mark.parametrize("a,w", [(1e-38, 1e30), (1e30, 1e-38), (1e-44, 1e38), (1e-36, 1e20), (1e-42, 1.0), (1.0, 1e-41),
                                 (1e-20, 1e-22), (1e-10, 1e-15), (1e-30, 1e-12), (1e18, 1e19)])
def test_scaled(M, N, K, a, w):
    _check(_randn(M, K, 1) * a, _randn(N, K, 2) * w)


@pytest.mark.parametrize("M,N,K", [(300, 128, 96), (20000, 272, 160)])
def test_mixed(M, N, K):
    """Small operands in some rows, columns and places only; zeros beside them; sums that only small operands make."""
    A, W = _randn(M, K, 3), _randn(N, K, 4)
    A[::7] *= 1e-39
    A[3::11] = 0.0
    A[5, :] = 0.0
    A[5, 17] = 1e-44
    W[::5] *= 1e25
    W[1::5, 3] = 1e-42
    W[2] = 0.0
    W[2, 17] = 3e37
    _check(A, W)


def test_small_operands_cost_ordinary_rows_nothing():
    """A single tiny operand leaves every other row's bits alone."""
    A, W = _randn(5000, 256, 5), _randn(256, 256, 6)
    ref = _run(A, W)
    A[2500, 8] = 1e-40
    W[7, 9] = -1e-41
    got = _run(A, W)
    keep = torch.ones(5000, dtype=torch.bool, device="cuda")
    keep[2500] = False
    cols = torch.arange(256, device="cuda") != 7
    assert torch.equal(got[keep][:, cols], ref[keep][:, cols])


def test_sums_that_pass_the_largest_float_on_the_way():
    """Products that cancel in the order of k: multiply-adds one after the other stay finite."""
    A, W = torch.zeros(200, 64, device="cuda"), torch.zeros(64, 64, device="cuda")
    A[:, 0::4], A[:, 1::4], A[:, 2::4] = 2e19, -2e19, 1e19
    W[:, :] = 1.6e19
    got = _run(A, W)
    want = torch.zeros((), device="cuda", dtype=torch.float64)
    a, w = A[0].double(), W[0].double()
    for k in range(64):
        want = (want + a[k] * w[k]).float().double()
    assert torch.equal(got, torch.full_like(got, float(want)))


@pytest.mark.parametrize("tiny", [0.0, 1e-40])
def test_zero_sums(tiny):
    """Zero columns of W and zero rows of A over many tiles a CTA, alone and with small operands in later rows: zero
    sums stay zero, and those that only small operands make are found."""
    M, N, K = 60000, 256, 160
    A, W = _randn(M, K, 7), _randn(N, K, 8)
    W[5::64] = 0.0
    A[::97] = 0.0
    if tiny:
        W[5::64, 9] = 1e20
        A[:, 9] = 0.0
        A[40000::31, 9] = tiny
        A[59999, 9] = tiny
    _check(A, W)
