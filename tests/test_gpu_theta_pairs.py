"""Column translation in float pairs (1024, 2048 and 4096 points) against extended-precision
transforms: every number of coordinates, rows of unlike and of extreme size, few and many
columns, in place, and values that are not finite."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")
# a transform there and back in float pairs: 24 additions and multiplications deep, each
# within 2^-46 of the row's size, growing as the root of their number
TOL = 2.0 ** -42


def _fft(x, sign):
    n = x.shape[-1]
    if n == 1:
        return x
    e, o = _fft(x[..., 0::2], sign), _fft(x[..., 1::2], sign)
    ang = 2 * PI * np.arange(n // 2).astype(LD) / LD(n)
    t = (np.cos(ang) + np.clongdouble(1j * sign) * np.sin(ang)) * o
    return np.concatenate([e + t, e - t], -1)


def _exact(X, rho, derivative):
    N = X.shape[-1]
    k = np.fft.fftfreq(N, 1.0 / N).astype(LD)
    ph = k * rho.astype(LD)[:, None]
    H = np.cos(ph) + np.clongdouble(1j) * np.sin(ph)
    nyq = np.cos(LD(N // 2) * rho.astype(LD))
    if derivative:
        H, nyq = H * (np.clongdouble(1j) * k), 0 * nyq
    H[:, N // 2] = nyq
    return (_fft(_fft(X.astype(np.clongdouble), -1) * H, 1) / LD(N)).real


def _check(X, rho, derivative):
    N = X.shape[-1]
    want = _exact(X.numpy(), rho.numpy(), derivative)
    got = tms.theta_translate(X.cuda(), rho.cuda(), derivative=derivative).cpu().numpy()
    size = np.abs(X.numpy()).max(-1, keepdims=True) * (N / 2 if derivative else 1)
    assert (np.abs(got.astype(LD) - want) <= TOL * size).all()
    Y = X.cuda()
    tms.theta_translate(Y, rho.cuda(), derivative=derivative, out=Y)
    assert np.array_equal(Y.cpu().numpy(), got)
    return got


@pytest.mark.parametrize("N", [1024, 2048, 4096])
@pytest.mark.parametrize("C,M", [(1, 1), (2, 3), (3, 2), (4, 5)])
@pytest.mark.parametrize("derivative", [False, True])
def test_against_extended_precision(N, C, M, derivative):
    g = torch.Generator().manual_seed(N + 10 * C + M)
    X = torch.randn(C, M, N, generator=g, dtype=torch.float64)
    rho = torch.rand(M, generator=g, dtype=torch.float64) * 200.0 - 100.0
    rho[0] = 0.0 if C == 2 else rho[0]
    _check(X, rho, derivative)


def test_rows_of_unlike_and_extreme_size():
    g = torch.Generator().manual_seed(5)
    X = torch.randn(4, 3, 1024, generator=g, dtype=torch.float64)
    f = torch.tensor([[1.0, 1e-9, 1e30], [1e-12, 0.0, 1e-200], [1e290, 3.0, 0.0], [1e-305, 1e-4, 1e-290]],
                     dtype=torch.float64)
    X = X * f[:, :, None]
    rho = torch.tensor([0.3, -7.0, 1e7], dtype=torch.float64)
    got = _check(X, rho, False)
    assert not got[1, 1].any() and not got[2, 2].any()
    # subnormal rows
    tiny = torch.randn(2, 1, 1024, generator=g, dtype=torch.float64) * 1e-310
    got = tms.theta_translate(tiny.cuda(), 1.7).cpu().numpy()
    want = _exact(tiny.numpy(), np.array([1.7]), False)
    assert (np.abs(got.astype(LD) - want) <= 2 * LD(5e-324)).all()


@pytest.mark.parametrize("M", [500, 1213])
def test_many_columns_give_each_its_own(M):
    """Blocks that stay for several rows: every column as it comes alone."""
    g = torch.Generator().manual_seed(M)
    X = torch.randn(3, M, 1024, generator=g, dtype=torch.float64).cuda()
    rho = (torch.rand(M, generator=g, dtype=torch.float64) * 6.0).cuda()
    whole = tms.theta_translate(X, rho)
    for m in (0, 1, M // 3, M // 2, M - 1):
        one = tms.theta_translate(X[:, m:m + 1].contiguous(), rho[m:m + 1])
        assert torch.equal(one[:, 0], whole[:, m])
    same = tms.theta_translate(X, 1.25)
    assert torch.equal(same, tms.theta_translate(X, torch.full((M,), 1.25, dtype=torch.float64).cuda()))


def test_rows_that_are_not_finite():
    g = torch.Generator().manual_seed(8)
    X = torch.randn(4, 3, 2048, generator=g, dtype=torch.float64).cuda()
    plain = tms.theta_translate(X, 2.4)
    X[1, 2, 77] = float("inf")
    X[2, 0, 5] = float("nan")
    got = tms.theta_translate(X, 2.4)
    assert not torch.isfinite(got[1, 2]).any() and not torch.isfinite(got[2, 0]).any()
    for c, m in ((0, 0), (0, 1), (1, 1), (2, 1), (2, 2), (3, 2)):
        assert torch.equal(got[c, m], plain[c, m])


def test_a_small_common_shift_keeps_fp64():
    """Below 1000 / N a common shift's arguments are nearly exact in FP64."""
    g = torch.Generator().manual_seed(9)
    X = torch.randn(2, 2, 1024, generator=g, dtype=torch.float64)
    got = tms.theta_translate(X.cuda(), 0.01).cpu().numpy()
    want = _exact(X.numpy(), np.array([0.01, 0.01]), False)
    assert np.abs(got.astype(LD) - want).max() <= 2.0 ** -47 * float(X.abs().max())
