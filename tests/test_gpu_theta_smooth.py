"""Column translation and derivative of smooth rows (a few harmonics, as a manifold's columns
are) hold what a plain FP64 transform holds: shifts of 0, small and large ones, as an array
and common; and rows of unlike size that share a transform."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
from tests.test_gpu_theta_pairs import LD, _exact

pytestmark = pytest.mark.gpu

RHO = [0.0, 1e-4, 0.7, -3.1, 97.3]


def _rows(C, M, N, seed):
    g = torch.Generator().manual_seed(seed)
    th = 2 * np.pi * torch.arange(N, dtype=torch.float64) / N
    k = torch.arange(7, dtype=torch.float64)
    a, b = (torch.randn(C, M, 7, generator=g, dtype=torch.float64) for _ in range(2))
    kt = k[:, None] * th
    return torch.einsum("cmk,kn->cmn", a, torch.cos(kt)) + torch.einsum("cmk,kn->cmn", b, torch.sin(kt))


def _radix2(x, sign):
    n = x.shape[-1]
    if n == 1:
        return x
    e, o = _radix2(x[..., 0::2], sign), _radix2(x[..., 1::2], sign)
    t = np.exp(sign * 2j * np.pi * np.arange(n // 2) / n) * o
    return np.concatenate([e + t, e - t], -1)


def _fp64(X, rho, derivative):
    """The same transform in FP64, radix 2, the multiplier rounded from extended precision."""
    N = X.shape[-1]
    k = np.fft.fftfreq(N, 1.0 / N).astype(LD)
    ph = k * rho.astype(LD)[:, None]
    H = np.cos(ph) + np.clongdouble(1j) * np.sin(ph)
    if derivative:
        H = H * (np.clongdouble(1j) * k)
    H[:, N // 2] = 0 if derivative else np.cos(LD(N // 2) * rho.astype(LD))
    return (_radix2(_radix2(X.astype(np.complex128), -1) * H.astype(np.complex128), 1) / N).real


def _rms(v):
    return np.sqrt((v.astype(LD) ** 2).mean(-1)).astype(np.float64)


@pytest.mark.parametrize("N", [256, 1024, 2048, 4096])
@pytest.mark.parametrize("derivative", [False, True])
def test_smooth_rows(N, derivative):
    # both errors are sums of 2 log2 N rounding errors a value; the kernel's twiddles are
    # products of two, at most three roundings where the model's have one
    X = _rows(4, len(RHO), N, N)
    rho = np.array(RHO)
    want = _exact(X.numpy(), rho, derivative)
    bound = 4.0 * _rms(_fp64(X.numpy(), rho, derivative) - want)
    got = tms.theta_translate(X.cuda(), torch.from_numpy(rho).cuda(), derivative=derivative)
    assert (_rms(got.cpu().numpy() - want) <= bound).all()
    for m, r in enumerate(RHO):
        one = tms.theta_translate(X[:, m:m + 1].contiguous().cuda(), r, derivative=derivative)
        assert torch.equal(one[:, 0], got[:, m])


@pytest.mark.parametrize("ratio", [1e-12, 1e-6, 2.0, 1e9, 1e300])
def test_rows_of_unlike_size_share_a_transform(ratio):
    X = _rows(2, len(RHO), 512, 3)
    rho = torch.tensor(RHO, dtype=torch.float64).cuda()
    alone = [tms.theta_translate(X[c:c + 1].cuda(), rho) for c in (0, 1)]
    X[1] *= ratio
    both = tms.theta_translate(X.cuda(), rho).cpu().numpy()
    for c, f in ((0, 1.0), (1, ratio)):
        size = float(X[c].abs().max())
        # two transforms, each within 2 log2 N places (2^-52) of the row's size, and the
        # rounding of the scaled row
        assert np.abs(both[c] - alone[c][0].cpu().numpy() * f).max() <= 2.0 ** -46 * size
