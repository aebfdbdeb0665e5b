"""Phase alignment costs in float pairs (circles of 192 points or more) and in the FP64
loop beside it: tile and cluster edges, every number of coordinates, values at both
ends of the exponent range, ties, and values that are not finite."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
from oracle import theta as T

pytestmark = pytest.mark.gpu

# a distance in float pairs is within 2^-45 (its square's sum within 2^-46 a coordinate
# of eight), and so is a sum of them
RTOL = 2.0 ** -45


def _circles(N, C, A, seed, scale=1.0):
    g = torch.Generator().manual_seed(seed)
    Wp = torch.randn(A, C, N, generator=g, dtype=torch.float64) * scale
    Wr = torch.roll(Wp, 5 % N, dims=-1) + 1e-4 * scale * torch.randn(A, C, N, generator=g, dtype=torch.float64)
    return Wr, Wp


def _check(Wr, Wp):
    shift, cost = tms.phase_align(Wr.cuda(), Wp.cuda())
    for a in range(Wr.shape[0]):
        m, want = T.phase_align(Wr[a].numpy(), Wp[a].numpy())
        assert np.abs(cost[a].cpu().numpy() - want).max() <= RTOL * want.max()
        assert np.allclose(cost[a].cpu().numpy(), want, rtol=RTOL, atol=0)
        assert int(shift[a]) == m
    return cost


@pytest.mark.parametrize("N", [1, 2, 3, 33, 191, 192, 193, 255, 511, 512, 513, 1023, 1025, 1100])
def test_edges(N):
    _check(*_circles(N, 4, 2, N))


@pytest.mark.parametrize("C", range(1, 9))
@pytest.mark.parametrize("N", [130, 257])
def test_coordinates(C, N):
    _check(*_circles(N, C, 3, C))


@pytest.mark.parametrize("scale", [1e-140, 1e-30, 1e30, 1e150])
def test_scales(scale):
    _check(*_circles(300, 3, 1, 4, scale))


def test_coordinates_of_unlike_size():
    Wr, Wp = _circles(300, 4, 1, 9)
    f = torch.tensor([1.0, 1e-4, 1e3, 1e-9], dtype=torch.float64)[None, :, None]
    _check(Wr * f, Wp * f)


def test_equal_circles_and_ties():
    """A roll of a circle costs nothing at its shift; a circle of period N / 2 has every
    cost twice, the same number both times, and the first shift wins."""
    _, Wp = _circles(400, 4, 1, 2)
    shift, cost = tms.phase_align(torch.roll(Wp, 123, dims=-1).cuda(), Wp.cuda())
    assert int(shift[0]) == 123 and float(cost[0, 123]) == 0.0
    half = Wp[:, :, :200]
    W = torch.cat([half, half], dim=2)
    other = torch.cat([torch.roll(half, 7, dims=2)] * 2, dim=2) + 0.25
    shift, cost = tms.phase_align(other.cuda(), W.cuda())
    assert torch.equal(cost[0, :200], cost[0, 200:])
    assert int(shift[0]) == int(torch.argmin(cost[0, :200]))
    same = torch.full((1, 4, 256), 0.3, dtype=torch.float64)
    shift, cost = tms.phase_align((same + 1.0).cuda(), same.cuda())
    assert int(shift[0]) == 0 and torch.equal(cost[0], cost[0, :1].expand(256))
    zero = torch.zeros_like(same)
    shift, cost = tms.phase_align(zero.cuda(), zero.cuda())
    assert int(shift[0]) == 0 and not cost.any()


def test_not_finite():
    """An alignment with an infinity or a NaN gives the FP64 loop's costs, and its
    neighbours in the batch their own."""
    Wr, Wp = _circles(256, 2, 3, 6)
    plain = tms.phase_align(Wr.cuda(), Wp.cuda())[1]
    Wr[0, 1, 10] = float("inf")
    Wr[2, 0, 3] = float("nan")
    cost = tms.phase_align(Wr.cuda(), Wp.cuda())[1]
    assert torch.isinf(cost[0]).all() and torch.isnan(cost[2]).all()
    assert torch.equal(cost[1], plain[1])
