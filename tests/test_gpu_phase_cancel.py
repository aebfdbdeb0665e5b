"""Phase alignment costs where most of the circles' size cancels out of the distances (a large
coordinate that is constant or nearly so, circles that agree to a few places, coordinates
that are tiny most of the way) against extended precision: within a float pair's 2^-45 of
themselves, not of the largest coordinate, and equal where their terms are."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms

pytestmark = pytest.mark.gpu

RTOL = 2.0 ** -45
LD = np.longdouble


def _circles(N, C, seed):
    g = torch.Generator().manual_seed(seed)
    k = torch.arange(1, 7, dtype=torch.float64)
    kt = k[:, None] * (2 * np.pi * torch.arange(N, dtype=torch.float64) / N)
    a = torch.randn(2, C, 6, generator=g, dtype=torch.float64) / k
    return torch.einsum("ck,kn->cn", a[0], torch.cos(kt)) + torch.einsum("ck,kn->cn", a[1], torch.sin(kt))


def _exact(Wr, Wp):
    r, p = Wr.numpy().astype(LD), Wp.numpy().astype(LD)
    return np.array([np.sqrt(((np.roll(r, -m, axis=1) - p) ** 2).sum(0)).sum() for m in range(r.shape[1])])


def _constant(N, big, small):
    p = _circles(N, 4, 1) * small
    r = torch.roll(p, 9, dims=1) + 1e-3 * small * _circles(N, 4, 2)
    p[0] = r[0] = big
    return r, p


def _offset(N, big, small):
    p = _circles(N, 4, 3) * small
    r = p + 1e-3 * small * _circles(N, 4, 4)
    p[2] += big
    r[2] += big
    return r, p


def _near(N, d):
    p = _circles(N, 3, 5)
    return torch.roll(p * (1 + d * _circles(N, 3, 6)), -11, dims=1), p


def _bumps(N, d):
    x = torch.linspace(-1, 1, N, dtype=torch.float64)
    p = torch.stack([torch.exp(-200 * (x - c) ** 2) for c in (-0.3, 0.1, 0.4)])
    return torch.roll(p * (1 + d), 5, dims=1), p


CASES = [(_constant, (1e6, 1e-6)), (_constant, (1e30, 1.0)), (_constant, (3.0, 1e-12)), (_offset, (1e4, 1e-3)),
         (_offset, (1e6, 1.0)), (_offset, (1e8, 1e-3)), (_offset, (1e10, 1.0)), (_near, (1e-9,)), (_near, (1e-14,)),
         (_bumps, (1e-8,)), (_bumps, (1e-3,))]


@pytest.mark.parametrize("N", [150, 300, 1025])
@pytest.mark.parametrize("make,args", CASES, ids=[f"{f.__name__[1:]}-{a}" for f, a in CASES])
def test_costs(make, args, N):
    Wr, Wp = make(N, *args)
    want = _exact(Wr, Wp)
    shift, cost = tms.phase_align(torch.stack([Wr, Wp]).cuda(), torch.stack([Wp, Wp]).cuda())
    assert (np.abs(cost[0].cpu().numpy() - want) <= RTOL * want).all()
    assert int(shift[0]) == int(np.argmin(cost[0].cpu().numpy()))
    assert int(shift[1]) == 0 and float(cost[1, 0]) == 0.0


def test_equal_terms_give_equal_costs():
    """Circles of period N / 2 under a large constant coordinate: every cost twice."""
    p, r = _circles(700, 3, 7) * 1e-8, _circles(700, 3, 8) * 1e-8
    p, r = torch.cat([p, p], dim=1), torch.cat([r, r], dim=1)
    p[1] = r[1] = 1.0
    shift, cost = tms.phase_align(r[None].cuda(), p[None].cuda())
    assert torch.equal(cost[0, :700], cost[0, 700:]) and int(shift[0]) < 700
