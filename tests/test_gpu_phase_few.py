"""Phase alignment costs that a few of the distances make: as near the exact ones as FP64 sums
of those distances, where a float pair's error would not average out."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
from tests.test_gpu_phase_cancel import _exact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [150, 192, 257, 700, 1030])
@pytest.mark.parametrize("C", [2, 4])
def test_costs_of_few_distances(N, C):
    """At most four distances differ from zero at any shift: each within C / 2 + 2 roundings
    (2^-53), their sum within three more."""
    g = torch.Generator().manual_seed(N + C)
    Wr, Wp = torch.zeros(C, N, dtype=torch.float64), torch.zeros(C, N, dtype=torch.float64)
    for W in (Wr, Wp):
        W[:, torch.randperm(N, generator=g)[:2]] = torch.randn(C, 2, generator=g, dtype=torch.float64)
    want = _exact(Wr, Wp)
    shift, cost = tms.phase_align(Wr[None].cuda(), Wp[None].cuda())
    got = cost[0].cpu().numpy()
    assert (np.abs(got - want) <= (C / 2 + 5) * 2.0 ** -53 * want).all()
    assert int(shift[0]) == int(np.argmin(got))
