"""A search whose every list starts at one record: each list in turn costs a run, one more for
every level of the trees, and the hits are those of a search with room."""
import math

import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


def _strips(n):
    """A strip of the (x, y) plane, and one along it that waves through the plane about once
    in ten quads: the nodes of every level overlap in a band along the diagonal."""
    t = torch.arange(n, dtype=torch.float64) / n
    A, B = torch.zeros(4, 2, n, dtype=torch.float64), torch.zeros(4, 2, n, dtype=torch.float64)
    A[0], A[1, 1] = t, 1e-3
    B[0], B[1] = t + 0.37 / n, 5e-4
    B[2] = 1e-3 * torch.sin(2 * math.pi * (n / 20.97) * t + 0.3)
    B[3, 0], B[3, 1] = -4e-4, 6e-4
    s = torch.tensor([0.0, 1.0], dtype=torch.float64)
    return [tms.Mesh.from_grid(synth.MeshGrid(X, s, False)) for X in (A, B)]


@pytest.mark.parametrize("n,levels", [(1 << 12, 0), (1 << 16, 1), (1 << 21, 4)])
def test_every_list_from_one_record(n, levels):
    A, B = _strips(n)
    kw = dict(hit_capacity=1 << 19)
    want = gpu_records(tms.search(A, B, **kw))
    got = gpu_records(tms.search(A, B, inject=33, **kw))
    # node pairs of each level, patch pairs, candidates, kept quads, raw hits
    assert tms.last_stats()["retries"] >= levels + 4
    assert all(np.array_equal(got[k], want[k]) for k in want)
    assert abs(len(want["triA"]) - n / 10.485) < 3
