"""Hits that fall on a few triangles of A, up to and past what a bucket of the short merge
takes: the hits of the search with the meshes exchanged, whose A side spreads them, in order;
a batch in which one pair's hits crowd; and one retry for a plan that finds it so."""
import math

import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


def _sheets(waves, n=16384):
    """A strip of two triangles, and a fine one that waves through its plane."""
    t = torch.arange(n, dtype=torch.float64) / n
    A, B = torch.zeros(4, 2, 2, dtype=torch.float64), torch.zeros(4, 2, n, dtype=torch.float64)
    A[0, :, 1], A[1, 1] = 1.0, 1e-3
    B[0], B[1] = 0.01 + 0.98 * t, 5e-4 * (1.0 - 0.9 * t)
    B[2] = 1e-3 * torch.sin(2 * math.pi * waves * t + 0.3)
    B[3, 0], B[3, 1] = -4e-4, 6e-4
    s = torch.tensor([0.0, 1.0], dtype=torch.float64)
    return [tms.Mesh.from_grid(synth.MeshGrid(X, s, False)) for X in (A, B)]


def _keys(r, swapped=False):
    return list(zip(r["triB"], r["triA"]) if swapped else zip(r["triA"], r["triB"]))


@pytest.mark.parametrize("waves", [100, 540, 570, 600, 1500, 3000])
def test_few_triangles(waves):
    A, B = _sheets(waves)
    out = torch.zeros((1 << 14, tms.HIT_BYTES), dtype=torch.uint8, device="cuda")
    got = gpu_records(tms.search(A, B, out=out))
    crowded = max(np.bincount(got["triA"])) > 1024
    assert (tms.last_stats()["retries"] == 1) == crowded
    again = gpu_records(tms.search(A, B, out=out))
    assert tms.last_stats()["retries"] == 0
    want = gpu_records(tms.search(B, A))
    assert _keys(got) == sorted(_keys(want, True)) == _keys(again)
    assert abs(len(got["triA"]) - 2 * waves) <= 2


def test_a_pair_of_a_batch():
    A, B = _sheets(2000)
    p = synth.build_pair(9, 300, 100, 280, 90, stretch="exp", n_folds=3, sites=(16, 4), n_hits=0)
    C, D = tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)
    whole = tms.search_batched([C, A, C], [D, B, D])
    r, off = gpu_records(whole), whole.offsets.cpu().numpy()
    for i, (x, y) in enumerate(((C, D), (A, B), (C, D))):
        one = gpu_records(tms.search(x, y))
        assert [k[off[i]:off[i + 1]].tolist() for k in (r["triA"], r["triB"])] == \
            [one["triA"].tolist(), one["triB"].tolist()]
