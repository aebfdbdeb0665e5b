"""The face level's candidates where boxes are unbounded (coordinates beyond FP32's range on
both sides, in every dimension): every face of one mesh with every face of the other, each
once, for tiles that the faces do not fill."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


def _mesh(n, m, seed, periodic=True):
    """Neighbouring vertices on opposite sides, all coordinates between 5e38 and 5e39."""
    g = torch.Generator().manual_seed(seed)
    sign = 1.0 - 2.0 * ((torch.arange(m)[:, None] + torch.arange(n)[None, :]) % 2).to(torch.float64)
    X = sign * (5e38 + 4.5e39 * torch.rand(4, m, n, generator=g, dtype=torch.float64))
    return tms.Mesh.from_grid(synth.MeshGrid(X, torch.linspace(0, 1, m, dtype=torch.float64), periodic))


@pytest.mark.parametrize("na,ma,nb,mb", [(4, 2, 3, 2), (4, 3, 10, 4), (10, 4, 9, 2), (30, 8, 34, 6)])
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("face_level", [0, 1])
def test_every_pair_once(na, ma, nb, mb, periodic, face_level):
    A, B = _mesh(na, ma, 1, periodic), _mesh(nb, mb, 2, periodic)
    quads = lambda n, m: (n if periodic else n - 1) * (m - 1)
    pairs = quads(na, ma) * quads(nb, mb) * (1 if face_level else 4)
    kw = dict(face_level=face_level, patch=0, hit_capacity=1 << 17)
    got = gpu_records(tms.search(A, B, **kw))
    if not (periodic and (na % 2 or nb % 2)):      # (else neighbours round the seam agree in sign)
        assert tms.last_stats()["candidates"] == pairs
    want = gpu_records(tms.search(A, B, precision=0, narrow_filter=0, **kw))
    assert all(np.array_equal(got[k], want[k]) for k in want)
