"""A launch that is refused while the search's graph is captured, or without a graph, is an
error of that search, each time, and of no other."""
import numpy as np
import pytest

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("patch", [0, 1])
def test_refused_launch(use_graph, patch):
    p = synth.build_pair(32, 300, 100, 280, 90, stretch="exp", n_folds=3, sites=(16, 4), n_hits=0)
    A, B = tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)
    kw = dict(patch=patch, use_graph=use_graph)
    want = gpu_records(tms.search(A, B, **kw))
    for _ in range(3):
        with pytest.raises(tms.TmsError) as e:
            tms.search(A, B, inject=128, **kw)
        assert e.value.status == tms.TMS_ERR_CUDA and "merge" in str(e.value)
        got = gpu_records(tms.search(A, B, **kw))
        assert all(np.array_equal(got[k], want[k]) for k in want)
