"""A search follows what its stream holds before it, with and without a graph, in the
default stream and others, and from several threads at once."""
import threading

import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


def _pair():
    return synth.build_pair(61, 300, 120, 280, 100, stretch="exp", n_folds=3, sites=(16, 8), n_hits=0)


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("use_graph", [0, 1])
def test_order_in_a_stream(own, use_graph):
    p = _pair()
    A, B = tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)
    want = gpu_records(tms.search(A, B))
    torch.cuda.synchronize()
    st = torch.cuda.Stream() if own else torch.cuda.default_stream()
    away = A.X + 1e3
    home = A.X.clone()
    big = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    for _ in range(3):
        with torch.cuda.stream(st):
            A.X.copy_(away)
            big.fill_(1)
            assert len(tms.search(A, B, use_graph=use_graph)) == 0
            big.fill_(2)
            A.X.copy_(home)
            h = tms.search(A, B, use_graph=use_graph)
            got = gpu_records(h)
        assert all(np.array_equal(want[k], got[k]) for k in want)


def test_threads_on_their_own_streams():
    p = _pair()
    A, B = tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)
    want = [gpu_records(tms.search(A, B)), gpu_records(tms.search(B, A))]
    wrong = []

    def work(k):
        torch.cuda.set_device(0)
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(20):
                got = gpu_records(tms.search(*((A, B) if k % 2 == 0 else (B, A))))
                if not all(np.array_equal(want[k % 2][q], got[q]) for q in got):
                    wrong.append(k)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong
