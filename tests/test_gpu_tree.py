"""The patch pairs from the meshes' trees against the quads in the grid (patch = 0): the
same candidates and hits for meshes of one patch, of part of one, at the edges of a
node's 4 x 4 children and tall and wide ones, with one, two and three levels above the
patches, periodic and open, in both precisions and in one batch."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


def _pair(na, ma, nb, mb, periodic=True):
    p = synth.build_pair(900 + na + mb, max(na, 8), max(ma, 3), max(nb, 8), max(mb, 3), stretch="exp", n_folds=3,
                         sites=(max(2, nb // 12 & ~1), max(1, mb // 8)), n_hits=0)
    s = lambda x, n, m: synth.MeshGrid(x.X[:, :m, :n].contiguous(), x.s[:m].contiguous(), periodic)
    return s(p.A, na, ma), s(p.B, nb, mb)


SIZES = [(3, 2, 3, 2), (8, 5, 8, 5), (9, 6, 7, 3), (32, 17, 33, 18), (31, 16, 65, 5), (128, 65, 129, 66),
         (1030, 6, 40, 70), (260, 70, 515, 33), (700, 300, 600, 350)]


def _same(A, B, **kw):
    kw.setdefault("hit_capacity", 1 << 17)
    tree = gpu_records(tms.search(A, B, **kw))
    nt = tms.last_stats()["candidates"]
    grid = gpu_records(tms.search(A, B, patch=0, **kw))
    assert nt == tms.last_stats()["candidates"] or kw.get("narrow_filter", 1)
    for k in tree:
        assert np.array_equal(tree[k], grid[k]), k
    return tree


@pytest.mark.parametrize("size", SIZES, ids=[f"{a}x{b}-{c}x{d}" for a, b, c, d in SIZES])
@pytest.mark.parametrize("periodic", [True, False])
def test_tree_equals_grid(size, periodic):
    ga, gb = _pair(*size, periodic=periodic)
    A, B = tms.Mesh.from_grid(ga), tms.Mesh.from_grid(gb)
    _same(A, B)
    # without the patch frames every quad pair with overlapping boxes is a candidate
    _same(A, B, narrow_filter=0)
    _same(A, B, narrow_filter=0, precision=0)
    _same(A, A, narrow_filter=0)


def test_uneven_batch():
    meshes = [_pair(*s) for s in SIZES]
    As, Bs = [tms.Mesh.from_grid(a) for a, _ in meshes], [tms.Mesh.from_grid(b) for _, b in meshes]
    for kw in (dict(), dict(precision=0)):
        tree = tms.search_batched(As, Bs, **kw)
        grid = tms.search_batched(As, Bs, patch=0, **kw)
        assert torch.equal(tree.offsets, grid.offsets)
        a, b = gpu_records(tree), gpu_records(grid)
        assert all(np.array_equal(a[k], b[k]) for k in a)


def test_three_levels():
    """More than 2^22 pairs of nodes two levels up: three levels above the patches."""
    p = synth.build_pair(5, 4001, 509, 4093, 511, stretch="exp", n_folds=3, sites=(128, 24), n_hits=0)
    A, B = tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)
    assert len(_same(A, B)["triA"]) > 1000
    A = tms.Mesh.from_grid(p.A, k0=3, k1=400)
    B = tms.Mesh.from_grid(p.B, k0=100)
    _same(A, B, precision=0)


def test_node_lists_grow():
    """The node pairs' lists from one record up (inject bits 0 and 3 at the patch level)."""
    ga, gb = _pair(700, 300, 600, 350)
    A, B = tms.Mesh.from_grid(ga), tms.Mesh.from_grid(gb)
    ref = gpu_records(tms.search(A, B))
    for bit in (1, 8):
        got = gpu_records(tms.search(A, B, inject=bit))
        assert tms.last_stats()["retries"] >= 1
        assert all(np.array_equal(ref[k], got[k]) for k in ref)


def test_a_vertex_that_is_not_finite_is_found_each_time():
    ga, gb = _pair(128, 65, 129, 66)
    X = ga.X.cuda()
    A, B = tms.Mesh(X, ga.s), tms.Mesh.from_grid(gb)
    ref = gpu_records(tms.search(A, B))
    keep = X[1, 64, 127].clone()
    for v in (float("nan"), float("inf"), float("-inf")):
        X[1, 64, 127] = v
        for _ in range(2):
            with pytest.raises(tms.TmsError) as e:
                tms.search(A, B)
            assert e.value.status == tms.TMS_ERR_ARG
    X[1, 64, 127] = keep
    got = gpu_records(tms.search(A, B))
    assert all(np.array_equal(ref[k], got[k]) for k in ref)
