"""The merge of raw hits by its two routes -- buckets (up to 32768 raw hits) and
the radix sort (more, or with the look-back test switch, inject bit 4, which has
nothing to wait for on one sort tile) -- bit for bit, meshes shared between the
pairs of a batch, and the adjoint at the edges of its blocks."""
import numpy as np
import pytest
import torch

import oracle
import paper_2109_14814_gb300 as tms
import synth
from tests import meshcases
from tests.parity import compare, gpu_records

pytestmark = pytest.mark.gpu


def _identical(a, b):
    assert a.keys() == b.keys()
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def _hand(name):
    A, B, _, _ = meshcases.ALL_CASES[name]()
    return synth.MeshPair(A, B, None)


PAIRS = {n: (lambda n=n: _hand(n)) for n in meshcases.ALL_CASES}
PAIRS["config1"] = synth.config1
PAIRS["730 crossings"] = lambda: synth.build_pair(31, 200, 60, 190, 64, stretch="exp", n_folds=3, sites=(40, 16),
                                                  n_hits=20)


@pytest.mark.parametrize("name", sorted(PAIRS))
@pytest.mark.parametrize("kw", [dict(), dict(precision=0, narrow_filter=0), dict(tau=1e-3)], ids=["", "plain", "tau"])
def test_short_merge_equals_the_sort(name, kw):
    p = PAIRS[name]()
    A, B = tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)
    short = gpu_records(tms.search(A, B, **kw))
    raw = tms.last_stats()["raw_hits"]
    assert raw <= 2048                       # one sort tile
    _identical(short, gpu_records(tms.search(A, B, inject=16, **kw)))
    assert tms.last_stats()["raw_hits"] == raw
    # a short output buffer: the count, and the first records
    if len(short["triA"]) > 1:
        out = torch.zeros((1, tms.HIT_BYTES), dtype=torch.uint8, device="cuda")
        with pytest.raises(tms.TmsError) as e:
            tms.search(A, B, out=out, **kw)
        assert e.value.status == tms.TMS_ERR_CAPACITY
        one = gpu_records(tms.Hits(out))
        assert all(np.array_equal(one[k], short[k][:1]) for k in short)


def test_short_merge_of_a_batch():
    """Pairs with no hits, with merged ones and with many, offsets included; the
    same handles in several pairs, on either side and both."""
    grids = [PAIRS[n]() for n in ("parallel", "vertex", "config1", "coplanar", "730 crossings", "diagonal", "seam",
                                  "near_miss_out")]
    A = [tms.Mesh.from_grid(p.A) for p in grids]
    B = [tms.Mesh.from_grid(p.B) for p in grids]
    pairs = [(A[k], B[k]) for k in range(len(grids))]
    pairs += [(A[4], B[4]), (B[4], A[4]), (A[2], A[2]), (A[1], B[5]), (A[4], B[4])]
    As, Bs = [a for a, _ in pairs], [b for _, b in pairs]
    h = tms.search_batched(As, Bs)
    offs, rec = h.offsets.cpu().numpy(), gpu_records(h)
    assert offs[0] == 0 and offs[-1] == len(h)
    for p, (a, b) in enumerate(pairs):
        one = gpu_records(tms.search(a, b))
        for k in one:
            if k != "pair":
                assert np.array_equal(rec[k][offs[p]:offs[p + 1]], one[k]), (p, k)
        assert (rec["pair"][offs[p]:offs[p + 1]] == p).all()
    # the first nine pairs by the sort (their raw hits make one sort tile)
    h2 = tms.search_batched(As[:9], Bs[:9], inject=16)
    assert tms.last_stats()["raw_hits"] <= 2048
    _identical({k: v[:offs[9]] for k, v in rec.items()}, gpu_records(h2))
    assert np.array_equal(offs[:10], h2.offsets.cpu().numpy())


def test_more_hits_than_the_short_merge_takes():
    """Over 32768 raw hits: the sort, which the plan finds on its first search;
    against the same mesh in column ranges of fewer hits each (the short merge)."""
    p = synth.build_pair(77, 2048, 512, 2048, 512, stretch="exp", n_folds=3, sites=(512, 128), n_hits=0)
    X, s = p.A.X.cuda().contiguous(), p.A.s
    B = tms.Mesh.from_grid(p.B)
    full = tms.Mesh(X, s)
    for _ in range(2):
        whole = gpu_records(tms.search(full, B))
        assert tms.last_stats()["raw_hits"] > 32768
    got, cuts = [], [0, 100, 200, 300, 400, 511]
    for k0, k1 in zip(cuts[:-1], cuts[1:]):
        r = gpu_records(tms.search(tms.Mesh(X, s, k0=k0, k1=k1 + 1), B))
        assert tms.last_stats()["raw_hits"] <= 32768
        r["triA"] = r["triA"] + 2 * full.N * k0
        got.append(r)
    for k in ("triA", "triB", "z", "P", "rho", "margin"):
        assert np.array_equal(np.concatenate([r[k] for r in got]), whole[k]), k


@pytest.mark.parametrize("n", [1, 15, 16, 17, 100])
def test_adjoint_at_block_edges(n):
    pair = synth.family_pair(99, 0.5, N=128, M=40, n_hits=60)
    pair2 = synth.build_pair(31, 200, 60, 190, 64, stretch="exp", n_folds=3, sites=(40, 16), n_hits=20, alpha=0.5,
                             with_dalpha=True)
    p = pair2 if n > 40 else pair
    XA, XB = p.A.X.cuda().contiguous(), p.B.X.cuda().contiguous()
    A, B = tms.Mesh(XA, p.A.s), tms.Mesh(XB, p.B.s)
    hits = tms.search(A, B)
    m = min(n, len(hits))
    hits = tms.Hits(hits.raw[:m])
    g = torch.Generator().manual_seed(n)
    gP, gZ = (torch.randn(m, 4, generator=g, dtype=torch.float64) for _ in range(2))
    gA, gB = torch.zeros_like(XA), torch.zeros_like(XB)
    ga = torch.full((m + 1,), 7.0, dtype=torch.float64, device="cuda")
    tms.backward(A, B, hits, gP=gP.cuda(), gZ=gZ.cuda(), gradA=gA, gradB=gB, dA_dalpha=p.A.dXdalpha.cuda(),
                 dB_dalpha=p.B.dXdalpha.cuda(), galpha=ga)
    assert float(ga[m]) == 7.0
    OA, OB = oracle.OMesh.from_grid(p.A), oracle.OMesh.from_grid(p.B)
    rA, rB, ra = oracle.hit_grads(OA, OB, hits.triA.cpu().numpy(), hits.triB.cpu().numpy(), gP.numpy(), gZ.numpy(),
                                  p.A.dXdalpha.numpy(), p.B.dXdalpha.numpy())
    # two backward-stable solves of one system: apart by its condition, bounded by 1 / rho
    tol = 1e-13 / max(float(hits.rho.min()), 1e-6)
    scale = max(np.abs(rA).max(), np.abs(rB).max())
    assert np.abs(gA.cpu().numpy() - rA).max() <= tol * scale
    assert np.abs(gB.cpu().numpy() - rB).max() <= tol * scale
    assert np.abs(ga[:m].cpu().numpy() - ra).max() <= tol * scale * 10
    # one side or one upstream gradient missing
    gB2 = torch.zeros_like(XB)
    tms.backward(A, B, hits, gP=gP.cuda(), gZ=gZ.cuda(), gradB=gB2)
    assert torch.allclose(gB2, gB, rtol=0, atol=1e-12 * scale)
