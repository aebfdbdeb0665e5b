"""The autotuner times no setting twice: at the patch level, which has no grid, one cell
multiplier, and tiles of 8 rows only where they do not run in the place of 4."""
import pytest

import paper_2109_14814_gb300 as tms
import synth

pytestmark = pytest.mark.gpu


def _meshes(n, m, pairs):
    out = []
    for i in range(pairs):
        p = synth.build_pair(60 + i, n, m + 8 * i, n, m, stretch="exp", n_folds=3, sites=(8, 4), n_hits=0)
        out.append((tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)))
    return [a for a, _ in out], [b for _, b in out]


@pytest.mark.parametrize("size", [(96, 40), (2048, 256)])
@pytest.mark.parametrize("pairs", [1, 3])
def test_one_multiplier_at_the_patch_level(size, pairs, tmp_path):
    As, Bs = _meshes(*size, pairs)
    cache = tmp_path / "tune.txt"
    best, _ = tms.autotune(As, Bs, cache_path=str(cache))
    assert best["patch"] == 1                       # (the faster at these sizes)
    assert abs(best["cell_mult"] - 1.0625) < 1e-6
    if size[0] == 2048:
        assert best["tile_rows"] == 4
    lines = cache.read_text().splitlines()
    assert all(float(l.split()[-1]) == 1.0625 for l in lines if l.startswith("C|"))


def test_a_known_class_keeps_its_line(tmp_path):
    As, Bs = _meshes(96, 40, 3)
    cache = tmp_path / "tune.txt"
    tms.autotune(As, Bs, cache_path=str(cache))
    classes = [l for l in cache.read_text().splitlines() if l.startswith("C|")]
    cache.write_text("".join(l.rsplit(" ", 1)[0] + " 2.5\n" for l in classes))
    best, _ = tms.autotune(As, Bs, cache_path=str(cache))
    if best["patch"] == 1:
        lines = [l for l in cache.read_text().splitlines() if l.startswith("C|")]
        assert lines and all(l.endswith(" 2.5") for l in lines) and len(lines) == len(classes)
