"""The refinement where B's sheet is the frame's (alpha_s = alpha_ref: its sums are taken
once) against the oracle and against the walk of B's sheet, which takes them apart, for
numbers of harmonics and folds from the smallest to the largest and numbers of seeds at
the edges of a warp's eight."""
import pytest

import synth
from oracle import refine as R
from tests.test_gpu_refine import _gpu_continue, _gpu_refine, _near_site_seeds, compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha_u", [0.5, 0.47])
@pytest.mark.parametrize("folds,stretch", [(0, "exp"), (3, "exp"), (4, "linear")])
@pytest.mark.parametrize("n", [1, 8, 9, 41])
def test_sheet_at_the_frames_parameter(n, folds, stretch, alpha_u):
    p = synth.build_pair(31 + folds, 40, 20, 36, 24, stretch=stretch, n_folds=folds, sites=(6, 2), n_hits=0,
                         alpha=0.5, with_dalpha=True)
    assert p.surface.alpha == p.surface.alpha_ref
    seeds = _near_site_seeds(p.surface, n, 1e-3, n)
    sp = R.with_alphas(p.surface, alpha_u, 0.5)
    one = _gpu_refine(sp, seeds)
    compare(one, R.damped_newton(sp, seeds), 1e-10)
    walk = _gpu_continue(sp, seeds, [], param="s", rho_turn=0.0, max_jump=1e9)
    compare({k: v[:, 0] for k, v in walk.items()}, one, 1e-10)
