"""Grid-solver paths that the sizes in test_gpu_grid_paths.py do not reach: FP32 corrections with variable
coefficients past the one-launch limit (general rows, three launches per iteration), coded rows
with reaction terms and with the flower, and one-launch CG over more iterations than a launch
takes (1000).  Solves to a relative residual of 1e-12 agree to 1e-9 of max |u|, as there."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _problem(**kw):
    import paper_2210_14907_gb300 as nbm
    return nbm.Problem(nbm.ProblemDesc(**{**dict(geometry=nbm.GEOM_SPHERE, r0=0.47, mu_plus=10.0), **kw}))


@pytest.mark.parametrize("n", [131, 166])
@pytest.mark.parametrize("solution", [0, 1], ids=["coded", "general"])
@pytest.mark.parametrize("geometry,k", [(1, 0.7), (2, 0.0), (2, 0.7)])
def test_refined_past_the_limit(n, solution, geometry, k):
    prob = _problem(geometry=geometry, solution=solution, k_minus=k, k_plus=2 * k)
    u, _, _, ok = prob.grid_cg_solve(n, rtol=1e-12)
    v, _, rr, ok2 = prob.grid_solve_refined(n, rtol=1e-12)
    assert ok and ok2 and rr <= 1e-12
    assert float((u - v).abs().max()) <= 1e-9 * float(u.abs().max())


def test_more_iterations_than_one_launch():
    """CG's recurrence residual goes on falling at its rate past the FP64 accuracy of x: 1e-40 takes
    about 40/12 of the iterations of 1e-12 (at 128^3 more than a launch's 1000)."""
    prob = _problem()
    u, it, _, ok = prob.grid_cg_solve(128, rtol=1e-12)
    v, it2, rr, ok2 = prob.grid_cg_solve(128, rtol=1e-40, max_iter=20000)
    assert ok and ok2 and rr <= 1e-40
    assert 1000 < it2 <= 1.25 * it * 40 / 12
    assert float((u - v).abs().max()) <= 1e-9 * float(u.abs().max())
    w, it3, _, ok3 = prob.grid_cg_solve(128, rtol=1e-40, max_iter=1003)
    assert it3 == 1003 and not ok3 and float((u - w).abs().max()) <= 1e-9 * float(u.abs().max())
