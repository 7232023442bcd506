"""The grid solvers' paths against one another: rows decided by FP32 level-set values
against the full FP64 rows, and CG in one launch (up to 130 cells per axis) against three
launches per iteration (refined: with coded rows), at sizes on both sides of the limit.  Solves to a
relative residual of 1e-12 agree to 1e-9 of max |u| (condition number about n^2 <= 3e4)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _solve(n, refined=False, **kw):
    import paper_2210_14907_gb300 as nbm
    prob = nbm.Problem(nbm.ProblemDesc(**{**dict(geometry=nbm.GEOM_SPHERE, r0=0.47, mu_plus=10.0), **kw}))
    u, it, rr, ok = (prob.grid_solve_refined if refined else prob.grid_cg_solve)(n, rtol=1e-12)
    assert ok and rr <= 1e-12
    return u, it


@pytest.mark.parametrize("n", [3, 24, 57, 130, 131, 164, 165])
def test_fp64_and_refined_solves_agree(n):
    u, it = _solve(n)
    v, _ = _solve(n, refined=True)
    assert it > 0 and float((u - v).abs().max()) <= 1e-9 * float(u.abs().max())


@pytest.mark.parametrize("n", [20, 61])
@pytest.mark.parametrize("k", [0.0, 0.7])
@pytest.mark.parametrize("solution", [0, 1])
def test_rows_by_fp32_signs_match_full_rows(n, k, solution):
    # a lobe count that is not an integer takes the full rows; 1e-13 off is the same flower
    kw = dict(geometry=2, n_hidden=3, k_minus=k, k_plus=2 * k, solution=solution, grid_jump=2)
    u, it = _solve(n, lobes_theta=5.0, **kw)
    v, it2 = _solve(n, lobes_theta=5.0 + 1e-13, **kw)
    assert it == it2 and float((u - v).abs().max()) <= 1e-9 * float(u.abs().max())


def test_iteration_limit_and_counts():
    import paper_2210_14907_gb300 as nbm
    prob = nbm.Problem(nbm.ProblemDesc(mu_plus=10.0))
    for limit in (1, 7, 25):
        _, it, _, ok = prob.grid_cg_solve(64, rtol=1e-12, max_iter=limit)
        assert it == limit and not ok
    _, it, _, ok = prob.grid_cg_solve(64, rtol=1e-12)
    assert ok and it % 10 == 0  # looked at every ten iterations


def test_solves_on_two_threads_and_streams():
    """Each thread its own problem and stream: the one-launch solves take turns on the GPU."""
    import concurrent.futures as cf

    import paper_2210_14907_gb300 as nbm
    ref, _ = _solve(40)

    def work(_):
        with torch.cuda.stream(torch.cuda.Stream()):
            prob = nbm.Problem(nbm.ProblemDesc(geometry=nbm.GEOM_SPHERE, r0=0.47, mu_plus=10.0))
            return [prob.grid_cg_solve(40, rtol=1e-12) for _ in range(5)]

    with cf.ThreadPoolExecutor(2) as ex:
        for runs in ex.map(work, range(2)):
            assert all(ok and torch.equal(u, ref) for u, _, _, ok in runs)
