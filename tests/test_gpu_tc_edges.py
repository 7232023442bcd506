"""The tensor-core forward and evaluation kernels at the edges of their tiles: 8 points
to a forward tile (its work items and 48-row groups, with all kinds of points mixed),
64 and 128 points to an evaluation tile, and evaluation batches that grow, shrink and
grow again, from one thread or two.  Tolerances: the per-point bound of the mixed path
(tests/parity.py) and its 2e-3 norm-wise from 1000 points on; evaluation against FP32
evaluation, 2e-3 (FP16) and 1e-2 (BF16) of the root mean square norm-wise, five times
that at each point."""
import numpy as np
import pytest
import torch

from oracle import pyoracle as O
from tests import inputs, parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,h,fp64", [(2, 2 / 64, 0), (3, 2 / 128, 0), (4, 2 / 64, 0),
                                      (2, 2 / 128, 1), (3, 2 / 64, 1), (4, 2 / 1024, 1)])
@pytest.mark.parametrize("geometry", [O.GEOM_SPHERE, O.GEOM_FLOWER])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 47, 48, 49, 385, 2431])
def test_forward_kernel_tiles(L, h, fp64, geometry, n):
    import paper_2210_14907_gb300 as nbm
    prob = nbm.Problem(nbm.ProblemDesc(geometry=geometry, n_hidden=L, width=128, mu_minus=1.0,
                                       mu_plus=10.0, h=h, precision=nbm.PREC_BF16,
                                       fp64_stencil=fp64))
    o = O.make_problem(geometry=geometry, n_hidden=L, width=128, mu_minus=1.0, mu_plus=10.0, h=h)
    pts = inputs.mixed_points(n, n, seed=n + L)
    pts = pts[np.random.default_rng(n).permutation(len(pts))[:n]]  # kinds mixed in each tile
    th = inputs.glorot_params(128, L, seed=n, bias_scale=0.1)
    L_ref, r2_ref = O.loss(o, th.astype(np.float64), pts, want_r2=True)
    loss, r2 = prob.residual(torch.from_numpy(th).cuda(), torch.from_numpy(pts.astype(np.float32)).cuda())
    got = r2.cpu().numpy()
    assert got.shape == (n,) and abs(loss - got.astype(np.float64).mean()) <= 1e-5 * loss
    parity.check_points(o, th, pts, got, r2_ref, *parity.bf16_tols(L), label=f"L{L} n{n}")
    if n >= 1000:
        e = np.linalg.norm(np.sqrt(got) - np.sqrt(r2_ref)) / np.linalg.norm(np.sqrt(r2_ref))
        assert e <= 2e-3


@pytest.mark.parametrize("L", [2, 3, 4])
@pytest.mark.parametrize("prec,tol", [(2, 2e-3), (1, 1e-2)], ids=["fp16", "bf16"])
@pytest.mark.parametrize("geometry", ["GEOM_SPHERE", "GEOM_ALL_MINUS"])
def test_eval_tiles_and_batches_that_grow_and_shrink(L, prec, tol, geometry):
    import paper_2210_14907_gb300 as nbm
    prob = nbm.Problem(nbm.ProblemDesc(geometry=getattr(nbm, geometry), n_hidden=L, width=128))
    pts = np.concatenate([inputs.uniform_points(90000, 3), inputs.shell_points(30000, 4)])
    x = torch.from_numpy(pts[np.random.default_rng(L).permutation(len(pts))].astype(np.float32)).cuda()
    th = torch.from_numpy(inputs.glorot_params(128, L, seed=L, bias_scale=0.2)).cuda()
    ref = prob.eval_points(th, x, precision=nbm.PREC_FP32).double()
    rms = float(ref.pow(2).mean().sqrt())
    for n in (1, 63, 64, 65, 120000, 1, 127, 129, 383, 385, 19457, 64, 120000, 31):
        got = prob.eval_points(th, x[:n].contiguous(), precision=prec).double()
        d = (got - ref[:n]).abs()
        assert got.shape[0] == n and float(d.max()) <= 5 * tol * rms, n
        if n >= 1000:
            assert float(d.pow(2).mean().sqrt()) <= tol * rms, n


def test_eval_from_two_threads_on_one_problem():
    import threading
    import paper_2210_14907_gb300 as nbm
    prob = nbm.Problem(nbm.ProblemDesc(geometry=nbm.GEOM_SPHERE, n_hidden=3, width=128))
    xs = [torch.from_numpy(inputs.uniform_points(n, n).astype(np.float32)).cuda() for n in (3001, 70000)]
    ths = [torch.from_numpy(inputs.glorot_params(128, 3, seed=s, bias_scale=0.2)).cuda() for s in (1, 2)]
    want = [prob.eval_points(t, x, precision=nbm.PREC_FP16).clone() for t, x in zip(ths, xs)]
    bad = []

    def run(t, x, w):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(40):
                if not torch.equal(prob.eval_points(t, x, precision=nbm.PREC_FP16), w):
                    bad.append(1)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=run, args=a) for a in zip(ths, xs, want)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not bad
