"""The narrow FP32 step kernel (width <= 32) over its widths, depths and warp tiles, against
the FP64 oracle: a warp takes min(4, 32 / width) points, so batches around that number
and one that gives the warps several tiles.  Tolerances of the FP32 path (loss 1e-5,
gradient 1e-4), as the convergence-study tests take them."""
import numpy as np
import pytest
import torch

from oracle import pyoracle as O
from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,L", [(1, 2), (5, 3), (8, 5), (10, 5), (11, 4), (16, 5), (17, 2), (32, 5)])
@pytest.mark.parametrize("act", [0, 1], ids=["tanh", "sine"])
@pytest.mark.parametrize("n,h", [(1, 2 / 32), (5, 2 / 8), (301, 2 / 64), (9001, 2 / 32)])
def test_narrow_step(H, L, act, n, h):
    import paper_2210_14907_gb300 as nbm
    kw = dict(geometry=O.GEOM_SPHERE, n_hidden=L, width=H, mu_minus=1.0, mu_plus=10.0, h=h, activation=act)
    prob = nbm.Problem(nbm.ProblemDesc(precision=nbm.PREC_FP32, **kw))
    o = O.make_problem(**kw)
    pts = inputs.mixed_points(n, n // 3 + 2, seed=H + L + n)[-n:]
    th = inputs.glorot_params(H, L, seed=n, bias_scale=0.1)
    L_ref, g_ref = O.loss_grad(o, th.astype(np.float64), pts)
    tp, tx = torch.from_numpy(th).cuda(), torch.from_numpy(pts.astype(np.float32)).cuda()
    loss, g = prob.loss_grad(tp, tx)
    again, g2 = prob.loss_grad(tp, tx)
    loss3, r2 = prob.residual(tp, tx)
    assert abs(loss - L_ref) <= 1e-5 * L_ref and abs(loss3 - L_ref) <= 1e-5 * L_ref
    assert np.linalg.norm(g.cpu().numpy() - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
    assert loss == again and torch.equal(g, g2)
