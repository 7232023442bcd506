"""The FP32 step kernel at the edges of its 16-point tiles, against the FP64 oracle.

Every instance (width, depth) at batch sizes around one tile, and one size whose
tiles exceed the CTAs, so that a CTA accumulates several tiles' weight gradients and
changes network.  Tolerances are those of the FP32 path (loss 1e-5, gradient 1e-4).
"""
import numpy as np
import pytest
import torch

from oracle import pyoracle as O
from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,L", [(64, 2), (64, 3), (64, 4), (128, 2), (128, 3), (128, 4)])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 6001])
def test_fp32_step_tile_edges(H, L, n):
    import paper_2210_14907_gb300 as nbm
    kw = dict(geometry=O.GEOM_FLOWER, n_hidden=L, width=H, mu_minus=1.0, mu_plus=10.0, h=2 / 32)
    prob = nbm.Problem(nbm.ProblemDesc(precision=nbm.PREC_FP32, **kw))
    o = O.make_problem(**kw)
    pts = inputs.mixed_points(n, n // 3 + 2, seed=H + L + n)[-n:]
    th = inputs.glorot_params(H, L, seed=n, bias_scale=0.1)
    L_ref, g_ref = O.loss_grad(o, th.astype(np.float64), pts)
    tp, tx = torch.from_numpy(th).cuda(), torch.from_numpy(pts.astype(np.float32)).cuda()
    loss, g = prob.loss_grad(tp, tx)
    again, g2 = prob.loss_grad(tp, tx)
    assert abs(loss - L_ref) <= 1e-5 * L_ref
    assert np.linalg.norm(g.cpu().numpy() - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
    assert loss == again and torch.equal(g, g2)  # the tiles add up in a fixed order
