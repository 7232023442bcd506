"""Gradient sums of tiny terms in the plain FP32 step: output weights of about 1e-32 make the
hidden weights' gradient about 1e-35, and its parts from the tiles, down to subnormal ones, are
below what a reduction in memory adds exactly.  A tile's parts and their sum are good to 2^-149 each
(1250 tiles at most: 1e-6 of 1e-36), and the FP32 path's gradient tolerance is 1e-4."""
import numpy as np
import pytest
import torch

from oracle import pyoracle as O
from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,L", [(64, 2), (64, 4), (128, 2), (128, 3), (128, 4)])
def test_weight_gradient_of_subnormal_terms(H, L):
    import paper_2210_14907_gb300 as nbm
    kw = dict(geometry=O.GEOM_SPHERE, n_hidden=L, width=H, mu_minus=1.0, mu_plus=10.0, h=2 / 32)
    prob = nbm.Problem(nbm.ProblemDesc(precision=nbm.PREC_FP32, **kw))
    o = O.make_problem(**kw)
    pts = inputs.uniform_points(20001, 3)
    th, g0 = inputs.glorot_params(H, L, seed=2, bias_scale=0.1), 4 * H
    P, hid = th.size // 2, (L - 1) * (H * H + H)
    for s in (0, P):
        th[s + g0 + hid:s + P] *= 1e-32
    ref = O.loss_grad(o, th.astype(np.float64), pts)[1]
    g = prob.loss_grad(torch.from_numpy(th).cuda(), torch.from_numpy(pts).float().cuda())[1].cpu().numpy()
    for s in (0, P):
        a, b = (v[s + g0:s + g0 + hid].astype(np.float64) for v in (g, ref))
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
