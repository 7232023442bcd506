"""Rounding of the narrow step's gradient sums: the mean error of eight gradients of 16,384
points against the FP64 oracle.  Bound 6.4e-8: kernels that add tile by tile (8 points
at a time) err by 5.65e-8 on these inputs, with a spread of 0.7e-8 from seed to seed, so the mean of
eight is below 6.4e-8 (three standard deviations); one chain over a CTA's 48 partial sums errs by
7.3e-8."""
import numpy as np
import pytest
import torch

from oracle import pyoracle as O
from tests import inputs

pytestmark = pytest.mark.gpu


def test_gradient_sums_of_a_cta():
    import paper_2210_14907_gb300 as nbm
    kw = dict(n_hidden=5, width=10, h=2 / 32, activation=1, solution=1)
    prob = nbm.Problem(nbm.ProblemDesc(precision=nbm.PREC_FP32, **kw))
    o = O.make_problem(geometry=O.GEOM_SPHERE, mu_minus=1.0, **kw)
    off = []
    for seed in range(8):
        th, x = inputs.glorot_params(10, 5, seed=seed, bias_scale=0.1), inputs.uniform_points(16384, 100 + seed)
        ref = O.loss_grad(o, th.astype(np.float64), x)[1]
        _, g = prob.loss_grad(torch.from_numpy(th).cuda(), torch.from_numpy(x).float().cuda())
        off.append(np.linalg.norm(g.cpu().numpy() - ref) / np.linalg.norm(ref))
    assert np.mean(off) <= 6.4e-8
