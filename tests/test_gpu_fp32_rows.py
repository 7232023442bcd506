"""The plain FP32 rows divide by D = 6 mu + h^2 k (a rounded reciprocal would shift every
row by the same relative error).  With networks that are 0 everywhere and the plus side's
source f = -6 mu, an interior row is r = h^2 6 mu / (6 mu): h^2 to the last bit, for a spacing that is a
power of two.  The values of mu are some for which 6 mu times its rounded reciprocal is not 1."""
import pytest
import torch

from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,L", [(10, 5), (32, 2), (64, 2), (128, 3)])
@pytest.mark.parametrize("mu", [41.0, 47.0, 53.0, 55.0])
@pytest.mark.parametrize("fp64", [0, 1])
def test_rows_of_the_zero_network(H, L, mu, fp64):
    import paper_2210_14907_gb300 as nbm
    prob = nbm.Problem(nbm.ProblemDesc(geometry=nbm.GEOM_ALL_PLUS, n_hidden=L, width=H, mu_plus=mu, h=2 / 32,
                                       precision=nbm.PREC_FP32, fp64_stencil=fp64))
    x = torch.from_numpy(0.9 * inputs.uniform_points(601, 7)).float().cuda()
    loss, r2 = prob.residual(torch.zeros(prob.P, device="cuda"), x)
    assert bool((r2 == 2.0 ** -16).all()) and loss == 2.0 ** -16
