"""The narrow step's results depend on its inputs alone: the same gradient call, with another
kernel in between that leaves other values in the SMs' shared memory, gives the same bits.
At widths where 32 / width points do not fill a warp, some lanes own no unit."""
import pytest
import torch

from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,L", [(5, 3), (10, 5), (11, 4), (16, 5), (20, 5)])
@pytest.mark.parametrize("act", [0, 1], ids=["tanh", "sine"])
def test_same_bits_after_another_kernel(H, L, act):
    import paper_2210_14907_gb300 as nbm
    prob = nbm.Problem(nbm.ProblemDesc(n_hidden=L, width=H, precision=nbm.PREC_FP32, mu_plus=10.0,
                                       h=2 / 32, activation=act))
    mesh = nbm.Problem(nbm.ProblemDesc(mu_plus=10.0))
    wide = nbm.Problem(nbm.ProblemDesc(n_hidden=3, width=128, precision=nbm.PREC_FP32, mu_plus=10.0, h=2 / 32))
    th = torch.from_numpy(inputs.glorot_params(H, L, seed=H, bias_scale=0.1)).cuda()
    tw = torch.from_numpy(inputs.glorot_params(128, 3, seed=3, bias_scale=0.1)).cuda()
    x = torch.from_numpy(inputs.uniform_points(16384, 5)).float().cuda()
    loss, g = prob.loss_grad(th, x)
    for between in (lambda: mesh.grid_cg_solve(128, rtol=1e-12, max_iter=20), lambda: wide.loss_grad(tw, x)):
        between()
        again, g2 = prob.loss_grad(th, x)
        assert loss == again and torch.equal(g, g2)
