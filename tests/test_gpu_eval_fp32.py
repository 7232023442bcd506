"""FP32 evaluation at the edges of its tiles (32 and 128 points) and of its 1024-point
chunks, against a plain FP64 torch evaluation of each point's network.  Tolerance: the
FP32 evaluation's 1e-5 (norm-wise relative)."""
import numpy as np
import pytest
import torch

from tests import inputs

pytestmark = pytest.mark.gpu


def _reference(th, H, L, x, minus):
    out = torch.empty(x.shape[0], dtype=torch.float64, device=x.device)
    for s, sel in ((0, minus), (1, ~minus)):
        p, a, at = th[s * (th.numel() // 2):], x[sel], 0
        for i in [3] + [H] * (L - 1):
            W, b = p[at:at + i * H].view(H, i), p[at + i * H:at + i * H + H]
            a, at = torch.tanh(a @ W.t() + b), at + i * H + H
        out[sel] = a @ p[at:at + H] + p[at + H]
    return out


@pytest.mark.parametrize("H,L", [(64, 2), (64, 4), (128, 2), (128, 3), (128, 4)])
@pytest.mark.parametrize("geometry", ["sphere", "all_minus", "all_plus"])
@pytest.mark.parametrize("n", [1, 31, 33, 9859, 19600, 41003])
def test_eval_points_fp32_tiles(H, L, geometry, n):
    import paper_2210_14907_gb300 as nbm
    geo = {"sphere": nbm.GEOM_SPHERE, "all_minus": nbm.GEOM_ALL_MINUS, "all_plus": nbm.GEOM_ALL_PLUS}
    prob = nbm.Problem(nbm.ProblemDesc(geometry=geo[geometry], n_hidden=L, width=H))
    pts = np.concatenate([inputs.uniform_points(n, 3), inputs.shell_points(n // 2, 4)])[-n:]
    x = torch.from_numpy(pts).cuda()
    th = torch.from_numpy(inputs.glorot_params(H, L, seed=n, bias_scale=0.2)).cuda()
    got = prob.eval_points(th, x.float().contiguous(), precision=nbm.PREC_FP32)
    minus = x.norm(dim=1) <= 0.5 if geometry == "sphere" else torch.full_like(x[:, 0], geometry == "all_minus").bool()
    ref = _reference(th.double(), H, L, x, minus)
    assert float((got.double() - ref).norm() / ref.norm()) <= 1e-5
    assert float((got.double() - ref).abs().max()) <= 1e-4  # every point (a wrong side or slot is O(1))
