"""The LF weights of many uneven views in one launch per step against the oracle:
images smaller than, equal to and just beyond a Sobel tile (32 x 32), flat images
(every magnitude equal: one key in every digit), and percentiles at the ends."""
import numpy as np
import pytest
import torch

from paper_2511_02510_gb300 import litevoxel as L

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 3), (31, 33), (32, 32), (33, 31), (65, 64), (400, 7), (5, 300), (257, 129)]


def _params(ppm):
    p = L.lv_lf_params()
    p.eps, p.gamma_max, p.t0, p.t1, p.pctl_ppm = 1e-3, 0.6, 300.0, 600.0, ppm
    return p


@pytest.mark.parametrize("ppm", [0, 500000, 990000, 1000000])
@pytest.mark.parametrize("flat", [False, True])
def test_uneven_views_match_the_oracle(ora, ppm, flat):
    rng = np.random.default_rng(ppm + flat)
    W, H = [w for w, _ in SIZES], [h for _, h in SIZES]
    gts = [np.full((w * h, 3), 0.25, np.float32) if flat else rng.uniform(0, 1, (w * h, 3)).astype(np.float32)
           for w, h in SIZES]
    rgbs = [np.clip(g + 0.1 * rng.standard_normal(g.shape), 0, 1).astype(np.float32) for g in gts]
    gt, rgb = (torch.as_tensor(np.concatenate(x), device="cuda") for x in (gts, rgbs))
    ws = torch.empty(L.lv_lf_workspace_size(W, H), dtype=torch.uint8, device="cuda")
    loss, grad = torch.empty(len(W), device="cuda"), torch.empty_like(rgb)
    L.lv_lf_weighted_loss(rgb, gt, W, H, 450.0, _params(ppm), loss, grad, ws)
    ref = ora.lf_loss(np.concatenate(rgbs), np.concatenate(gts), SIZES, gamma=ora.lf_gamma(450.0, 300.0, 600.0, 0.6),
                      eps=1e-3, pctl_ppm=ppm)
    # a magnitude is within about 8 roundings of its sums (at most 4), so s is within 2e-6 / P, and close
    # to s = 1 a weight moves by gamma (1e-3)^(gamma - 1) = 38 times that, P about 0.7 here
    np.testing.assert_allclose(loss.cpu().numpy(), ref["loss"], rtol=2e-4)
    assert np.abs(grad.cpu().numpy() - ref["dL_drgb"]).max() <= 2e-4 * np.abs(ref["dL_drgb"]).max()
