"""The raster backward at two pixels per thread with FP32 moments (8x8 blocks, a lane's
pixels four rows apart) against the oracle: lists around the staged batch, more visits
than slots, ragged images and tiles, alphas at the 0.99 clamp, and non-finite loss
gradients, which stay with the Gaussians their pixels blend."""
import numpy as np
import pytest
import torch

from test_gpu_parity import _check_grad, _oracle_all, _run_forward, _sum_slots, _unstable_gaussians, gs  # noqa: F401
from test_gpu_raster_blocks import _pile

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [(16, 16), (16, 32)])
@pytest.mark.parametrize("n,w,h,opaque", [(1, 16, 16, 0), (63, 5, 3, 1), (64, 16, 16, 0), (65, 17, 9, 0), (128, 33, 40, 3),
                                          (257, 18, 21, 0), (700, 16, 32, 5)])
def test_matches_oracle(gs, orc, tile, n, w, h, opaque):  # noqa: F811
    gsstep, step_mod = gs
    scene, cam = _pile(n, n, w, h)
    scene.opacities[:opaque] = 0.999
    b, p, P, r = _oracle_all(orc, scene, cam, tile)
    out = []
    for bad in (False, True):
        tr = _run_forward(step_mod, scene, [cam], tile=tile, capacity=64 * n + 4096,
                          tpt=tile[0] * tile[1] // 2)
        dl64 = np.random.default_rng(n).normal(size=(h, w, 3)).astype(np.float32).astype(np.float64) / (3 * w * h)
        dl = torch.from_numpy(dl64.astype(np.float32).reshape(-1, 3)).cuda()
        if bad:
            dl[0] = float("nan")
        tr.dl.copy_(dl)
        gsstep.gs_raster_bwd(tr.plan, tr.ws, tr.image, tr.dl)
        off = tr.buffer(1, n + 1).cpu().numpy().view(np.uint32).astype(np.int64)
        gr = gsstep.gs_gradient_records(tr.plan, tr.ws, b.K).cpu().numpy()
        out.append(_sum_slots(gr, off, tr.buffer(0, n).cpu().numpy().view(np.uint32)))
    g2 = orc.raster_bwd64(cam, P, b, dl64, (0, 0, 0), *tile)
    good = (b.count > 0) & ~_unstable_gaussians(P, r, cam)
    if good.any():
        _check_grad(out[0], g2, good, f"grad2d {tile} n={n} {w}x{h}")
    assert np.isfinite(out[0]).all()
    # the first pixel's gradient reaches only Gaussians within 3 sigma of it
    dx, dy = 0.5 - P[:, 4], 0.5 - P[:, 5]
    near = P[:, 9] * dx * dx + 2 * P[:, 10] * dx * dy + P[:, 11] * dy * dy <= 9.0 * (1 + 1e-3)
    assert not (~np.isfinite(out[1]).all(1) & ~near).any()
