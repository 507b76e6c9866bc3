"""The L1 + SSIM kernel at the edges of 32x31 and 16x16 tiles and their 10-pixel
halos, against the FP64 oracle, at the tolerances of test_gpu_ssim: views one
pixel below, at and above a tile and a tile plus its halo, several views in one
launch, masked and not; and a non-finite pixel, which reaches the gradients of
the pixels that share a window with it and no others."""
import numpy as np
import pytest
import torch

from paper_2605_00219_gb300 import synth

from test_gpu_ssim import _flat, _grad_err, _plan, _split, gs  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(31, 30), (32, 31), (33, 32), (64, 62), (65, 63), (41, 93), (42, 94), (5, 40), (11, 11), (75, 3)]


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("smooth", [False, True])
def test_tile_edges_match_oracle(gs, orc, masked, smooth):  # noqa: F811
    gsstep, _ = gs
    imgs, tgts = synth.loss_images(SHAPES, seed=5 + smooth, smooth=smooth)
    plan, ws = _plan(gsstep, SHAPES)
    img_d, tgt_d = _flat(imgs, 3), _flat(tgts, 4)
    dl = torch.full_like(img_d, float("nan"))
    (gsstep.gs_loss_l1_ssim_masked if masked else gsstep.gs_loss_l1_ssim)(plan, ws, img_d, tgt_d, 0.2, dl)
    loss = gsstep.gs_read_stats(plan, ws).loss
    masks = [orc.rgba8_alpha(t) if masked else np.ones(t.shape[:2]) for t in tgts]
    ref_loss, ref_g = orc.l1_ssim_loss_grad(imgs, [orc.rgba8_to_float(t) for t in tgts], 0.2,
                                            masks=masks if masked else None)
    assert abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)
    for got, ref, img, t, m in zip(_split(dl.cpu().numpy(), SHAPES), ref_g, imgs, tgts, masks):
        tie = np.abs(m[..., None] * (img.astype(np.float64) - orc.rgba8_to_float(t))) < 1e-6
        assert _grad_err(got, ref, tie).max() <= 1e-3


@pytest.mark.parametrize("y,x", [(15, 16), (46, 48), (0, 0), (30, 31), (69, 89)])
def test_non_finite_pixel_stays_in_its_windows(gs, y, x):  # noqa: F811
    gsstep, _ = gs
    w, h = 90, 70
    imgs, tgts = synth.loss_images([(w, h)], seed=3)
    plan, ws = _plan(gsstep, [(w, h)])
    out = []
    for bad in (False, True):
        img = imgs[0].copy()
        if bad:
            img[y, x, 1] = np.nan
        dl = torch.empty((w * h, 3), device="cuda")
        gsstep.gs_loss_l1_ssim(plan, ws, _flat([img], 3), _flat(tgts, 4), 0.2, dl)
        out.append(dl.view(h, w, 3).cpu().numpy())
    yy, xx = np.mgrid[0:h, 0:w]
    near = (np.abs(yy - y) <= 10) & (np.abs(xx - x) <= 10)      # windows of windows
    assert np.isnan(out[1][..., 1][near]).all()
    assert np.isfinite(out[1][..., 1][~near]).all()
    # the other channels, and the pixels out of reach, are as before (a shift of
    # the moments moves rounding only)
    np.testing.assert_array_equal(out[1][..., [0, 2]], out[0][..., [0, 2]])
    rms = np.sqrt((out[0] ** 2).mean())
    assert np.abs(out[1][..., 1] - out[0][..., 1])[~near].max() <= 1e-4 * rms
