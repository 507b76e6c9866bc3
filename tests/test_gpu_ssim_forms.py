"""The two forms of the L1 + SSIM kernel, 32x31 tiles with BF16 moments and pairs of
16x16 tiles with FP32 moments, at the edges of both tilings, against the FP64 oracle at
the tolerances of test_gpu_ssim."""
import numpy as np
import pytest
import torch

from paper_2605_00219_gb300 import synth

from test_gpu_ssim import _flat, _grad_err, _split, gs  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(15, 15), (16, 16), (17, 17), (31, 31), (32, 32), (33, 33), (48, 16), (49, 47), (1, 1), (64, 1), (3, 70)]


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("bf16_moments", [False, True])
def test_forms_match_oracle(gs, orc, masked, bf16_moments):  # noqa: F811
    gsstep, _ = gs
    imgs, tgts = synth.loss_images(SHAPES, seed=11)
    plan = gsstep.Plan([16], [(w, h, 0) for w, h in SHAPES],
                       storage_flags=gsstep.STORE_MOMENTS_BF16 if bf16_moments else 0)
    ws = torch.empty(plan.workspace_bytes(), dtype=torch.uint8, device="cuda")
    gsstep.gs_workspace_init(plan, ws)
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
