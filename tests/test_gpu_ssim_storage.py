"""The L1 + SSIM loss and its gradient depend on the images alone: a plan that stores
its Adam moments as BF16 gets the bits of one that stores them as FP32, on hard edges
(periods that meet the kernel's tiles and ones that do not), ramps, flat images and
noise, masked and not."""
import numpy as np
import pytest
import torch

from test_gpu_ssim import _flat, gs  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(200, 150), (97, 70), (64, 62), (33, 31), (16, 16), (5, 40), (1, 1)]


def _image(kind, w, h, rng):
    y, x = np.mgrid[0:h, 0:w]
    if kind.startswith("edges"):
        p = int(kind[5:])
        a = ((x // p + y // p) % 2).astype(np.float64)
    else:
        a = {"ramp": (x + 2.0 * y) / (w + 2.0 * h), "flat": np.full((h, w), 0.4), "noise": rng.random((h, w))}[kind]
    return np.clip(a[..., None] * [1.0, 0.7, 0.4] + 0.02 * rng.normal(size=(h, w, 3)), 0, 1)


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("kind", ["edges48", "edges16", "edges31", "ramp", "flat", "noise"])
def test_same_bits_for_both_storage_types(gs, kind, masked):  # noqa: F811
    gsstep, _ = gs
    rng = np.random.default_rng(3)
    imgs = [_image(kind, w, h, rng).astype(np.float32) for w, h in SHAPES]
    tgts = [np.concatenate([np.rint(255 * _image(kind, w, h, rng)), rng.integers(0, 256, (h, w, 1))], -1).astype(np.uint8)
            for w, h in SHAPES]
    img_d, tgt_d = _flat(imgs, 3), _flat(tgts, 4)
    out = []
    for flags in (0, gsstep.STORE_MOMENTS_BF16, gsstep.STORE_MOMENTS_BF16 | gsstep.STORE_SH_BF16):
        plan = gsstep.Plan([16], [(w, h, 0) for w, h in SHAPES], storage_flags=flags)
        ws = torch.empty(plan.workspace_bytes(), dtype=torch.uint8, device="cuda")
        gsstep.gs_workspace_init(plan, ws)
        dl = torch.full_like(img_d, float("nan"))
        (gsstep.gs_loss_l1_ssim_masked if masked else gsstep.gs_loss_l1_ssim)(plan, ws, img_d, tgt_d, 0.2, dl)
        out.append((dl.cpu().numpy(), gsstep.gs_read_stats(plan, ws).loss))
    assert np.isfinite(out[0][0]).all()
    for dl, loss in out[1:]:
        np.testing.assert_array_equal(dl, out[0][0])
        assert loss == out[0][1]
