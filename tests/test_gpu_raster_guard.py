"""Values that must not reach a Gaussian's record from pixels that do not blend it: a
product of a loss gradient and a colour that overflows although both are finite, and
the colour still to come in front of an infinite background.  Small and large grids
(the raster backward's lane groups of 16 and 8), one and two pixels per thread."""
import numpy as np
import pytest
import torch

from paper_2605_00219_gb300 import synth

from test_gpu_parity import LR, gs  # noqa: F401

pytestmark = pytest.mark.gpu

# (tile, threads per tile, BF16 moments)
FORMS = [((8, 8), 0, False), ((16, 16), 0, False), ((16, 16), 128, False), ((16, 16), 128, True), ((16, 16), 64, False),
         ((16, 32), 0, False), ((16, 32), 256, False), ((16, 32), 256, True), ((16, 32), 128, False)]


def _scene(n=40):
    """n Gaussians whose footprints cover the image centre and, in front of them, one
    of radius 0.29 pixels between four pixel centres, which no pixel blends."""
    rng = np.random.default_rng(1)
    sc = synth.uniform_scene(n, 1)
    sc.means = rng.normal(0, 0.01, size=(n, 3)).astype(np.float32)
    sc.scales = np.exp(rng.normal(-3.3, 0.3, size=(n, 3))).astype(np.float32)
    sc.opacities = rng.uniform(0.02, 0.1, size=n).astype(np.float32)
    sc.means[0], sc.scales[0], sc.opacities[0] = (0, 0, -0.5), 1e-4, 0.0045
    return sc


def _cam(size):
    return synth.Camera(np.eye(3, dtype=np.float32), np.array([0, 0, 4], np.float32), 150.0, 150.0, size / 2.0 + 3.0,
                        size / 2.0 + 2.0, size, size)


def _records(gsstep, tr, n):
    K = tr.stats().k_required
    off = tr.buffer(1, n + 1).cpu().numpy().view(np.uint32).astype(np.int64)
    rec = gsstep.gs_gradient_records(tr.plan, tr.ws, K).cpu().numpy()
    return [rec[off[g]:off[g + 1]] for g in range(n)]


def _trainer(step_mod, sc, size, form, bg=None):
    tile, tpt, bf16 = form
    tr = step_mod.Trainer([sc], [_cam(size)], capacity=8192, tile=tile, threads_per_tile=tpt, mom_bf16=bf16, bg=bg, lr=LR)
    tr.forward()
    return tr


@pytest.mark.parametrize("size", [32, 912])
@pytest.mark.parametrize("form", FORMS)
def test_product_that_overflows(gs, form, size):  # noqa: F811
    gsstep, step_mod = gs
    sc = _scene()
    k = 7
    sc.sh[k] = 0
    sc.sh[k, 0] = 1e20
    tr = _trainer(step_mod, sc, size, form)
    img = tr.image.view(size, size, 3)[..., 0]
    hot = (img > 1e10).cpu().numpy()          # pixels that blend the bright Gaussian
    assert hot.any() and bool(torch.isfinite(img).all())
    # the pixels of its 8x4 blocks that do not blend it
    b = hot.reshape(size // 4, 4, size // 8, 8).any((1, 3))
    cold = np.repeat(np.repeat(b, 4, 0), 8, 1) & ~hot
    assert cold.any()
    tr.dl.copy_(torch.from_numpy(np.where(cold, np.float32(1e20), np.float32(0))).cuda().reshape(-1, 1).expand(-1, 3))
    gsstep.gs_raster_bwd(tr.plan, tr.ws, tr.image, tr.dl)
    rec = _records(gsstep, tr, sc.n)
    assert all(np.isfinite(r).all() for r in rec)
    assert not rec[k].any()                   # its own pixels have no loss gradient
    assert any(r.any() for r in rec)


@pytest.mark.parametrize("size", [32, 912])
@pytest.mark.parametrize("form", FORMS)
def test_infinite_background(gs, form, size):  # noqa: F811
    gsstep, step_mod = gs
    sc = _scene()
    tr = _trainer(step_mod, sc, size, form, bg=(float("inf"), 0.0, 0.5))
    tr.dl.copy_(torch.randn(tr.dl.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2)))
    gsstep.gs_raster_bwd(tr.plan, tr.ws, tr.image, tr.dl)
    rec = _records(gsstep, tr, sc.n)
    assert len(rec[0]) and not rec[0].any()   # listed, blended by no pixel
    assert any(not np.isfinite(r).all() for r in rec[1:])
