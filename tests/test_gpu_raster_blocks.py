"""The raster kernels' 4x4-block walk at its edges, against the oracle: tile
lists around the staged chunk and batch lengths, images smaller than a block
and than a tile, and values that must not leave the pixels they belong to
(a lane group's pixels that do not blend still run the packed arithmetic)."""
import numpy as np
import pytest
import torch

from paper_2605_00219_gb300 import synth

from test_gpu_parity import _check_grad, _oracle_all, _run_forward, _sum_slots, _unstable_gaussians, gs  # noqa: F401

pytestmark = pytest.mark.gpu


def _pile(n, seed, w, h):
    """n Gaussians whose footprints all cross the image centre, faint enough
    that pixels blend most of them."""
    rng = np.random.default_rng(seed)
    sc = synth.uniform_scene(n, seed)
    sc.means = (rng.normal(0, 0.01, size=(n, 3))).astype(np.float32)
    sc.scales = np.exp(rng.normal(-3.3, 0.6, size=(n, 3))).astype(np.float32)
    sc.opacities = rng.uniform(0.01, 0.08, size=n).astype(np.float32)
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.array([0, 0, 4], np.float32), 150.0, 140.0, w / 2.0, h / 2.0,
                       w, h)
    return sc, cam


@pytest.mark.parametrize("tile", [(8, 8), (16, 16), (16, 32)])
@pytest.mark.parametrize("n,w,h", [(1, 16, 16), (31, 3, 5), (32, 16, 16), (63, 16, 32), (64, 16, 16), (65, 17, 9),
                                   (96, 16, 16), (97, 16, 16), (127, 16, 16), (128, 33, 7), (129, 16, 16),
                                   (257, 18, 21), (700, 16, 16)])
def test_list_lengths_and_ragged_images(gs, orc, tile, n, w, h):  # noqa: F811
    gsstep, step_mod = gs
    scene, cam = _pile(n, n, w, h)
    b, p, P, r = _oracle_all(orc, scene, cam, tile)
    tr = _run_forward(step_mod, scene, [cam], tile=tile, capacity=64 * n + 4096)
    assert tr.stats().status == 0 and tr.stats().k_required == b.K
    img = tr.image.view(h, w, 3).cpu().numpy().astype(np.float64)
    ok = ~r.unstable_px
    assert np.abs(img - r.image)[ok].max() <= 1e-5
    np.testing.assert_array_equal(tr.buffer(5, w * h).cpu().numpy().reshape(h, w)[ok], r.nlast[ok])
    dl64 = np.random.default_rng(n).normal(size=(h, w, 3)).astype(np.float32).astype(np.float64) / (3 * w * h)
    tr.dl.copy_(torch.from_numpy(dl64.astype(np.float32).reshape(-1, 3)))
    gsstep.gs_raster_bwd(tr.plan, tr.ws, tr.image, tr.dl)
    g2 = orc.raster_bwd64(cam, P, b, dl64, (0, 0, 0), *tile)
    good = (b.count > 0) & ~_unstable_gaussians(P, r, cam)
    off = tr.buffer(1, n + 1).cpu().numpy().view(np.uint32).astype(np.int64)
    gr = gsstep.gs_gradient_records(tr.plan, tr.ws, b.K).cpu().numpy()
    got = _sum_slots(gr, off, tr.buffer(0, n).cpu().numpy().view(np.uint32))
    if good.any():
        _check_grad(got, g2, good, f"grad2d {tile} n={n} {w}x{h}")
    assert np.isfinite(got).all()


@pytest.mark.parametrize("tile", [(8, 8), (16, 16), (16, 32)])
def test_non_finite_values_stay_where_they_belong(gs, orc, tile):  # noqa: F811
    """An infinite colour reaches only the pixels its Gaussian blends, and a
    non-finite loss gradient only the Gaussians its pixel blends."""
    gsstep, step_mod = gs
    scene, _, cams = synth.tiny_workload(5)
    cam = cams[0]
    b, p, P, r = _oracle_all(orc, scene, cam, tile)
    k = int(np.argmax(np.where(np.abs(P[:, 4] - 60) + np.abs(P[:, 5] - 60) < 40, b.count, 0)))
    ys, xs = np.mgrid[0:128, 0:128]
    def d2(q):
        dx, dy = xs + 0.5 - q[4], ys + 0.5 - q[5]
        return q[9] * dx * dx + 2 * q[10] * dx * dy + q[11] * dy * dy
    reach = d2(P[k]) <= 9.0 * (1 + 1e-3)
    hot = scene.copy()
    hot.sh[k, 0, 0] = np.inf
    img = _run_forward(step_mod, hot, cams, tile=tile).image.view(128, 128, 3).cpu().numpy()
    bad = ~np.isfinite(img).all(-1)
    assert bad.any() and not (bad & ~reach).any()
    # loss gradient: one pixel of infinity, one of NaN
    tr = _run_forward(step_mod, scene, cams, tile=tile)
    dl = torch.full((128 * 128, 3), 1e-5, device="cuda")
    pix = [(61, 58, float("inf")), (37, 90, float("nan"))]
    for y, x, val in pix:
        dl[y * 128 + x] = val
    gsstep.gs_raster_bwd(tr.plan, tr.ws, tr.image, dl)
    off = tr.buffer(1, scene.n + 1).cpu().numpy().view(np.uint32).astype(np.int64)
    gr = gsstep.gs_gradient_records(tr.plan, tr.ws, b.K).cpu().numpy()
    near = np.zeros(scene.n, bool)
    for y, x, _ in pix:
        dx, dy = x + 0.5 - P[:, 4], y + 0.5 - P[:, 5]
        near |= P[:, 9] * dx * dx + 2 * P[:, 10] * dx * dy + P[:, 11] * dy * dy <= 9.0 * (1 + 1e-3)
    got = _sum_slots(gr, off, tr.buffer(0, scene.n).cpu().numpy().view(np.uint32))
    nonfinite = ~np.isfinite(got).all(1)
    assert nonfinite.any() and not (nonfinite & ~near).any()
