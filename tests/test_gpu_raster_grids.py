"""The raster backward's kernels for 16-wide tiles, chosen by the grid: one tile's records
are the same bits in a grid of one tile (long lists: a warp per block), of a few (lane
groups of 16, or a warp per block) and of thousands (groups of 8, or 8x8 blocks), for
lists around the staged batches, more visits than slots, alphas at the 0.99 clamp and a
non-finite loss gradient; and the records of the large grid match the oracle."""
import numpy as np
import pytest
import torch

from paper_2605_00219_gb300 import synth

from test_gpu_parity import _check_grad, _oracle_all, _run_forward, _sum_slots, _unstable_gaussians, gs  # noqa: F401

pytestmark = pytest.mark.gpu


def _pile(n, opaque):
    """n faint Gaussians over the first tile, one to a depth, the last `opaque` of them
    at the 0.99 clamp."""
    rng = np.random.default_rng(n)
    sc = synth.uniform_scene(n, n)
    sc.means = rng.normal(0, 0.01, size=(n, 3)).astype(np.float32)
    sc.means[:, 2] = 1e-4 * rng.permutation(n)
    sc.scales = np.exp(rng.normal(-3.6, 0.5, size=(n, 3))).astype(np.float32)
    sc.opacities = rng.uniform(0.006, min(0.08, 30.0 / n + 0.007), size=n).astype(np.float32)
    sc.opacities[np.argsort(sc.means[:, 2])[n - opaque:]] = 0.999
    return sc


def _cam(w, h):
    return synth.Camera(np.eye(3, dtype=np.float32), np.array([0, 0, 4], np.float32), 150.0, 140.0, 8.3, 8.1, w, h)


def _dl(w, h, seed, tile, bad):
    """Loss gradient of a w x h image, the same numbers in the first tile for any size."""
    d = np.random.default_rng(seed).normal(size=(max(h, 32), 16, 3)).astype(np.float32) / 768
    out = np.zeros((h, w, 3), np.float32)
    out[:min(h, tile[1]), :16] = d[:min(h, tile[1])]
    if bad:
        out[5, 9] = np.nan
    return out


# (tile, threads per tile, BF16 moments)
FORMS = [((16, 16), 0, False), ((16, 16), 128, False), ((16, 16), 128, True),
         ((16, 32), 0, False), ((16, 32), 256, False), ((16, 32), 256, True)]


@pytest.mark.parametrize("n,opaque,bad", [(1, 0, False), (63, 2, False), (64, 0, True), (65, 1, False), (257, 3, True),
                                          (700, 0, False), (2600, 2, True), (12400, 0, False)])
@pytest.mark.parametrize("form", FORMS)
def test_one_tile_in_grids_of_any_size(gs, form, n, opaque, bad):  # noqa: F811
    gsstep, step_mod = gs
    tile, tpt, bf16 = form
    sc = _pile(n, opaque)
    out = []
    for w, h in ((16, tile[1]), (64, 64), (912, 912)):
        tr = step_mod.Trainer([sc], [_cam(w, h)], capacity=12 * n + 4096, tile=tile, threads_per_tile=tpt, mom_bf16=bf16)
        tr.forward()
        st = tr.stats()
        assert st.status == 0
        K = int(st.k_required)
        a, b = (int(x) for x in tr.buffer(4, 2).cpu().numpy().view(np.uint32))
        tr.dl.copy_(torch.from_numpy(_dl(w, h, n, tile, bad).reshape(-1, 3)))
        gsstep.gs_raster_bwd(tr.plan, tr.ws, tr.image, tr.dl)
        slot = tr.buffer(9, K).cpu().numpy().view(np.uint32)[a:b]
        out.append((tr.buffer(3, K).cpu().numpy()[a:b], gsstep.gs_gradient_records(tr.plan, tr.ws, K).cpu().numpy()[slot]))
    assert len(out[0][0]) > n // 2 and np.nan_to_num(out[0][1]).any()
    assert np.isnan(out[0][1]).any() == bad
    for ids, rec in out[1:]:
        np.testing.assert_array_equal(ids, out[0][0])
        np.testing.assert_array_equal(rec, out[0][1])


@pytest.mark.parametrize("n,opaque", [(63, 2), (64, 0), (65, 1), (257, 3)])
@pytest.mark.parametrize("form", FORMS)
def test_large_grid_matches_oracle(gs, orc, form, n, opaque):  # noqa: F811
    gsstep, step_mod = gs
    tile, tpt, bf16 = form
    w, h = 907, 905
    sc, cam = _pile(n, opaque), _cam(w, h)
    b, p, P, r = _oracle_all(orc, sc, cam, tile)
    tr = step_mod.Trainer([sc], [cam], capacity=64 * n + 4096, tile=tile, threads_per_tile=tpt, mom_bf16=bf16)
    tr.forward()
    assert tr.stats().status == 0 and tr.stats().k_required == b.K
    rng = np.random.default_rng(n)
    dl = (rng.normal(size=(h, w, 3)) / 768).astype(np.float32)
    tr.dl.copy_(torch.from_numpy(dl.reshape(-1, 3)))
    gsstep.gs_raster_bwd(tr.plan, tr.ws, tr.image, tr.dl)
    off = tr.buffer(1, n + 1).cpu().numpy().view(np.uint32).astype(np.int64)
    gr = gsstep.gs_gradient_records(tr.plan, tr.ws, b.K).cpu().numpy()
    got = _sum_slots(gr, off, tr.buffer(0, n).cpu().numpy().view(np.uint32))
    g2 = orc.raster_bwd64(cam, P, b, dl.astype(np.float64), (0, 0, 0), *tile)
    good = (b.count > 0) & ~_unstable_gaussians(P, r, cam)
    assert good.sum() > 0.5 * n
    _check_grad(got, g2, good, f"grad2d {form} n={n}")
