"""The sort's set-up at the edges of its paths: one block up to 4,096 tiles (pairs
summed by the block itself up to 64 groups of 1,024, by k_sort_sums beyond) and three
launches above, several scenes of uneven view counts, footprints placed by a lane, by
a warp and by a repeated traversal: counts, offsets, ranges, sorted keys and pairs
bit-exact against the oracle, and an overflow that leaves every list empty."""
import numpy as np
import pytest
import torch

from paper_2605_00219_gb300 import synth

from test_gpu_parity import gs  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(orc, tr, scenes, cams, tile):
    off_t = off_k = 0
    q0 = np.cumsum([0] + [s.n * sum(c.scene == k for c in cams) for k, s in enumerate(scenes)])
    pairs = int(q0[-1])
    count = tr.buffer(0, pairs).cpu().numpy().view(np.uint32).astype(np.int64)
    offs = tr.buffer(1, pairs + 1).cpu().numpy().view(np.uint32).astype(np.int64)
    K = int(tr.stats().k_required)
    np.testing.assert_array_equal(offs, np.concatenate([[0], np.cumsum(count)]))
    assert K == offs[-1]
    keys = tr.buffer(2, K).cpu().numpy().view(np.uint32)
    pids = tr.buffer(3, K).cpu().numpy().view(np.uint32).astype(np.int64)
    ranges = tr.buffer(4, 2 * tr.plan.tiles).cpu().numpy().view(np.uint32).reshape(-1, 2).astype(np.int64)
    pair_base = 0
    seen = [0] * len(scenes)
    for c in cams:
        sc = scenes[c.scene]
        b = orc.bin32(sc, c, *tile)
        nt = -(-c.width // tile[0]) * -(-c.height // tile[1])
        np.testing.assert_array_equal(keys[off_k:off_k + b.K], b.keys)
        np.testing.assert_array_equal(pids[off_k:off_k + b.K] - pair_base, b.gidx)
        r = ranges[off_t:off_t + nt]
        np.testing.assert_array_equal(np.where(r[:, 1:] > r[:, :1], r - off_k, 0), b.ranges)
        nv = sum(x.scene == c.scene for x in cams)
        np.testing.assert_array_equal(count[q0[c.scene] + seen[c.scene]:q0[c.scene + 1]:nv], b.count)
        seen[c.scene] += 1
        off_t, off_k, pair_base = off_t + nt, off_k + b.K, pair_base + sc.n
    return K


def _scene(n, seed, big=0):
    sc = synth.cluster_scene(n, 8, 3.0, seed=seed, log_scale=(-3.5, 0.7), logit_opacity=(0.0, 1.5))
    if big:
        sc.scales[:big] = np.exp(np.random.default_rng(seed).uniform(-2.0, 0.5, size=(big, 3))).astype(np.float32)
        sc.opacities[:big] = 0.9
    return sc


@pytest.mark.parametrize("w,h,tile", [(512, 512, (8, 8)), (520, 512, (8, 8)), (203, 149, (16, 16)),
                                      (1030, 1030, (16, 16)), (330, 700, (16, 32))])
@pytest.mark.parametrize("n,big", [(1, 1), (1023, 40), (70_000, 200)])
def test_one_view(gs, orc, w, h, tile, n, big):  # noqa: F811
    _, step_mod = gs
    sc = _scene(n, n, big)
    cam = synth.look_at([0, -5, 1.5], [0, 0, 0], w, h, 0.8 * w)
    tr = step_mod.Trainer([sc], [cam], tile=tile, capacity=16 * n + 3_000_000)
    tr.forward()
    assert tr.stats().status == 0
    _check(orc, tr, [sc], [cam], tile)


def test_scenes_of_uneven_views(gs, orc):  # noqa: F811
    _, step_mod = gs
    scenes = [_scene(n, k, 20) for k, n in enumerate((257, 5000, 1024, 33))]
    cams = [synth.look_at([0, -5, 1 + 0.2 * i], [0, 0, 0], 96 + 16 * i, 80, 90.0, scene=s)
            for i, s in enumerate((0, 1, 1, 1, 3, 1, 0, 3, 2))]
    tr = step_mod.Trainer(scenes, cams, capacity=2_000_000)
    tr.forward()
    assert tr.stats().status == 0
    K = _check(orc, tr, scenes, cams, (16, 16))
    small = step_mod.Trainer(scenes, cams, capacity=K - 2048)
    small.forward()
    st = small.stats()
    assert st.status == 1 and st.k_required == K
    assert not small.buffer(4, 2 * small.plan.tiles).any()
    assert not small.image.any()
