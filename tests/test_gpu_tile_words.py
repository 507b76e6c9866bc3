"""The tile sort by 32-bit words at the edges of its paths: list lengths around one
warp's words, the groups' and chunks' limits and merged chunks; depths all different,
in runs of 32 equal ones (still put in order afterwards) and in few, long runs (64-bit
keys instead); views of 19 and 20 bits of depth: keys and Gaussians bit-exact against
the oracle."""
import numpy as np
import pytest

from paper_2605_00219_gb300 import synth

from test_gpu_parity import gs  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(1040, 1024), (960, 960)])
@pytest.mark.parametrize("depths", ["spread", "runs", "few"])
@pytest.mark.parametrize("n", [1, 8, 9, 255, 257, 1023, 2047, 4096, 4097, 8192, 8193, 16385, 24600])
def test_words(gs, orc, w, h, depths, n):  # noqa: F811
    _, step_mod = gs
    rng = np.random.default_rng(n)
    m = rng.uniform(-0.004, 0.004, (n, 3))
    if depths == "spread":
        m[:, 2] = rng.uniform(-0.5, 0.5, n)
    else:
        values = np.linspace(-0.5, 0.5, -(-n // 32) if depths == "runs" else 3)
        m[:, 2] = rng.permutation(np.resize(values, n))
    sc = synth.Scene(m.astype(np.float32), np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                     np.full((n, 3), 1e-3, np.float32), np.full(n, 0.5, np.float32),
                     np.zeros((n, 16, 3), np.float32))
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.array([0, 0, 4], np.float32), 800.0, 800.0, 520.0, 520.0, w, h, 0)
    b = orc.bin32(sc, cam)
    assert (b.ranges[:, 1] - b.ranges[:, 0]).max() == n
    tr = step_mod.Trainer([sc], [cam], capacity=2 * n + 4096)
    tr.forward()
    assert tr.stats().status == 0
    np.testing.assert_array_equal(tr.buffer(2, b.K).cpu().numpy().view(np.uint32), b.keys)
    np.testing.assert_array_equal(tr.buffer(3, b.K).cpu().numpy().view(np.uint32), b.gidx)
