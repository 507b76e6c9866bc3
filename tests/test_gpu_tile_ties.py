"""The tile sort on lists whose equal depth codes are too many for words: runs that show in
256 sorted words, runs that appear only after the merges, and one run among different
depths: keys and Gaussians bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2605_00219_gb300 import synth

from test_gpu_parity import gs  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("run", [33, 40, 41, 100, 300, -33, -300])
@pytest.mark.parametrize("n", [254, 256, 257, 300, 1022, 1030, 2046, 4096, 4100, 8192, 9000])
def test_runs(gs, orc, n, run):  # noqa: F811
    """run > 0: every depth that many times; run < 0: one depth that often, the others once."""
    _, step_mod = gs
    rng = np.random.default_rng(n)
    m = rng.uniform(-0.004, 0.004, (n, 3))
    z = np.linspace(-0.5, 0.5, n)
    if run > 0:
        z = np.resize(np.linspace(-0.5, 0.5, -(-n // run)), n)
    else:
        z[n // 3:n // 3 - run] = z[n // 3]
    m[:, 2] = rng.permutation(z)
    sc = synth.Scene(m.astype(np.float32), np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                     np.full((n, 3), 1e-3, np.float32), np.full(n, 0.5, np.float32),
                     np.zeros((n, 16, 3), np.float32))
    cam = synth.Camera(np.eye(3, dtype=np.float32), np.array([0, 0, 4], np.float32), 800.0, 800.0, 520.0, 520.0, 1040,
                       1024, 0)
    b = orc.bin32(sc, cam)
    assert (b.ranges[:, 1] - b.ranges[:, 0]).max() == n
    tr = step_mod.Trainer([sc], [cam], capacity=2 * n + 4096)
    tr.forward()
    assert tr.stats().status == 0
    np.testing.assert_array_equal(tr.buffer(2, b.K).cpu().numpy().view(np.uint32), b.keys)
    np.testing.assert_array_equal(tr.buffer(3, b.K).cpu().numpy().view(np.uint32), b.gidx)
