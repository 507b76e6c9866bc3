"""gs_loss_l1_noalloc at the edges of its tiles and its grid, aligned and not:
gradient bit-equal to sign / n, loss within 2^-22 of the float64 mean (two
compensated sums and a tree of eight values and 13 levels: under 2 ulp each)."""
import numpy as np
import pytest
import torch

from test_zz_no_alloc import gs  # noqa: F401

pytestmark = pytest.mark.gpu
TILE, BLOCKS = 2048, 152 * 8


@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 3, 4, 255, TILE - 1, TILE, TILE + 1, 3 * TILE + 5, BLOCKS * TILE - 1, BLOCKS * TILE,
                               BLOCKS * TILE + 1, 3 * BLOCKS * TILE + 777])
def test_sizes(gs, n, shift):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(n)
    img, tgt = (torch.rand(n + 4, device="cuda", generator=g)[shift:shift + n] for _ in range(2))
    tgt[::7] = img[::7]
    buf = torch.full((n + 8,), 7.0, device="cuda")
    dl, loss = buf[4 + shift:4 + shift + n], torch.zeros(1, device="cuda")
    for _ in range(2):
        gs.gs_loss_l1_noalloc(img, tgt, dl, loss)
    assert torch.equal(dl, torch.sign(img - tgt) * np.float32(1.0) / np.float32(n))
    assert float(buf[:4 + shift].min()) == 7.0 and float(buf[4 + shift + n:].min()) == 7.0     # nothing outside
    ref = float((img - tgt).abs().double().mean())
    assert abs(float(loss) - ref) <= 2.0 ** -22 * ref
