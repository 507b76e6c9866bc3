"""gs_loss_l1_noalloc on values whose sum is infinite: the loss is infinite as a plain
sum's is (its compensated sums must not turn infinity - infinity into NaN), NaN only
where an input is, and the gradient the sign of each difference."""
import numpy as np
import pytest
import torch

from test_zz_no_alloc import gs  # noqa: F401

pytestmark = pytest.mark.gpu
TILE, BLOCKS = 2048, 152 * 8


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("where", ["first", "last", "all", "overflow", "nan"])
@pytest.mark.parametrize("n", [1, 5, TILE, TILE + 1, 300 * TILE, 2 * BLOCKS * TILE + 777])
def test_infinite_sums(gs, n, where, shift):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(n)
    img, tgt = (torch.rand(n + 4, device="cuda", generator=g)[shift:shift + n] for _ in range(2))
    if where == "overflow":
        img.fill_(3e38)
        tgt.fill_(-3e38 if n == 1 else 0.0)
    else:
        img[{"first": slice(0, 1), "last": slice(n - 1, n), "all": slice(0, n), "nan": slice(n // 2, n // 2 + 1)}[where]] = \
            float("nan") if where == "nan" else -float("inf")
    dl, loss = torch.empty(n, device="cuda"), torch.zeros(1, device="cuda")
    for _ in range(2):
        gs.gs_loss_l1_noalloc(img, tgt, dl, loss)
    got = float(loss)
    assert np.isnan(got) if where == "nan" else got == float("inf")
    want = torch.nan_to_num(torch.sign(img - tgt), nan=0.0)
    assert torch.equal(dl, want * np.float32(1.0) / np.float32(n))
