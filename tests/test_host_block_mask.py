"""The raster kernels' 4x4-block mask, emulated with numpy float32 operation
by operation, never drops a block that holds a pixel the kernels would blend:
their own FP32 decision (exponent >= -4.5 log2 e and o 2^p >= 1/255) over every
pixel of the tile, for round, elongated and nearly degenerate conics, means
inside and far outside the tile, opacities from 1/255 to 1."""
import numpy as np
import pytest

f32 = np.float32


def _fma(a, b, c):
    return (a.astype(np.float64) * b + c).astype(f32)


def _mask(x, y, a, b, c, op, TW, TH):
    """(n, TH/4, TW/4) booleans; the kernel's approximate functions are
    replaced by exactly rounded ones widened to their 2-ulp error."""
    with np.errstate(all="ignore"):
        ac = a * c
        det = ac - b * b
        kappa = ac / det
        r2 = _fma(np.minimum(f32(9), f32(2) * np.log(op * f32(255))), _fma(f32(4e-6) * np.ones_like(kappa), kappa, f32(1.002)),
                  f32(1e-3)) * f32(1 - 1e-6)
        s = r2 / det
        ex, ey = np.sqrt(s * c), np.sqrt(s * a)
        mg = _fma(f32(1e-5) * np.ones_like(x), ex + ey + np.abs(x) + np.abs(y), f32(0.02))
        ia = f32(1) / a
        k, u, w = -b * ia, r2 * ia * f32(1.00001), det * ia * ia
        ys = -b * (ex / c)
        ylo, yhi = -ey - mg, ey + mg
        out = np.zeros((len(x), TH // 4, TW // 4), bool)
        for by in range(TH // 4):
            lo, hi = np.maximum(f32(4 * by) - y, ylo), np.minimum(f32(4 * by + 3) - y, yhi)
            dR, dL = np.minimum(np.maximum(ys, lo), hi), np.minimum(np.maximum(-ys, lo), hi)
            hR, hL = (np.sqrt(np.maximum(f32(0), _fma(-w * d, d, u))) for d in (dR, dL))
            xr, xl = x + _fma(k, dR, hR) + mg, x + _fma(k, dL, -hL) - mg
            b0, b1 = np.maximum(0, np.ceil((xl - f32(3)) * f32(0.25))), np.minimum(TW // 4 - 1, np.floor(xr * f32(0.25)))
            for bx in range(TW // 4):
                out[:, by, bx] = (lo <= hi) & (b0 <= bx) & (bx <= b1)
    all_on = ~(det > 0) | ~(kappa < f32(1e5))
    out[all_on] = True
    out[~(op * f32(255) > f32(1))] = False
    return out


def _hits(x, y, a, b, c, op, TW, TH):
    """The kernels' decision for every pixel (mean relative to the first
    pixel's centre)."""
    l2e = f32(1.4426950408889634)
    A, B, C = f32(-0.5) * l2e * a, -l2e * b, f32(-0.5) * l2e * c
    dx = np.arange(TW, dtype=f32)[None, :] - x[:, None]
    dy = np.arange(TH, dtype=f32)[None, :] - y[:, None]
    adx2, bdx = (A[:, None] * dx) * dx, B[:, None] * dx
    t = _fma(C[:, None, None], dy[:, :, None], bdx[:, None, :])
    p = _fma(dy[:, :, None], t, adx2[:, None, :])
    G = np.exp2(p.astype(np.float64)) * (1 + 1e-6)
    return (p >= f32(-4.5) * l2e) & ((op[:, None, None] * G).astype(f32) >= f32(1 / 255.0))


@pytest.mark.parametrize("TW,TH", [(8, 8), (16, 16), (16, 32)])
@pytest.mark.parametrize("spread", [1.0, 30.0, 1000.0])
def test_block_mask_keeps_every_blending_block(TW, TH, spread):
    rng = np.random.default_rng(int(spread) + TW + TH)
    n = 40_000
    # covariance: low-pass 0.3 plus a rotated pair of variances, axis ratio up to `spread`
    s1 = np.exp(rng.uniform(-2, 3, n))
    s2 = s1 * np.exp(rng.uniform(0, np.log(spread) + 1e-9, n))
    th = rng.uniform(0, np.pi, n)
    v = [s1 ** 2, s2 ** 2]
    ca = 0.3 + v[0] * np.cos(th) ** 2 + v[1] * np.sin(th) ** 2
    cc = 0.3 + v[0] * np.sin(th) ** 2 + v[1] * np.cos(th) ** 2
    cb = (v[0] - v[1]) * np.sin(th) * np.cos(th)
    det = ca * cc - cb * cb
    a, b, c = (q.astype(f32) for q in (cc / det, -cb / det, ca / det))
    r = np.minimum(3 * s2, 2000)
    x = (rng.uniform(0, TW, n) + rng.uniform(-1, 1, n) * r).astype(f32)
    y = (rng.uniform(0, TH, n) + rng.uniform(-1, 1, n) * r).astype(f32)
    op = (1.0 / (1.0 + np.exp(-rng.normal(-1, 2.5, n)))).astype(f32)
    op[: n // 8] = (f32(1 / 255.0) * (1 + rng.uniform(-1e-3, 2e-2, n // 8))).astype(f32)
    hit = _hits(x, y, a, b, c, op, TW, TH).reshape(n, TH // 4, 4, TW // 4, 4).any((2, 4))
    mask = _mask(x, y, a, b, c, op, TW, TH)
    assert hit.any(1).any(1).sum() > n // 10
    assert not (hit & ~mask).any()
    if spread == 1.0:      # round footprints: few blocks beyond the needed ones
        assert mask.sum() < 1.1 * hit.sum()
