"""Densification's output rows at the edges of its scan blocks and for one-sided
fates, against torch indexing: sources in the documented order (kept, clones, first
and second split products), copied rows bit for bit, zero moments for new rows,
split means within 2e-6 of float64, split scales the correctly rounded quotients."""
import numpy as np
import pytest
import torch

from test_gpu_densify import gs  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("n,mix", [(1, "keep"), (1, "split"), (8, "mixed"), (4095, "mixed"), (4096, "mixed"),
                                   (4097, "mixed"), (8192, "split"), (12289, "clone"), (50_001, "mixed")])
def test_rows(gs, n, mix, bf16):  # noqa: F811
    gsstep, step_mod = gs
    g = torch.Generator(device="cuda").manual_seed(n)
    dt = torch.bfloat16 if bf16 else torch.float32
    sh = torch.randn((6, n, 8) if bf16 else (12, n, 4), device="cuda", generator=g).to(dt)
    sb = step_mod.SceneBuffers(n, torch.randn((3, n, 4), device="cuda", generator=g), sh,
                               torch.randn((15, n, 4), device="cuda", generator=g).to(dt),
                               torch.rand((15, n, 4), device="cuda", generator=g).to(dt))
    # fate: 0 pruned, 1 kept, 2 cloned, 3 split
    one = {"keep": 1, "clone": 2, "split": 3}
    fate = torch.randint(0, 4, (n,), device="cuda", generator=g) if mix == "mixed" else \
        torch.full((n,), one[mix], device="cuda")
    fate[0] = max(1, int(fate[0]))
    sb.geom[2, :, :3] = torch.rand((n, 3), device="cuda", generator=g) * 0.01 + 0.001
    sb.geom[2, fate == 3, 1] = 0.05
    sb.geom[2, :, 3] = torch.where(fate == 0, 0.001, 0.5)
    sb.stats = torch.stack([torch.where(fate >= 2, 1e-3, 1e-5), torch.ones(n, device="cuda")], 1).contiguous()
    cfg = gsstep.make_densify_cfg(2.0)
    scratch = torch.empty(gsstep.gs_densify_scratch_bytes(n), dtype=torch.uint8, device="cuda")
    gsstep.gs_densify_count(sb, sb.storage_flags, cfg, scratch)
    counts = gsstep.gs_densify_counts(scratch)
    ik, ic, isp = (torch.nonzero(x)[:, 0] for x in ((fate == 1) | (fate == 2), fate == 2, fate == 3))
    assert counts == (len(ik), len(ic), len(isp), len(ik) + len(ic) + 2 * len(isp))
    out = step_mod.SceneBuffers.empty_like_layout(sb, counts[3])
    eps = torch.randn((n, 6), device="cuda", generator=g)
    gsstep.gs_densify_apply(sb, sb.storage_flags, cfg, eps, scratch, out)
    src = torch.cat([ik, ic, isp, isp])
    first = len(ik) + len(ic)
    assert torch.equal(out.sh, sb.sh[:, src]) and torch.equal(out.geom[1], sb.geom[1, src])
    assert torch.equal(out.geom[:, :first], sb.geom[:, src[:first]])
    for a, b in ((out.m, sb.m), (out.v, sb.v)):
        assert torch.equal(a[:, :len(ik)], b[:, ik]) and not a[:, len(ik):].any()
    assert not out.stats.any()
    if len(isp):
        q = sb.geom[1, isp].double()
        w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                         2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                         2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
        s = sb.geom[2, isp, :3].double()
        for k in range(2):
            at = slice(first + k * len(isp), first + (k + 1) * len(isp))
            mean = sb.geom[0, isp, :3].double() + (R @ (s * eps[isp, 3 * k:3 * k + 3].double())[:, :, None])[:, :, 0]
            assert float((out.geom[0, at, :3] - mean).abs().max()) <= 2e-6
            assert torch.equal(out.geom[0, at, 3], sb.geom[0, isp, 3])
            ref = (sb.geom[2, isp, :3].cpu().numpy() / np.float32(1.6)).astype(np.float32)
            np.testing.assert_array_equal(out.geom[2, at, :3].cpu().numpy(), ref)
            assert torch.equal(out.geom[2, at, 3], sb.geom[2, isp, 3])
    # an output of another size is left alone
    bad = step_mod.SceneBuffers.empty_like_layout(sb, counts[3] + 1)
    bad.geom.fill_(7.0)
    gsstep.gs_densify_apply(sb, sb.storage_flags, cfg, eps, scratch, bad)
    assert bool((bad.geom == 7.0).all())
