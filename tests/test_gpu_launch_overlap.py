"""Kernels whose blocks are scheduled before the previous kernel has ended: steps issued
back to back on a stream of their own give the bits of steps with a synchronisation after
every call, and of replayed graphs, also with other work of the stream in between."""
import numpy as np
import pytest
import torch

from paper_2605_00219_gb300 import gsstep, synth

from test_gpu_parity import gs  # noqa: F401

pytestmark = pytest.mark.gpu


def _trainer(step_mod, n, size, loss):
    scene = synth.cluster_scene(n, 8, 3.0, seed=n, log_scale=(-3.5, 0.7), logit_opacity=(0.0, 1.5))
    cam = synth.look_at([0, -5, 1.5], [0, 0, 0], *size, 0.8 * size[0])
    tr = step_mod.Trainer([scene], [cam], capacity=16 * n + 3_000_000, loss=loss, seed=3)
    g = torch.Generator(device="cuda").manual_seed(1)
    t = torch.rand(tr.target.shape, device="cuda", generator=g)
    tr.target.copy_(t if tr.target.dtype == torch.float32 else (255 * t).to(torch.uint8))
    gsstep.gs_workspace_set_step(tr.plan, tr.ws, 100)
    return tr


@pytest.mark.parametrize("n,size,loss", [(500, (64, 48), "l1"), (2000, (128, 128), "l1_ssim"),
                                         (70_000, (640, 360), "l1"), (70_000, (1100, 1000), "l1_ssim_masked")])
def test_back_to_back(gs, monkeypatch, n, size, loss):  # noqa: F811
    _, step_mod = gs
    steps = 12
    fast, slow, graph = (_trainer(step_mod, n, size, loss) for _ in range(3))
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        for k in range(steps):
            fast.step(0, side)
            if k % 3 == 1:      # work of another library between the kernels
                fast.scenes[0].geom.mul_(1.0)
    side.synchronize()
    graph.capture()
    for _ in range(steps):
        graph.replay()
    names = ("gs_project_fwd", "gs_bin_sort", "gs_raster_fwd", "gs_loss_l1", "gs_loss_l1_ssim",
             "gs_loss_l1_ssim_masked", "gs_raster_bwd", "gs_project_bwd_adam")
    for name in names:
        def call(*a, _f=getattr(gsstep, name), **k):
            r = _f(*a, **k)
            torch.cuda.synchronize()
            return r
        monkeypatch.setattr(gsstep, name, call)
    for _ in range(steps):
        slow.step(0)
    torch.cuda.synchronize()
    for other in (fast, graph):
        for a, b in zip((slow.image, slow.scenes[0].geom, slow.scenes[0].sh, slow.scenes[0].m, slow.scenes[0].v),
                        (other.image, other.scenes[0].geom, other.scenes[0].sh, other.scenes[0].m, other.scenes[0].v)):
            np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())
