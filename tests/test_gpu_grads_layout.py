"""gs_project_bwd_grads writes the gradients of gs_project_bwd_adam's gradient mode,
bit for bit, in the layout and type of each scene's buffers (BF16 SH rounded to
nearest), for several scenes at the edges of its 128-Gaussian blocks; bad arguments
are refused before anything is launched."""
import ctypes

import pytest
import torch

from paper_2605_00219_gb300 import synth

from test_gpu_parity import gs  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("sizes", [(1,), (127, 129, 256), (5, 3000)])
def test_same_gradients_in_stored_layout(gs, sizes, bf16):  # noqa: F811
    gsstep, step_mod = gs
    scenes = [synth.uniform_scene(n, 3 + k) for k, n in enumerate(sizes)]
    cams = [synth.Camera(*synth.tiny_camera().__dict__.values()) for _ in range(2 * len(sizes))]
    for i, c in enumerate(cams):
        c.scene = i // 2
        c.t = c.t + 0.1 * (i % 2)
    tr = step_mod.Trainer(scenes, cams, sh_bf16=bf16)
    tr.forward()
    tr.dl.normal_(generator=torch.Generator(device="cuda").manual_seed(1))
    gsstep.gs_raster_bwd(tr.plan, tr.ws, tr.image, tr.dl)
    N = sum(sizes)
    ref = torch.empty((15, N, 4), device="cuda")
    gsstep.gs_project_bwd_adam(tr.plan, tr.ws, tr.scenes, tr.cams, None, ref)
    grads = [(torch.full_like(b.geom, 7.0), torch.full_like(b.sh, 7.0)) for b in tr.scenes]
    gsstep.gs_project_bwd_grads(tr.plan, tr.ws, tr.scenes, tr.cams, grads)
    o = 0
    for n, (dgeom, dsh) in zip(sizes, grads):
        assert torch.equal(dgeom, ref[:3, o:o + n])
        want = ref[3:, o:o + n]
        if bf16:
            want = want.reshape(6, 2, n, 4).permute(0, 2, 1, 3).reshape(6, n, 8).to(torch.bfloat16)
        assert torch.equal(dsh, want)
        o += n
    L = gsstep.lib()
    bufs, cp = gsstep.scene_bufs(tr.scenes), ctypes.c_void_p(tr.cams.data_ptr())
    ws, st = ctypes.c_void_p(tr.ws.data_ptr()), None
    assert L.gs_project_bwd_grads(tr.plan.handle, ws, bufs, cp, None, st) == 1
    arr = (gsstep.gs_scene_buf * len(sizes))()
    assert L.gs_project_bwd_grads(tr.plan.handle, ws, bufs, cp, arr, st) == 1          # null buffers, n = 0
    for i, (b, (dgeom, dsh)) in enumerate(zip(tr.scenes, grads)):
        arr[i] = gsstep.gs_scene_buf(b.n, dgeom.data_ptr() + 4, dsh.data_ptr(), None, None, None)
    assert L.gs_project_bwd_grads(tr.plan.handle, ws, bufs, cp, arr, st) == 1          # misaligned
