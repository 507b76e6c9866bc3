"""The buffers that Renderer's backward hands to gs_project_bwd_grads hold what the
library writes for the plan (FP32 geometry float4[3][n]; SH float4[12][n], or uint4[6][n]
with BF16 storage), whatever type and shape the scene tensors have: the native calls
are replaced by ones that record the buffers, so nothing is read or written out of
range here."""
import types

import pytest
import torch

from paper_2605_00219_gb300 import autograd, gsstep

N = 5


def _backward(monkeypatch, sh_bf16, geom, sh):
    seen = []
    for name in ("gs_project_fwd", "gs_bin_sort", "gs_raster_fwd", "gs_raster_bwd"):
        monkeypatch.setattr(gsstep, name, lambda *a, **k: None)

    def grads_call(plan, ws, scenes, cams, grads, stream=None):
        for g, s in grads:
            seen.append((g.nbytes, s.nbytes))
            g.fill_(1.0)
            s.fill_(2.0)

    monkeypatch.setattr(gsstep, "gs_project_bwd_grads", grads_call)
    r = types.SimpleNamespace(plan=types.SimpleNamespace(pixels=6), ws=None, cams=None, bg=None,
                              device=torch.device("cpu"), scene_sizes=[N], sh_bf16=sh_bf16, generation=0)
    geom, sh = geom.requires_grad_(), sh.requires_grad_()
    img = autograd._GSRender.apply(r, geom, sh)
    error = None
    try:
        img.sum().backward()
    except RuntimeError as e:
        error = e
    return seen, geom.grad, sh.grad, error


@pytest.mark.parametrize("sh_bf16", [False, True])
@pytest.mark.parametrize("geom_dtype", [torch.float32, torch.float16, torch.bfloat16, torch.float64])
@pytest.mark.parametrize("sh_dtype", [torch.float32, torch.bfloat16, torch.float16])
def test_buffers_hold_what_the_kernel_writes(monkeypatch, sh_bf16, geom_dtype, sh_dtype):
    sh = torch.zeros((6, N, 8) if sh_bf16 and sh_dtype == torch.bfloat16 else (12, N, 4), dtype=sh_dtype)
    seen, dgeom, dsh, error = _backward(monkeypatch, sh_bf16, torch.zeros((3, N, 4), dtype=geom_dtype), sh)
    assert error is None
    assert seen == [(48 * N, (96 if sh_bf16 else 192) * N)]
    assert dgeom.dtype == geom_dtype and dsh.dtype == sh_dtype      # autograd casts them
    assert bool((dgeom == 1).all()) and bool((dsh == 2).all())


@pytest.mark.parametrize("sh_bf16", [False, True])
@pytest.mark.parametrize("geom_shape,sh_shape", [((12 * N,), (12, N, 4)), ((N, 12), (12, N, 4)), ((3, N, 4), (48 * N,)),
                                                 ((3, N, 3), (12, N, 4)), ((3, N, 4), (6, N, 8))])
def test_other_shapes_are_refused(monkeypatch, geom_shape, sh_shape, sh_bf16):
    seen, _, _, error = _backward(monkeypatch, sh_bf16, torch.zeros(geom_shape), torch.zeros(sh_shape))
    assert seen == [(48 * N, (96 if sh_bf16 else 192) * N)]
    assert error is not None and "shape" in str(error)
