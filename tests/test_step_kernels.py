"""bench.step_kernels is the number of this library's kernels in a step: the kernel nodes
of a captured step, for each form of the sort's set-up (one block up to 4,096 tiles, which
also sums the pairs up to 64 groups of 1,024, and three launches above)."""
import ctypes
import types

import pytest
import torch

import bench

CASES = [(2000, 128, 128, 10), (65536, 128, 128, 10), (65537, 128, 128, 11), (70000, 1024, 1024, 11),
         (1000, 1040, 1024, 12), (70000, 1040, 1024, 12)]


@pytest.mark.parametrize("n,w,h,kernels", CASES)
def test_kernels_of_a_plan(n, w, h, kernels):
    tiles = -(-w // 16) * -(-h // 16)
    assert bench.step_kernels(types.SimpleNamespace(tiles=tiles, pairs=n)) == kernels


@pytest.mark.gpu
@pytest.mark.parametrize("n,w,h,kernels", CASES)
def test_kernel_nodes_of_a_captured_step(n, w, h, kernels):
    from paper_2605_00219_gb300 import build, step, synth
    build.build()
    if not hasattr(torch.cuda.CUDAGraph, "raw_cuda_graph"):
        pytest.skip("this PyTorch does not hand out the graph")
    scene = synth.uniform_scene(n, 1)
    cam = synth.tiny_camera()
    cam.width, cam.height = w, h
    tr = step.Trainer([scene], [cam], capacity=40 * n)
    g = torch.cuda.CUDAGraph(keep_graph=True)
    side = torch.cuda.Stream()
    with torch.cuda.graph(g, stream=side):
        tr.step(0, side)
    cu = ctypes.CDLL("libcuda.so.1")
    graph, count = ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    kinds = []
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    assert kinds.count(0) == kernels == bench.step_kernels(tr.plan)      # 0: kernel node
