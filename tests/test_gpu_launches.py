"""The number of kernels that the benchmark states for a step, against the
kernel nodes of the step captured as a graph."""

import ctypes
import os

import pytest
import torch

import bench
import synth

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")
from paper_2410_04974_gb300 import build  # noqa: E402


def _kernel_nodes(call):
    rt = ctypes.CDLL(os.path.join(build.cuda_libdir(build.nvcc()), "libcudart.so"))   # the library's own runtime
    stream = torch.cuda.Stream()
    handle, graph, count = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert rt.cudaStreamBeginCapture(handle, 2) == 0
    call(stream)
    assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    kinds = []
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    assert rt.cudaGraphDestroy(graph) == 0
    return kinds.count(0)


@pytest.mark.parametrize("n,views,size,kernels", [(3_000, 1, 800, 8), (3_000, 1, 128, 7), (3_000, 50, 64, 8)])
def test_step_launches(n, views, size, kernels):
    scene = synth.scene_cube(n, 5)
    r = sx.Renderer(n, scene.sh_degree, synth.ring_cameras(views, size, size), dup_capacity=4 << 20)
    params = sx.params_to_device(scene)
    img = r.forward(params)
    target, grads = torch.zeros_like(img), r.new_grads(params)
    torch.cuda.synchronize()
    assert _kernel_nodes(lambda s: r.step(params, img, target, None, grads, s)) == kernels
    assert bench.step_launches(r.plan) == kernels
