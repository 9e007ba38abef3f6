"""bench.py's count of the kernels of one run, against a captured run's."""
import ctypes

import pytest
import torch

import bench
import paper_2506_23364_gb300 as awo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,r,levels,quantised", [
    (256, 256, 0, 1, False), (1021, 763, 0, 9, True), (500, 300, 2, 4, True), (300, 500, -1, 8, False),
    (4096, 4096, 0, 2, True), (4097, 4096, 0, 7, True),            # scan of its own from 2^24 cells
    (2048, 2048, 1, 1, True), (2052, 2048, 1, 1, True),            # ... of 2^24 texels
    (8192, 8192, -1, 14, True), (8194, 8192, -1, 1, True)])
def test_launches_of_a_run(W, H, r, levels, quantised):
    ov = awo.Overlay(W, H, 10.0, quantised=quantised, levels=levels, want_normals=False, release_log2=r)
    ov.h.zero_()
    if quantised:
        ov.q.zero_()
    p = awo.SimParams.make(traj_per_cell=1, max_steps=1)
    ov.run(30.0, 45.0, p)  # flat: no release cell
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        ov.run(30.0, 45.0, p)
    nodes = ctypes.c_size_t(0)
    assert ctypes.CDLL("libcuda.so.1").cuGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None,
                                                       ctypes.byref(nodes)) == 0
    assert nodes.value == bench.launches_per_step(awo, W, H, r, levels)
