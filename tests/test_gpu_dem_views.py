"""Texture views of DEM buffers: the sizes that get one, and that many small
DEMs never take the place of a large one's view (in a process of its own: views
are kept for the life of a process)."""
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import paper_2506_23364_gb300 as awo
from paper_2506_23364_gb300 import inputs

pytestmark = pytest.mark.gpu

MANY = """
import torch
import paper_2506_23364_gb300 as awo
buf = torch.zeros((1 << 20) + 300 * 128, device="cuda")
def path(i, h, w):
    return awo.awo_dem_gather_path(buf[128 * i:128 * i + h * w].reshape(h, w), awo.grid(w, h, 10.0))
first, last = %r
for (h, w) in (first, last):
    paths = [path(i, h, w) for i in range(300)]
    assert paths == ["texture"] * 256 + ["loads"] * 44, (h, w, paths.count("texture"))
    assert [path(i, h, w) for i in range(300)] == paths  # a view is found again
"""


@pytest.mark.parametrize("order", [((512, 1024), (1024, 1024)), ((1024, 1024), (512, 1024))])
def test_small_and_large_views_do_not_compete(order):
    subprocess.run([sys.executable, "-c", MANY % (order,)], check=True, timeout=300)


@pytest.mark.parametrize("h,want", [(512, "texture"), (511, "loads")])
def test_smallest_grid_with_a_view(h, want):
    """2^19 cells and one row fewer, both ways of fetching against the oracle."""
    w = 1024
    dem = np.ascontiguousarray(inputs.fbm(w, 0.8, seed=h, relief=1500.0)[:h]).astype(np.float32)
    cells = np.arange(0, h * w, 101).astype(np.uint32)
    kw = dict(traj_per_cell=6, max_steps=200, seed=4)
    dh, g = torch.from_numpy(dem).cuda(), awo.grid(w, h, 10.0)
    assert awo.awo_dem_gather_path(dh, g) == want
    dc = torch.from_numpy(cells.view(np.int32)).cuda()
    count, maxe = torch.zeros((h, w), dtype=torch.int32, device="cuda"), torch.zeros((h, w), device="cuda")
    stats = torch.zeros(6, dtype=torch.int64, device="cuda")
    ws = torch.empty(awo.awo_simulate_workspace_bytes(cells.size), dtype=torch.uint8, device="cuda")
    awo.awo_simulate(dh, g, dc, None, cells.size, awo.SimParams.make(**kw), count, maxe, stats, ws)
    c64, want_e, st = oracle.simulate_threaded(dem, 10.0, cells, oracle.SimParams(**kw))
    assert {k: awo.stats_dict(stats)[k] for k in st} == st
    assert np.array_equal(count.cpu().numpy().view(np.uint32), oracle.counts_u32(c64))
    assert np.array_equal(maxe.cpu().numpy(), want_e)


def test_soft_calls_at_the_smallest_view():
    """Deposits and weight gradients do not depend on the way of fetching."""
    h, w = 512, 1024
    dem = np.ascontiguousarray(inputs.fbm(w, 0.8, seed=1, relief=1500.0)[:h]).astype(np.float32)
    buf = torch.empty(h * w + 1, device="cuda")
    cells = torch.arange(0, h * w, 211, dtype=torch.int32, device="cuda")
    n, g = cells.numel(), awo.grid(w, h, 10.0)
    weight, grad = torch.linspace(0.5, 1.5, n, device="cuda"), torch.linspace(-1.0, 1.0, h * w, device="cuda").reshape(h, w)
    ws = torch.empty(awo.awo_soft_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    p = awo.SimParams.make(drag_k=1e-3, traj_per_cell=5, max_steps=200, seed=2, flags=1)
    got = []
    for dh, path in ((torch.from_numpy(dem).cuda(), "texture"), (buf[1:].reshape(h, w), "loads")):
        dh.copy_(torch.from_numpy(dem))
        assert awo.awo_dem_gather_path(dh, g) == path
        q = torch.zeros((h, w), dtype=torch.int64, device="cuda")
        stats = torch.zeros(6, dtype=torch.int64, device="cuda")
        awo.awo_soft_forward(dh, g, cells, None, n, weight, p, 1.0, q, stats, ws)
        gt = torch.empty(2, dtype=torch.float64, device="cuda")
        gw = torch.empty(n, device="cuda")
        awo.awo_soft_backward(dh, g, cells, None, n, weight, p, 1.0, grad, gt, gw, ws)
        got.append((q, stats, gw, gt))
    (q0, s0, w0, t0), (q1, s1, w1, t1) = got
    assert torch.equal(q0, q1) and torch.equal(s0, s1) and int(s0[0]) > 0
    # sums in FP64 by atomics, in any order (5 terms; 12 k terms), the weights' rounded to FP32 at the end
    assert torch.allclose(w0, w1, rtol=2.0 ** -22, atol=1e-12)
    assert torch.allclose(t0, t1, rtol=1e-9, atol=1e-7)
