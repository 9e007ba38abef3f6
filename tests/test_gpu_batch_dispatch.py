"""The batched call's ways of running a request -- all requests of a kind in
one launch, or a launch of its own for one with many particles or alone of its
kind; with and without the look at a cell's maximum; with and without drag --
give every request the rasters and statistics of awo_simulate on it alone."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2506_23364_gb300 as awo
from paper_2506_23364_gb300 import inputs

pytestmark = pytest.mark.gpu

LARGE = 3_000_000  # particles from which a request has a launch of its own, in a batch that looks at the maxima


class Region:
    """A request and what awo_simulate gives for it alone."""

    def __init__(self, dem, cells, kw, n_max=None, r=0):
        H, W = dem.shape
        self.g, self.n, self.dem, self.list, self.kw = awo.grid(W, H, 10.0), len(cells), dem, cells, kw
        self.h = torch.from_numpy(dem).cuda()
        self.cells = torch.zeros(max(n_max or len(cells), 1), dtype=torch.int32, device="cuda")
        self.cells[:len(cells)] = torch.from_numpy(np.asarray(cells, np.uint32).view(np.int32)).cuda()
        self.n_dev = torch.tensor([len(cells)], dtype=torch.int32, device="cuda")
        self.n_max = n_max if n_max is not None else len(cells)
        self.p = awo.SimParams.make(**kw, release_log2=r, flags=1)
        self.count = torch.empty((H, W), dtype=torch.int32, device="cuda")
        self.maxe = torch.empty((H, W), device="cuda")
        self.stats = torch.zeros(6, dtype=torch.int64, device="cuda")
        ws = torch.empty(awo.awo_simulate_workspace_bytes(self.n_max), dtype=torch.uint8, device="cuda")
        awo.awo_simulate(self.h, self.g, self.cells, self.n_dev, self.n_max, self.p, self.count, self.maxe, self.stats, ws)
        self.want = self.count.clone(), self.maxe.clone(), self.stats.clone()
        self.count.fill_(9)
        self.maxe.fill_(1e9)

    def request(self):
        return awo.sim_request(self.h, self.g, self.cells, self.n_dev, self.n_max, self.p, self.count, self.maxe)


def _run(regions, tuning=None):
    reqs = (awo.SimRequest * len(regions))(*[q.request() for q in regions])
    ws = torch.empty(awo.awo_simulate_batched_workspace_bytes(reqs), dtype=torch.uint8, device="cuda")
    stats = torch.full((len(regions), 6), -1, dtype=torch.int64, device="cuda")
    awo.awo_simulate_batched(reqs, ws, tuning, stats)
    torch.cuda.synchronize()
    for i, q in enumerate(regions):
        count, maxe, st = q.want
        assert torch.equal(q.count, count), i
        assert torch.equal(q.maxe, maxe), i
        assert torch.equal(stats[i], st), (i, stats[i], st)
    return stats


def _slope(h, w, seed):
    return inputs.fbm(max(h, w), 0.8, seed=seed, relief=1.5 * max(h, w))[:h, :w].astype(np.float32)


SHAPES = [(512, 1024), (96, 130), (64, 64), (33, 200), (513, 1024), (80, 81)]  # texture gathers: the first and fifth


@pytest.mark.parametrize("tuning", [None, (64, 0, 0), (256, 0, 0), (128, 100, 0), (64, 0, 1), (128, 0, 1), (256, 4096, 1)])
@pytest.mark.parametrize("drag", [0.0, 1e-3])
@pytest.mark.parametrize("look", [False, True])
def test_regions_equal_single_runs(look, drag, tuning):
    regions = []
    for i, (h, w) in enumerate(SHAPES):
        every, n = (1, 16) if look else (7, 1 + i)
        cells = np.arange(0, h * w, every)
        regions.append(Region(_slope(h, w, i), cells, dict(traj_per_cell=n, max_steps=30, drag_k=drag, seed=i)))
    total, cells = sum(q.n * q.kw["traj_per_cell"] for q in regions), sum(q.g.cells for q in regions)
    lanes = 1280 * torch.cuda.get_device_properties(0).multi_processor_count
    assert (total >= 32 * lanes or total >= 7 * cells) == look
    paths = [awo.awo_dem_gather_path(q.h, q.g) for q in regions]
    assert paths == ["texture", "loads", "loads", "loads", "texture", "loads"]
    _run(regions, awo.Tuning(*tuning, 0) if tuning else None)


@pytest.mark.parametrize("times", [0.97, 1.03])
def test_either_side_of_the_look_line(times):
    lanes = 1280 * torch.cuda.get_device_properties(0).multi_processor_count
    dem = _slope(512, 1024, 3)
    regions = []
    for i, s in enumerate((1.0, 0.5)):  # a particle at half steps counts twice
        n = int(times * 32 * lanes * s / 2 / 64)
        regions.append(Region(dem, np.arange(n) % dem.size, dict(traj_per_cell=64, max_steps=2, seed=i, step_scale=s)))
    assert sum(q.n * 64 for q in regions) < 7 * 2 * dem.size
    _run(regions)


@pytest.mark.parametrize("n", [1, 2, 3, 33, 128])
def test_numbers_of_requests(n):
    """Texel and cell lists, empty requests, capped ones, entries outside the grid."""
    dem = _slope(40, 56, 1)
    regions = []
    for i in range(n):
        r = (0, 0, 0, 1, -1)[i % 5]
        cells = np.arange(i % 3, 560, 1 + i % 7)
        kw = dict(traj_per_cell=(3, 33, 0, 1, 100, 5)[i % 6], max_steps=(50, 0, 1, 2, 400)[i % 5 if i % 11 else 1], seed=i)
        if i % 9 == 4:
            cells = cells[:0]
        elif i % 9 == 7:
            cells = np.concatenate([cells, [dem.size << 4, 0xFFFFFFFF]])
        regions.append(Region(dem, cells, kw, r=r))
    _run(regions)


@pytest.mark.parametrize("look", [False, True])
@pytest.mark.parametrize("n_cells", [LARGE // 256, LARGE // 256 + 1])
def test_either_side_of_a_launch_of_its_own(n_cells, look):
    dem = _slope(512, 1024, 2)
    kw = dict(traj_per_cell=256, max_steps=2)
    lanes = 1280 * torch.cuda.get_device_properties(0).multi_processor_count
    n_big = 3 if look else 2
    big = [Region(dem, (np.arange(n_cells) * 22) % dem.size, dict(kw, seed=i), n_max=dem.size) for i in range(n_big)]
    small = [Region(_slope(64, 64, i), np.arange(0, 4096, 9), dict(traj_per_cell=20, max_steps=90, seed=i)) for i in range(2)]
    assert (sum(q.n * q.kw["traj_per_cell"] for q in big + small) >= 32 * lanes) == look
    _run([*big[:1], small[0], *big[1:], small[1]])


def test_against_the_oracle():
    regions = [Region(_slope(h, w, 20 + i), np.arange(0, h * w, 11), dict(traj_per_cell=9, max_steps=200, seed=i))
               for i, (h, w) in enumerate(SHAPES)]
    _run(regions)
    for q in regions:
        c64, maxe, st = oracle.simulate_threaded(q.dem, 10.0, np.asarray(q.list, np.uint32), oracle.SimParams(**q.kw))
        assert np.array_equal(q.count.cpu().numpy().view(np.uint32), oracle.counts_u32(c64))
        assert np.array_equal(q.maxe.cpu().numpy(), maxe)


def test_launches_do_not_grow_with_the_requests():
    """A call over many small regions makes a handful of launches."""
    dem = _slope(64, 64, 0)
    regions = [Region(dem, np.arange(0, 4096, 20), dict(traj_per_cell=4, max_steps=50, seed=i)) for i in range(100)]
    for q in regions:
        q.p.flags = 0  # no raster to clear
    reqs = (awo.SimRequest * len(regions))(*[q.request() for q in regions])
    ws = torch.empty(awo.awo_simulate_batched_workspace_bytes(reqs), dtype=torch.uint8, device="cuda")
    awo.awo_simulate_batched(reqs, ws)  # occupancy queries outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        awo.awo_simulate_batched(reqs, ws)
    nodes = ctypes.c_size_t(0)
    assert ctypes.CDLL("libcuda.so.1").cuGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None,
                                                       ctypes.byref(nodes)) == 0
    assert 3 <= nodes.value <= 8
