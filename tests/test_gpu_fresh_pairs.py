"""The particle kernel's fresh pairs, pool and general direction against the
oracle, bit for bit, at the sizes where they can go wrong: particle counts
around a warp, caps inside and just past the first pair, every particle
leaving the grid, random parts whose scaled form is not exact, both instances
(with and without the look at a cell's maximum) on both footprint paths."""
import numpy as np
import pytest
import torch

import oracle
import paper_2506_23364_gb300 as awo
from paper_2506_23364_gb300 import inputs

pytestmark = pytest.mark.gpu

LANES = 194_560  # 152 SMs x 1280: the look pays from 32 particles a lane, or 7 a cell of the grid


def _check(dem, cs, cells, kw):
    H, W = dem.shape
    ov = awo.Overlay(W, H, cs, quantised=False, want_normals=False, want_mask=False)
    ov.load_dem(dem)
    ov.simulate(awo.SimParams.make(**kw), cells=torch.from_numpy(cells.astype(np.int32)).cuda(), n_cells=cells.size)
    torch.cuda.synchronize()
    c64, maxe, st = oracle.simulate_threaded(dem, cs, cells, oracle.SimParams(**kw))
    got = ov.stats_dict()
    assert {k: got[k] for k in st} == st
    assert np.array_equal(ov.count.cpu().numpy().view(np.uint32), oracle.counts_u32(c64))
    assert np.array_equal(ov.maxe.cpu().numpy(), maxe)
    return st


def _slope(h=61, w=83):
    return np.ascontiguousarray(inputs.tiny_dem()[60:60 + h, 90:90 + w])


@pytest.mark.parametrize("cap", [1, 2, 3, 64])
@pytest.mark.parametrize("n", [1, 5, 31, 32, 33, 70])
def test_counts_around_a_warp(n, cap):
    dem = _slope()
    cells = np.arange(7, dem.size, 29).astype(np.uint32)
    _check(dem, 10.0, cells, dict(traj_per_cell=n, max_steps=cap, seed=n + cap))


@pytest.mark.parametrize("kw", [
    dict(randomness=0.0), dict(randomness=2.0 ** -110), dict(randomness=2.0 ** -103), dict(randomness=2.0 ** 127),
    dict(randomness=0.5, persistence=0.0), dict(persistence=1.0), dict(step_scale=0.37, drag_k=2e-3)])
def test_random_parts_and_options(kw):
    dem = _slope()
    dem[20:30, 30:50] = dem[25, 40]  # flat ground inside the slope
    cells = np.arange(0, dem.size, 11).astype(np.uint32)
    _check(dem, 10.0, cells, dict(dict(traj_per_cell=9, max_steps=300, seed=3), **kw))


@pytest.mark.parametrize("shape", [(1, 40), (40, 1), (2, 2), (33, 31)])
def test_particles_leave_small_grids(shape):
    y, x = np.mgrid[0:shape[0], 0:shape[1]]
    dem = (1000.0 - 9.0 * (x + y)).astype(np.float32)
    cells = np.arange(dem.size, dtype=np.uint32)
    st = _check(dem, 10.0, cells, dict(traj_per_cell=40, max_steps=200, seed=1))  # 40 a cell: the look is taken
    assert st["n_exited"] > 0


@pytest.mark.parametrize("side", [1024, 1022])  # texture gathers, loads
@pytest.mark.parametrize("per_lane", [1, 33])
def test_large_lists_with_and_without_the_look(side, per_lane):
    dem = inputs.fbm(side, 0.8, seed=5, relief=1700.0).astype(np.float32)
    _, t2, _ = oracle.normals(dem, 10.0)
    _, cells = oracle.release(t2, 43.0, 45.0)
    n = -(-per_lane * LANES // cells.size)
    _check(dem, 10.0, cells, dict(traj_per_cell=n, max_steps=60, seed=2))


@pytest.mark.parametrize("kw", [{}, dict(step_scale=0.5)])
@pytest.mark.parametrize("times", [0.85, 0.99, 1.0, 1.01, 1.09, 1.17])
def test_one_instance_runs_on_either_side_of_the_line(times, kw):
    """Particle counts around 32 a lane (16 at half steps), few for the grid."""
    side = 1024
    y, x = np.mgrid[0:side, 0:side]
    dem = (9000.0 - 4.0 * x - 3.0 * y).astype(np.float32)
    total = int(times * 32 * LANES * kw.get("step_scale", 1.0))
    n = 2048
    cells = np.arange(3000, 3000 + 17 * (total // n), 17).astype(np.uint32)
    _check(dem, 10.0, cells, dict(traj_per_cell=n, max_steps=1, seed=8, mu=0.2, **kw))
