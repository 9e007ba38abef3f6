"""The caller's statistics hold the last call's until a call's own are
complete, then these, at any alignment."""
import numpy as np
import pytest
import torch

import paper_2506_23364_gb300 as awo
from paper_2506_23364_gb300 import inputs

pytestmark = pytest.mark.gpu


def _overlay():
    dem = inputs.tiny_dem()
    ov = awo.Overlay(dem.shape[1], dem.shape[0], 10.0, quantised=False)
    ov.load_dem(dem)
    ov.terrain(30.0, 45.0)
    return ov


def _watch(stats, host, stream, done):
    """Distinct values of `stats`, read on a stream of its own until `done` is reached."""
    seen = set()
    with torch.cuda.stream(stream):
        while True:
            ended = done.query()
            host.copy_(stats, non_blocking=True)
            stream.synchronize()
            seen.add(tuple(host.tolist()))
            if ended:
                return seen


@pytest.mark.parametrize("batched", [False, True])
def test_no_partial_sums_in_the_callers_buffer(batched):
    ov = _overlay()
    p = awo.SimParams.make(traj_per_cell=512, max_steps=1000, seed=3, flags=1)  # tens of milliseconds
    reqs = (awo.SimRequest * 1)(awo.sim_request(ov.h, ov.g, ov.cells, ov.n_rel, ov.n_tex, p, ov.count, ov.maxe))
    ws = torch.empty(awo.awo_simulate_batched_workspace_bytes(reqs), dtype=torch.uint8, device="cuda")
    call = (lambda: awo.awo_simulate_batched(reqs, ws, None, ov.stats)) if batched else (lambda: ov.simulate(p))
    call()
    torch.cuda.synchronize()
    final = tuple(ov.stats.cpu().tolist())
    before = (11, 22, 33, 44, 55, 66)
    ov.stats.copy_(torch.tensor(before))
    # made before the call: page-locked memory is only had when the GPU is idle
    host, stream, done = torch.empty(6, dtype=torch.int64, pin_memory=True), torch.cuda.Stream(), torch.cuda.Event()
    done.record()
    _watch(ov.stats, host, stream, done)
    call()
    done.record()
    seen = _watch(ov.stats, host, stream, done)
    assert seen <= {before, final} and final in seen, seen
    assert before in seen  # the call was still running


@pytest.mark.parametrize("off", [0, 1, 4, 7])
@pytest.mark.parametrize("n", [1, 5])
def test_any_alignment(n, off):
    ov = _overlay()
    ps = [awo.SimParams.make(traj_per_cell=2 + i, max_steps=40, seed=i, flags=1) for i in range(n)]
    want = []
    outs = [(torch.empty_like(ov.count), torch.empty_like(ov.maxe)) for _ in ps]
    for p in ps:
        ov.simulate(p)
        want.append(ov.stats.clone())
    reqs = (awo.SimRequest * n)(*[awo.sim_request(ov.h, ov.g, ov.cells, ov.n_rel, ov.n_tex, p, c, e)
                                  for p, (c, e) in zip(ps, outs)])
    ws = torch.empty(awo.awo_simulate_batched_workspace_bytes(reqs), dtype=torch.uint8, device="cuda")
    buf = torch.full((48 * n + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    st = awo.lib().awo_simulate_batched(reqs, n, None, buf.data_ptr() + off, ws.data_ptr(), ws.numel(),
                                        torch.cuda.current_stream().cuda_stream)
    assert st == awo.AWO_OK
    torch.cuda.synchronize()
    got = buf.cpu().numpy()
    assert np.array_equal(got[off:off + 48 * n].copy().view(np.int64).reshape(n, 6), torch.stack(want).cpu().numpy())
    assert (got[:off] == 0xA5).all() and (got[off + 48 * n:] == 0xA5).all()
