"""Normals and release in one pass against the oracle, bit for bit: tile edges
and remainders, rows that are and are not 16-byte aligned, values outside the
range of the fast divisions (the general form of a run), signed zeros; and the
row groups of the release texture on few rows."""
import numpy as np
import pytest
import torch

import oracle
import paper_2506_23364_gb300 as awo

pytestmark = pytest.mark.gpu

SHAPES = [(4, 1), (4, 1025), (8, 513), (12, 700), (1024, 4), (1028, 9), (4096, 3), (8192, 2), (13, 50), (1, 7)]  # W, H


def _dem(W, H, special):
    rng = np.random.default_rng(W * 1000 + H)
    h = (rng.random((H, W)) * 30.0).astype(np.float32)
    h.ravel()[rng.integers(0, W * H, W * H // 3)] = 7.0  # equal neighbours: zero differences
    if special:
        vals = np.array([-0.0, 0.0, 1e-40, -1e-30, 1e-20, 3e25, -1e20, 1e12], np.float32)
        at = rng.integers(0, W * H, max(1, W * H // 5))
        h.ravel()[at] = vals[rng.integers(0, vals.size, at.size)]
    return h


@pytest.mark.parametrize("special", [False, True])
@pytest.mark.parametrize("W,H", SHAPES)
def test_normals_release_fp32(W, H, special):
    dem = _dem(W, H, special)
    ov = awo.Overlay(W, H, 10.0, quantised=False, want_slope=True)
    ov.load_dem(dem)
    ov.terrain(20.0, 60.0)
    torch.cuda.synchronize()
    nrm, t2, _ = oracle.normals(dem, 10.0)
    mask, cells = oracle.release(t2, 20.0, 60.0)
    assert np.array_equal(ov.tan2.cpu().numpy().view(np.uint32), t2.view(np.uint32))
    assert np.array_equal(ov.normal.cpu().numpy().view(np.uint32), np.asarray(nrm).view(np.uint32))
    assert np.array_equal(ov.mask.cpu().numpy().ravel(), np.asarray(mask).ravel())
    assert np.array_equal(ov.release_cells(), cells)


@pytest.mark.parametrize("want_mask", [True, False])
@pytest.mark.parametrize("W,H", SHAPES)
def test_normals_release_u16(W, H, want_mask):
    rng = np.random.default_rng(W + H)
    q = rng.integers(0, 400, (H, W)).astype(np.uint16)
    ov = awo.Overlay(W, H, 10.0, quantised=True, want_mask=want_mask, want_normals=False)
    ov.load_dem(q)
    ov.terrain(30.0, 55.0)
    torch.cuda.synchronize()
    h = oracle.decode_u16(q, 0.1)
    _, t2, _ = oracle.normals(h, 10.0)
    _, cells = oracle.release(t2, 30.0, 55.0)
    assert np.array_equal(ov.h.cpu().numpy(), h)
    assert np.array_equal(ov.tan2.cpu().numpy().view(np.uint32), t2.view(np.uint32))
    assert np.array_equal(ov.release_cells(), cells)


@pytest.mark.parametrize("r,W", [(1, 2048), (2, 1024)])
@pytest.mark.parametrize("H", [2, 3, 6])
def test_texture_row_groups_on_few_rows(r, W, H):
    dem = _dem(W, H, False)
    ov = awo.Overlay(W, H, 10.0, quantised=False, release_log2=r)
    ov.load_dem(dem)
    ov.terrain(20.0, 60.0)
    torch.cuda.synchronize()
    _, t2, _ = oracle.normals(dem, 10.0)
    mask, texels = oracle.release_texture(t2, r, 20.0, 60.0)
    assert np.array_equal(ov.mask.cpu().numpy().ravel(), np.asarray(mask).ravel())
    assert np.array_equal(ov.release_cells(), texels)
