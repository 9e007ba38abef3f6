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


@pytest.mark.parametrize("tan2_off,mask_off", [(0, 0), (1, 0), (0, 3)])
@pytest.mark.parametrize("r,W,H", [(1, 2048, 4), (1, 4096, 2), (2, 1024, 5), (2, 3072, 2)])
def test_texture_row_groups_ends_and_offsets(r, W, H, tan2_off, mask_off):
    """Runs at the row ends, the vector and scalar loads and stores, values that no weight may touch."""
    rng = np.random.default_rng(W + H)
    t2 = (rng.random((H, W)) * 2.0).astype(np.float32)
    vals = np.array([0.0, 1e-42, 3e38, np.inf, np.nan, 1.0], np.float32)
    for col in (0, 1, 2, W - 3, W - 2, W - 1, 7, 8, W // 2):
        t2[:, col] = vals[rng.integers(0, vals.size, H)]
    buf = torch.zeros(W * H + tan2_off, device="cuda")
    d_t2 = buf[tan2_off:]
    d_t2.copy_(torch.from_numpy(t2.ravel()))
    g = awo.grid(W, H, 10.0)
    wr, hr = awo.awo_release_texture_dims(g, r)
    mask = torch.full((wr * hr + mask_off,), 9, dtype=torch.uint8, device="cuda")
    texels = torch.zeros(wr * hr, dtype=torch.int32, device="cuda")
    n = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(awo.awo_release_texture_workspace_bytes(g, r), dtype=torch.uint8, device="cuda")
    awo.awo_release_texture(d_t2, g, r, 30.0, 50.0, mask[mask_off:], texels, n, ws)
    torch.cuda.synchronize()
    want_mask, want = oracle.release_texture(t2, r, 30.0, 50.0)
    assert np.array_equal(mask[mask_off:].cpu().numpy(), np.asarray(want_mask).ravel())
    assert np.array_equal(texels[:int(n)].cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("size", [16, 4096, 16384, 16387, 40000])
def test_mask_bytes_of_any_value(size):
    rng = np.random.default_rng(size)
    m = np.where(rng.random(size) < 0.5, 0, rng.choice([1, 2, 0x7f, 0x80, 0xff], size)).astype(np.uint8)
    g = awo.grid(size, 1, 10.0)
    cells = torch.zeros(size, dtype=torch.int32, device="cuda")
    n = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(awo.awo_release_workspace_bytes(g), dtype=torch.uint8, device="cuda")
    awo.awo_release_from_mask(torch.from_numpy(m).cuda(), g, cells, n, ws)
    torch.cuda.synchronize()
    assert np.array_equal(cells[:int(n)].cpu().numpy(), np.flatnonzero(m))


@pytest.mark.parametrize("W,H", [(1, 5000), (3, 3000), (83, 61), (1023, 9), (4097, 3), (4100, 1), (2, 2049), (1799, 1391)])
@pytest.mark.parametrize("off", [0, 1])
def test_single_cells_of_any_width_and_offset(W, H, off):
    """The pass for ragged rows and unaligned buffers, alone and with the release, on values for every form."""
    dem = _dem(W, H, True)
    n = W * H
    nrm, t2, deg = oracle.normals(dem, 10.0)
    _, cells = oracle.release(t2, 20.0, 60.0)
    d_h = torch.zeros(n + off, device="cuda")[off:]
    d_h.copy_(torch.from_numpy(dem.ravel()))
    g = awo.grid(W, H, 10.0)
    out = [torch.full((k * n + off,), 7.0, device="cuda")[off:] for k in (3, 1)]
    awo.awo_normals(d_h, g, out[0], out[1], None)
    mask = torch.full((n + off,), 9, dtype=torch.uint8, device="cuda")[off:]
    lst, cnt = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(awo.awo_release_workspace_bytes(g), dtype=torch.uint8, device="cuda")
    both = [torch.full((k * n + off,), 7.0, device="cuda")[off:] for k in (3, 1)]
    awo.awo_terrain(d_h, g, None, d_h, both[0], both[1], None, 20.0, 60.0, mask, lst, cnt, ws)
    torch.cuda.synchronize()
    for a, b in (out, both):
        assert np.array_equal(a.cpu().numpy().view(np.uint32), np.ascontiguousarray(nrm).ravel().view(np.uint32))
        assert np.array_equal(b.cpu().numpy().view(np.uint32), t2.ravel().view(np.uint32))
    assert np.array_equal(lst[:int(cnt)].cpu().numpy().view(np.uint32), cells)
    assert np.array_equal(np.flatnonzero(mask.cpu().numpy()), cells)


@pytest.mark.parametrize("r", [-1, -2, -3])
@pytest.mark.parametrize("W,H", [(8, 8), (17, 700), (1030, 77), (2047, 33)])
def test_coarse_texture_texels(r, W, H):
    rng = np.random.default_rng(W * 7 + H)
    t2 = (rng.random((H, W)) * 2.0).astype(np.float32)
    t2.ravel()[rng.integers(0, W * H, W * H // 20)] = np.inf
    t2.ravel()[rng.integers(0, W * H, W * H // 20)] = np.nan
    g = awo.grid(W, H, 10.0)
    wr, hr = awo.awo_release_texture_dims(g, r)
    mask = torch.full((wr * hr,), 9, dtype=torch.uint8, device="cuda")
    texels, n = torch.zeros(wr * hr, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(awo.awo_release_texture_workspace_bytes(g, r), dtype=torch.uint8, device="cuda")
    awo.awo_release_texture(torch.from_numpy(t2).cuda().view(-1), g, r, 30.0, 50.0, mask, texels, n, ws)
    torch.cuda.synchronize()
    want_mask, want = oracle.release_texture(t2, r, 30.0, 50.0)
    assert np.array_equal(mask.cpu().numpy(), np.asarray(want_mask).ravel())
    assert np.array_equal(texels[:int(n)].cpu().numpy().view(np.uint32), want)
