"""Mipmap chains deeper than one fused launch and the snow pass on planes that
are not 16-byte aligned, against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import paper_2506_23364_gb300 as awo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,levels", [(700, 521, 11), (129, 4097, 14), (64, 64, 8), (1, 3000, 16), (256, 130, 7)])
def test_deep_mipmap(W, H, levels):
    rng = np.random.default_rng(W + H)
    count = rng.integers(0, 2 ** 32, (H, W), dtype=np.uint64).astype(np.uint32)  # saturates within a few levels
    count[rng.random((H, W)) < 0.9] = 3
    maxe = (rng.random((H, W)) * 400).astype(np.float32)
    g = awo.grid(W, H, 10.0)
    shapes = awo.lod_shapes(g, levels)[1:]
    vel = torch.empty((H, W), device="cuda")
    cl = [torch.empty(s, dtype=torch.int32, device="cuda") for s in shapes]
    vl = [torch.empty(s, dtype=torch.float32, device="cuda") for s in shapes]
    awo.awo_finalize_lod(torch.from_numpy(maxe).cuda(), torch.from_numpy(count.view(np.int32)).cuda(), g, 9.81, levels,
                         vel, cl, vl)
    want_vel = oracle.finalize(maxe, 9.81)
    want_c, want_v = oracle.lod(count, want_vel, levels)
    assert np.array_equal(vel.cpu().numpy(), want_vel)
    for l in range(1, levels):
        assert np.array_equal(cl[l - 1].cpu().numpy().view(np.uint32), want_c[l]), l
        assert np.array_equal(vl[l - 1].cpu().numpy(), want_v[l]), l


@pytest.mark.parametrize("off_h", [0, 1, 2])
@pytest.mark.parametrize("off_nz", [0, 1, 2, 3])
@pytest.mark.parametrize("W,H", [(37, 11), (1, 3), (64, 33)])
def test_snow_unaligned_inputs(W, H, off_h, off_nz):
    n = W * H
    rng = np.random.default_rng(n + off_nz)
    h = (rng.random((H, W)) * 1200 + 900).astype(np.float32)
    nz = (rng.random((H, W)) * 0.4 + 0.6).astype(np.float32)
    hb, zb = torch.empty(n + 4, device="cuda"), torch.empty(n + 4, device="cuda")
    ht, zt = hb[off_h:off_h + n], zb[off_nz:off_nz + n]
    ht.copy_(torch.from_numpy(h.ravel()))
    zt.copy_(torch.from_numpy(nz.ravel()))
    alpha = torch.empty((H, W), device="cuda")
    rgba = torch.empty((H, W, 4), dtype=torch.uint8, device="cuda")
    awo.awo_snow_cover(ht, zt, awo.grid(W, H, 10.0), awo.SnowParams(1500.0, 300.0, 36.0, 4.0), alpha, rgba)
    want_a, want_rgba = oracle.snow_cover(h, nz, 1500.0, 300.0, 36.0, 4.0)
    assert np.array_equal(alpha.cpu().numpy(), np.asarray(want_a).reshape(H, W))
    assert np.array_equal(rgba.cpu().numpy(), np.asarray(want_rgba).reshape(H, W, 4))


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("off_in,off_out", [(0, 0), (2, 0), (1, 0), (0, 1), (0, 2)])
@pytest.mark.parametrize("W,H", [(4, 1), (4, 130), (68, 5), (132, 33), (66, 7), (67, 64), (128, 65)])
def test_mipmap_widths_and_alignments(W, H, off_in, off_out, in_place):
    """Rows of whole groups of four, of pairs and odd ones; inputs and level 1 off 16 and 8 bytes."""
    n, levels = W * H, 4
    rng = np.random.default_rng(n + off_in)
    count = rng.integers(0, 2 ** 32, (H, W), dtype=np.uint64).astype(np.uint32)
    count[rng.random((H, W)) < 0.7] = 5
    maxe = (rng.random((H, W)) * 400).astype(np.float32)
    g = awo.grid(W, H, 10.0)

    def buf(size, dtype, off):
        return torch.zeros(size + off, dtype=dtype, device="cuda")[off:]

    c0, e0 = buf(n, torch.int32, off_in), buf(n, torch.float32, off_in)
    c0.copy_(torch.from_numpy(count.view(np.int32).ravel()))
    e0.copy_(torch.from_numpy(maxe.ravel()))
    vel = e0 if in_place else buf(n, torch.float32, off_in)
    sizes = [a * b for a, b in awo.lod_shapes(g, levels)[1:]]
    cl = [buf(s, torch.int32, off_out) for s in sizes]
    vl = [buf(s, torch.float32, off_out) for s in sizes]
    awo.awo_finalize_lod(e0, c0, g, 9.81, levels, vel, cl, vl)
    want_vel = oracle.finalize(maxe, 9.81)
    want_c, want_v = oracle.lod(count, want_vel, levels)
    assert np.array_equal(vel.cpu().numpy(), want_vel.ravel())
    cl2, vl2 = [torch.zeros_like(t) for t in cl], [torch.zeros_like(t) for t in vl]
    awo.awo_overlay_lod(c0, vel, g, levels, cl2, vl2)
    for l in range(1, levels):
        for c, v in ((cl, vl), (cl2, vl2)):
            assert np.array_equal(c[l - 1].cpu().numpy().view(np.uint32), want_c[l].ravel()), l
            assert np.array_equal(v[l - 1].cpu().numpy(), want_v[l].ravel()), l


@pytest.mark.parametrize("hit", [0.0, 0.02, 0.5, 1.0])
@pytest.mark.parametrize("count_min,alpha", [(0, 0.7), (1, 0.7), (1, 0.0), (3, 1.0), (2 ** 32 - 1, 0.5)])
@pytest.mark.parametrize("n_stops", [2, 5, 16])
def test_compose_groups_without_hits(n_stops, count_min, alpha, hit):
    """Groups below count_min, among hit ones and alone, over a base and in place of it; several groups a thread."""
    W, H = 1283, 977  # more groups than one sweep of the smallest grid, and a tail
    rng = np.random.default_rng(n_stops + int(100 * hit))
    value = (rng.random((H, W)) * 80 - 10).astype(np.float32)
    at = rng.integers(0, W * H, 2000)
    value.ravel()[at] = np.array([np.nan, np.inf, -np.inf, -0.0], np.float32)[at % 4]
    count = rng.integers(0, 6, (H, W)).astype(np.uint32)
    count[np.repeat(rng.random(W * H // 7 + 1), 7)[:W * H].reshape(H, W) >= hit] = 0  # runs that straddle groups
    base = rng.integers(0, 256, (H, W, 4)).astype(np.uint8)
    x = np.linspace(0.0, 60.0, n_stops)
    stops = [(float(x[k]), tuple(int(c) for c in rng.integers(0, 256, 3))) for k in range(n_stops)]
    cm = awo.Colormap.make(stops, alpha=alpha, count_min=count_min)
    g = awo.grid(W, H, 10.0)
    v, c = torch.from_numpy(value).cuda(), torch.from_numpy(count.view(np.int32)).cuda()
    b = torch.from_numpy(base).cuda()
    out = torch.empty_like(b)
    awo.awo_compose(v, c, g, cm, b, out)
    bare = torch.empty_like(b)
    awo.awo_compose(v, c, g, cm, None, bare)
    awo.awo_compose(v, c, g, cm, b, b)
    want = oracle.compose(value, count, stops, alpha, count_min, base)
    assert np.array_equal(out.cpu().numpy(), want)
    assert np.array_equal(b.cpu().numpy(), want)
    assert np.array_equal(bare.cpu().numpy(), oracle.compose(value, count, stops, alpha, count_min))
