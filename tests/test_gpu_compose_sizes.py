"""Compose on either side of the sizes at which its launch changes (groups of
four texels per thread of the GPU), with and without a base, against the
oracle, byte for byte; a buffer off 16 bytes takes single texels."""
import numpy as np
import pytest
import torch

import oracle
import paper_2506_23364_gb300 as awo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("rows_less", [0, 1])
@pytest.mark.parametrize("groups_a_thread", [24, 40, 64])
def test_compose_sizes(groups_a_thread, rows_less, off):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    W, H = sms * (1 if off else 4), 256 * groups_a_thread - rows_less
    n = W * H
    rng = np.random.default_rng(groups_a_thread)
    value = (rng.random(n, dtype=np.float32) * 80 - 10)
    count = rng.integers(0, 3, n).astype(np.uint32)
    count[: n // 2] = 0  # half without a hit
    base = rng.integers(0, 256, (n, 4), dtype=np.uint8)
    stops = [(0.0, (40, 40, 200)), (10.0, (0, 190, 230)), (25.0, (40, 200, 60)), (45.0, (250, 220, 0)), (70.0, (220, 30, 30))]
    cm = awo.Colormap.make(stops, alpha=0.7, count_min=1)
    v = torch.empty(n + off, device="cuda")[off:]
    v.copy_(torch.from_numpy(value))
    c, b = torch.from_numpy(count.view(np.int32)).cuda(), torch.from_numpy(base).cuda()
    g = awo.grid(W, H, 10.0)
    out = torch.empty_like(b)
    for bt, bn in ((b, base.reshape(H, W, 4)), (None, None)):
        awo.awo_compose(v, c, g, cm, bt, out)
        want = oracle.compose(value.reshape(H, W), count.reshape(H, W), stops, 0.7, 1, *([bn] if bn is not None else []))
        assert np.array_equal(out.cpu().numpy(), np.asarray(want).reshape(n, 4))
