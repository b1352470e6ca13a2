"""Several percentiles of disks whose tile footprint exceeds 65535 pixels for some tile shapes, on an
image of several waves of tiles, at sampled pixels."""
import numpy as np
import pytest

import datagen
import oracle
from helpers import to_device, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,r,pcts", [("u16", 120, (25, 50, 75)), ("u8", 128, (25, 50, 75)),
                                          ("f32", 114, (25, 50, 75)), ("u16", 100, (5, 50, 95)),
                                          ("u16", 128, (0, 50, 100))])
def test_sampled_pixels(dtype, r, pcts):
    import torch
    import paper_2505_22938_gb300 as fim
    h, w = 1500, 1701
    img = datagen.image_for(dtype, 31, h, w)
    store, _ = to_device(img)
    outs = fim.percentiles(store, fim.fim_create_kernel_circle(r), pcts)
    torch.cuda.synchronize()
    assert fim.fim_sync_status() == 0
    rng = np.random.default_rng(r)
    ys = np.concatenate([rng.integers(0, h, 300), [0, 0, h - 1, h - 1]])
    xs = np.concatenate([rng.integers(0, w, 300), [0, w - 1, 0, w - 1]])
    off = oracle.disk_offsets(r)
    for pct, out in zip(pcts, outs):
        exp = oracle.median_points(img, off, xs, ys, rank=oracle.percentile_rank(len(off), pct))
        got = to_host(out)[ys, xs]
        assert np.array_equal(got.view(np.uint8), exp.view(np.uint8)), pct
