"""A disk whose tile's box has 256 rows (r = 64 on 128-row tiles) runs on the span membership test."""
import numpy as np
import pytest

import datagen
import oracle
from helpers import assert_bit_exact, fim_kernel, gpu_filter, to_device, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["u8", "u16", "f32"])
def test_r64_on_128_rows(dtype, monkeypatch):
    import torch
    import paper_2505_22938_gb300 as fim
    monkeypatch.setenv("FIM_TILE", "64,128,8,2")
    img = datagen.image_for(dtype, 64, 270, 231)
    off = oracle.disk_offsets(64)
    k = fim_kernel("circle", 64)
    exp = oracle.median_filter(img, off)
    assert_bit_exact(gpu_filter(img, k), exp, dtype)
    store, _ = to_device(img)
    low, mid = fim.percentiles(store, k, (10, 50))
    small, large = fim.median_radii(store, [fim_kernel("circle", 20), k])
    torch.cuda.synchronize()
    assert fim.fim_sync_status() == 0
    assert_bit_exact(to_host(low), oracle.median_filter(img, off, rank=oracle.percentile_rank(len(off), 10)), "p10")
    assert_bit_exact(to_host(mid), exp, "p50")
    assert_bit_exact(to_host(large), exp, "radii 64")
    assert_bit_exact(to_host(small), oracle.median_filter(img, oracle.disk_offsets(20)), "radii 20")
