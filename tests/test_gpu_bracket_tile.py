"""Training rows and learned launches of the rank bracket take the same tile, and the rows' features are
what they are documented to be."""
import numpy as np
import pytest

import datagen
import oracle
from helpers import assert_bit_exact, to_device, to_host

pytestmark = pytest.mark.gpu
CODE = {"u8": 0, "u16": 1, "f32": 2}


def collect(img, dtype, k):
    import torch
    import paper_2505_22938_gb300 as fim
    h, w = img.shape
    store, _ = to_device(img)
    out = torch.empty_like(store)
    rows = torch.zeros((4096, 42), dtype=torch.float32, device="cuda")
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    fim.fim_collect_seed_samples(store.data_ptr(), out.data_ptr(), w, h, store.stride(0) * store.element_size(),
                                 CODE[dtype], k, rows.data_ptr(), 4096, count.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert fim.fim_sync_status() == 0
    return rows[:int(count.item())].cpu().numpy(), to_host(out)


@pytest.mark.parametrize("dtype", ["u8", "u16", "f32"])
def test_r64_rows_and_launches_share_a_tile(dtype):
    import torch
    import paper_2505_22938_gb300 as fim
    h, w = 300, 200
    img = datagen.image_for(dtype, 64, h, w)
    k = fim.fim_create_kernel_circle(64)
    rows, out = collect(img, dtype, k)
    exp = oracle.median_filter(img, oracle.disk_offsets(64))
    assert_bit_exact(out, exp, "training launch")
    seeds = 16 * -(-w // 64) * -(-h // 128)  # 8 bands of 2 seeds in each 64 x 128 tile
    assert len(rows) == seeds
    store, _ = to_device(img)
    out = torch.empty_like(store)
    stats = torch.zeros(5, dtype=torch.int64, device="cuda")
    fim.fim_median_learned(store.data_ptr(), out.data_ptr(), w, h, store.stride(0) * store.element_size(), CODE[dtype],
                           k, fim.Model.create(seed=3), torch.cuda.current_stream().cuda_stream, stats.data_ptr())
    torch.cuda.synchronize()
    assert fim.fim_sync_status() == 0
    assert_bit_exact(to_host(out), exp, "learned launch")
    assert int(stats[0]) == seeds


def test_rank_features_of_a_large_footprint():
    """r = 48: a 64 x 128 tile's footprint has 33644 pixels, more than 15 bits of ranks. The last nine
    features are the ranks, over the footprint's size, of the 3 x 3 pixels at the seed's centre."""
    import paper_2505_22938_gb300 as fim
    r, h, w = 48, 128, 64  # one tile
    img = np.random.default_rng(48).permutation(h * w).reshape(h, w).astype(np.float32)
    rows, _ = collect(img, "f32", fim.fim_create_kernel_circle(r))
    half = [int(np.floor(np.sqrt(r * r - dy * dy))) for dy in range(-r, r + 1)]
    values = []
    for y in range(-r, h + r):  # row y of the footprint: the widest kernel row that reaches it
        reach = max(half[y - t + r] for t in range(h) if abs(y - t) <= r)
        xs = np.clip(np.arange(-reach, w + reach), 0, w - 1)
        values.append(img[min(max(y, 0), h - 1), xs])
    values = np.sort(np.concatenate(values))
    n = len(values)
    assert n == 33644
    want = {}
    for band in range(8):
        for s in (16, 48):
            box = img[16 * band + 7:16 * band + 10, s - 1:s + 2].ravel()
            want[(band, s)] = (np.searchsorted(values, box, "left"), np.searchsorted(values, box, "right"))
    assert len(rows) == len(want)
    for row in rows:
        ranks = np.rint(row[32:41].astype(np.float64) * n)
        assert any(np.all((lo <= ranks) & (ranks < hi)) for lo, hi in want.values()), ranks
