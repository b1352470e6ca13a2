"""The sort by equalised codes on tiles that take it: images with several tiles whose whole box lies
inside (test_planner.py checks that every plan here sorts by codes and has such tiles), bit for bit
against the oracle, on value distributions that decide how many pixels share a code and how many of
those lie in one window.
"""
import numpy as np
import pytest

import datagen
import oracle
from helpers import assert_bit_exact, fim_kernel, gpu_filter, oracle_offsets, to_device, to_host
from test_gpu_sort_codes import image as basic_image

pytestmark = pytest.mark.gpu

H, W = 330, 300
HEX = ("polygon", oracle.regular_polygon_vertices(6, 30.0))
# (dtype, kernel, tile): CTAs of 256, 512 and 1024 threads
PLANS = [("f32", ("circle", 15), "64,64,2,2"), ("f32", ("circle", 24), "64,64,4,2"), ("f32", ("circle", 20), "64,64,8,2"),
         ("f32", ("circle", 33), "64,128,8,2"), ("f32", ("circle", 64), "64,64,8,2"), ("f32", HEX, "64,64,8,2"),
         ("u16", ("circle", 24), "64,64,4,2"), ("u16", ("circle", 28), "64,64,4,2"),
         ("u16", ("ellipse", 40, 22), "64,64,4,2")]
KINDS = ["photo", "constant", "narrow", "levels", "impulses", "ends", "mixed", "uniform", "clusters", "one group"]


def image(kind, dtype):
    rng = np.random.default_rng(23)
    if kind == "uniform":  # codes of one to four pixels and a few more
        a = rng.random((H, W)) * 60000.0
    elif kind == "clusters":  # about five pixels within a few units in the last place: one code, different keys
        a = rng.integers(1, 3000, (H, W)) * (19.0 if dtype == "u16" else 1e3) + rng.integers(0, 3, (H, W)) * (1 if dtype == "u16" else 0.25)
    elif kind == "one group":  # smooth, but for 40 pixels of neighbouring values in every tile: the exact sort
        a = datagen.image_for("f32", 5, H, W).astype(np.float64)
        if dtype == "u16":
            a = 20000 + 300 * a
        a[::8, ::8] = (5000.0 if dtype == "u16" else 1e6) + rng.integers(0, 2, a[::8, ::8].shape) * (1 if dtype == "u16" else 0.0625)
    elif kind == "ends" and dtype == "u16":
        a = rng.choice([0, 1, 2, 65533, 65534, 65535], size=(H, W))
    elif kind == "mixed" and dtype == "u16":  # dense and spread values
        a = np.where(rng.random((H, W)) < 0.5, 30000 + rng.integers(0, 40, (H, W)), rng.integers(0, 65536, (H, W)))
    else:
        return basic_image(kind, dtype, H, W)
    return a.clip(-3e38, 3e38).astype({"u16": np.uint16, "f32": np.float32}[dtype])


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("dtype,spec,tile", PLANS)
def test_median(dtype, spec, tile, kind, monkeypatch):
    monkeypatch.setenv("FIM_TILE", tile)
    img = image(kind, dtype)
    assert_bit_exact(gpu_filter(img, fim_kernel(*spec)), oracle.median_filter(img, oracle_offsets(*spec)), kind)


@pytest.mark.parametrize("kind", ["photo", "clusters", "mixed"])
@pytest.mark.parametrize("dtype,spec,tile", [PLANS[1], PLANS[2], PLANS[5], PLANS[6]])
def test_percentiles_map_and_batch(dtype, spec, tile, kind, monkeypatch):
    import torch
    import paper_2505_22938_gb300 as fim
    monkeypatch.setenv("FIM_TILE", tile)
    img = image(kind, dtype)
    off, k = oracle_offsets(*spec), fim_kernel(*spec)
    store, _ = to_device(img)
    got = fim.percentiles(store, k, (0, 25, 50, 100))
    pct = np.tile(np.linspace(0.0, 100.0, W, dtype=np.float32), (H, 1))
    mapped = fim.percentile_map(store, k, torch.from_numpy(pct).cuda())
    out = [torch.zeros_like(store) for _ in range(2)]
    jobs = [fim.make_job(store.data_ptr(), o.data_ptr(), W, H, W * store.element_size(), fim.DTYPES[dtype], k) for o in out]
    torch.cuda.synchronize()
    batch = fim.fim_batch_create(jobs, [k])
    batch.run(torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert fim.fim_sync_status() == 0
    for p, o in zip((0, 25, 50, 100), got):
        assert_bit_exact(to_host(o), oracle.median_filter(img, off, rank=oracle.percentile_rank(len(off), p)), f"{kind} p{p}")
    ranks = oracle.percentile_rank_map(len(off), pct)
    assert_bit_exact(to_host(mapped), oracle.rank_map_filter(img, off, ranks), f"{kind} map")
    exp = oracle.median_filter(img, off)
    for o in out:
        assert_bit_exact(to_host(o), exp, f"{kind} batch")
