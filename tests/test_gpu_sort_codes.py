"""Parity of the sort by equalised codes and of the radix sort (16-bit data in smaller CTAs) with
the oracle, bit for bit (the output is a selected input value), on the value distributions
that decide which pixels share a code: smooth data, values that differ in their last bits only,
few distinct values, constants, impulses, both ends of the float order, and a mixture that must
fall back to the exact sort. Sizes span several tiles of each shape with ragged edges.
"""
import numpy as np
import pytest

import datagen
import oracle
from helpers import assert_bit_exact, fim_kernel, gpu_filter, oracle_offsets

pytestmark = pytest.mark.gpu


def image(kind, dtype, h, w):
    rng = np.random.default_rng(17)
    if kind == "photo":
        return datagen.image_for(dtype, 71, h, w)
    if kind == "constant":
        a = np.full((h, w), 1000.25)
    elif kind == "narrow":  # a ramp of a few thousand neighbouring values
        a = 1000.0 + (np.arange(h)[:, None] * 3 + np.arange(w)[None, :] % 7) / 16384.0
        if dtype == "u16":
            a = 1000 + (np.arange(h)[:, None] // 9 + np.arange(w)[None, :] % 3)
    elif kind == "levels":  # few distinct values
        a = rng.integers(0, 12, (h, w)) / 4.0 + 1.0
        if dtype == "u16":
            a = a * 64
    elif kind == "impulses":
        a = rng.normal(size=(h, w)) * 100 + 20000
        a[rng.random((h, w)) < 0.2] = 65535
        a[rng.random((h, w)) < 0.2] = 0
    elif kind == "ends":
        a = rng.choice([0.0, -0.0, 1e-45, -1e-45, 3e38, -3e38, np.inf, -np.inf, 1.0, -1.0], size=(h, w))
    elif kind == "mixed":  # two magnitudes of dense values: pairs of them share codes in large groups
        a = np.where(rng.random((h, w)) < 0.5, 1.0 + rng.integers(0, 40, (h, w)) * 2.0 ** -23,
                     rng.standard_cauchy((h, w)) * 1e20)
    return a.astype({"u16": np.uint16, "f32": np.float32}[dtype])


@pytest.mark.parametrize("kind", ["photo", "constant", "narrow", "levels", "impulses", "ends", "mixed"])
@pytest.mark.parametrize("r,tile", [(2, None), (8, "32,32,2,1"), (20, "64,64,8,2"), (33, "64,128,8,2"),
                                    (15, "64,64,2,2"), (24, "64,64,4,2")])
def test_f32(kind, r, tile, monkeypatch):
    if tile:
        monkeypatch.setenv("FIM_TILE", tile)
    img = image(kind, "f32", 131, 117)
    assert_bit_exact(gpu_filter(img, fim_kernel("circle", r)), oracle.median_filter(img, oracle.disk_offsets(r)), kind)


@pytest.mark.parametrize("kind", ["photo", "constant", "narrow", "levels", "impulses"])
@pytest.mark.parametrize("spec,tile", [(("circle", 8), "32,32,2,1"), (("ellipse", 21, 9), "32,32,4,1"),
                                       (("circle", 90), "32,64,4,1"), (("circle", 24), "64,64,4,2")])
@pytest.mark.parametrize("pct", [None, 0.0, 93.0])
def test_u16_smaller_ctas(kind, spec, tile, pct, monkeypatch):
    monkeypatch.setenv("FIM_TILE", tile)
    img = image(kind, "u16", 93, 107)
    off = oracle_offsets(*spec)
    rank = None if pct is None else oracle.percentile_rank(len(off), pct)
    assert_bit_exact(gpu_filter(img, fim_kernel(*spec), percentile=pct), oracle.median_filter(img, off, rank=rank),
                     f"{kind} {spec} {pct}")
