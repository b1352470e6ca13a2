"""Parity of the vertical sweep's forms with the oracle, bit for bit (the output is a selected input
value): the packed slide with signed and with unsigned 16-bit ranks, the slide of kernels of a
few columns, the block scan and the span test with 8-bit and 16-bit coordinates. The kernels are
the ones whose column lists, padding or rank ranges sit on an edge of one of those forms.
"""
import numpy as np
import pytest

import datagen
import oracle
from helpers import assert_bit_exact, fim_kernel, gpu_filter, oracle_offsets

pytestmark = pytest.mark.gpu


def check(img, spec, percentile=None):
    off = oracle_offsets(*spec)
    rank = None if percentile is None else oracle.percentile_rank(len(off), percentile)
    got = gpu_filter(img, fim_kernel(*spec), percentile=percentile)
    assert_bit_exact(got, oracle.median_filter(img, off, rank=rank), f"{spec} {percentile} {img.dtype}")


@pytest.mark.parametrize("tile", [None, "64,64,8,2", "32,32,1,1", "32,96,3,1", "128,64,4,2"])
@pytest.mark.parametrize("spec", [
    ("spans", [0] * 9, [0] * 9, -4),                       # one column: an empty list of odd columns
    ("spans", [-1] * 5, [0] * 5, -2),                      # two columns
    ("spans", [-6], [6], 0),                               # one row of 13
    ("spans", list(range(-12, 1)), list(range(0, 13)), 3),  # skewed, off centre
    ("circle", 5), ("circle", 6),                          # either side of the few-columns rule
])
def test_column_lists(spec, tile, monkeypatch):
    if tile:
        monkeypatch.setenv("FIM_TILE", tile)
    check(datagen.image_for("u16", 31, 101, 139), spec)


@pytest.mark.parametrize("dtype,tile,spec,pct", [
    ("u16", "64,128,8,2", ("circle", 47), None),      # 32972 footprint pixels: ranks relative to the feasible ones
    ("u16", "64,128,8,2", ("circle", 47), 0.0),       # their ends: the least and the greatest member
    ("u16", "64,128,8,2", ("circle", 47), 100.0),
    ("u8", "64,64,8,2", ("circle", 128), None),       # over 65535 pixels, feasible ranks beyond signed 16 bits
    ("f32", "64,128,8,2", ("ellipse", 40, 60), None),
    ("f32", "64,128,8,2", ("ellipse", 100, 21), None),  # box beyond 256 columns: 16-bit coordinates
    ("u8", "64,128,8,2", ("circle", 64), 30.0),       # a 128-row tile whose box is 256 rows: 16-bit coordinates
])
def test_rank_and_coordinate_ranges(dtype, tile, spec, pct, monkeypatch):
    monkeypatch.setenv("FIM_TILE", tile)
    check(datagen.image_for(dtype, 57, 141, 77), spec, pct)


def test_equal_values_and_long_scans():
    """Two flat halves with a seam (scans of half the omnigram), under a disk and a polygon."""
    img = np.zeros((150, 170), np.uint16)
    img[:, 83:] = 40000
    img[70:72, :] = 65535
    check(img, ("circle", 33))
    check(img, ("polygon", oracle.regular_polygon_vertices(6, 30.0)))
