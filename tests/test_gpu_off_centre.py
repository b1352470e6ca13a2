"""Kernels that lie far from their centre: no window holds its centre pixel, and the footprint lies far
from the tile."""
import pytest

import datagen
import oracle
from helpers import assert_bit_exact, fim_kernel, gpu_filter, oracle_offsets

pytestmark = pytest.mark.gpu

SPECS = [
    ("spans", [600] * 5, [606] * 5, 500),           # right of and below every pixel
    ("spans", [-900] * 40, [-870] * 40, -1000),     # left of and above; more rows than a warp's lanes
    ("spans", [40, 39, 38], [44, 45, 46], -60),
]


@pytest.mark.parametrize("spec", SPECS)
@pytest.mark.parametrize("dtype,tile", [("u16", None), ("u8", "64,64,8,2"), ("f32", "64,64,4,2")])
def test_matches_oracle(spec, dtype, tile, monkeypatch):
    if tile:
        monkeypatch.setenv("FIM_TILE", tile)
    img = datagen.image_for(dtype, 9, 140, 170)
    assert_bit_exact(gpu_filter(img, fim_kernel(*spec)), oracle.median_filter(img, oracle_offsets(*spec)), str(spec[1:]))
