"""fim_median_host with kernels that lie above or below their centre: the rows a band needs are copied
before it runs, also where these are repeats of the first or last row alone."""
import numpy as np
import pytest

import datagen
import oracle
from helpers import assert_bit_exact, fim_kernel, oracle_offsets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dy0", [-700, -95, 90, 700])
def test_bands(dy0):
    import paper_2505_22938_gb300 as fim
    spec = ("spans", [-2, -3, -2], [2, 3, 2], dy0)
    img = datagen.image_for("u16", 3, 640, 210)
    for _ in range(3):
        out = np.zeros_like(img)
        fim.fim_median_host(img.ctypes.data, out.ctypes.data, 210, 640, 420, fim.FIM_U16, fim_kernel(*spec), 0)
        assert_bit_exact(out, oracle.median_filter(img, oracle_offsets(*spec)), f"dy0={dy0}")
