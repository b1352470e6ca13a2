"""fim_median_noalloc on the tiles it takes where the library's default does not fit its workspace."""
import pytest

import datagen
from helpers import fim_kernel
from test_zz_no_alloc import _run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,spec", [("f32", ("circle", 50)), ("u16", ("ellipse", 104, 52)),
                                        ("f32", ("ellipse", 104, 52))])
def test_same_bytes_as_fim_median(dtype, spec):
    _run_both(datagen.image_for(dtype, 104, 700, 1300), fim_kernel(*spec))
