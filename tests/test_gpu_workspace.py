"""The workspace of a stream holds nothing that one call leaves for the next."""
import numpy as np
import pytest

import datagen
import oracle
from helpers import assert_bit_exact, to_device, to_host

pytestmark = pytest.mark.gpu


def test_call_between_a_capture_and_its_first_replay():
    """The workspace is allocated while a stream captures (relaxed mode) from memory that held other
    data; a call on that stream before the graph has run finds its own tile queue."""
    import torch
    import paper_2505_22938_gb300 as fim
    img = datagen.image_for("u16", 5, 1800, 1900)  # several waves of the radius's tiles
    k = fim.fim_create_kernel_circle(4)
    store, _ = to_device(img)
    outs = [torch.zeros_like(store) for _ in range(3)]
    st = torch.cuda.Stream()
    junk = torch.full((256 << 20,), 0x7f, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    fim.fim_release_workspace()
    del junk
    torch.cuda.empty_cache()

    def call(out):
        fim.fim_median(store.data_ptr(), out.data_ptr(), 1900, 1800, 3800, fim.FIM_U16, k, st.cuda_stream)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        g.capture_begin(capture_error_mode="relaxed")
        call(outs[0])
        g.capture_end()
        call(outs[1])
    st.synchronize()
    with torch.cuda.stream(st):
        g.replay()
        call(outs[2])
    st.synchronize()
    assert fim.fim_sync_status(st.cuda_stream) == 0
    exp = oracle.median_filter(img, oracle.disk_offsets(4))
    for i, out in enumerate(outs):
        assert_bit_exact(to_host(out), exp, f"call {i}")
    del g
    fim.fim_release_workspace()


@pytest.mark.parametrize("size", [(32, 8), (64, 40), (700, 500), (1024, 1024)])
def test_one_wave_and_queued_grids(size):
    """Grids with a CTA per tile (no queue) and grids that take several tiles per CTA, in turn on one
    stream."""
    import torch
    import paper_2505_22938_gb300 as fim
    w, h = size
    img = datagen.image_for("u8", w, h, w)
    store, _ = to_device(img)
    for r in (2, 30, 2):
        out = fim.median(store, fim.fim_create_kernel_circle(r))
        torch.cuda.synchronize()
        assert fim.fim_sync_status() == 0
        assert_bit_exact(to_host(out), oracle.median_filter(img, oracle.disk_offsets(r)), f"{size} r={r}")
