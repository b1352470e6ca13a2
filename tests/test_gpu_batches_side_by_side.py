"""Several batches at once: one of smaller plans leaves an earlier one of the same kernels as it was."""
import pytest
import torch

import datagen
import oracle
from helpers import assert_bit_exact, to_device, to_host

pytestmark = pytest.mark.gpu


def make(r, seed):
    import paper_2505_22938_gb300 as fim
    imgs = [datagen.image_for("u16", seed + i, 150, 140 + 10 * i) for i in range(2)]
    ins = [to_device(x)[0] for x in imgs]
    outs = [torch.zeros_like(x) for x in ins]
    k = fim.fim_create_kernel_circle(r)
    jobs = [fim.make_job(i.data_ptr(), o.data_ptr(), i.shape[1], i.shape[0], i.shape[1] * 2, fim.FIM_U16, k)
            for i, o in zip(ins, outs)]
    torch.cuda.synchronize()
    return fim.fim_batch_create(jobs, [k]), imgs, ins, outs


def test_run_the_larger_after_creating_the_smaller():
    import paper_2505_22938_gb300 as fim
    made = [(72, make(72, 1)), (34, make(34, 7))]  # one class kernel: 1024-thread CTAs, other shared memory
    for r, (batch, imgs, _, outs) in made + made[:1]:
        batch.run(torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert fim.fim_sync_status() == 0
        for img, out in zip(imgs, outs):
            assert_bit_exact(to_host(out), oracle.median_filter(img, oracle.disk_offsets(r)), f"r={r}")
            out.zero_()
