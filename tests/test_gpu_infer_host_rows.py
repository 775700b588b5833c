"""The perceptron's inference on rows in pinned host memory (mapped into the
device's address space), which it reads in place: the same bits as on a copy of
them in device memory."""
import numpy as np
import pytest

import paper_2603_04942_gb300 as tpx
from test_gpu_infer_groups import rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [100, 128 * 152 + 1])
def test_rows_in_pinned_memory(n):
    import torch
    h = 160
    p = (0.1 * np.random.default_rng(n).normal(size=int(tpx.Context.tpx_refiner_params(h)))).astype(np.float32)
    x = torch.from_numpy(rows(n, n)).pin_memory()
    ctx = tpx.Context(tpx.Config(), max_packets=16)
    try:
        packed = ctx.tpx_refiner_pack(torch.from_numpy(p).cuda(), h)
        want = ctx.tpx_refiner_infer(packed, h, x.cuda())[:n]
        out = torch.zeros((n, 6), device="cuda")
        assert tpx.lib().tpx_refiner_infer(ctx._h, packed.data_ptr(), h, x.data_ptr(), n, out.data_ptr()) == 0
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    finally:
        ctx.close()
