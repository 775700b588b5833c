"""The CNN's inference where its patches are shared out over rounds of groups of
fewer than 44: a row's outputs do not depend on the group it is in, so calls of
other sizes give the bits that a large call gives for the same rows."""
import numpy as np
import pytest

import oracle.refiner as orf
import paper_2603_04942_gb300 as tpx
from test_gpu_infer_groups import check, rows

pytestmark = pytest.mark.gpu


def test_rounds():
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    one = 44 * sms
    x = rows(9 * one, 3)
    p = (0.15 * np.random.default_rng(6).normal(size=49750)).astype(np.float32)
    bits = torch.from_numpy((x.view(np.uint32) >> 16).astype(np.uint16).view(np.int16)).cuda()
    ctx = tpx.Context(tpx.Config(), max_packets=16)
    try:
        packed = ctx.tpx_cnn_pack(torch.from_numpy(p).cuda())
        want = ctx.tpx_cnn_infer(packed, bits)                    # beyond the rounds that are evened out
        for n in (1, 4, 5, sms, 4 * sms + 1, 8 * sms, 20 * sms - 1, 40 * sms, 40 * sms + 1, one - 1, one, one + 1, 48 * sms, 2 * one, 2 * one + 1,
                  96 * sms, 7 * one + 5, 8 * one, 8 * one + 1):
            got = ctx.tpx_cnn_infer(packed, bits[:n])
            assert torch.equal(got[:n], want[:n]), n
        assert ctx.tpx_sync(check=False)[0] == 0
    finally:
        ctx.close()
    check(want[:300].cpu().numpy().astype(np.float64), orf.cnn_forward_bf16(p, x[:300]))
