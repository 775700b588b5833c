"""Inference kernels at the edges of their groups and tiles: the CNN's groups
of patches (44) over one, all and more SMs, the perceptron's tiles of 128 rows
per SM and of 256 beyond. A row's outputs do not depend on its place: the same
rows shifted by some, in calls of other sizes, give the same bits; and they
agree with the oracle's inference precision as in the networks' own tests."""
import numpy as np
import pytest

import oracle.refiner as orf
import paper_2603_04942_gb300 as tpx

pytestmark = pytest.mark.gpu


def rows(n, seed):
    rng = np.random.default_rng(seed)
    x = np.where(rng.random((n, 162)) < 0.3, rng.random((n, 162)), 0).astype(np.float32)
    return (x.view(np.uint32) & 0xFFFF0000).view(np.float32)   # exact in bf16


def check(g, o):
    scale = max(1.0, np.abs(o).max())
    err = np.abs(g - o).max(axis=1)
    assert np.mean(err <= 1e-3 * scale) >= 0.95 and err.max() <= 5e-2 * scale, np.sort(err)[-5:]


@pytest.mark.parametrize("n", [1, 43, 44, 45, 89, 44 * 152 - 1, 44 * 152 + 1])
def test_cnn_groups(n):
    import torch
    x = rows(n + 17, n)
    p = (0.15 * np.random.default_rng(5).normal(size=49750)).astype(np.float32)
    ctx = tpx.Context(tpx.Config(), max_packets=16)
    try:
        packed = ctx.tpx_cnn_pack(torch.from_numpy(p).cuda())
        bits = torch.from_numpy((x.view(np.uint32) >> 16).astype(np.uint16).view(np.int16)).cuda()
        a = ctx.tpx_cnn_infer(packed, bits)[: n + 17].cpu().numpy()
        # rows 8 on (the buffer stays 16-byte aligned), and the first n alone
        b = ctx.tpx_cnn_infer(packed, bits[8:].contiguous())[: n + 9].cpu().numpy()
        c = ctx.tpx_cnn_infer(packed, bits[:n].contiguous())[:n].cpu().numpy()
        assert ctx.tpx_sync(check=False)[0] == 0
    finally:
        ctx.close()
    assert np.array_equal(a[8:], b) and np.array_equal(a[:n], c)
    check(a[:200].astype(np.float64), orf.cnn_forward_bf16(p, x[:200]))


@pytest.mark.parametrize("h", [64, 160])
@pytest.mark.parametrize("n", [1, 127, 129, 128 * 152, 128 * 152 + 1, 256 * 153 + 3])
def test_perceptron_tiles(h, n):
    import torch
    x = rows(n + 5, n + h)
    size = int(tpx.Context.tpx_refiner_params(h))
    p = (0.1 * np.random.default_rng(h).normal(size=size)).astype(np.float32)
    ctx = tpx.Context(tpx.Config(), max_packets=16)
    try:
        packed = ctx.tpx_refiner_pack(torch.from_numpy(p).cuda(), h)
        d = torch.from_numpy(x).cuda()
        a = ctx.tpx_refiner_infer(packed, h, d)[: n + 5].cpu().numpy()
        b = ctx.tpx_refiner_infer(packed, h, d[5:])[:n].cpu().numpy()   # 8-byte, not 16-byte aligned
        c = ctx.tpx_refiner_infer(packed, h, d[:100])[: min(n + 5, 100)].cpu().numpy()
        torch.cuda.synchronize()
    finally:
        ctx.close()
    assert np.array_equal(a[5:], b) and np.array_equal(a[: c.shape[0]], c)
    check(a[:300].astype(np.float64), orf.forward_bf16(p.astype(np.float64), h, x[:300]))
