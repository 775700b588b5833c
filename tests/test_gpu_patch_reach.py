"""Patch extraction where a cluster's packets lie far apart in the stream (in
the tile's margins, in the wider search's reach, beyond both), at the tiles'
edges, with cells hit twice by equal charges, with records in another order
than ascending, and into a buffer that is not aligned to pairs: equal to the
oracle's patches, bit for bit."""
import numpy as np
import pytest

import oracle.refiner as orf
import paper_2603_04942_gb300 as tpx
import synth

pytestmark = pytest.mark.gpu

PERIOD = 640_000


def crowded(rng, shots, per_shot, lead=0):
    """Shots of `per_shot` pixels in clusters of 20, read out in random order; `lead` packets before the first trigger."""
    t0 = 50_000_000
    out = [synth.encode_pixels(rng.integers(0, 256, lead), rng.integers(0, 256, lead), rng.integers(0, 9, lead), t0 - 5000 + np.zeros(lead, np.int64))]
    for k in range(shots):
        m = per_shot // 20
        cx, cy, ct = rng.integers(0, 251, m), rng.integers(0, 252, m), rng.integers(0, 60_000, m)
        i = np.arange(20)
        x, y = cx[:, None] + i % 5, cy[:, None] + i // 5
        x[:, 19], y[:, 19] = x[:, 7], y[:, 7]                      # a cell twice
        tot = rng.integers(0, 1024, (m, 20))
        tot[:, 19] = np.where(rng.random(m) < 0.5, tot[:, 7], tot[:, 19])
        t = ct[:, None] + rng.integers(0, 12, (m, 20))
        o = rng.permutation(m * 20)
        out.append(synth.encode_tdcs(np.array([t0 + k * PERIOD])))
        out.append(synth.encode_pixels(x.ravel()[o], y.ravel()[o], tot.ravel()[o], t0 + k * PERIOD + t.ravel()[o]))
    return np.concatenate(out)


def clustered(pk):
    import torch
    d = torch.from_numpy(pk.view(np.int64)).cuda()
    ctx = tpx.Context(tpx.Config(), max_packets=pk.size)
    out = ctx.alloc_outputs(pk.size, labels=True)
    ctx.tpx_process(d, out)
    ctx.tpx_sync()
    return ctx, d, out, int(out["n_clusters"].item())


@pytest.mark.parametrize("shots,per_shot,lead", [(3, 1000, 0), (8, 1000, 1047), (4, 2040, 7), (2, 5000, 1), (1, 40_000, 0)])
@pytest.mark.parametrize("bf16", [False, True])
def test_reach(shots, per_shot, lead, bf16):
    import torch
    pk = crowded(np.random.default_rng(per_shot + lead), shots, per_shot, lead)
    want, sel, centre, _ = orf.patches(pk, 12)
    ctx, d, out, n = clustered(pk)
    try:
        f = ctx.tpx_refine_patches_bf16 if bf16 else ctx.tpx_refine_patches
        got = f(d, out["labels"], out["clusters"], n, 12)
        torch.cuda.synchronize()
        m = int(got["n"].item())
        assert m == sel.size > 0 and got["status"] == 0
        p = got["patches"][:m]
        p = p.view(torch.bfloat16).float() if bf16 else p
        assert np.array_equal(p.cpu().numpy(), want)
        assert np.array_equal(got["sel"][:m].cpu().numpy(), sel)
        assert np.array_equal(got["centre"][:m].cpu().numpy(), centre)
    finally:
        ctx.close()


def test_records_in_another_order():
    import torch
    pk = crowded(np.random.default_rng(3), 3, 1000)
    want, sel, _, _ = orf.patches(pk, 12)
    ctx, d, out, n = clustered(pk)
    try:
        words = out["clusters"][: n * 88].view(torch.int64).view(n, 11)
        back = torch.flip(words, [0]).contiguous().view(-1).view(torch.uint8)
        got = ctx.tpx_refine_patches(d, out["labels"], back, n, 12)
        m = int(got["n"].item())
        assert m == sel.size
        assert np.array_equal(got["patches"][:m].cpu().numpy(), want[::-1])
        assert np.array_equal(got["sel"][:m].cpu().numpy(), n - 1 - sel[::-1])
    finally:
        ctx.close()


@pytest.mark.parametrize("bf16", [False, True])
def test_unaligned_patches(bf16):
    import torch
    pk = crowded(np.random.default_rng(4), 3, 1000)
    want, sel, _, _ = orf.patches(pk, 12)
    ctx, d, out, n = clustered(pk)
    try:
        size = 2 if bf16 else 4
        buf = torch.zeros(n * 162 + 4, dtype=torch.int16 if bf16 else torch.float32, device="cuda")
        idx = torch.empty(n, dtype=torch.int64, device="cuda")
        cen = torch.empty((n, 2), dtype=torch.int32, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
        f = tpx.lib().tpx_refine_patches_bf16 if bf16 else tpx.lib().tpx_refine_patches
        rc = f(ctx._h, d.data_ptr(), pk.size, 0, out["labels"].data_ptr(), out["clusters"].data_ptr(), n, 12,
               buf.data_ptr() + size, idx.data_ptr(), cen.data_ptr(), n, cnt.data_ptr())
        torch.cuda.synchronize()
        m = int(cnt.item())
        assert rc == 0 and m == sel.size
        p = buf[1: 1 + m * 162].view(m, 162)
        p = p.contiguous().view(torch.bfloat16).float() if bf16 else p
        assert np.array_equal(p.cpu().numpy(), want)
        assert int(buf[0]) == 0
    finally:
        ctx.close()
