"""Patch extraction on dense shots, whose clusters are read out over more
packets than a tile's margins: in calls where few or many patches go on to the
wider search (bit for bit the oracle's patches), in calls large enough that the
tiles hand theirs on untried (the definition, vectorised), and at a cost per
packet that does not grow with the density."""
import time

import numpy as np
import pytest

import oracle.refiner as orf
import paper_2603_04942_gb300 as tpx
import synth
from test_gpu_patch_reach import PERIOD, clustered, crowded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shots,per_shot,lead", [(6, 2200, 0), (4, 5120, 1019), (3, 9200, 3), (2, 20_000, 11)])
@pytest.mark.parametrize("bf16", [False, True])
def test_few_and_many_go_on(shots, per_shot, lead, bf16):
    import torch
    pk = crowded(np.random.default_rng(per_shot), shots, per_shot, lead)
    want, sel, centre, _ = orf.patches(pk, 12)
    ctx, d, out, n = clustered(pk)
    try:
        f = ctx.tpx_refine_patches_bf16 if bf16 else ctx.tpx_refine_patches
        got = f(d, out["labels"], out["clusters"], n, 12)
        m = int(got["n"].item())
        assert m == sel.size > 0 and got["status"] == 0
        p = got["patches"][:m]
        p = p.view(torch.bfloat16).float() if bf16 else p
        assert np.array_equal(p.cpu().numpy(), want)
        assert np.array_equal(got["centre"][:m].cpu().numpy(), centre)
    finally:
        ctx.close()


def acquisition(rng, shots, per_shot):
    """`shots` shots of clusters of 20 pixels (a 4 x 5 block), read out in random order."""
    m = per_shot // 20
    cx, cy = rng.integers(0, 252, (shots, m, 1)), rng.integers(0, 251, (shots, m, 1))
    i = np.arange(20)
    x, y = cx + i % 4, cy + i // 4
    t = rng.integers(0, 60_000, (shots, m, 1)) + rng.integers(0, 8, x.shape) + 50_000_000 + PERIOD * np.arange(shots)[:, None, None]
    o = np.argsort(rng.random((shots, per_shot)), axis=1)
    x, y, t, tot = (np.take_along_axis(v.reshape(shots, per_shot), o, axis=1) for v in (x, y, t, rng.integers(1, 1024, x.shape)))
    px = synth.encode_pixels(x.ravel(), y.ravel(), tot.ravel(), t.ravel()).reshape(shots, per_shot)
    tdc = synth.encode_tdcs(50_000_000 + PERIOD * np.arange(shots)).reshape(shots, 1)
    z = np.zeros((shots, 1), np.int64)
    words = [np.hstack([a, b]).ravel() for a, b in ((tdc, px), (z, x), (z, y), (z, tot), (z, t))]
    return words[0], words[1:]


def by_definition(values, labels, sel, centre):
    """The patches of the clusters labelled sel: per cell the brightest member, the later of equal ones."""
    x, y, tot, t = values
    slot = np.full(labels.size, -1)
    slot[sel] = np.arange(sel.size)
    q = np.flatnonzero(labels >= 0)
    s = slot[labels[q]]
    q, s = q[s >= 0], s[s >= 0]
    dx, dy = x[q] - centre[s, 0] + 4, y[q] - centre[s, 1] + 4
    inside = (dx >= 0) & (dx < 9) & (dy >= 0) & (dy < 9)
    q, s, cell = q[inside], s[inside], (dy * 9 + dx)[inside]
    best = np.full((sel.size, 81), -1, np.int64)
    np.maximum.at(best, (s, cell), (tot[q] << 32) | q)
    out = np.zeros((sel.size, 162), np.float32)
    i, c = np.nonzero(best >= 0)
    w = best[i, c] & 0xFFFFFFFF
    bits = (tot[w].astype(np.float32) / np.float32(1023)).view(np.uint32).astype(np.int64)
    out[i, c] = ((bits + 0x7FFF + ((bits >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32)
    d = (t[w] - t[sel[i]]).astype(np.float32) / np.float32(32)
    out[i, 81 + c] = np.clip(d, -8, 8).astype(np.float16)
    return out


def extract(pk, mode=0, min_pixels=12):
    import torch
    d = torch.from_numpy(pk.view(np.int64)).cuda()
    ctx = tpx.Context(tpx.Config(mode=mode), max_packets=pk.size)
    try:
        out = ctx.alloc_outputs(pk.size, labels=True)
        ctx.tpx_process(d, out)
        ctx.tpx_sync()
        n = int(out["n_clusters"].item())
        times = []
        for _ in range(4):
            t0 = time.perf_counter()
            got = ctx.tpx_refine_patches(d, out["labels"], out["clusters"], n, min_pixels, capacity=n)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
        m = int(got["n"].item())
        rec = np.frombuffer(out["clusters"][: 88 * n].cpu().numpy().tobytes(), tpx.CLUSTER_DTYPE)
        return (out["labels"].cpu().numpy(), rec["label"][got["sel"][:m].cpu().numpy()], got["centre"][:m].cpu().numpy(),
                got["patches"][:m].cpu().numpy(), min(times))
    finally:
        ctx.close()


@pytest.mark.parametrize("shots,per_shot,mode", [(700, 4000, 0), (160, 20_000, 0), (1400, 2000, 1)])
def test_large_calls(shots, per_shot, mode):
    """2.8e6 packets and more: far more tiles than run at a time, so that the later ones see what became of the
    first ones' patches. (PAPER mode: a record's count is not its label's, none of the searches completes one.)"""
    pk, values = acquisition(np.random.default_rng(per_shot + mode), shots, per_shot)
    labels, root, centre, got, _ = extract(pk, mode, 12 if mode == 0 else 3)
    assert root.size > 8192
    assert np.array_equal(got, by_definition(values, labels, root, centre))


def test_cost_per_packet():
    """Shots of 4000 pixels cost a few times as much as of 500 at most, per packet (65 times, with a search for each patch)."""
    rng = np.random.default_rng(8)
    a, b = (extract(acquisition(rng, shots, per)[0])[4] for shots, per in ((16_000, 500), (2000, 4000)))
    assert b < 6 * a, (a, b)
