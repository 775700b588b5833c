"""Big ranges of a batch whose clusters are joined by many threads at once (14,000
pixels within 300 ticks): every pixel carries its cluster's label, in every one
of many runs, as the oracle has it."""
import numpy as np
import pytest

import paper_2603_04942_gb300 as tpx
from gpu_common import assert_clusters_equal, oracle_run, to_device
from test_gpu_cell_table import stream

pytestmark = pytest.mark.gpu


def dense(rng, n):
    cx, cy = rng.integers(0, 250, (n // 25, 1)), rng.integers(0, 250, (n // 25, 1))
    i, o = np.arange(25), rng.permutation(n)
    return (cx + i % 5).ravel()[o], (cy + i // 5).ravel()[o], rng.integers(1, 900, n), 500 + rng.integers(0, 300, n)


@pytest.mark.parametrize("tile", [tpx.TILE_4096, tpx.TILE_2048])
@pytest.mark.parametrize("r,dt", [(1, 32), (3, 32), (7, 32), (2, 300)])
def test_every_pixel_has_its_cluster(r, dt, tile):
    import torch
    rng = np.random.default_rng(10 * r + dt)
    runs = [stream([dense(rng, 14_000) for _ in range(4)]) for _ in range(8)]
    offs = np.concatenate([[0], np.cumsum([x.size for x in runs])]).astype(np.int64)
    pk = np.concatenate(runs)
    o = [oracle_run(x, rx=r, ry=r, dt=dt, index_base=int(a)) for x, a in zip(runs, offs)]
    labels = torch.from_numpy(np.concatenate([x["labels"] for x in o])).cuda()
    ctx = tpx.Context(tpx.Config(rx=r, ry=r, dt_ticks=dt, tile_geometry=tile), max_packets=pk.size)
    try:
        out = ctx.alloc_batch_outputs(pk.size, 8, labels=True, is_peak=True, cluster_capacity=pk.size, trig_capacity=64)
        d = to_device(pk)
        for _ in range(25):
            ctx.tpx_process_batch(d, offs, out)
            rc, cnt = ctx.tpx_sync(check=False)
            assert rc == 0 and cnt["redone"] == 0
            assert torch.equal(out["labels"][: pk.size], labels)
        g = ctx.collect_batch(out, rc, cnt)
    finally:
        ctx.close()
    assert_clusters_equal(g["clusters"], np.concatenate([x["clusters"] for x in o]))
