"""Big ranges of a batch with boxes of other radii than the eight neighbours:
the pairs come from the cell chains or from the time windows, whichever has less
to compare. Both, at the sensor's edges, with cells hit many times and with a
time radius over the whole shot, against the oracle on each run alone."""
import numpy as np
import pytest

import paper_2603_04942_gb300 as tpx
import synth
from gpu_common import assert_clusters_equal, oracle_run, to_device

pytestmark = pytest.mark.gpu

PERIOD = 640_000


def run_of(rng, sizes, spread):
    """Shots of clusters (rectangles of up to 3 x 3), stray pixels at the edges, and a cell hit many times."""
    parts = []
    for k, n in enumerate(sizes):
        m = n // 12
        cx, cy, ct = rng.integers(0, 254, (m, 1)), rng.integers(0, 254, (m, 1)), rng.integers(0, spread, (m, 1))
        i = np.arange(9)
        x, y, t = cx + i % 3, cy + i // 3, ct + rng.integers(0, 25, (m, 9))
        e = n - 9 * m
        x = np.concatenate([x.ravel(), rng.choice([0, 1, 77, 254, 255], e)])
        y = np.concatenate([y.ravel(), rng.choice([0, 1, 133, 255], e)])
        t = np.concatenate([t.ravel(), rng.integers(0, spread, e)])
        o = rng.permutation(n)
        parts += [synth.encode_tdcs(np.array([50_000_000 + k * PERIOD])),
                  synth.encode_pixels(x[o], y[o], rng.integers(1, 30, n), 50_000_000 + k * PERIOD + t[o])]
    return np.concatenate(parts)


@pytest.mark.parametrize("tile", [tpx.TILE_4096, tpx.TILE_2048])
@pytest.mark.parametrize("rx,ry,dt", [(2, 1, 32), (1, 2, 32), (2, 2, 0), (3, 3, 32), (7, 7, 32), (7, 0, 32), (0, 7, 32), (2, 2, 3000), (1, 3, 70_000), (7, 7, 70_000)])
def test_wide_boxes(rx, ry, dt, tile):
    rng = np.random.default_rng(100 * rx + 10 * ry + dt)
    runs = [run_of(rng, s, spread) for s, spread in (((9000, 300, 11_000), 60_000), ((16_000,), 40_000), ((400, 8300, 8300), 2000))]
    offs = np.concatenate([[0], np.cumsum([r.size for r in runs])]).astype(np.int64)
    pk = np.concatenate(runs)
    ctx = tpx.Context(tpx.Config(rx=rx, ry=ry, dt_ticks=dt, tile_geometry=tile), max_packets=pk.size)
    try:
        out = ctx.alloc_batch_outputs(pk.size, offs.size - 1, labels=True, is_peak=True, cluster_capacity=pk.size, trig_capacity=64)
        ctx.tpx_process_batch(to_device(pk), offs, out)
        rc, cnt = ctx.tpx_sync(check=False)
        g = ctx.collect_batch(out, rc, cnt)
    finally:
        ctx.close()
    assert rc == 0 and cnt["redone"] == 0
    for r, run in enumerate(runs):
        o = oracle_run(run, rx=rx, ry=ry, dt=dt, index_base=int(offs[r]))
        assert np.array_equal(g["labels"][offs[r]: offs[r + 1]], o["labels"])
        assert np.array_equal(g["is_peak"][offs[r]: offs[r + 1]], o["is_peak"])
        assert_clusters_equal(g["clusters"][g["run_clusters"][r]: g["run_clusters"][r + 1]], o["clusters"])
