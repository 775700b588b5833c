"""tpx_process_host on a call that the fused kernel cannot hold: the outputs
that reach the host are those of the exact redo, also where the call is not one
of the autotuner's samples (too small, or a fixed tile geometry)."""
import numpy as np
import pytest

import paper_2603_04942_gb300 as tpx
import synth
from gpu_common import assert_clusters_equal, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [tpx.TILE_DEFAULT, tpx.TILE_2048])
def test_an_oversize_shot_reaches_the_host(tile):
    rng = np.random.default_rng(3)
    t0, parts = 40_000_000, []
    for k, n in enumerate((500, 12_000, 700)):
        parts.append(synth.encode_tdcs(np.array([t0 + k * 640_000])))
        parts.append(synth.encode_pixels(rng.integers(0, 256, n), rng.integers(0, 256, n), rng.integers(1, 900, n),
                                         t0 + k * 640_000 + rng.integers(0, 60_000, n)))
    pk = np.concatenate(parts)
    o = oracle_run(pk)
    ctx = tpx.Context(tpx.Config(tile_geometry=tile), max_packets=pk.size)
    try:
        lab, peak = np.empty(pk.size, np.int64), np.empty(pk.size, np.uint8)
        cl, tr = np.empty(pk.size, tpx.CLUSTER_DTYPE), np.empty(16, np.int64)
        rc, ncl, ntr = ctx.tpx_process_host(pk, lab, peak, cl, tr)
    finally:
        ctx.close()
    assert rc == 0 and ncl == o["clusters"].size and ntr == 3
    assert np.array_equal(lab, o["labels"]) and np.array_equal(peak, o["is_peak"])
    assert np.array_equal(tr[:3], o["triggers"])
    assert_clusters_equal(cl[:ncl], o["clusters"])
