"""The unwrap pre-pass against the oracle at its switch points: one warp's
scan (up to 32 tiles), a block's (up to 1024, one launch), and the general
scan beyond; with a pixel wrap in the stream's first, a middle and the last
tile. Compared exactly, as in the other parity tests."""
import numpy as np
import pytest

import oracle
import paper_2603_04942_gb300 as tpx
import synth
from gpu_common import assert_parity, gpu_run, oracle_run

pytestmark = pytest.mark.gpu

PERIOD = 640_000


@pytest.mark.parametrize("tiles,extra", [(1, -1), (1, 0), (2, 1), (31, 33), (32, 0), (33, -64), (1024, 0), (1025, -1), (1026, 1)])
@pytest.mark.parametrize("wrap_at", [0.0, 0.5, 1.0])
def test_prepass_sizes(tiles, extra, wrap_at):
    n = tiles * 2048 + extra
    shots = n / 51.1   # two particles a shot: many triggers in every tile
    pk, _, _ = synth.generate(synth.small(n_shots=int(1.1 * shots) + 20, particles_per_shot=2.0,
                                          t_start_ticks=(1 << 34) - int(wrap_at * shots * PERIOD) + 1000))
    assert pk.size >= n
    assert_parity(gpu_run(pk[:n], tile=2), oracle_run(pk[:n]))


@pytest.mark.parametrize("tiles", [1, 3, 40, 1030])
def test_wraps_before_the_first_value(tiles):
    """A state of wraps without a value yet (a slice taken up after them)."""
    import torch
    shots = tiles * 2048 / 51.1
    pk, _, _ = synth.generate(synth.small(n_shots=int(1.1 * shots) + 20, particles_per_shot=2.0,
                                          t_start_ticks=3 * (1 << 34) + (1 << 34) // 2 + (1 << 36)))
    pk = pk[: tiles * 2048]
    o = oracle.run(pk, oracle.Config(epoch0_pix=7, epoch0_tdc=1))
    ctx = tpx.Context(tpx.Config(tile_geometry=tpx.TILE_2048), max_packets=pk.size)
    try:
        ctx.tpx_set_state(dict(pixels=0, pix_last_raw=0, pix_wraps=7, triggers=0, tdc_last_raw=0, tdc_wraps=1))
        out = ctx.alloc_outputs(pk.size, True, True, pk.size, pk.size)
        ctx.tpx_process(torch.from_numpy(pk.view(np.int64)).cuda(), out)
        rc, counters = ctx.tpx_sync(check=False)
        assert counters["redone"] == 0
        assert_parity(ctx.collect(out, rc, counters), o)
    finally:
        ctx.close()
