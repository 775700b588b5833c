"""The unwrap pre-pass against the oracle at its switch points: one warp's
scan (up to 32 tiles), a block's (up to 1024, one launch), and the general
scan beyond; with a pixel wrap in the stream's first, a middle and the last
tile. Compared exactly, as in the other parity tests."""
import numpy as np
import pytest

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
