"""Trigger times of a stream whose TDC counter steps up and down again among a
few hundred packets (two triggers read out in the wrong order at its wrap):
the call reports decreasing triggers, and the times it leaves behind are the
oracle's, also where the two wrap steps cancel in a part's sum."""
import numpy as np
import pytest

import paper_2603_04942_gb300 as tpx
import synth
from gpu_common import oracle_run, to_device

pytestmark = pytest.mark.gpu

PERIOD, WRAP = 640_000, 1 << 36


@pytest.mark.parametrize("lead", [0, 1, 97, 470, 2100])
def test_opposite_steps(lead):
    rng = np.random.default_rng(lead)
    trig = WRAP + PERIOD * (np.arange(12) - 6) + 1000

    def pixels(n, t):
        return synth.encode_pixels(rng.integers(0, 256, n), rng.integers(0, 256, n), rng.integers(1, 99, n), t + rng.integers(0, 50_000, n))

    pk = np.concatenate([pixels(lead, int(trig[0]) - 60_000), synth.encode_tdcs(trig[:5]), synth.encode_tdcs(trig[[6, 5]]),   # low, then high again
                         pixels(4200, int(trig[5])), synth.encode_tdcs(trig[7:]), pixels(300, int(trig[11]))])
    o = oracle_run(pk)
    assert o["status"] == -4 and (np.diff(o["triggers"]) < 0).any()
    ctx = tpx.Context(tpx.Config(), max_packets=pk.size)
    try:
        d = ctx.tpx_decode(to_device(pk))
        rc, _ = ctx.tpx_sync(check=False)
        assert rc == -4
        assert int(d["n_trig"].item()) == o["triggers"].size
        assert np.array_equal(d["trig"][: o["triggers"].size].cpu().numpy(), o["triggers"])
    finally:
        ctx.close()
