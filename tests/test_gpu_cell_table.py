"""The fused kernel's cell table against the oracle, where it can go wrong:
the sensor's edges, cells hit more than once, cells that several shots of a
range share, more clusters than threads, pairs whose times chain (every pair
adjacent, their ends not), more pairs to unite than the queue holds, and a
pixel wrap inside a range. Everything is compared exactly, as in the other
parity tests."""
import numpy as np
import pytest

import synth
from gpu_common import assert_parity, gpu_run, oracle_run

pytestmark = pytest.mark.gpu

PERIOD = 640_000
WRAP = 1 << 34


def stream(shots, t0=50_000_000):
    """Packets of shots given as (x, y, tot, time after the trigger) arrays."""
    parts = []
    for k, (x, y, tot, t) in enumerate(shots):
        parts.append(synth.encode_tdcs(np.array([t0 + k * PERIOD])))
        parts.append(synth.encode_pixels(x, y, tot, t0 + k * PERIOD + np.asarray(t, np.int64)))
    return np.concatenate(parts)


def edges(rng):
    e = np.array([0, 1, 2, 253, 254, 255])
    return stream([(rng.choice(e, 70), rng.choice(e, 70), rng.integers(1, 40, 70), 500 + rng.integers(0, 90, 70)) for _ in range(60)])


def second_hits(rng):
    return stream([(100 + rng.integers(0, 4, 120), 60 + rng.integers(0, 4, 120), rng.integers(1, 30, 120), 500 + rng.integers(0, 700, 120))
                   for _ in range(50)])


def shared_cells(rng):
    return stream([(rng.integers(0, 12, 6), rng.integers(0, 256, 6), rng.integers(1, 9, 6), 700 + rng.integers(0, 40, 6)) for _ in range(900)])


def many_clusters(rng):
    shots = []
    for _ in range(4):
        c = rng.permutation(128 * 128)[:1900]
        shots.append((2 * (c % 128), 2 * (c // 128), rng.integers(1, 1024, c.size), rng.integers(0, 60_000, c.size)))
    return stream(shots)


def chained_times(rng):
    shots = []
    for _ in range(30):
        y, x = np.mgrid[40:52, 100:140]
        o = rng.permutation(x.size)
        shots.append((x.ravel()[o], y.ravel()[o], rng.integers(1, 1024, x.size), (600 + 20 * (x - 100) + 17 * (y - 40)).ravel()[o]))
    return stream(shots)


def full_queue(rng):
    shots = []
    for _ in range(6):
        y, x = np.mgrid[30:80, 30:80]
        shots.append((x.ravel(), y.ravel(), rng.integers(1, 9, x.size), 600 + rng.integers(0, 60, x.size)))
    return stream(shots)


def pixel_wrap(rng):
    # the wrap of the pixel counter falls among the pixels of shot 6, read out
    # in another order than they arrived
    t0 = WRAP - 6 * PERIOD - 9_000
    shots = [(rng.integers(0, 30, 400), rng.integers(0, 30, 400), rng.integers(1, 99, 400), rng.integers(0, 18_000, 400)) for _ in range(12)]
    return stream(shots, t0)


STREAMS = dict(edges=edges, second_hits=second_hits, shared_cells=shared_cells, many_clusters=many_clusters, chained_times=chained_times,
               full_queue=full_queue, pixel_wrap=pixel_wrap)


@pytest.mark.parametrize("tile", [1, 2])
@pytest.mark.parametrize("mode,r", [(0, 1), (0, 2), (1, 1), (1, 3)])
@pytest.mark.parametrize("name", STREAMS)
def test_against_the_oracle(name, mode, r, tile):
    pk = STREAMS[name](np.random.default_rng(sum(map(ord, name))))
    g = gpu_run(pk, rx=r, ry=r, mode=mode, tile=tile, index_base=11)
    o = oracle_run(pk, rx=r, ry=r, mode=mode, index_base=11)
    assert g["status"] == 0 and g["counters"]["redone"] == 0
    assert_parity(g, o)
