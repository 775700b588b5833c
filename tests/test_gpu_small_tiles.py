"""The tiles of 1024 packets, which calls of up to one such tile per SM take when
the geometry is left to the library: the cell table's adversarial streams, the
pre-pass at its switch points and at the largest such call and the next, ranges
up to and past the capacity (eight tiles on), as many records as packets, and
the context's memory. Compared exactly, as in the other parity tests."""
import numpy as np
import pytest

import paper_2603_04942_gb300 as tpx
import synth
from gpu_common import assert_parity, gpu_run, oracle_run
from test_gpu_cell_table import PERIOD, STREAMS, stream

pytestmark = pytest.mark.gpu

T, C = 1024, 8192


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("mode,r", [(0, 1), (0, 2), (1, 1), (1, 3)])
@pytest.mark.parametrize("name", STREAMS)
def test_adversarial_streams(name, mode, r):
    pk = STREAMS[name](np.random.default_rng(1 + sum(map(ord, name))))
    assert pk.size <= sms() * T
    g = gpu_run(pk, rx=r, ry=r, mode=mode, index_base=11)
    assert g["status"] == 0 and g["counters"]["redone"] == 0
    assert_parity(g, oracle_run(pk, rx=r, ry=r, mode=mode, index_base=11))


@pytest.mark.parametrize("tiles,extra", [(1, -1), (1, 0), (2, 1), (8, -31), (31, 33), (32, 0), (33, -64), (0, -1), (0, 0), (0, 1)])
@pytest.mark.parametrize("wrap_at", [0.0, 0.5, 1.0])
def test_sizes(tiles, extra, wrap_at):
    n = (tiles or sms()) * T + extra   # 0: a tile for each SM
    shots = n / 51.1                   # two particles a shot: many triggers in every tile
    pk, _, _ = synth.generate(synth.small(n_shots=int(1.1 * shots) + 20, particles_per_shot=2.0,
                                          t_start_ticks=(1 << 34) - int(wrap_at * shots * PERIOD) + 1000))
    assert pk.size >= n
    assert_parity(gpu_run(pk[:n]), oracle_run(pk[:n]))


def pixels(rng, n):
    return rng.integers(0, 256, n), rng.integers(0, 256, n), rng.integers(1, 900, n), rng.integers(0, 60_000, n)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("first", [0, 1, 700, 1023])   # the long shot's trigger, in a tile
@pytest.mark.parametrize("end,redone", [(C - T - 1, 0), (C - T, 0), (C - 2, 0), (C - 1, 0), (C, 1), (C + 1, 1), (9 * T, 1)])   # the next trigger, from the tile's start
def test_range_capacity(first, end, redone, mode):
    rng = np.random.default_rng(first + end)
    pk = stream([pixels(rng, T + first - 1), pixels(rng, end - first - 1), pixels(rng, 300)])   # the first shot: the tile before
    assert (pk[[T + first, T + end]] >> np.uint64(60) == 6).all()
    g = gpu_run(pk, mode=mode)
    assert g["status"] == 0 and g["counters"]["redone"] == redone
    assert_parity(g, oracle_run(pk, mode=mode))


@pytest.mark.parametrize("n,redone", [(C - 1, 0), (C, 0), (C + 1, 1), (9 * T + 1, 1)])
def test_range_to_the_end(n, redone):
    pk = stream([pixels(np.random.default_rng(n), n - 1)])
    g = gpu_run(pk)
    assert g["status"] == 0 and g["counters"]["redone"] == redone
    assert_parity(g, oracle_run(pk))


@pytest.mark.parametrize("per", [61, 900, 5000, 7100])
def test_a_record_for_every_pixel(per):
    """No two pixels adjacent: the staging is full where the ranges are."""
    rng = np.random.default_rng(per)
    n = sms() * T
    shots = []
    for _ in range(n // (per + 1)):
        c = rng.permutation(128 * 128)[:per]
        shots.append((2 * (c % 128), 2 * (c // 128), rng.integers(1, 1024, per), rng.integers(0, 60_000, per)))
    pk = stream(shots)
    g = gpu_run(pk)
    assert g["counters"]["redone"] == 0 and g["n_clusters"] == pk.size - len(shots)
    assert_parity(g, oracle_run(pk))


@pytest.mark.parametrize("n,megabytes", [(17_723, 12), (65_536, 24), (155_648, 48)])
def test_context_memory(n, megabytes):
    """A record range for each CTA of the larger tiles' grids, no more: 6, 17 and 38 MB."""
    import torch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = tpx.Context(tpx.Config(), max_packets=n)
    used = before - torch.cuda.mem_get_info()[0]
    ctx.close()
    assert used <= megabytes << 20
