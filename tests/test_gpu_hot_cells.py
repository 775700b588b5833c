"""Cells hit many times over (a noisy pixel): their hits lie outside the cell
table, in chains, and are met row by row of the box, narrow and wide, at the
sensor's edges and corners too. Against the oracle, exactly."""
import numpy as np
import pytest

from gpu_common import assert_parity, gpu_run, oracle_run
from test_gpu_cell_table import stream

pytestmark = pytest.mark.gpu


def hot(rng, n):
    """Half of a shot's pixels in six cells, three of them side by side, the rest around those or anywhere."""
    hx, hy = np.array([0, 255, 100, 101, 102, 31]), np.array([0, 255, 60, 60, 60, 254])
    k = rng.integers(0, 6, n)
    u = rng.random(n)
    d = rng.integers(-8, 9, (2, n)) * (u > 0.5)
    x = np.where(u < 0.9, np.clip(hx[k] + d[0], 0, 255), rng.integers(0, 256, n))
    y = np.where(u < 0.9, np.clip(hy[k] + d[1], 0, 255), rng.integers(0, 256, n))
    return x, y, rng.integers(1, 30, n), rng.integers(0, 20_000, n)


@pytest.mark.parametrize("tile", [0, 1, 2])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("rx,ry,dt", [(1, 1, 32), (2, 2, 400), (3, 2, 32), (2, 3, 32), (7, 7, 32), (7, 1, 5000)])
def test_against_the_oracle(rx, ry, dt, mode, tile):
    rng = np.random.default_rng(rx + 10 * ry + dt)
    pk = stream([hot(rng, int(n)) for n in rng.integers(200, 1500, 14)])
    g = gpu_run(pk, rx=rx, ry=ry, dt=dt, mode=mode, tile=tile)
    assert g["status"] == 0 and g["counters"]["redone"] == 0
    assert_parity(g, oracle_run(pk, rx=rx, ry=ry, dt=dt, mode=mode))
