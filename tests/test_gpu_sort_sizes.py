"""The general path's sort, segments and record placing at the edges of their
tiles of 4096 hits, with 32- and 64-bit keys (few and very many shots), all
digits in use, equal keys (ties keep stream order), compared exactly with the
oracle; and tpx_centroid on hits whose stream indices span more than its rank
table holds."""
import numpy as np
import pytest

from test_gpu_general import check_unfused
import synth

pytestmark = pytest.mark.gpu

PERIOD = 640_000


def stream(rng, hits, shots):
    """`hits` kept pixels over `shots` shots, in random times and few cells (so that clusters form)."""
    per = np.bincount(rng.integers(0, shots, hits), minlength=shots)
    out = []
    for k in range(shots):
        t0 = 50_000_000 + k * PERIOD
        out.append(synth.encode_tdcs(np.array([t0])))
        m = int(per[k])
        if m:
            out.append(synth.encode_pixels(rng.integers(100, 110, m), rng.integers(100, 110, m), rng.integers(0, 1024, m),
                                           t0 + rng.integers(0, 60_000, m) // 16 * 16))
    return np.concatenate(out)


@pytest.mark.parametrize("hits,shots", [(1, 1), (4095, 1), (4096, 2), (4097, 255), (8192, 256), (12_289, 257), (40_000, 300), (5000, 9000)])
def test_sort_sizes(hits, shots):
    check_unfused(stream(np.random.default_rng(hits + shots), hits, shots))


@pytest.mark.parametrize("mode", [0, 1])
def test_sparse_indices(mode):
    # one kept pixel in a hundred: the indices span a hundred times the hits
    rng = np.random.default_rng(5)
    t0 = 50_000_000
    out = []
    for k in range(40):
        m = 3000
        t = t0 + k * PERIOD + np.where(rng.random(m) < 0.01, rng.integers(0, 600, m), rng.integers(70_000, 600_000, m))
        out += [synth.encode_tdcs(np.array([t0 + k * PERIOD])), synth.encode_pixels(rng.integers(0, 12, m), rng.integers(0, 12, m), rng.integers(0, 1024, m), t)]
    check_unfused(np.concatenate(out), mode=mode, index_base=7)
