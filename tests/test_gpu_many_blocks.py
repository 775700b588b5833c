"""The counts of more than 4096 blocks, which one block scans instead of every
placing block adding them up: the unfused calls on more than 4096 blocks of 4096
hits (against the oracle), and the choice of the clusters that get a patch from
more than 4096 blocks of 512 records (against the records)."""
import numpy as np
import pytest

import paper_2603_04942_gb300 as tpx
import synth
from test_gpu_general import check_unfused

pytestmark = pytest.mark.gpu


def test_unfused_hits():
    g, _ = check_unfused(synth.generate(synth.small(n_shots=36_000, seed=31))[0])
    assert g["hits"]["index"].size > 4096 * 4096


def test_selected_records():
    import torch
    pk = synth.generate(synth.small(n_shots=115_000, seed=32))[0]
    ctx = tpx.Context(tpx.Config(), max_packets=pk.size)
    try:
        d = torch.from_numpy(pk.view(np.int64)).cuda()
        out = ctx.alloc_outputs(pk.size, labels=True, cluster_capacity=2_400_000)
        ctx.tpx_process(d, out)
        ctx.tpx_sync()
        n = int(out["n_clusters"].item())
        assert n > 4096 * 512
        rec = np.frombuffer(out["clusters"][: 88 * n].cpu().numpy().tobytes(), tpx.CLUSTER_DTYPE)
        want = np.flatnonzero(rec["n"] > 24)
        assert want.size > 100_000 and want[-1] > 4096 * 512
        got = ctx.tpx_refine_patches(d, out["labels"], out["clusters"], n, 24, capacity=want.size)
        assert got["status"] == 0 and int(got["n"].item()) == want.size
        assert np.array_equal(got["sel"].cpu().numpy(), want)
        r = rec[want]
        for k, s in enumerate(("s_x", "s_y")):
            assert np.array_equal(got["centre"][:, k].cpu().numpy(), (2 * r[s] + r["s_tot"]) // (2 * r["s_tot"]))
        # the charge of a patch is a part of its cluster's, and of most all of it
        tot = got["patches"][:, :81].double().sum(1).cpu().numpy() * 1023 / r["s_tot"]
        assert tot.max() < 1.004 and np.median(tot) > 0.996   # bf16: 2^-9 relative
    finally:
        ctx.close()
