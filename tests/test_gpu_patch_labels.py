"""Patch extraction with a negative packet_index_base: a label below zero is no
cluster's, so the records that carry one get empty patches, whichever kernel
meets them; the others' patches are the oracle's, bit for bit."""
import numpy as np
import pytest

import oracle.refiner as orf
import paper_2603_04942_gb300 as tpx
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base", [-1500, -(1 << 40)])
def test_labels_below_zero(base):
    import torch
    pk = synth.generate(synth.small(n_shots=12))[0]
    want, sel, centre, _ = orf.patches(pk, 12, idx_base=base)
    assert (want == 0).all(axis=1).any() and (want != 0).any() == (base + pk.size > 0)
    ctx = tpx.Context(tpx.Config(), max_packets=pk.size)
    try:
        d = torch.from_numpy(pk.view(np.int64)).cuda()
        out = ctx.alloc_outputs(pk.size, labels=True)
        ctx.tpx_process(d, out, base)
        ctx.tpx_sync()
        got = ctx.tpx_refine_patches(d, out["labels"], out["clusters"], int(out["n_clusters"].item()), 12, index_base=base)
        m = int(got["n"].item())
        assert m == sel.size
        assert np.array_equal(got["patches"][:m].cpu().numpy(), want)
        assert np.array_equal(got["centre"][:m].cpu().numpy(), centre)
    finally:
        ctx.close()
