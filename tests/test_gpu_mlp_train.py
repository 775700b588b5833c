"""The perceptron refiner's fused training step against the float64 oracle at
the edges of its tiles: one row, rows short of and past a CTA's 32 and a
cluster's eighth, widths of one column to the widest it takes (160), and the
general GEMMs one past that."""
import numpy as np
import pytest

import oracle.refiner as orf
import paper_2603_04942_gb300 as tpx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h", [1, 33, 64, 80, 160, 161])
@pytest.mark.parametrize("n", [1, 31, 257, 2049])
def test_step_matches_the_oracle(h, n):
    import torch
    rng = np.random.default_rng(1000 * h + n)
    x = np.where(rng.random((n, 162)) < 0.3, rng.random((n, 162)), 0).astype(np.float32)
    y = np.concatenate([rng.integers(1, 3, (n, 1)), rng.normal(size=(n, 4))], axis=1).astype(np.float32)
    p0 = (0.1 * rng.normal(size=int(tpx.Context.tpx_refiner_params(h)))).astype(np.float32)
    m0 = (1e-3 * rng.normal(size=p0.size)).astype(np.float32)
    v0 = (1e-6 + 1e-5 * rng.random(p0.size)).astype(np.float32)
    w, lr, step = 0.7, 1e-3, 41
    ctx = tpx.Context(tpx.Config(), max_packets=16)
    try:
        P, m, v = (torch.from_numpy(a.copy()).cuda() for a in (p0, m0, v0))
        g = torch.zeros_like(P)
        work = torch.empty(n * (4 * h + 12), dtype=torch.float32, device="cuda")
        loss = torch.zeros(1, dtype=torch.float32, device="cuda")
        ctx.tpx_refiner_train_step(P, m, v, g, h, step, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), lr, w, work, loss)
        torch.cuda.synchronize()
        P, m, v, g, loss = (t.cpu().numpy().astype(np.float64) for t in (P, m, v, g, loss))
    finally:
        ctx.close()
    pd = p0.astype(np.float64)
    og = orf.grad(pd, h, x, y, w)
    op, om, ov = orf.adam(pd, m0.astype(np.float64), v0.astype(np.float64), og, step, lr)
    # fp32 sums of at most 2049 products, each chain below 400: relative error
    # of the summed magnitudes below 400 * 2^-24 = 2.4e-5
    gs = np.abs(og).max()
    assert abs(loss[0] - orf.loss(pd, h, x, y, w)) <= 1e-5 * abs(loss[0]) + 1e-6
    assert np.abs(g - og).max() <= 1e-4 * gs
    assert np.abs(m - om).max() <= 1e-5 * gs + 1e-9
    assert np.abs(v - ov).max() <= 1e-6 * gs * gs + 1e-5 * ov.max()
    # v stays far from zero, so the update follows m's and v's relative errors
    assert np.abs(P - op).max() <= 1e-6 + 1e-2 * lr
