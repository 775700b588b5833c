"""The work that a user of this framework has it do, as measurable cases.

Each case names a public path (`kind`) and its sizes. Inputs are synthetic
TPX3 packet streams drawn on the GPU with the charge-cloud model of `synth`
(particles uniform over the sensor, Gaussian clouds thresholded at ToT 10,
readout ordered by ToA + 16 ToT + U(0, 1 us), a pixel dead while over
threshold), or refiner patches of such clouds.

  process   tpx_process + tpx_sync on packets in device memory
  batch     tpx_process_batch + tpx_sync: many runs in one launch
  host      tpx_process_host: pinned host buffers in and out
  unfused   tpx_decode, tpx_cluster, tpx_centroid
  stream    one chunk through an open Stream: submit, poll
  patches   tpx_refine_patches(_bf16) of a clustered stream
  infer     the learned refiner's network on patches, and its decision
  train     one minibatch step (loss, gradients, Adam)
"""
import math
import random

import numpy as np
import torch

import paper_2603_04942_gb300 as tpx
from paper_2603_04942_gb300 import refiner

PERIOD = 640_000                          # 1 kHz trigger period in ticks of 1.5625 ns
T_START = (1 << 34) - 320_000_000 - 3_200  # shot 500 straddles the first pixel wrap
WRAP_THR = 12_800_000_000
PIX_PER_PARTICLE = 23.9                   # times sigma^2: packets of a mean cloud (the pixels over threshold, less those at the edges and in dead time)
TICK = 1.5625


def listed():
    return [
        # a preview of a few shots while the acquisition is set up: the latency of one call
        dict(name="preview_37_shots", kind="process", shots=37, particles=20.0, poisson=False, mode="cc", radius=1, peaks=True),
        # the small run of the benchmark's configuration: 1 s of acquisition
        dict(name="run_1000_shots", kind="process", shots=1000, particles=20.0, poisson=False, mode="cc", radius=1, peaks=True),
        # a whole acquisition, the headline workload: 50 particles a shot, 5% overlapping pairs
        dict(name="acquisition_600k_shots", kind="process", shots=600_000, particles=50.0, poisson=True, pairs=0.05, mode="cc", radius=1),
        # the paper's own per-maximum neighbourhoods with a wider box, a timewalk table and int32 labels
        dict(name="paper_mode_radius2", kind="process", shots=20_011, particles=30.0, poisson=True, mode="paper", radius=2, timewalk=True, labels32=True),
        # independent runs of a parameter scan in one launch: electron- and ion-like, 1 to 500 particles a shot
        dict(name="batch_64_uneven_runs", kind="batch", runs=64, shots_lo=10, shots_hi=3000, particles_lo=1.0, particles_hi=500.0),
        # from host memory to host memory, the compact outputs
        dict(name="host_to_host_40k_shots", kind="host", shots=40_000, particles=20.0, poisson=True, compact=True),
        # dense ion shots, flight times over the whole period: the path in three calls
        dict(name="unfused_dense_ions", kind="unfused", shots=151, mhits=40.0),
        # live monitoring at 40 Mhit/s: a chunk of 5 to 45 ms in, the closed shots' records out
        dict(name="stream_chunk_40mhits", kind="stream", mhits=40.0, chunks=96, ms_lo=5.0, ms_hi=45.0),
        # the overlap refiner's windows of every cluster of an acquisition
        dict(name="patches_bf16_20k_shots", kind="patches", shots=20_000, particles=20.0, bf16=True),
        # which clusters hold two particles, and where: both networks
        dict(name="mlp_infer_1m", kind="infer", net="mlp", rows=1_000_003),
        dict(name="cnn_infer_1m", kind="infer", net="cnn", rows=1_000_003),
        # training the refiner, its default minibatch
        dict(name="mlp_train_4096", kind="train", net="mlp", rows=4096),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["process"] * 4 + ["paper", "batch", "host", "unfused", "stream", "patches", "infer", "infer", "train", "train"])
    if kind in ("process", "paper"):
        particles = log(1.0, 110.0)
        shots = int(min(log(20, 400_000), 2.5e7 / particles))
        c = dict(kind="process", shots=shots, particles=round(particles, 3), poisson=True, pairs=rng.choice([0.0, 0.05, 0.3]), mode="cc", radius=1,
                 peaks=rng.random() < 0.4, labels32=rng.random() < 0.3, records64=rng.random() < 0.2, timewalk=rng.random() < 0.3,
                 dark=rng.choice([0.0, 0.0, 2.0]))
        if kind == "paper":
            c.update(mode="paper", radius=rng.choice([1, 2, 3]), shots=int(min(shots, 1e6 / particles) + 3))
        elif rng.random() < 0.2:
            c.update(radius=2, shots=int(min(shots, 4e6 / particles) + 3))
        return c
    if kind == "batch":
        return dict(kind="batch", runs=int(log(8, 96)), shots_lo=10, shots_hi=int(log(100, 3000)), particles_lo=1.0, particles_hi=round(log(20, 500), 2))
    if kind == "host":
        return dict(kind="host", shots=int(log(200, 40_000)), particles=round(log(5, 50), 2), poisson=True, compact=rng.random() < 0.5)
    if kind == "unfused":
        return dict(kind="unfused", shots=int(log(20, 200)), mhits=round(log(5, 40), 2))
    if kind == "stream":
        return dict(kind="stream", mhits=round(log(10, 80), 1), chunks=int(rng.uniform(24, 64)), ms_lo=2.0, ms_hi=round(rng.uniform(20, 80), 1))
    if kind == "patches":
        return dict(kind="patches", shots=int(log(500, 30_000)), particles=round(log(5, 40), 2), bf16=rng.random() < 0.5)
    if kind == "infer":
        return dict(kind="infer", net=rng.choice(["mlp", "cnn"]), rows=int(log(1000, 2_000_000)))
    return dict(kind="train", net=rng.choice(["mlp", "cnn"]), rows=rng.choice([1024, 2048, 4096, 4096, 6000, 8192]))


# ------------------------------------------------------------------ inputs
def _gen(seed, part=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1_000_003 + part) & 0x7FFFFFFFFFFFFFFF)


def _clouds(g, shots, particles, poisson, sigma, tof_ns, pairs):
    """The hits (shot, x, y, ToT, ToA relative to the trigger, particle) of `shots` shots."""
    dev = "cuda"
    if poisson:
        counts = torch.poisson(torch.full((shots,), float(particles), device=dev), generator=g).long()
    else:
        counts = torch.full((shots,), int(particles), device=dev, dtype=torch.int64)
    shot = torch.repeat_interleave(torch.arange(shots, device=dev), counts)
    u = torch.rand((9, shot.numel()), device=dev, generator=g)
    cx, cy, peak = u[0] * 256, u[1] * 256, 200 + 823 * u[2]
    t0 = (tof_ns[0] + (tof_ns[1] - tof_ns[0]) * u[3]) / TICK
    if pairs:
        two = torch.nonzero(u[4] < pairs).flatten()
        sep, ang = 4 * u[5][two], 2 * math.pi * u[6][two]
        shot = torch.cat([shot, shot[two]])
        cx, cy = torch.cat([cx, cx[two] + sep * torch.cos(ang)]), torch.cat([cy, cy[two] + sep * torch.sin(ang)])
        t0 = torch.cat([t0, t0[two] + 20 / TICK * u[7][two]])
        peak = torch.cat([peak, peak[two] * (0.3 + 0.7 * u[8][two])])
    r = int(math.ceil(sigma * math.sqrt(2 * math.log(102.3))))
    off = torch.arange(-r, r + 1, device=dev)
    x, y = cx.round().long()[:, None] + off, cy.round().long()[:, None] + off
    ex = torch.exp(-(x - cx[:, None]) ** 2 / (2 * sigma * sigma)) * ((x >= 0) & (x < 256))
    ey = torch.exp(-(y - cy[:, None]) ** 2 / (2 * sigma * sigma)) * ((y >= 0) & (y < 256))
    amp = (peak[:, None, None] * ex[:, :, None]) * ey[:, None, :]
    p, i, j = torch.nonzero(amp >= 10, as_tuple=True)
    tot = amp[p, i, j].long().clamp_(max=1023)
    toa = (t0[p] + 3 / TICK * torch.randn(p.numel(), device=dev, generator=g)).round().long().clamp_(min=0)
    return shot[p], x[p, i], y[p, j], tot, toa, p


def _live(shot, x, y, tot, toa, p):
    """Without the hits of a pixel that is still over threshold."""
    key = (((shot << 16) | (y << 8) | x) << 24) | toa
    key, order = torch.sort(key, stable=True)
    shot, x, y, tot, toa, p = (v[order] for v in (shot, x, y, tot, toa, p))
    busy = torch.zeros_like(key, dtype=torch.bool)
    busy[1:] = ((key[1:] >> 24) == (key[:-1] >> 24)) & (toa[1:] < toa[:-1] + 16 * tot[:-1])
    live = ~busy
    return (v[live] for v in (shot, x, y, tot, toa, p))


def _pixel_words(x, y, tot, t):
    c = torch.div(t + 15, 16, rounding_mode="floor")
    ftoa = c * 16 - t
    c = c & ((1 << 30) - 1)
    return (torch.full_like(t, (0xB << 60) - (1 << 64)) | ((x >> 1) << 53) | ((y >> 2) << 47) | ((((x & 1) << 2) | (y & 3)) << 44)
            | ((c & 0x3FFF) << 30) | (tot << 20) | (ftoa << 16) | (c >> 14))


def _acquisition(seed, shots, particles, poisson=True, sigma=1.0, tof_ns=(1000.0, 10000.0), pairs=0.0, dark=0.0, t_start=T_START, each=0):
    """The packets (int64 on the GPU) of an acquisition. `each`: that many pixels in every shot, and in one piece, so that pixels may be read out after later triggers."""
    per = shots if each else max(1, int(4e5 / max(1.0, particles)))
    parts = []
    for k, s0 in enumerate(range(0, shots, per)):
        n = min(per, shots - s0)
        g = _gen(seed, k)
        shot, x, y, tot, toa, p = _live(*_clouds(g, n, particles, poisson, sigma, tof_ns, pairs))
        if each:   # the first clouds of every shot
            by = torch.sort(p, stable=True).indices
            counts = torch.bincount(shot, minlength=n)
            assert int(counts.min()) >= each
            at = torch.arange(by.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(counts, 0) - counts, counts)
            shot, x, y, tot, toa = (v[by[at < each]] for v in (shot, x, y, tot, toa))
            toa = toa.clamp(max=PERIOD - 2)
        if dark:
            nd = int(n * dark)
            u = torch.rand((5, nd), device="cuda", generator=g)
            more = [(u[0] * n).long(), (u[1] * 256).long(), (u[2] * 256).long(), 10 + (51 * u[3]).long(), (u[4] * (PERIOD - 20_000)).long()]
            shot, x, y, tot, toa = (torch.cat([a, b]) for a, b in zip((shot, x, y, tot, toa), more))
        t = shot * PERIOD + toa
        late = torch.randint(0, 641, t.shape, device="cuda", generator=g)
        trig = torch.arange(n, device="cuda") * PERIOD
        key = torch.cat([2 * (t + 16 * tot + late) + 1, 2 * trig])
        t0 = t_start + s0 * PERIOD
        tdc = (torch.full_like(trig, 0x6 << 60)) | ((((trig + t0) >> 1) & ((1 << 35) - 1)) << 9)
        words = torch.cat([_pixel_words(x, y, tot, t + t0), tdc])
        parts.append(words[torch.sort(key, stable=True).indices])
    return torch.cat(parts)


def _per_shot(particles, sigma=1.0, pairs=0.0, dark=0.0):
    return particles * PIX_PER_PARTICLE * sigma * sigma * (1.0 + 0.6 * pairs) + dark + 1


def _buffer(seed, shots, particles, poisson=True, sigma=1.0, tof_ns=(1000.0, 10000.0), pairs=0.0, dark=0.0, t_start=T_START):
    """The first packets of an acquisition of about `shots` shots, as many for every seed: a receive buffer, which ends inside a shot."""
    n = int(shots * _per_shot(particles, sigma, pairs, dark)) | 1
    more = shots + shots // 16 + 4
    while True:
        pk = _acquisition(seed, more, particles, poisson, sigma, tof_ns, pairs, dark, t_start)
        if pk.numel() >= n:
            return pk[:n].clone()
        more += more // 4 + 8


def _ions(seed, shots, mhits):
    """Dense ion shots of mhits * 1000 pixels each, flight times over the whole period."""
    return _acquisition(seed, shots, mhits * 1e3 / (0.85 * PIX_PER_PARTICLE * 1.44), False, 1.2, (0.0, 999_999.0), each=int(mhits * 1e3))


def _runs(case):
    """The runs of a batch: shots, particles a shot, sigma, flight times, start."""
    r = random.Random(case["runs"] * 7 + 1)
    out = []
    for k in range(case["runs"]):
        shots = int(round(math.exp(r.uniform(math.log(case["shots_lo"]), math.log(case["shots_hi"])))))
        mean = math.exp(r.uniform(math.log(case["particles_lo"]), math.log(case["particles_hi"])))
        ion = r.random() < 0.5
        out.append((shots, mean, 1.2 if ion else 0.6, (1000.0, 20000.0) if ion else (0.0, 50.0), 2 * r.randrange(1 << 33)))
    return out


def _timewalk():
    """A timewalk table of Eq. 1's form: 1500 ns / (ToT + 5)."""
    return torch.round(1500 / TICK / (torch.arange(1024, dtype=torch.float64) + 5)).to(torch.int16).cuda()


def _patches(seed, rows):
    """Patches of one- and two-particle clouds as the extraction leaves them: ToT/1023 rounded to bf16, times in 1/32 units."""
    g = _gen(seed, 1)
    out = torch.empty((rows, 162), dtype=torch.float32, device="cuda")
    ax = torch.arange(-4, 5, device="cuda", dtype=torch.float32)
    for a in range(0, rows, 250_000):
        n = min(250_000, rows - a)
        u = torch.rand((8, n), device="cuda", generator=g)
        amp = torch.zeros((n, 9, 9), device="cuda")
        for k in range(2):
            px, py = 3 * (u[2 * k] - 0.5), 3 * (u[2 * k + 1] - 0.5)
            h = (200 + 823 * u[4]) * (1.0 if k == 0 else (u[5] < 0.5) * (0.3 + 0.7 * u[6]))
            amp += h[:, None, None] * torch.exp(-(ax - py[:, None]) ** 2 / 2)[:, :, None] * torch.exp(-(ax - px[:, None]) ** 2 / 2)[:, None, :]
        tot = torch.where(amp >= 10, amp.clamp(max=1023).floor(), 0.0)
        dt = torch.where(tot > 0, torch.randint(0, 24, tot.shape, device="cuda", generator=g) / 32, 0.0)
        out[a:a + n, :81] = (tot / 1023).to(torch.bfloat16).float().reshape(n, 81)
        out[a:a + n, 81:] = dt.reshape(n, 81)
    return out


def _weights(seed, net):
    """A network's parameters as training leaves them: scaled uniform weights, small biases (the layout of the framework's parameter vector)."""
    rng = np.random.default_rng(seed)
    h = refiner.HIDDEN
    layers = [(162, 162 * h, h), (h, h * h, h), (h, 6 * h, 6)] if net == "mlp" else [(18, 288, 16), (144, 2304, 16), (144, 4608, 32), (288, 41472, 144), (144, 864, 6)]
    return np.concatenate([np.concatenate([rng.uniform(-1, 1, size) * math.sqrt(6 / fan), 0.05 * rng.standard_normal(bias)])
                           for fan, size, bias in layers]).astype(np.float32)


def _net(ctx, case, seed):
    net = refiner.Refiner(ctx) if case["net"] == "mlp" else refiner.CnnRefiner(ctx)
    net.params.copy_(torch.from_numpy(_weights(seed, case["net"])))
    return net


def _targets(case, seed):
    """Training targets: the count and the offsets of one or two particles; Adam's moments of a run under way."""
    g = _gen(seed, 2)
    y = 3 * (torch.rand((case["rows"], 5), device="cuda", generator=g) - 0.5)
    y[:, 0] = 1 + (y[:, 0] > 0)
    y[y[:, 0] == 1, 3:] = 0
    n = _weights(0, case["net"]).size
    m = 1e-3 * torch.randn(n, device="cuda", generator=g)
    v = 1e-6 + 1e-5 * torch.rand(n, device="cuda", generator=g)
    return y, m, v


def _packets(case, seed):
    kind = case["kind"]
    if kind == "batch":
        runs = [_buffer(seed * 131 + k, s, m, True, sig, tof, t_start=t0) for k, (s, m, sig, tof, t0) in enumerate(_runs(case))]
        return torch.cat(runs), np.concatenate([[0], np.cumsum([r.numel() for r in runs])]).astype(np.int64)
    if kind == "unfused":
        return _ions(seed, case["shots"], case["mhits"])
    return _buffer(seed, case["shots"], case["particles"], case.get("poisson", True), pairs=case.get("pairs", 0.3 if kind == "patches" else 0.0),
                        dark=case.get("dark", 0.0))


def _config(case):
    r = case.get("radius", 1)
    return tpx.Config(rx=r, ry=r, mode=tpx.MODE_PAPER if case.get("mode") == "paper" else tpx.MODE_CC, timewalk_lut=_timewalk() if case.get("timewalk") else None,
                      labels32=bool(case.get("labels32")), records64=bool(case.get("records64")),
                      tof_max_ticks=PERIOD - 1 if case["kind"] in ("unfused", "stream") else 64_000)


def _records(buf, words):
    """The whole numbers and the 64-bit floats of a record buffer, as views of it."""
    r = {"whole": buf.view(torch.int64).view(-1, words)[:, :8]}
    if words == 11:
        r["float"] = buf.view(torch.float64).view(-1, words)[:, 8:]
    return r


def _cleared(out):
    for v in out.values():
        if isinstance(v, torch.Tensor):
            v.zero_()
    return out


def _caps(case, n):
    """Record and trigger capacities as a program sizes them: from the particles that it expects, twice over."""
    shots = sum(r[0] for r in _runs(case)) if case["kind"] == "batch" else case["shots"]
    if case.get("mode") == "paper" or case["kind"] == "batch":
        return max(4096, n // 4), shots + shots // 8 + 64
    return min(n, int(1.5 * shots * (case["particles"] + case.get("dark", 0)) + 4096)), shots + shots // 8 + 64


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind in ("process", "batch"):
        pk = _packets(case, seed)
        pk, s["runs"] = pk if kind == "batch" else (pk, None)
        n = pk.numel()
        cap, tcap = _caps(case, n)
        cfg = _config(case)
        ctx = tpx.Context(cfg, max_packets=n)
        if kind == "batch":
            out = ctx.alloc_batch_outputs(n, case["runs"], labels=True, cluster_capacity=cap, trig_capacity=tcap)
        else:
            out = ctx.alloc_outputs(n, True, bool(case.get("peaks")), cap, tcap)
        _cleared(out)
        res = _records(out["clusters"], 8 if cfg.records64 else 11)
        res.update({k: out[k] for k in ("labels", "is_peak", "n_clusters", "n_trig", "trig", "run_clusters", "run_trig") if out.get(k) is not None})
        s.update(ctx=ctx, cfg=cfg, pk=pk, out=out, res=res)
    elif kind == "host":
        pk = _packets(case, seed)
        n = pk.numel()
        cap, tcap = _caps(case, n)
        cfg = tpx.Config(labels32=case["compact"], records64=case["compact"])

        def pinned(size, dtype):
            return torch.zeros(size, dtype=dtype, pin_memory=True).numpy()

        host = torch.empty(n, dtype=torch.int64, pin_memory=True)
        host.copy_(pk)
        rec = pinned(cap * (8 if case["compact"] else 11), torch.int64)
        s.update(ctx=tpx.Context(cfg, max_packets=n), cfg=cfg, keep=host, pk=host.numpy().view(np.uint64), labels=pinned(n, torch.int32 if case["compact"] else torch.int64),
                 rec=rec, clusters=rec.view(cfg.record_dtype()), trig=pinned(tcap, torch.int64))
        words = rec.reshape(-1, 8 if case["compact"] else 11)
        s["res"] = {"whole": words[:, :8], "labels": s["labels"], "trig": s["trig"]}
        if not case["compact"]:
            s["res"]["float"] = rec.view(np.float64).reshape(-1, 11)[:, 8:]
    elif kind == "unfused":
        pk = _packets(case, seed)
        s.update(ctx=tpx.Context(_config(case), max_packets=pk.numel()), pk=pk, room=pk.numel() - case["shots"])
    elif kind == "stream":
        r = random.Random(case["chunks"] * 31 + 5)
        ms = [r.uniform(case["ms_lo"], case["ms_hi"]) for _ in range(case["chunks"])]
        pk = _ions(seed, int(sum(ms)), case["mhits"])
        host = torch.empty(pk.numel(), dtype=torch.int64, pin_memory=True)
        host.copy_(pk)
        cuts = np.concatenate([[0], np.cumsum(ms)]) / sum(ms) * host.numel()
        cuts = cuts.astype(np.int64)
        words = host.numpy().view(np.uint64)
        s.update(keep=host, chunks=[words[a:b] for a, b in zip(cuts[:-1], cuts[1:])], at=0, cfg=_config(case), stream=None,
                 room=int(max(cuts[1:] - cuts[:-1])), hold=int(case["mhits"] * 1e3 * 6))
        shots = int(sum(ms)) + 8
        s.update(rec=np.zeros((int(shots * case["mhits"] * 40), 11), np.int64), trig=np.zeros(shots, np.int64))
        _open(s)
    elif kind == "patches":
        pk = _packets(case, seed)
        n = pk.numel()
        cap, tcap = _caps(case, n)
        ctx = tpx.Context(tpx.Config(), max_packets=n)
        out = ctx.alloc_outputs(n, True, False, cap, tcap)
        ctx.tpx_process(pk, out)
        ctx.tpx_sync()
        s.update(ctx=ctx, pk=pk, out=out, n=int(out["n_clusters"].item()), room=int(1.3 * case["shots"] * case["particles"]) + 1024)
    elif kind == "infer":
        ctx = tpx.Context(tpx.Config(), max_packets=1 << 16)
        n = case["rows"]
        x = _patches(seed, n)
        g = _gen(seed, 3)
        rec = torch.zeros((n, 11), dtype=torch.int64, device="cuda")
        rec.view(torch.float64)[:, 8:10] = 256 * torch.rand((n, 2), device="cuda", generator=g, dtype=torch.float64)
        s.update(ctx=ctx, net=_net(ctx, case, seed), rec=rec, sel=torch.arange(n, device="cuda"), centre=rec.view(torch.float64)[:, 8:10].round().to(torch.int32).contiguous(),
                 x=x if case["net"] == "mlp" else x.to(torch.bfloat16).view(torch.int16))
    else:
        ctx = tpx.Context(tpx.Config(), max_packets=1 << 16)
        net = _net(ctx, case, seed)
        y, m, v = _targets(case, seed)
        net.m.copy_(m)
        net.v.copy_(v)
        n = case["rows"]
        work = torch.empty(n * (4 * refiner.HIDDEN + 12) if case["net"] == "mlp" else int(tpx.lib().tpx_cnn_work_floats(n)), dtype=torch.float32, device="cuda")
        s.update(ctx=ctx, net=net, x=_patches(seed, n), y=y, work=work, loss=torch.zeros(1, device="cuda"))
    return s


def _open(s):
    s["stream"] = tpx.Stream(s["cfg"], max_chunk_packets=s["room"], max_hold_packets=s["hold"], hold_triggers=2, slots=4)
    s["at"], s["used"] = 0, (0, 0)


# -------------------------------------------------------------- the passes
def run(s):
    kind = s["kind"]
    if kind == "process":
        s["ctx"].tpx_process(s["pk"], s["out"])
        s["ctx"].tpx_sync()
        return s["res"]
    if kind == "batch":
        s["ctx"].tpx_process_batch(s["pk"], s["runs"], s["out"])
        s["ctx"].tpx_sync()
        return s["res"]
    if kind == "host":
        _, n_cl, n_tr = s["ctx"].tpx_process_host(s["pk"], s["labels"], None, s["clusters"], s["trig"])
        return dict(s["res"], n_clusters=n_cl, n_trig=n_tr)
    if kind == "unfused":
        ctx = s["ctx"]
        d = ctx.tpx_decode(s["pk"], hits_capacity=s["room"], trig_capacity=s["case"]["shots"])
        n = int(d["n_hits"].item())
        c = ctx.tpx_cluster(d["hits"], n, is_peak=True)
        r = ctx.tpx_centroid(d["hits"], c["labels"], c["is_peak"], n, cluster_capacity=s["room"] // 16)
        m = int(r["n_clusters"].item())
        r["clusters"][88 * m:].zero_()   # the buffer's free end, so that it is the same each time
        return dict(_records(r["clusters"], 11), labels=c["labels"], is_peak=c["is_peak"], n_trig=d["n_trig"], trig=d["trig"], **d["hits"])
    if kind == "stream":
        if s["at"] == len(s["chunks"]):   # the acquisition is over: the next one begins
            s["stream"].close()
            _open(s)
        t = s["stream"].submit(s["chunks"][s["at"]])
        r = s["stream"].poll(t)
        s["at"] += 1
        # the records and trigger times join the acquisition's
        a, b = s["used"]
        m, k = r["clusters"].size, r["triggers"].size
        s["rec"][a:a + m] = r["clusters"].view(np.int64).reshape(-1, 11)
        s["trig"][b:b + k] = r["triggers"]
        s["used"] = (a + m, b + k)
        return {"whole": s["rec"][:, :8], "float": s["rec"].view(np.float64)[:, 8:], "trig": s["trig"], "n": a + m, "n_trig": b + k, "first_shot": r["first_shot"]}
    if kind == "patches":
        f = s["ctx"].tpx_refine_patches_bf16 if s["case"]["bf16"] else s["ctx"].tpx_refine_patches
        p = f(s["pk"], s["out"]["labels"], s["out"]["clusters"], s["n"], capacity=s["room"])
        n = int(p["n"].item())
        res = {k: p[k] for k in ("patches", "sel", "centre")}
        for v in res.values():
            v[n:].zero_()   # the buffers' free ends, so that they are the same each time
        return dict(res, n=n)
    if kind == "infer":
        n = s["case"]["rows"]
        logits = s["net"].infer(s["x"], n)
        return {"logits": logits, "hits": s["ctx"].tpx_refine_decide(logits, s["rec"], s["sel"], s["centre"], n, 0.8)}
    net, n = s["net"], s["case"]["rows"]
    if s["case"]["net"] == "mlp":
        s["ctx"].tpx_refiner_train_step(net.params, net.m, net.v, net.grad, net.h, 500, s["x"], s["y"], 1e-3, 1.0, s["work"], s["loss"], n=n)
    else:
        s["ctx"].tpx_cnn_train_step(net.params, net.m, net.v, net.grad, 500, s["x"], s["y"], 1e-3, 1.0, s["work"], s["loss"], n=n)
    return {"params": net.params, "m": net.m, "v": net.v, "grad": net.grad, "loss": s["loss"]}


def work(case):
    kind = case["kind"]
    if kind in ("infer", "train"):
        n, mlp = case["rows"], case["net"] == "mlp"
        fl = 105_664 if mlp else 311_040
        p = _weights(0, case["net"]).size
        if kind == "infer":
            return {"bytes": n * ((648 if mlp else 324) + 24 + 88 + 16 + 20) + 4 * p, "flops": n * fl}
        return {"bytes": n * (648 + 20) + 4 * p * 7, "flops": 3 * n * fl}
    if kind == "stream":
        px = 0.5 * (case["ms_lo"] + case["ms_hi"]) * case["mhits"] * 1e3
        return {"bytes": (8 + 88 / (PIX_PER_PARTICLE * 1.44)) * px, "flops": 0}
    if kind == "batch":
        runs = _runs(case)
        px = sum(a * _per_shot(b, c) for a, b, c, _, _ in runs)
        return {"bytes": 16 * px + 56 * sum(r[0] * r[1] for r in runs) + 8 * sum(r[0] for r in runs), "flops": 0}
    shots = case["shots"]
    if kind == "unfused":   # packets in; hits out; hits in, labels and peaks out; hits, labels and peaks in
        px = shots * case["mhits"] * 1e3
        hits = 8 * 3 + 4 + 1 + 1 + 2
        return {"bytes": px * (8 + 3 * hits + 2 * 9 + 88 / (PIX_PER_PARTICLE * 1.44)) + 8 * shots, "flops": 0}
    px = shots * _per_shot(case["particles"], 1.0, case.get("pairs", 0.3 if kind == "patches" else 0.0), case.get("dark", 0.0))
    if kind == "patches":
        return {"bytes": 16 * px + shots * case["particles"] * (88 + (324 if case["bf16"] else 648) + 16), "flops": 0}
    lab = 4 if case.get("labels32") or case.get("compact") else 8
    return {"bytes": px * (8 + lab + (1 if case.get("peaks") else 0)) + 56 * shots * case["particles"] + 8 * shots, "flops": 0}


# ------------------------------------------- what the outputs are, in 64 bits
def _unwrap(raw, period):
    if raw.numel() == 0:
        return raw
    d = raw[1:] - raw[:-1]
    step = (d < -WRAP_THR).long() - (d > WRAP_THR).long()
    return raw + period * torch.cat([torch.zeros(1, dtype=torch.int64, device=raw.device), torch.cumsum(step, 0)])


def _decoded(w, tof_max, lut):
    """Kept pixels in stream order: index, shot, t (corrected), trigger time, x, y, ToT."""
    head = (w >> 60) & 15
    ip, it = torch.nonzero(head == 0xB).flatten(), torch.nonzero(head == 0x6).flatten()
    p, q = w[ip], w[it]
    t = _unwrap((((((p & 0xFFFF) << 14) | ((p >> 30) & 0x3FFF)) * 16) - ((p >> 16) & 15)) & ((1 << 34) - 1), 1 << 34)
    trig = _unwrap((2 * ((q >> 9) & ((1 << 35) - 1))), 1 << 36)
    shot = torch.searchsorted(trig, t, right=True) - 1
    base = trig[shot.clamp(min=0)]
    keep = torch.nonzero((shot >= 0) & (t - base <= tof_max)).flatten()
    ip, p, t, shot, base = ip[keep], p[keep], t[keep], shot[keep], base[keep]
    pix = (p >> 44) & 7
    tot = (p >> 20) & 1023
    if lut is not None:
        t = t - lut.long()[tot]
    return ip, shot, t, base, 2 * ((p >> 53) & 127) + (pix >> 2), 4 * ((p >> 47) & 63) + (pix & 3), tot


def _pairs(shot, x, y, tof, r, dt):
    """Adjacent pixels (a, b), each pair once: box neighbours of one shot, |dt| within the radius."""
    span, bias = 1 << 21, 1 << 16
    key = (((shot * 272) + y + 8) * 272 + x + 8) * span + tof + bias
    key, order = torch.sort(key)
    cell, time = torch.div(key, span, rounding_mode="floor"), key % span
    me = torch.arange(key.numel(), device=key.device)
    found = []
    for dy in range(r + 1):
        for dx in range(-r if dy else 0, r + 1):
            at = (cell + 272 * dy + dx) * span
            lo = me + 1 if dx == dy == 0 else torch.searchsorted(key, at + time - dt)
            n = torch.searchsorted(key, at + time + dt, right=True) - lo
            a = torch.repeat_interleave(me, n)
            b = torch.arange(a.numel(), device=key.device) - torch.repeat_interleave(torch.cumsum(n, 0) - n, n) + torch.repeat_interleave(lo, n)
            found.append(torch.stack([order[a], order[b]]))
    return torch.cat(found, 1)


def _centroids(w, tof_max, lut, paper, r, dt=32):
    """x, y, tof of every record of a stream, in ascending label order (float64 [records x 3])."""
    index, shot, t, base, x, y, tot = _decoded(w, tof_max, lut)
    n, tof = index.numel(), t - base
    a, b = _pairs(shot, x, y, tof, r, dt)
    # (time, position) order, time first
    rank = torch.empty(n, dtype=torch.int64, device=w.device)
    rank[torch.sort(t * 1, stable=True).indices] = torch.arange(n, device=w.device)
    if paper:
        dim = torch.zeros(n, dtype=torch.bool, device=w.device)
        first = (tot[a] > tot[b]) | ((tot[a] == tot[b]) & (index[a] > index[b]))
        dim[torch.where(first, b, a)] = True
        owner = torch.cat([a, b, torch.arange(n, device=w.device)])
        member = torch.cat([b, a, torch.arange(n, device=w.device)])
        live = torch.nonzero(~dim[owner]).flatten()
        owner, member = owner[live], member[live]
        roots = torch.nonzero(~dim).flatten()
    else:
        byrank = torch.sort(rank).indices
        lab = rank.clone()
        ra, rb = rank[a], rank[b]
        lab = torch.arange(n, device=w.device)     # over ranks: the earliest member's rank
        while True:
            m = torch.minimum(lab[ra], lab[rb])
            new = lab.clone()
            new.scatter_reduce_(0, lab[ra], m, "amin")
            new.scatter_reduce_(0, lab[rb], m, "amin")
            new.scatter_reduce_(0, ra, m, "amin")
            new.scatter_reduce_(0, rb, m, "amin")
            for _ in range(3):
                new = new[new]
            if torch.equal(new, lab):
                break
            lab = new
        owner, member = byrank[lab[rank]], torch.arange(n, device=w.device)
        roots = torch.nonzero(owner == member).flatten()
    tmin = torch.full((n,), 1 << 60, dtype=torch.int64, device=w.device).scatter_reduce_(0, owner, tof[member], "amin")
    sums = []
    for v in (torch.ones_like(tot), x, y):
        sums.append(torch.zeros(n, dtype=torch.int64, device=w.device).index_add_(0, owner, (tot * v)[member]))
    st = torch.zeros(n, dtype=torch.int64, device=w.device).index_add_(0, owner, tot[member] * (tof[member] - tmin[owner]))
    s = [v[roots].double() for v in sums]
    return torch.stack([s[1] / s[0], s[2] / s[0], tmin[roots].double() + st[roots].double() / s[0]], 1)


def _network(p, net, x):
    """The plain network in the precision of p and x, logits [rows x 6]."""
    sizes, at, w = [], 0, []
    h = refiner.HIDDEN
    sizes = [(162, h), (h,), (h, h), (h,), (h, 6), (6,)] if net == "mlp" else [(16, 2, 3, 3), (16,), (16, 16, 3, 3), (16,), (32, 16, 3, 3), (32,), (144, 288), (144,), (6, 144), (6,)]
    for s in sizes:
        k = math.prod(s)
        w.append(p[at:at + k].view(s))
        at += k
    if net == "mlp":
        x = torch.relu(x @ w[0] + w[1])
        x = torch.relu(x @ w[2] + w[3])
        return x @ w[4] + w[5]
    x = x.view(-1, 2, 9, 9)
    for k in (0, 2, 4):
        # a valid convolution as a product, so that it is plain 64-bit arithmetic
        cols = torch.nn.functional.unfold(x, 3)
        side = x.shape[-1] - 2
        x = torch.relu(w[k].reshape(w[k].shape[0], -1) @ cols + w[k + 1][:, None]).view(x.shape[0], -1, side, side)
    x = torch.relu(x.flatten(1) @ w[6].T + w[7])
    return x @ w[8].T + w[9]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("process", "batch", "host"):
        if kind == "host" and case["compact"] or case.get("records64") or work(case)["bytes"] > 2e9:
            return None
        got = _packets(case, seed)
        w, offs = got if kind == "batch" else (got, [0, got.numel()])
        lut = _timewalk() if case.get("timewalk") else None
        rows = torch.cat([_centroids(w[a:b], 64_000, lut, case.get("mode") == "paper", case.get("radius", 1)) for a, b in zip(offs[:-1], offs[1:])])
        full = torch.zeros((_caps(case, w.numel())[0], 3), dtype=torch.float64, device="cuda")
        full[: rows.shape[0]] = rows
        return {"float": full}
    if kind == "unfused":
        rows = _centroids(_packets(case, seed), PERIOD - 1, None, False, 1)
        full = torch.zeros((int(case["mhits"] * 1e3) * case["shots"] // 16, 3), dtype=torch.float64, device="cuda")
        full[: rows.shape[0]] = rows
        return {"float": full}
    if kind == "infer":
        p = torch.from_numpy(_weights(seed, case["net"])).cuda().double()
        x = _patches(seed, case["rows"])
        return {"logits": torch.cat([_network(p, case["net"], x[a:a + 50_000].double()) for a in range(0, x.shape[0], 50_000)])}
    if kind == "train":
        p = torch.from_numpy(_weights(seed, case["net"])).cuda().double().requires_grad_(True)
        x = _patches(seed, case["rows"]).double()
        y, m, v = (t.double() for t in _targets(case, seed))
        o = _network(p, case["net"], x)
        two = (y[:, 0] == 2)
        ce = torch.nn.functional.cross_entropy(o[:, :2], two.long())
        off = ((o[:, 2:4] - y[:, 1:3]) ** 2).sum(1) + torch.where(two, ((o[:, 4:6] - y[:, 3:5]) ** 2).sum(1), 0.0)
        loss = ce + 0.5 * off.mean()
        loss.backward()
        g = p.grad
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        step = 1e-3 * (m / (1 - 0.9 ** 500)) / ((v / (1 - 0.999 ** 500)).sqrt() + 1e-8)
        return {"params": p.detach() - step, "m": m, "v": v, "grad": g, "loss": loss.detach().reshape(1)}
    return None
