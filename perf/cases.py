"""What a user of the codec has it do, as measurable cases.

Every case goes through the Python entry points (`zc`, `collectives`,
`selector`).  `listed()` gives the fixed cases, `draw()` more of the same
ranges.  Operations (`op`):

  roundtrip  compress one tensor, decompress the stream
  compress   compress one tensor
  decompress decompress one stream
  ring       ring Allreduce of P rank buffers
  redoub     recursive-doubling Allreduce of P rank buffers
  scatter    pack of P uneven segments into P streams
  batch      many uneven messages in one launch, and back
  select     statistics, networks, selection, grouped batch of 64 KiB chunks
  train      one epoch of the selector's network

Output buffers are zero-filled once, so that the bytes behind a stream's end
compare like the stream itself.
"""
import math

import numpy as np
import torch

from paper_2308_05199_gb300 import collectives, selector, workloads, zc

DEV = "cuda"
BLOCKS = (16, 32, 64, 128)


# ---- cases ------------------------------------------------------------------------

def listed():
    return [
        # the smallest messages of a gradient exchange (4 KiB): launches and latency
        {"name": "message_4k", "op": "roundtrip", "data": "tdist", "n": 1024, "dtype": "f32",
         "block": 32, "mode": "abs", "eb": 1e-3, "heads": False},
        # a 4 MiB 1-D signal, the small correctness workload of the bench
        {"name": "signal_4m", "op": "roundtrip", "data": "signal", "n": 1 << 20, "dtype": "f32",
         "block": 32, "mode": "abs", "eb": 1e-4, "heads": False},
        # a BF16 gradient bucket of odd length
        {"name": "bucket_bf16", "op": "roundtrip", "data": "tdist", "n": 13000001, "dtype": "bf16",
         "block": 128, "mode": "abs", "eb": 1e-3, "heads": False},
        # a snapshot of a simulation on a 203^3 grid at a tight bound
        {"name": "field_203_tight", "op": "compress", "data": "field", "n": 203 ** 3,
         "dtype": "f32", "block": 64, "mode": "rel", "eb": 1e-4, "heads": False},
        # a 512^3 volume, the size of the paper's RTM snapshots: writing it ...
        {"name": "field_512_write", "op": "compress", "data": "field", "n": 1 << 27,
         "dtype": "f32", "block": 32, "mode": "rel", "eb": 1e-3, "heads": False},
        # ... and reading it back
        {"name": "field_512_read", "op": "decompress", "data": "field", "n": 1 << 27,
         "dtype": "f32", "block": 32, "mode": "rel", "eb": 1e-3, "heads": False},
        # the image-stacking Allreduce, 8 ranks of 8192^2 pixels
        {"name": "ring_8x8192sq", "op": "ring", "P": 8, "n": 1 << 26, "block": 32, "eb": 1e-3},
        # a remainder rank count and ragged buffers, whole-buffer exchanges
        {"name": "redoub_5x1m", "op": "redoub", "P": 5, "n": 1000003, "block": 32, "eb": 1e-3},
        # a root's compressed Scatterv of a volume to 8 ranks
        {"name": "scatterv_8", "op": "scatter", "P": 8, "n": 50000000, "dtype": "f32", "block": 32,
         "mode": "rel", "eb": 1e-2},
        # gradient buckets, 4 KiB - 64 MiB, half FP32 and half BF16, one launch each way
        {"name": "batch_250", "op": "batch", "messages": 250, "lo": 4096, "hi": 64 << 20,
         "block": 128},
        # a mixed workload cut into 64 KiB chunks, each stored as the selector picks
        {"name": "select_1g", "op": "select", "bytes": 1 << 30, "link": 12.5},
        # training of the selector's network, one epoch at the default minibatch
        {"name": "train_epoch", "op": "train", "rows": 10000, "batch": 256},
    ]


def _log(rng, lo, hi):
    """Log-uniform integer in [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["roundtrip", "roundtrip", "compress", "decompress", "ring", "redoub",
                     "scatter", "batch", "select", "train"])
    if op in ("roundtrip", "compress", "decompress"):
        data = rng.choice(["signal", "field", "tdist", "offset"])
        mode = "abs" if data == "tdist" else rng.choice(["abs", "rel"])
        eb = {"tdist": 1e-3, "signal": 1e-4, "field": 1e-3, "offset": 1e-3}[data] * \
            rng.choice([0.5, 1.0, 4.0])
        return {"op": op, "data": data, "n": _log(rng, 1 << 10, 1 << 24 if op == "roundtrip" else 1 << 26),
                "dtype": rng.choice(["f32", "f32", "bf16"]), "block": rng.choice(BLOCKS),
                "mode": mode, "eb": eb, "heads": rng.random() < 0.2}
    if op == "ring":
        P = rng.randint(2, 8)
        return {"op": op, "P": P, "n": _log(rng, 1 << 16, (1 << 28) // P), "block": rng.choice(BLOCKS),
                "eb": 1e-3}
    if op == "redoub":
        P = rng.randint(2, 8)
        return {"op": op, "P": P, "n": _log(rng, 1 << 14, (1 << 25) // P), "block": rng.choice(BLOCKS),
                "eb": 1e-3}
    if op == "scatter":
        return {"op": op, "P": rng.randint(2, 64), "n": _log(rng, 1 << 16, 1 << 26),
                "dtype": rng.choice(["f32", "bf16"]), "block": rng.choice(BLOCKS),
                "mode": rng.choice(["abs", "rel"]), "eb": 1e-2 * rng.choice([0.1, 1.0])}
    if op == "batch":
        return {"op": op, "messages": _log(rng, 8, 200), "lo": 4096, "hi": _log(rng, 1 << 16, 32 << 20),
                "block": rng.choice(BLOCKS)}
    if op == "select":
        return {"op": op, "bytes": _log(rng, 1 << 26, 1 << 29), "link": rng.choice([12.5, 100.0])}
    return {"op": op, "rows": _log(rng, 500, 10000), "batch": rng.choice([64, 256, 1000])}


# ---- inputs -----------------------------------------------------------------------

def _tensor(case, seed):
    """The tensor of a single-stream or scatter case."""
    n, data = case["n"], case.get("data", "field")
    if data == "tdist":
        x = workloads.student_t3(n, 1.0, seed, device=DEV)
    elif data == "signal":
        x = workloads.sinusoids_1d(n, seed=seed, device=DEV)
    else:
        side = max(2, math.ceil(round(n ** (1 / 3), 6)))
        x = workloads.grf_3d(side, seed=seed, device=DEV)[:n].clone()
        if data == "offset":
            x += 10.0
    return x.to(torch.bfloat16) if case.get("dtype") == "bf16" else x


def _bound(case, x):
    """The absolute FP32 bound of a case on its input, as the codec states it."""
    eb = case["eb"]
    if case["mode"] == "rel":
        lo, hi = float(x.min()), float(x.max())
        eb = eb * (hi - lo) if hi > lo else eb * max(abs(hi), 1.0)
    return float(np.float32(eb))


def _ranks(case, seed):
    """Stacking images (or the first n pixels of them), and the ring's bound."""
    side = math.isqrt(case["n"] - 1) + 1
    base = workloads.stacking_base(side, seed=seed, device=DEV)[:case["n"]].clone()
    xs = [workloads.stacking_rank(base, r, seed=seed) for r in range(case["P"])]
    eb = case["eb"] * max(float(x.max()) - float(x.min()) for x in xs)
    return xs, float(np.float32(eb))


def _segments(case):
    """Counts (uneven, given by the case) and displacements of a scatter case."""
    r = np.random.Generator(np.random.PCG64(case["n"]))
    w = r.uniform(0.5, 1.5, case["P"])
    ends = np.floor(np.cumsum(w) / w.sum() * case["n"]).astype(np.int64)
    ends[-1] = case["n"]
    b = [0] + [int(e) for e in ends]
    return [b[i + 1] - b[i] for i in range(case["P"])], b[:-1]


def _messages(case, seed):
    """Gradient-like messages (sizes, types and scales given by the case, values
    by the seed): views of one FP32 and one BF16 buffer, each message on a
    16-element boundary, and their absolute bounds."""
    specs = workloads.message_specs(m=case["messages"], lo_bytes=case["lo"], hi_bytes=case["hi"],
                                    seed=case["messages"])
    flat, views = {}, []
    for kind, dt in (("f32", torch.float32), ("bf16", torch.bfloat16)):
        total = sum((s["n"] + 15) // 16 * 16 for s in specs if s["dtype"] == kind)
        flat[kind] = workloads.student_t3(max(total, 16), 1.0, seed + (kind == "f32"), device=DEV)
        flat[kind] = [flat[kind], 0, dt]
    for s in specs:
        f = flat[s["dtype"]]
        views.append((f[0][f[1]:f[1] + s["n"]].mul_(s["sigma"]), s["dtype"]))
        f[1] += (s["n"] + 15) // 16 * 16
    bf = flat["bf16"][0].to(torch.bfloat16)
    out, at = [], 0
    for v, kind in views:
        if kind == "bf16":
            out.append(bf[at:at + v.numel()])
            at += (v.numel() + 15) // 16 * 16
        else:
            out.append(v)
    return out, [s["eb"] for s in specs]


def _networks(seed, link):
    """A bits network that is the piecewise-linear log2 of features 0..3 (16
    knots each), a time network near the codec's measured rates, and the cost
    model: what training leaves in a user's hands, made from the seed."""
    r = np.random.Generator(np.random.PCG64(seed))
    rates = np.array([1.10e-3, 1.00e-3, 0.95e-3, 0.93e-3])
    knots = np.geomspace(0.3, 26.0, 17)
    slopes = np.diff(np.log2(knots)) / np.diff(knots)
    nets = []
    for time_net in (False, True):
        W1, W2, W3 = np.zeros((64, 16)), np.eye(64), np.zeros((4, 64))
        b1, b2, b3 = np.zeros(64), np.zeros(64), np.full(4, np.log2(knots[0]))
        for k in range(4):
            for j in range(16):
                W1[16 * k + j, k] = 1.0
                b1[16 * k + j] = -knots[j]
                W3[k, 16 * k + j] = slopes[j] - (slopes[j - 1] if j else 0.0)
        if time_net:
            W3, b3 = W3 * 0.1, np.log2(rates)
        W1 += r.uniform(-1e-3, 1e-3, W1.shape)
        W2 += r.uniform(-1e-3, 1e-3, W2.shape)
        m = selector.Mlp(0, device=DEV)
        p = np.concatenate([a.reshape(-1) for a in (W1, b1, W2, b2, W3, b3)]).astype(np.float32)
        m.params.copy_(torch.from_numpy(p))
        nets.append(m)
    cfg = zc.ZcSelectCfg()
    cfg.link_gbs = link
    for k in range(4):
        cfg.ns_per_byte[k] = rates[k]
    cfg.raw_ns_per_byte = 6.0e-4
    cfg.judge_log2 = 1.0
    cfg.judge_time_log2 = 2.0
    return nets[0], nets[1], cfg


def _chunks(case, seed):
    """64 KiB chunks of signals, volumes, images and gradient-like messages in
    turn (sizes given by the case, values by the seed), and their bounds."""
    xs, ebs, total, k = [], [], 0, 0
    while total < case["bytes"]:
        s = 1000 * seed + k
        vol = workloads.grf_3d(256, seed=s, device=DEV)
        img = workloads.stacking_rank(workloads.stacking_base(1024, seed=s, device=DEV), k, seed=s)
        new = [(workloads.sinusoids_1d(1 << 20, seed=s, device=DEV), 1e-4),
               (vol, 2.0 * (1e-2, 1e-3, 1e-4)[k % 3]),
               (img, 1e-3 * float(img.max() - img.min()))]
        for j, sp in enumerate(workloads.message_specs(m=8, hi_bytes=16 << 20, seed=4000 + k)):
            sp["seed"] = 10 * s + j
            new.append((workloads.message(sp, device=DEV), sp["eb"]))
        xs += [x for x, _ in new]
        ebs += [e for _, e in new]
        total += sum(x.numel() * x.element_size() for x, _ in new)
        k += 1
    views, cebs = selector.split_chunks(xs, ebs)
    keep = [i for i, v in enumerate(views) if v.numel() >= 128]
    return [views[i] for i in keep], [cebs[i] for i in keep]


def _dataset(case, seed):
    """Rows like the chunk statistics (positive, a few units wide) and the
    log2 bits that go with them."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    X = torch.rand((case["rows"], 16), generator=g, device=DEV) * 12.0 + 0.5
    T = torch.log2(X[:, :4] * (1.0 + 0.05 * torch.randn((case["rows"], 4), generator=g, device=DEV)).clamp(min=0.5))
    return X, T


# ---- a user's program ---------------------------------------------------------------

def prepare(case, seed):
    op = case["op"]
    s = {"case": case}
    if op in ("roundtrip", "compress", "decompress"):
        x = _tensor(case, seed)
        n = x.numel()
        mode = zc.EB_REL if case["mode"] == "rel" else zc.EB_ABS
        cap = zc.zc_max_compressed_bytes_heads(n, case["block"]) if case["heads"] else \
            zc.zc_max_compressed_bytes(n, case["block"])
        s.update(x=x, n=n, mode=mode, ws=zc.Workspace(n, 1),
                 out=torch.zeros(cap, dtype=torch.uint8, device=DEV),
                 ob=torch.zeros(1, dtype=torch.int64, device=DEV))
        if op != "compress":
            s["y"] = torch.zeros_like(x)
        if op == "decompress":
            _compress(s)
            s["out"] = s["out"][:(int(s["ob"]) + 15) // 16 * 16].clone()
            del s["x"]
        return s
    if op in ("ring", "redoub"):
        xs, eb = _ranks(case, seed)
        cls = collectives.RingAllreduce if op == "ring" else collectives.RecursiveDoublingAllreduce
        s["all"] = cls(xs, eb, case["block"])
        return s
    if op == "scatter":
        x = _tensor(case, seed)
        counts, displs = _segments(case)
        cap = sum(zc.zc_max_compressed_bytes(c, case["block"]) for c in counts)
        s.update(x=x, counts=counts, displs=displs, ws=zc.Workspace(case["n"], case["P"]),
                 mode=zc.EB_REL if case["mode"] == "rel" else zc.EB_ABS,
                 out=torch.zeros(cap, dtype=torch.uint8, device=DEV),
                 off=torch.zeros(case["P"] + 1, dtype=torch.int64, device=DEV))
        return s
    if op == "batch":
        xs, ebs = _messages(case, seed)
        cap = sum(zc.zc_max_compressed_bytes(x.numel(), case["block"]) for x in xs)
        packed = torch.zeros(cap, dtype=torch.uint8, device=DEV)
        comp = zc.BatchCompress(xs, [case["block"]] * len(xs), ebs, packed=packed, cap=cap)
        flat, outs = {}, []
        for dt in (torch.float32, torch.bfloat16):
            flat[dt] = [torch.zeros(sum((x.numel() + 15) // 16 * 16 for x in xs if x.dtype == dt),
                                    dtype=dt, device=DEV), 0]
        for x in xs:
            f = flat[x.dtype]
            outs.append(f[0][f[1]:f[1] + x.numel()])
            f[1] += (x.numel() + 15) // 16 * 16
        s.update(comp=comp, dec=zc.BatchDecompress(packed, comp.msg_off, outs, ws=comp.ws),
                 f32=flat[torch.float32][0], bf16=flat[torch.bfloat16][0])
        return s
    if op == "select":
        views, ebs = _chunks(case, seed)
        cb = selector.ChunkBatch(views, ebs)
        cb.batch.packed.zero_()
        s["nets"] = _networks(seed, case["link"])
        s["cb"] = cb
        return s
    X, T = _dataset(case, seed)
    net = selector.Mlp(seed, device=DEV)
    net.set_norm(X)
    s.update(X=X, T=T, net=net, seed=seed)
    return s


def _compress(s):
    c = s["case"]
    zc.compress(s["x"], c["eb"], c["block"], mode=s["mode"], ws=s["ws"], out=s["out"],
                out_bytes=s["ob"], heads=c["heads"])


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "compress":
        _compress(s)
        return {"stream": s["out"], "bytes": s["ob"]}
    if op == "decompress":
        return {"y": zc.decompress(s["out"], s["n"], ws=s["ws"], out=s["y"])}
    if op == "roundtrip":
        _compress(s)
        zc.decompress(s["out"], s["n"], ws=s["ws"], out=s["y"])
        return {"stream": s["out"], "bytes": s["ob"], "y": s["y"]}
    if op in ("ring", "redoub"):
        return {"sums": list(s["all"].run()), "sizes": s["all"].sizes}
    if op == "scatter":
        zc.scatter_pack(s["x"], s["counts"], s["displs"], c["eb"], c["block"], mode=s["mode"],
                        ws=s["ws"], out=s["out"], seg_off=s["off"])
        return {"packed": s["out"], "offsets": s["off"]}
    if op == "batch":
        packed, off = s["comp"].run()
        s["dec"].run()
        return {"packed": packed, "offsets": off, "f32": s["f32"], "bf16": s["bf16"]}
    if op == "select":
        cb = s["cb"]
        bits, times, cfg = s["nets"]
        cb.run_selected(cfg, bits, times)
        return {"features": cb.feat, "bits": cb.pred, "times": cb.pred_time, "choice": cb.choice,
                "packed": cb.batch.packed, "offsets": cb.batch.msg_off}
    net = s["net"]
    net.fit(s["X"], s["T"], epochs=1, batch=c["batch"], seed=s["seed"])
    return {"params": net.params, "velocity": net.vel, "gradient": net.grad}


# ---- what a pass cannot do without -----------------------------------------------------

def _bits(case):
    """Stream bits per element, about (measured on the listed inputs)."""
    data = case.get("data", "field")
    if data == "tdist":
        return 13.5
    if data == "signal":
        return 13.7
    return {1e-2: 4.4, 1e-3: 7.7, 1e-4: 11.1}.get(case["eb"], 8.0)


def work(case):
    op = case["op"]
    es = 2 if case.get("dtype") == "bf16" else 4
    if op in ("roundtrip", "compress", "decompress", "scatter"):
        one = case["n"] * (es + _bits(case) / 8)
        return {"bytes": one * (2 if op == "roundtrip" else 1), "flops": 0}
    if op in ("ring", "redoub"):
        # every rank's input read, its result written, and the streams between ranks
        P, n, b = case["P"], case["n"], 4.5 / 8
        if op == "ring":
            return {"bytes": P * n * 8 + P * n * b * 2 + (P - 1) * n * b, "flops": 0}
        return {"bytes": P * n * 8 + P * n * b * 2 * int(math.log2(P)), "flops": 0}
    if op == "batch":
        # sizes are log-uniform: mean (hi - lo) / ln(hi / lo); half the bytes BF16
        raw = case["messages"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        packed = raw * (0.5 * 13.5 / 32 + 0.5 * 13.5 / 16)
        return {"bytes": 2 * (raw + packed), "flops": 0}
    if op == "select":
        return {"bytes": case["bytes"] * 1.4, "flops": case["bytes"] / 65536 * 2 * 2 * 5376}
    return {"bytes": case["rows"] * 20 * 4, "flops": case["rows"] * 6 * 5376}


# ---- the same in 64 bits -----------------------------------------------------------------

def _decoded(x, eb):
    """Reconstruction at the absolute bound eb: the nearest multiple of 2 eb."""
    two = 2.0 * eb
    return torch.round(x.double() / two) * two


def _bitlen(v):
    return torch.frexp(v.double())[1].to(torch.int64) * (v > 0)


def _stats(x, eb):
    """Chunk statistics of equal chunks x[G, n], bounds eb[G] (n >= 128)."""
    G, n = x.shape
    m = n // 128
    S = min(16, m)
    at = [128 * (j * (m - 1) // (S - 1)) if S > 1 else 0 for j in range(S)]
    v = torch.stack([x[:, a:a + 128] for a in at], 1).double()
    q = torch.round(v / (2.0 * eb)[:, None, None]).to(torch.int64)
    d = q[..., 1:] - q[..., :-1]
    d2 = d[..., 1:] - d[..., :-1]
    f = torch.zeros((G, 16), dtype=torch.float64, device=x.device)
    tot, nd, nd2 = S * 128, S * 127, S * 126
    for k, L in enumerate(BLOCKS):
        full = torch.cat([q[..., :1], d], -1).abs()
        blocks = full.reshape(G, S, 128 // L, L).clone()
        blocks[..., 0] = q.reshape(G, S, 128 // L, L)[..., 0].abs()
        w = blocks.amax(-1)
        b = torch.where(w > 0, (_bitlen(w) + 1) * L, torch.zeros_like(w))
        f[:, k] = b.sum((1, 2)).double() / tot + 8.0 / L + 256.0 / n
        if L == 32:
            f[:, 13] = (b.sum(2).double() / 128.0).std(1, correction=0)
    lg = lambda t: torch.log2(1.0 + t.double())  # noqa: E731
    f[:, 4] = lg(q.amax((1, 2)) - q.amin((1, 2)))
    f[:, 5] = lg(d.abs().sum((1, 2)).double() / nd)
    f[:, 6] = lg(d.abs().amax((1, 2)))
    f[:, 7] = (d == 0).sum((1, 2)).double() / nd
    f[:, 8] = (q == 0).sum((1, 2)).double() / tot
    f[:, 9] = lg(q.abs().sum((1, 2)).double() / tot)
    f[:, 10] = lg(d2.abs().sum((1, 2)).double() / nd2)
    f[:, 11] = (d[..., 1:] * d[..., :-1] < 0).sum((1, 2)).double() / nd2
    f[:, 12] = _bitlen(q[..., ::32].abs()).sum((1, 2)).double() / (S * 4) / 24.0
    f[:, 14] = 1.0 if x.dtype == torch.float32 else 0.5
    f[:, 15] = math.log2(n) / 16.0
    return f


def _layers(p):
    o = [0, 1024, 1088, 5184, 5248, 5504, 5508]
    W = [p[o[i]:o[i + 1]] for i in range(6)]
    return W[0].reshape(64, 16), W[1], W[2].reshape(64, 64), W[3], W[4].reshape(4, 64), W[5]


def _forward(p, norm, X):
    W1, b1, W2, b2, W3, b3 = _layers(p)
    h = torch.relu((X - norm[:16]) * norm[16:] @ W1.T + b1)
    return torch.relu(h @ W2.T + b2) @ W3.T + b3


def exact(case, seed):
    op = case["op"]
    if op == "compress" or op == "scatter":
        return None  # whole bytes and lengths only
    if op in ("decompress", "roundtrip"):
        x = _tensor(case, seed)
        y = _decoded(x, _bound(case, x))
        return {"y": y} if op == "decompress" else {"stream": None, "bytes": None, "y": y}
    if op in ("ring", "redoub"):
        # the sum that the collective approximates, the same for every rank
        xs, _ = _ranks(case, seed)
        t = torch.zeros(case["n"], dtype=torch.float64, device=DEV)
        for x in xs:
            t += x.double()
        return {"sums": [t] * case["P"], "sizes": None}
    if op == "batch":
        xs, ebs = _messages(case, seed)
        flat = {torch.float32: [], torch.bfloat16: []}
        for x, eb in zip(xs, ebs):
            y = _decoded(x, float(np.float32(eb)))
            flat[x.dtype].append(torch.nn.functional.pad(y, (0, -y.numel() % 16)))
        empty = torch.zeros(0, dtype=torch.float64, device=DEV)
        f32, bf16 = (torch.cat(flat[t]) if flat[t] else empty for t in (torch.float32, torch.bfloat16))
        return {"packed": None, "offsets": None, "f32": f32, "bf16": bf16}
    if op == "select":
        views, ebs = _chunks(case, seed)
        f = torch.zeros((len(views), 16), dtype=torch.float64, device=DEV)
        groups = {}
        for i, v in enumerate(views):
            groups.setdefault((v.numel(), v.dtype), []).append(i)
        eb = torch.tensor(np.array(ebs, np.float32), device=DEV).double()
        for ids in groups.values():
            at = torch.tensor(ids, device=DEV)
            f[at] = _stats(torch.stack([views[i] for i in ids]), eb[at])
        bits, times, _ = _networks(seed, case["link"])
        return {"features": f, "bits": _forward(bits.params.double(), bits.norm.double(), f),
                "times": _forward(times.params.double(), times.norm.double(), f),
                "choice": None, "packed": None, "offsets": None}
    X, T = _dataset(case, seed)
    net = selector.Mlp(seed, device=DEV)
    net.set_norm(X)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    at = torch.randperm(case["rows"], generator=g, device=DEV)
    p, v, norm = net.params.double(), torch.zeros_like(net.params, dtype=torch.float64), net.norm.double()
    grad = v
    for k in range(0, case["rows"], case["batch"]):
        i = at[k:k + case["batch"]]
        p = p.detach().requires_grad_(True)
        loss = ((_forward(p, norm, X[i].double()) - T[i].double()) ** 2).mean()
        grad, = torch.autograd.grad(loss, p)
        v = 0.9 * v + grad
        p = p.detach() - 0.02 * v
    return {"params": p, "velocity": v, "gradient": grad}
