"""Workloads of the library, as a user's program calls it: queries on resident graphs, list builds, the whole method
from host arrays, exact counts, batches of queries, and the learned proposal's parts.

Graphs follow the recipes of paper_2409_08975_gb300/synth.py (bursty Chung-Lu multigraphs, uniform repeats or Zipf(1.8)
pair multiplicities), generated on the GPU so that inputs of another seed are quick to make.
"""
import math

import numpy as np
import torch

from paper_2409_08975_gb300 import tc

SPAN = 100_000_000  # seconds
ZIPF, ZIPF_CAP = 1.8, 1000
MOTIFS = {
    "c4": [(0, 1), (1, 2), (2, 3), (3, 0)],                             # directed 4-cycle
    "chord": [(0, 1), (1, 2), (2, 3), (0, 3)],                          # path, then its chord
    "multi": [(0, 1), (1, 2), (1, 2), (2, 3), (3, 0), (0, 2)],          # several lists to count
    "late_mid": [(2, 3), (1, 2), (0, 1), (0, 3)],                       # middle edge not the second in time
    "triangle": [(0, 1), (0, 2), (1, 2)],                               # 3 vertices: wedge sampling
}
DELTAS = (600, 3600, 86400)


def listed():
    return [
        # the tiny configuration: uniform times, 20,000 edges, 1e5 samples; one short call after another
        dict(name="query_tiny", kind="query", graph="uniform", n=2000, m=20_000, unit="s", motif="c4", closed=False, delta=10_000, k=100_000),
        # the mid configuration: a 20M-edge communication-like graph, 1e8 samples of the path with a chord
        dict(name="query_mid", kind="query", graph="uniform_repeats", n=1_000_000, m=20_000_000, unit="s", motif="chord", closed=False, delta=3600, k=100_000_000),
        # the large configuration and the benchmark's step: 300M transaction-like edges, 1e9 samples of the 4-cycle
        dict(name="query_large", kind="query", graph="zipf", n=100_000_000, m=300_000_000, unit="s", motif="c4", closed=False, delta=3600, k=1_000_000_000),
        # millisecond time stamps (a span beyond 32 bits), closed windows, a motif with several lists, odd sizes
        dict(name="query_ms_multi", kind="query", graph="zipf", n=1_234_567, m=9_999_991, unit="ms", motif="multi", closed=True, delta=3600, k=5_000_011),
        # a new graph arrives on the device: its time-sorted lists, read back by the caller
        dict(name="build_mid", kind="build", graph="uniform_repeats", n=1_000_000, m=20_000_000, unit="s"),
        # the whole method from pinned host arrays: copy, lists, weights, samples (the profiling-size large graph)
        dict(name="host_large_small", kind="host", graph="zipf", n=10_000_000, m=30_000_000, unit="s", motif="c4", closed=False, delta=3600, k=30_000_000),
        # the exact count of a graph of the size of one 1% time slice of the large graph
        dict(name="exact_slice", kind="exact", graph="zipf", n=1_000_000, m=3_000_000, unit="s", motif="c4", closed=False, delta=3600),
        # many queries in one replayed launch: 24 rank orders of the 4-cycle x 3 windows on one graph, and small graphs
        dict(name="batch_small", kind="batch", graph="uniform_repeats", big_m=10_000_000, small=8, k_lo=100_000, k_hi=10_000_000),
        # per-edge inputs of the learned proposal: counts and sample statistics
        dict(name="features_mid", kind="features", graph="uniform_repeats", n=1_000_000, m=20_000_000, unit="s", motif="chord", closed=False, delta=3600, samples=1_000_000),
        # the network alone: logits of a table of rows, the gradient of a batch of them (ragged sizes)
        dict(name="mlp_rows", kind="mlp", rows=1_000_003, batch=100_003, objective="closure"),
        # training the proposal on the plain sampler's own paths, in the usual batches (a few steps: the optimizer
        # magnifies the last bits of a gradient in every further one)
        dict(name="train_mid", kind="train", graph="uniform_repeats", n=500_000, m=10_000_000, unit="s", motif="chord", closed=False, delta=3600, samples=100_000, batch=16_384, objective="variance"),
        # the learned configuration: inference over 1e8 edges, then 1e8 samples from the proposal
        dict(name="proposal_learned", kind="proposal", graph="uniform_repeats", n=20_000_000, m=100_000_000, unit="s", motif="chord", closed=False, delta=3600, k=100_000_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "build", "host", "exact", "batch", "features", "mlp", "train", "proposal"])
    if kind == "mlp":
        return dict(kind=kind, rows=_log(rng, 1000, 4_000_000), batch=_log(rng, 100, 400_000), objective=rng.choice(["closure", "variance", "bce"]))
    if kind == "batch":
        return dict(kind=kind, graph="uniform_repeats", big_m=_log(rng, 100_000, 10_000_000), small=rng.randint(1, 16), k_lo=10_000, k_hi=_log(rng, 100_000, 10_000_000))
    m = _log(rng, 20_000, {"query": 100_000_000, "build": 100_000_000, "host": 30_000_000, "exact": 3_000_000, "features": 30_000_000, "train": 10_000_000, "proposal": 100_000_000}[kind])
    case = dict(kind=kind, graph=rng.choice(["uniform_repeats", "zipf"]), n=max(100, int(m / rng.uniform(3, 20))), m=m, unit="s")
    if kind in ("query", "build", "host"):
        case["unit"] = rng.choice(["s", "s", "ms"])
    if kind == "build":
        return case
    case.update(motif="chord" if kind == "features" else rng.choice(["c4", "chord"] if kind in ("exact", "train", "proposal") else sorted(MOTIFS)),
                closed=kind in ("query", "host") and rng.random() < 0.3, delta=rng.choice(DELTAS[:2] if kind in ("exact", "proposal") else DELTAS))
    if kind in ("query", "host", "proposal"):
        case["k"] = _log(rng, 1000, 100_000_000)
    if kind == "features":
        case["samples"] = _log(rng, 20_000, 1_000_000)
    if kind == "train":
        case.update(batch=rng.choice([4096, 16_384, 65_536]), objective=rng.choice(["closure", "variance", "bce"]))
        case["samples"] = int(case["batch"] * rng.uniform(1.2, 6.0))
    return case


# ---------------------------------------------------------------------------
# Inputs


def _first_rank_offset(n, edges, top):
    """i0 of the vertex weights (i + i0)^(-10/11) that give the first vertex about `top` of `edges` draws."""
    a, b = 1.0 / 1.1, 1.0 - 1.0 / 1.1
    lo, hi = 1e-3, float(n)
    for _ in range(80):
        mid = math.sqrt(lo * hi)
        share = mid ** -a * b / ((n + mid) ** b - mid ** b)
        lo, hi = (mid, hi) if edges * share > top else (lo, mid)
    return hi


def _edges(case, seed):
    """(src, dst, t) on the GPU, in random input order."""
    n, m = case["n"], case["m"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    u = lambda k: torch.rand(k, generator=gen, device="cuda", dtype=torch.float64).clamp_(1e-12, 1.0 - 1e-12)  # noqa: E731
    below = lambda k, hi: (u(k) * hi).long()  # noqa: E731
    pareto = lambda k: u(k).pow_(-1.0 / 1.5).floor_().clamp_(max=2.0 ** 40).long()  # noqa: E731

    if case["graph"] == "uniform":  # unique-ish uniform pairs, uniform times in [0, 1e6)
        src = below(m, n)
        dst = (src + 1 + below(m, n - 1)) % n
        again = torch.nonzero(u(m) < 0.1)[:, 0]
        pick = below(len(again), m)
        src[again], dst[again] = src[pick], dst[pick]
        t = below(m, 1_000_000)
    else:
        zipf = case["graph"] == "zipf"
        mult = torch.arange(1, ZIPF_CAP + 1, device="cuda", dtype=torch.float64)
        p = mult ** -ZIPF
        mean = float((mult * p).sum() / p.sum())
        base = max(2, int(m / mean) if zipf else int(round(m * 0.7)))
        top = max(10.0, m / 200.0) if not zipf else max(10.0, m / 300.0)
        i0 = _first_rank_offset(n, base, top / mean if zipf else top)
        # bursts: sizes, vertex slots, the burst of every base edge
        count = int(base / 200 * 1.2) + 100
        sizes = torch.empty(count, device="cuda", dtype=torch.float64).geometric_(1.0 / 200, generator=gen).long()
        ends = torch.cumsum(sizes, 0)
        S = min(count, int(torch.searchsorted(ends, base)) + 1)
        sizes, ends = sizes[:S].clone(), ends[:S].clone()
        sizes[-1] += base - ends[-1]
        ends[-1] = base
        deg = torch.exp(math.log(1.5) + u(S) * (math.log(24.0) - math.log(1.5)))
        nv = torch.clamp((sizes / deg).round(), min=4).long()
        soff = torch.cumsum(nv, 0) - nv
        b = 1.0 - 1.0 / 1.1
        lo, hi = i0 ** b, (n + i0) ** b
        slots = ((lo + u(int(nv.sum())) * (hi - lo)) ** (1.0 / b) - i0).long().clamp_(0, n - 1)
        slots = (slots * 2654435761 + 12345) % n  # ranks to vertex ids
        burst = torch.repeat_interleave(torch.arange(S, device="cuda"), sizes)
        at, width = soff[burst], nv[burst]
        src = slots[at + (u(base) * width).long()]
        dst = slots[at + (u(base) * width).long()]
        for _ in range(3):
            same = torch.nonzero(src == dst)[:, 0]
            dst[same] = slots[at[same] + (u(len(same)) * width[same]).long()]
        same = torch.nonzero(src == dst)[:, 0]
        dst[same] = (src[same] + 1) % n
        del at, width
        cand = below(4 * S + 64, SPAN)
        if zipf:  # daily periodicity of burst starts
            keep = u(len(cand)) * 1.5 < 1.0 + 0.5 * torch.sin(2 * math.pi * cand / 86400.0)
            cand = torch.cat([cand[keep], below(S, SPAN)])
        gaps = pareto(base)
        gaps[ends - sizes] = 0
        cum = torch.cumsum(gaps, 0)
        t = torch.clamp(cand[:S][burst] + cum - cum[ends - sizes][burst], max=SPAN - 1)
        del gaps, cum, burst
        extra = m - base
        if zipf:
            more = torch.searchsorted(torch.cumsum(p / p.sum(), 0), u(base)).clamp_(max=ZIPF_CAP - 1)
            pick = torch.repeat_interleave(torch.arange(base, device="cuda"), more)[:extra]
            gsum = torch.cumsum(pareto(len(pick)), 0)
            begin = torch.cumsum(more, 0) - more
            before = torch.cat([torch.zeros(1, device="cuda", dtype=torch.int64), gsum])
            rt = t[pick] + gsum - before[begin[pick]]
            rest = below(extra - len(pick), base)
            pick, rt = torch.cat([pick, rest]), torch.cat([rt, t[rest] + pareto(len(rest))])
            del gsum, before, begin, more
        else:
            pick = below(extra, base)
            rt = t[pick] + pareto(extra)
        src, dst = torch.cat([src, src[pick]]), torch.cat([dst, dst[pick]])
        t = torch.cat([t, torch.clamp(rt, max=SPAN - 1)])
        del pick, rt
    if case["unit"] == "ms":
        t = t * 1000 + below(m, 1000)
    order = torch.randperm(m, generator=gen, device="cuda")
    return src[order].int(), dst[order].int(), t[order].contiguous()


def _delta(case):
    return case["delta"] * (1000 if case["unit"] == "ms" else 1)


def _motif(case):
    return tc.make_motif(MOTIFS[case["motif"]], window=tc.WINDOW_CLOSED if case["closed"] else tc.WINDOW_STRICT)


def _mlp_inputs(case, seed):
    """A feature table (log1p of skewed counts, as bf16 bits), the batch's rows and closure counts, the parameters."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 29)
    u = lambda *s: torch.rand(*s, generator=gen, device="cuda").clamp_(1e-6, 1.0)  # noqa: E731
    counts = (u(case["rows"], tc.FEATURE_STRIDE) ** -1.2).floor_() - 1.0
    feat = torch.log1p(counts).to(torch.bfloat16).view(torch.int16)
    rows = torch.randint(0, case["rows"], (case["batch"],), generator=gen, device="cuda", dtype=torch.int32)
    labels = torch.where(u(case["batch"]) < 0.3, (u(case["batch"]) ** -0.6).floor_(), torch.zeros((), device="cuda"))
    rng = np.random.default_rng(int(seed))
    fan = np.concatenate([np.full(64 * 16 + 64, 16.0), np.full(64 * 64 + 64, 64.0), np.full(64 + 1, 64.0)])
    params = ((2 * rng.random(tc.MLP_PARAMS) - 1) / np.sqrt(fan)).astype(np.float32)
    return feat, rows, labels, params


def _logits64(p, x):
    """The network of 16 inputs, two hidden layers of 64 and one output, in the precision of its arguments."""
    a = torch.relu(x @ p[:1024].view(64, 16).T + p[1024:1088])
    a = torch.relu(a @ p[1088:5184].view(64, 64).T + p[5184:5248])
    return a @ p[5248:5312] + p[5312]


def _batch_queries(case, seed):
    import itertools
    rng = np.random.default_rng(int(seed))
    c4 = MOTIFS["c4"]
    orders = [[c4[j] for j in p] for p in itertools.permutations(range(4))]
    ms = [case["big_m"]] + [int(np.exp(rng.uniform(np.log(1e4), np.log(max(2e4, case["big_m"] / 20))))) for _ in range(case["small"])]
    graphs = []
    for i, m in enumerate(ms):
        src, dst, t = _edges(dict(graph=case["graph"], n=max(1000, m // 20), m=m, unit="s"), int(seed) * 31 + i)
        graphs.append(tc.tc_build_temporal_csr(max(1000, m // 20), src, dst, t))
    k = lambda: int(np.exp(rng.uniform(np.log(case["k_lo"]), np.log(case["k_hi"]))))  # noqa: E731
    queries = [(graphs[0], o, d, k(), 0, 0) for o in orders for d in DELTAS]
    # a rank order per small graph, and every fourth a 3-vertex motif
    queries += [(graphs[1 + i], MOTIFS["triangle"] if i % 4 == 3 else orders[i % 24], DELTAS[i % 3], k(), 0, 0) for i in range(case["small"])]
    return queries


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        feat, rows, labels, params = _mlp_inputs(case, seed)
        mlp = tc.MLP(0)
        mlp.set_params(params)
        return dict(case=case, mlp=mlp, feat=feat, rows=rows, labels=labels)
    if kind == "batch":
        return dict(case=case, batch=tc.Batch(_batch_queries(case, seed)))
    src, dst, t = _edges(case, seed)
    if kind == "build":
        full = lambda: torch.zeros(case["m"] + 1, device="cuda", dtype=torch.int32)  # noqa: E731
        return dict(case=case, src=src, dst=dst, t=t, graph=None, pair_dst=full(), pair_eoff=full())
    if kind == "host":
        pin = lambda x: x.cpu().pin_memory()  # noqa: E731
        return dict(case=case, src=pin(src), dst=pin(dst), t=pin(t), motif=_motif(case), seed=int(seed) % 1000)
    g = tc.tc_build_temporal_csr(case["n"], src, dst, t)
    del src, dst, t
    s = dict(case=case, graph=g, motif=_motif(case), delta=_delta(case), seed=int(seed) % 1000)
    if kind == "query":
        s["weights"] = tc.alloc_weights(g)  # reused by a program that asks again and again
        return s
    s["weights"] = tc.tc_path_weights(g, s["motif"], s["delta"])
    if kind == "features":
        s["feat"] = tc.alloc_features(g)
    if kind in ("train", "proposal"):
        s["feat"] = tc.alloc_features(g)
        tc.tc_edge_features(g, s["motif"], s["delta"], s["weights"], out=s["feat"])
        tc.tc_sample_features(g, s["motif"], s["delta"], s["weights"], s["feat"], 500_000, seed=777)
        s["mlp"] = tc.MLP(s["seed"])
        s["params"] = s["mlp"].get_params()
    if kind == "proposal":
        # closure rates spread over (0, 1) as a trained network's are (training is not repeatable bit by bit): the last
        # layer scaled and shifted for logits of mean -1 and deviation 1.5 on a part of the rows
        x = s["feat"][:1_000_000].view(torch.bfloat16).double()
        z = _logits64(torch.from_numpy(s["params"]).cuda().double(), x[x[:, 0] > 0][:100_000])
        scale, mean = (1.5 / float(z.std()), float(z.mean())) if len(z) > 1 else (1.0, 0.0)
        s["params"][5312] = (s["params"][5312] - mean) * scale - 1.0
        s["params"][5248:5312] *= scale
        s["mlp"].set_params(s["params"])
    return s


# ---------------------------------------------------------------------------
# One pass


def _sums(es):
    """The integers of estimates as int64 limbs, and their floats."""
    low = 0xFFFFFFFFFFFFFFFF
    whole = [[e["W"], e["k"], e["sum_x"], e["sum_x2"] & low, e["sum_x2"] >> 64, e["hits"], e["checked"]] for e in es]
    return {"sums": np.array(whole, np.uint64).view(np.int64), "estimate": np.array([e["estimate"] for e in es]),
            "std_err": np.array([e["std_err"] for e in es])}


def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "query":
        w = tc.tc_path_weights(s["graph"], s["motif"], s["delta"], out=s["weights"])
        out = _sums([tc.tc_sample_estimate(s["graph"], s["motif"], s["delta"], w, c["k"], seed=s["seed"])])
        # after the 256-byte header, the window entries: 16 bytes an edge
        return dict(out, prefix=w.prefix, windows=w.index[256:256 + 16 * c["m"]].view(torch.int32))
    if kind == "build":
        g = tc.tc_build_temporal_csr(c["n"], s["src"], s["dst"], s["t"])
        out = {name: g.array(name) for name in tc.ARRAYS}
        for name in ("pair_dst", "pair_eoff"):  # as long as there are pairs: kept in the caller's buffers
            s[name][:len(out[name])] = out[name]
            out[name] = s[name]
        s["graph"] = g  # a program keeps the graph it built; the one before goes
        return out
    if kind == "host":
        return _sums([tc.tc_estimate_from_host(c["n"], s["src"], s["dst"], s["t"], s["motif"], _delta(c), c["k"], seed=s["seed"])])
    if kind == "exact":
        return _sums([tc.tc_exact_count(s["graph"], s["motif"], s["delta"], s["weights"])])
    if kind == "batch":
        return _sums(s["batch"].run())
    if kind == "features":
        f = tc.tc_edge_features(s["graph"], s["motif"], s["delta"], s["weights"], out=s["feat"])
        tc.tc_sample_features(s["graph"], s["motif"], s["delta"], s["weights"], s["feat"], c["samples"], seed=s["seed"])
        return {"counts": f[:, :12], "statistics": f[:, 12:]}
    if kind == "mlp":
        z = tc.tc_mlp_forward(s["mlp"], s["feat"])
        grad, loss = tc.tc_mlp_grad(s["mlp"], s["feat"], s["rows"], s["labels"], objective=c["objective"])
        return {"logits": z, "grad": grad, "loss": loss}
    if kind == "train":
        s["mlp"].set_params(s["params"])
        first, last = tc.tc_mlp_train(s["mlp"], s["graph"], s["motif"], s["delta"], s["weights"], s["feat"], c["samples"], seed=s["seed"], batch=c["batch"], objective=c["objective"])
        return {"losses": np.array([first, last], np.float32), "params": s["mlp"].get_params()}
    p = tc.tc_proposal_weights(s["mlp"], s["graph"], s["motif"], s["delta"], s["weights"], s["feat"])
    e = tc.tc_sample_estimate_q(s["graph"], s["motif"], s["delta"], s["weights"], p, c["k"], seed=s["seed"], want_bins=True)
    return dict(_sums([e]), h=p.h, qprefix=p.qprefix, bins=e["bins"].view(np.int64))


def work(case):
    """Each input read once, each output written once. A graph's lists: 16-byte out- and in-edges, 12 bytes of pair
    times and a 16-byte pair entry for most edges; windows and prefix 24 bytes an edge."""
    kind, m = case["kind"], case.get("m", 0)
    lists, index, net = 16 + 16 + 12 + 16, 16 + 8, 2 * (16 * 64 + 64 * 64 + 64)
    if kind == "query":
        return {"bytes": m * (lists + index), "flops": 0}
    if kind == "build":
        return {"bytes": m * (16 + 16 + 4 + 16 + 4 + 8 + 4 + 4 + 4), "flops": 0}
    if kind == "host":
        return {"bytes": m * (16 + lists + index), "flops": 0}
    if kind == "exact":
        return {"bytes": m * (lists + index), "flops": 0}
    if kind == "batch":  # 72 queries on the big graph share four anchor classes x three windows
        return {"bytes": case["big_m"] * (lists + 12 * index), "flops": 0}
    if kind == "features":
        return {"bytes": m * (lists + index + 32), "flops": 0}
    if kind == "mlp":
        return {"bytes": case["rows"] * 36 + case["batch"] * 40, "flops": case["rows"] * net + 3 * case["batch"] * net}
    if kind == "train":
        return {"bytes": case["samples"] * (32 + 32 + 8), "flops": case["samples"] * 3 * net}
    return {"bytes": m * (lists + index + 32 + 2 + 8), "flops": m * net}


# ---------------------------------------------------------------------------
# The computed outputs in 64 bits


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "features" and case["motif"] == "chord" and not case["closed"]:
        return {"counts": _exact_counts(case, seed), "statistics": None}
    return None  # integers, and floats formed from sampled integers


def _exact_mlp(case, seed):
    feat, rows, y, params = _mlp_inputs(case, seed)
    x = feat.view(torch.bfloat16).double()
    p = torch.from_numpy(params).cuda().double().requires_grad_(True)
    with torch.no_grad():
        z = torch.cat([_logits64(p, part) for part in x.split(500_000)])
    zb, y, eps = _logits64(p, x[rows.long()]), y.double(), 0.05
    if case["objective"] == "variance":
        h = eps + torch.sigmoid(zb)
        loss = h.mean() * (y * y / h).mean()
    else:
        if case["objective"] == "bce":
            y = (y > 0).double()
        loss = torch.where(y > 0, y * torch.nn.functional.softplus(-zb), torch.nn.functional.softplus(zb)).mean()
    loss.backward()
    return {"logits": z, "grad": p.grad, "loss": float(loss.detach())}


def _exact_counts(case, seed):
    """log1p of the 12 counts of every edge with a path (zero rows elsewhere), edges in (src, t, input index) order."""
    src, dst, t = (x.long() for x in _edges(case, seed))
    delta, BIG = _delta(case), 1 << 34
    t = t - t.min() + 2 * delta
    key_out, key_in, key_pair = src * BIG + t, dst * BIG + t, None
    order = torch.sort(key_out, stable=True)[1]
    src, dst, t = src[order], dst[order], t[order]
    outs, ins = torch.sort(key_out)[0], torch.sort(key_in)[0]
    at = lambda keys, v, x, right: torch.searchsorted(keys, v * BIG + x, right=right)  # noqa: E731
    span = lambda keys, v, lo, hi: at(keys, v, hi, True) - at(keys, v, lo, False)  # noqa: E731
    d1 = at(ins, src, t, False) - at(ins, src, t - delta, False)   # into the source, within delta before
    d3 = at(outs, dst, t + delta, True) - at(outs, dst, t, True)   # out of the destination, within delta after
    # pair lists: dense pair numbers, then the same searches
    pairs, number = torch.unique(src * case["n"] + dst, return_inverse=True)
    key_pair = torch.sort(number * BIG + t)[0]
    back = dst * case["n"] + src
    where = torch.searchsorted(pairs, back).clamp_(max=len(pairs) - 1)
    there = pairs[where] == back
    degree = lambda v: torch.bincount(v, minlength=case["n"])  # noqa: E731
    out_deg, in_deg = degree(src), degree(dst)
    lo, hi = t - delta, t + delta
    cols = [d1, d3, d1 * d3, span(ins, src, lo, hi), span(outs, src, lo, hi), span(ins, dst, lo, hi), span(outs, dst, lo, hi),
            span(key_pair, number, lo, hi), torch.where(there, span(key_pair, where, lo, hi), torch.zeros_like(t)),
            out_deg[src], in_deg[dst], in_deg[src]]
    live = (d1 * d3 > 0).double()
    return torch.stack([torch.log1p(c.double()) * live for c in cols], 1)
