"""The workloads this library is timed on: anneals over its kernels' real range, and the learned start.

A case is a dict of plain values.  `prepare` makes what a program holds before the call (graphs from
the seed alone, the annealing context or the network), `run` is one call of the public entry points as
a program makes it, with every result it reads back, `work` says what one call cannot do without, and
`exact` gives the network's outputs in 64 bits (an anneal's outputs are whole numbers and have to stay
what they are).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1908_00210_gb300 import (GDI_FLAG_STANDARD, GDI_METROPOLIS, GDI_PAPER_PF, Annealer, Schedule,
                                    learn)

NOISE = 8          # noise channels of the network's input
FEAT_SEED = 0x9E3779B9


def listed():
    sparse = dict(kind="anneal", A=1, B=4, mode="metropolis", t0=3.0, t1=0.05, start="random", tune=False,
                  standard=False)
    return [
        # one large power-law graph bisected on the whole GPU: the headline workload
        dict(sparse, name="ba1m_r8", graph="ba", count=1, n_lo=1_000_000, n_hi=1_000_000, d_lo=10.0, d_hi=10.0,
             signed=False, W=256, replicas=8, sweeps=500),
        # a medium graph, one replica, small windows: the latency of the whole-GPU path
        dict(sparse, name="ba20k_r1", graph="ba", count=1, n_lo=20_000, n_hi=20_000, d_lo=10.0, d_hi=10.0,
             signed=False, W=64, replicas=1, sweeps=300),
        # windows above 256 (closer to the paper's whole-class updates) on the whole-GPU path
        dict(sparse, name="ba100k_w1024", graph="ba", count=1, n_lo=99_991, n_hi=99_991, d_lo=10.0, d_hi=10.0,
             signed=False, W=1024, replicas=8, sweeps=100),
        # many replicas of a +-1 lattice, tuned once and annealed at length
        dict(sparse, name="torus100_r64", graph="torus", count=1, n_lo=10_000, n_hi=10_000, d_lo=4.0, d_hi=4.0,
             signed=True, W=256, replicas=64, sweeps=5000, tune=True),
        # the smallest anneal: one replica of one dense little graph
        dict(sparse, name="er800_r1", graph="er", count=1, n_lo=800, n_hi=800, d_lo=47.9, d_hi=47.9, signed=False,
             W=64, replicas=1, sweeps=1000),
        # a batch of uneven instances in one launch, tuned as such a program does
        dict(sparse, name="er_batch640", graph="er", count=640, n_lo=800, n_hi=3000, d_lo=3.0, d_hi=48.0,
             signed=True, W=256, replicas=1, sweeps=500, tune=True),
        # short low-temperature anneals from starts that lie on the device (a learned start's)
        dict(sparse, name="warm128_r8", graph="mix", count=128, n_lo=1000, n_hi=5000, d_lo=3.0, d_hi=48.0,
             signed=False, W=256, replicas=8, sweeps=25, t0=0.5, start="device"),
        # the paper's own setting: whole-class windows (the default) and its P_f schedule
        dict(sparse, name="er2000_default", graph="er", count=1, n_lo=2000, n_hi=2000, d_lo=20.0, d_hi=20.0,
             signed=False, W=0, replicas=8, sweeps=200, mode="paper"),
        # the paper's standard annealer (Algorithm 2), which the method is compared with
        dict(sparse, name="torus71_alg2", graph="torus", count=1, n_lo=5041, n_hi=5041, d_lo=4.0, d_hi=4.0,
             signed=False, W=0, replicas=8, sweeps=100, mode="paper", standard=True),
        # logits of the learned start for a set of held-out graphs, features included
        dict(kind="infer", name="infer128", graph="mix", count=128, n_lo=1000, n_hi=5000, d_lo=3.0, d_hi=48.0,
             signed=False, steps=256),
        # the same for a single graph
        dict(kind="infer", name="infer1", graph="er", count=1, n_lo=1999, n_hi=1999, d_lo=12.0, d_hi=12.0,
             signed=False, steps=256),
        # one training batch: forward, loss and every gradient, features at hand
        dict(kind="train", name="train16", graph="mix", count=16, n_lo=1000, n_hi=5000, d_lo=3.0, d_hi=48.0,
             signed=False, steps=0),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    pick = rng.choice(["ba", "ba", "wide", "torus", "er", "batch", "warm", "default", "standard", "infer", "train"])
    c = dict(kind="anneal", A=1, B=rng.choice([1, 4, 4]), mode=rng.choice(["metropolis", "metropolis", "paper"]),
             t0=3.0, t1=0.05, start="random", tune=False, standard=False, count=1, signed=False)
    if pick == "ba":
        n = spread(3000, 1_000_000)
        r = rng.choice([1, 2, 3, 8, 8, 11]) if n < 500_000 else rng.choice([1, 3, 8])
        c.update(graph="ba", n_lo=n, n_hi=n, d_lo=10.0, d_hi=10.0, W=rng.choice([32, 64, 100, 128, 256, 256]), replicas=r,
                 sweeps=spread(20, 300))
    elif pick == "wide":
        n = spread(20_000, 300_000)
        c.update(graph="ba", n_lo=n, n_hi=n, d_lo=10.0, d_hi=10.0, W=rng.choice([300, 512, 1024]),
                 replicas=rng.choice([1, 4, 8]), sweeps=spread(20, 100))
    elif pick == "torus":
        L = rng.randint(20, 100)
        c.update(graph="torus", n_lo=L * L, n_hi=L * L, d_lo=4.0, d_hi=4.0, signed=True,
                 W=rng.choice([32, 64, 128, 256, 256]), replicas=spread(1, 64), sweeps=spread(100, 2000), tune=True)
    elif pick == "er":
        n, d = spread(200, 3000), rng.uniform(3.0, 48.0)
        c.update(graph="er", n_lo=n, n_hi=n, d_lo=d, d_hi=d, signed=rng.random() < 0.5,
                 W=rng.choice([7, 32, 64, 128, 256]), replicas=rng.choice([1, 1, 2, 5, 8]), sweeps=spread(50, 800))
    elif pick == "batch":
        c.update(graph="er", count=spread(8, 400), n_lo=800, n_hi=3000, d_lo=3.0, d_hi=48.0, signed=True,
                 W=rng.choice([64, 256, 256]), replicas=1, sweeps=spread(50, 500), tune=True)
    elif pick == "warm":
        c.update(graph="mix", count=spread(4, 100), n_lo=1000, n_hi=5000, d_lo=3.0, d_hi=48.0, W=256,
                 replicas=rng.choice([1, 4, 8]), sweeps=rng.choice([25, 50, 100]), t0=0.5, start="device",
                 mode="metropolis")
    elif pick in ("default", "standard"):
        if rng.random() < 0.5:
            n = spread(500, 3000)
            c.update(graph="er", n_lo=n, n_hi=n, d_lo=16.0, d_hi=16.0)
        else:
            L = rng.randint(20, 71)
            c.update(graph="torus", n_lo=L * L, n_hi=L * L, d_lo=4.0, d_hi=4.0)
        c.update(W=0, replicas=rng.choice([1, 4, 8]), sweeps=spread(20, 200), mode="paper",
                 standard=pick == "standard")
    else:
        c = dict(kind=pick, graph="mix", count=spread(1, 110) if pick == "infer" else spread(2, 24),
                 n_lo=rng.randint(300, 1500), n_hi=rng.randint(2000, 5000), d_lo=3.0, d_hi=48.0, signed=False,
                 steps=rng.choice([32, 64, 256]) if pick == "infer" else 0)
        if rng.random() < 0.3:
            n = spread(200, 7000)
            c.update(count=1, n_lo=n, n_hi=n)
    return c


# ---------------------------------------------------------------------------------------------
# Graphs: made on the GPU from the seed, handed over as the host CSR that the library takes.

def _sizes(case):
    """Sizes and mean degrees of the case's graphs: the same for every seed, so that results keep their shapes."""
    rng = np.random.default_rng(case["count"])
    ns = rng.integers(case["n_lo"], case["n_hi"] + 1, case["count"])
    ds = rng.uniform(case["d_lo"], case["d_hi"], case["count"])
    return ns, ds


def _ba_edges(n, m, gen):
    """Preferential attachment (Batagelj-Brandes): slot k of vertex v copies a uniform earlier slot."""
    core = torch.combinations(torch.arange(m + 1, device="cuda"), 2)
    c = 2 * core.shape[0]
    k = torch.arange((n - m - 1) * m, device="cuda")
    vert = m + 1 + k // m
    pos = c + 2 * k
    to = (torch.rand(k.shape[0], generator=gen, device="cuda", dtype=torch.float64) * (pos + 1)).long()
    ptr = torch.arange(c + 2 * k.shape[0], device="cuda")
    ptr[pos + 1] = to
    val = torch.empty_like(ptr)
    val[:c] = core.reshape(-1)
    val[pos] = vert
    for _ in range(64):
        nxt = ptr[ptr]
        if torch.equal(nxt, ptr):
            break
        ptr = nxt
    return torch.cat([core[:, 0], vert]), torch.cat([core[:, 1], val[ptr[pos + 1]]])


def _graph(case, seed):
    """The disjoint union of the case's graphs: device CSR, vertex offsets, weights, colouring."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ns, ds = _sizes(case)
    ptr = np.concatenate([[0], np.cumsum(ns)]).astype(np.int64)
    N, color = int(ptr[-1]), None
    us, vs = [], []
    if case["graph"] == "ba":
        u, v = _ba_edges(N, 5, gen)
        us, vs = [u], [v]
    elif case["graph"] == "torus":
        L = math.isqrt(N)
        i = torch.arange(N, device="cuda")
        x, y = i % L, i // L
        us, vs = [i, i], [y * L + (x + 1) % L, ((y + 1) % L) * L + x]
        if L % 2 == 0:
            color = ((x + y) & 1).int().cpu().numpy()
    else:
        er = np.arange(case["count"]) % 2 == 0 if case["graph"] == "mix" else np.ones(case["count"], bool)
        m = np.where(er, (ns * ds / 2).astype(np.int64), 0)
        of = torch.repeat_interleave(torch.arange(len(ns), device="cuda"), torch.from_numpy(m).cuda())
        n_d, p_d = torch.from_numpy(ns).cuda()[of], torch.from_numpy(ptr).cuda()[of]
        for out in (us, vs):
            f = torch.rand(of.shape[0], generator=gen, device="cuda", dtype=torch.float64)
            out.append(p_d + (f * n_d).long())
        for g in np.nonzero(~er)[0]:     # random geometric: points in the unit square, joined within a radius
            n, d = int(ns[g]), 4.0 + 28.0 * (ds[g] - 3.0) / 45.0
            p = torch.rand((n, 2), generator=gen, device="cuda", dtype=torch.float64)
            near = (p[:, None, 0] - p[None, :, 0]) ** 2 + (p[:, None, 1] - p[None, :, 1]) ** 2 < d / (math.pi * (n - 1))
            uv = near.triu(1).nonzero() + int(ptr[g])
            us.append(uv[:, 0])
            vs.append(uv[:, 1])
    u, v = torch.cat(us), torch.cat(vs)
    keep = u != v
    key = torch.unique(torch.minimum(u, v)[keep] * N + torch.maximum(u, v)[keep])
    a, b = key // N, key % N
    w = torch.ones_like(a)
    if case["signed"]:       # +-1 weights; in a batch half of the instances keep unit weights
        w = 1 - 2 * torch.randint(0, 2, a.shape, generator=gen, device="cuda")
        if case["count"] > 1:
            odd = torch.repeat_interleave(torch.arange(len(ns), device="cuda") % 2, torch.from_numpy(ns).cuda())
            w = torch.where(odd[a] == 1, w, torch.ones_like(w))
    order = torch.argsort(torch.cat([a * N + b, b * N + a]))
    col = torch.cat([b, a])[order].int()
    deg = torch.bincount(torch.cat([a, b]), minlength=N)
    row_ptr = torch.cat([torch.zeros(1, dtype=torch.long, device="cuda"), torch.cumsum(deg, 0)])
    return SimpleNamespace(N=N, ptr=ptr, ns=ns, row_ptr=row_ptr, col=col, w=torch.cat([w, w])[order].int(), color=color)


def _schedule(case):
    if case["mode"] == "paper":
        scale = 5.0 if case["standard"] else 1.0
        return Schedule(sweeps=case["sweeps"], mode=GDI_PAPER_PF, pf0=0.02 * scale, pf1=0.0002 * scale)
    return Schedule(sweeps=case["sweeps"], mode=GDI_METROPOLIS, t0=case["t0"] * case["B"], t1=case["t1"] * case["B"])


def _features(g, seed):
    """Input features as training has them at hand: unit noise channels, then the degree channels."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    X = torch.zeros((g.N, learn.FIN), device="cuda")
    X[:, :NOISE] = torch.randn((g.N, NOISE), generator=gen, device="cuda")
    deg = (g.row_ptr[1:] - g.row_ptr[:-1]).double()
    of = torch.repeat_interleave(torch.arange(len(g.ns), device="cuda"), torch.from_numpy(g.ns).cuda())
    mean = torch.zeros(len(g.ns), dtype=torch.float64, device="cuda").index_add_(0, of, deg) / torch.from_numpy(g.ns).cuda()
    X[:, NOISE] = torch.log1p(deg).float()
    X[:, NOISE + 1] = (deg / mean[of].clamp_min(1e-30)).float()
    return X


def _labels(g, X, seed):
    """A balanced partition per graph that the features partly predict."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 2)
    score = X[:, 0] + torch.randn(g.N, generator=gen, device="cuda")
    y = torch.empty(g.N, dtype=torch.int8, device="cuda")
    for lo, hi in zip(g.ptr[:-1], g.ptr[1:]):
        n = int(hi - lo)
        s = torch.full((n,), -1, dtype=torch.int8, device="cuda")
        s[torch.argsort(score[lo:hi], descending=True, stable=True)[:n // 2]] = 1
        y[lo:hi] = s
    return y


def _params(seed):
    """Glorot-uniform weights and small biases, flat in the library's order."""
    rng = np.random.default_rng(seed + 3)
    parts = []
    for din, dout in learn.LAYER_DIMS:
        a = math.sqrt(6.0 / (din + dout))
        parts += [rng.uniform(-a, a, din * dout), rng.uniform(-a, a, din * dout), rng.uniform(-0.1, 0.1, dout)]
    a = math.sqrt(6.0 / 65)
    parts += [rng.uniform(-a, a, 64), rng.uniform(-0.1, 0.1, 1)]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    g = _graph(case, seed)
    if case["kind"] == "anneal":
        host = SimpleNamespace(n=g.N, row_ptr=g.row_ptr.cpu().numpy(), col=g.col.cpu().numpy(), w=g.w.cpu().numpy(),
                               color=g.color)
        ann = Annealer(host, A=case["A"], B=case["B"], W=case["W"], replicas=case["replicas"],
                       inst_ptr=g.ptr if case["count"] > 1 else None)
        s = SimpleNamespace(kind="anneal", ann=ann, schedule=_schedule(case), seed=seed, init=None,
                            flags=GDI_FLAG_STANDARD if case["standard"] else 0)
        if case["start"] == "device":    # a balanced start per graph, the same for every replica
            half = _labels(g, _features(g, seed), seed)
            s.init = half.repeat(case["replicas"])
            s.spins = torch.empty_like(s.init)
        if case["tune"]:
            ann.autotune(s.schedule, probe_sweeps=min(20, case["sweeps"]))
        return s
    batch = learn.GraphBatch(N=g.N, G=len(g.ns), max_n=int(g.ns.max()), graph_ptr_h=g.ptr, row_ptr=g.row_ptr,
                             col=g.col, graph_ptr=torch.from_numpy(g.ptr).cuda(),
                             graph_id=torch.arange(len(g.ns), dtype=torch.int32, device="cuda"), graphs=[])
    model = learn.MPNN(params=_params(seed), steps=case["steps"], feat_seed=FEAT_SEED)
    s = SimpleNamespace(kind=case["kind"], model=model, batch=batch)
    if case["kind"] == "train":
        s.X = _features(g, seed)
        s.y = _labels(g, s.X, seed)
    return s


def run(s):
    if s.kind == "anneal":
        stream = torch.cuda.current_stream()
        if s.init is not None:
            s.ann.anneal(s.schedule, s.seed, init_device_ptr=s.init.data_ptr(), flags=s.flags, stream=stream)
            s.ann.spins_to_device(s.spins.data_ptr())
            return {"spins": s.spins, **s.ann.results()}
        s.ann.anneal(s.schedule, s.seed, flags=s.flags, stream=stream)
        return {"spins": s.ann.spins(), **s.ann.results()}
    if s.kind == "infer":
        z, cache = s.model.forward(s.batch)
        return {"logits": z, "features": cache[0][0]}
    # the Adam update (one pass over 27k parameters) is left to the optimiser's step, so that the
    # weights stay those of the state
    z, cache = s.model.forward(s.batch, s.X)
    loss, stats = s.model.loss_and_backward(s.batch, s.y, z, cache)
    return {"logits": z, "loss": loss, "stats": stats, "grads": s.model.grads}


def work(case):
    """Bytes: the graph, the state and the results once.  Operations: an anneal draws and decides every
    spin in every sweep (a Philox block of about 100 operations for four spins, then about 10 for the
    threshold and the decision); the network multiplies dense layers and sums neighbours."""
    N = case["count"] * (case["n_lo"] + case["n_hi"]) / 2
    nnz = N * (case["d_lo"] + case["d_hi"]) / 2
    if case["kind"] == "anneal":
        R = case["replicas"]
        ops = 35.0 * N * R * case["sweeps"]
        if case["standard"]:
            ops += 2.0 * N * R * case["sweeps"] * (case["n_lo"] + case["n_hi"]) / 2
        return {"bytes": 4 * nnz + 8 * N + 2 * N * R, "flops": ops}
    dense = 2.0 * N * 64 * (2 * 16 + 2 * 64 + 2 * 64)
    gather = 2.0 * nnz * (16 + 64 + 64)
    if case["kind"] == "infer":
        return {"bytes": 4 * nnz + 8 * N + 64 * N + 4 * N, "flops": dense + gather + 2.0 * nnz * NOISE * case["steps"]}
    return {"bytes": 4 * nnz + 8 * N + 64 * N + 5 * N, "flops": 3 * dense + 2 * gather}


# ---------------------------------------------------------------------------------------------
# The network in 64 bits.

def _philox_sign(local, graph, seed):
    """Top bit of word 0 of Philox4x32-10 at counter (vertex, channel, graph, tag): [n, 8] signs."""
    lo32 = np.uint64(0xFFFFFFFF)
    ch = np.arange(NOISE, dtype=np.uint64)[None, :]
    c = [np.broadcast_to(x, (len(local), NOISE)).astype(np.uint64)
         for x in (local[:, None], ch, graph[:, None], np.uint64(0x4D504E4E))]
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & lo32, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & lo32]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & lo32, (k1 + np.uint64(0xBB67AE85)) & lo32
    return np.where(c[0] >> np.uint64(31), -1.0, 1.0)


def exact(case, seed):
    if case["kind"] == "anneal":
        return None
    g = _graph(case, seed)
    f64 = torch.float64
    deg = (g.row_ptr[1:] - g.row_ptr[:-1]).to(f64)
    of = torch.repeat_interleave(torch.arange(len(g.ns), device="cuda"), torch.from_numpy(g.ns).cuda())
    ns = torch.from_numpy(g.ns).cuda().to(f64)
    rows = torch.repeat_interleave(torch.arange(g.N, device="cuda"), deg.long())
    cols = g.col.long()

    def sparse(vals):
        return torch.sparse_csr_tensor(g.row_ptr, cols, vals, size=(g.N, g.N))

    def per_graph(v):
        return torch.zeros((len(g.ns),) + v.shape[1:], dtype=f64, device="cuda").index_add_(0, of, v)

    if case["kind"] == "infer":
        local = np.concatenate([np.arange(n, dtype=np.uint64) for n in g.ns])
        R = torch.from_numpy(_philox_sign(local, of.cpu().numpy().astype(np.uint64), FEAT_SEED)).cuda()
        walk = sparse(torch.rsqrt(deg[rows] * deg[cols]))
        for _ in range(case["steps"]):
            R = 0.5 * R + 0.5 * (walk @ R)
        R = R - (per_graph(R) / ns[:, None])[of]
        rms = torch.sqrt(per_graph(R * R) / ns[:, None]) + 1e-12
        X = torch.zeros((g.N, learn.FIN), dtype=f64, device="cuda")
        X[:, :NOISE] = R / rms[of]
        X[:, NOISE] = torch.log1p(deg)
        X[:, NOISE + 1] = deg / (per_graph(deg) / ns).clamp_min(1e-300)[of]
    else:
        X = _features(g, seed).to(f64)

    flat, layers, o = torch.from_numpy(_params(seed)).cuda(), [], 0
    for din, dout in learn.LAYER_DIMS:
        mats = [flat[o + k * din * dout:o + (k + 1) * din * dout].bfloat16().to(f64).reshape(din, dout) for k in (0, 1)]
        layers.append((mats[0], mats[1], flat[o + 2 * din * dout:o + 2 * din * dout + dout].to(f64)))
        o += 2 * din * dout + dout
    wo, bo = flat[o:o + 64].bfloat16().to(f64), flat[o + 64].to(f64)
    mean = sparse(1.0 / deg[rows])
    hs, aggs = [X], []
    for Ws, Wn, b in layers:
        aggs.append(mean @ hs[-1])
        hs.append(torch.relu(hs[-1] @ Ws + aggs[-1] @ Wn + b))
    z = hs[-1] @ wo + bo
    if case["kind"] == "infer":
        return {"logits": z, "features": X}

    y, lam = _labels(g, _features(g, seed), seed).to(f64), 0.1
    sp = torch.nn.functional.softplus
    L1, L2, m = per_graph(sp(-y * z)) / ns, per_graph(sp(y * z)) / ns, per_graph(torch.tanh(z)) / ns
    lg = torch.minimum(L1, L2) + lam * m * m
    t = torch.where(L1 <= L2, 1.0, -1.0)[of] * y
    dz = (-t * torch.sigmoid(-t * z) + 2 * lam * m[of] * (1 - torch.tanh(z) ** 2)) / (ns[of] * len(g.ns))
    grads = [dz.sum()[None], hs[-1].T @ dz]
    dh, back = dz[:, None] * wo, sparse(1.0 / deg[cols])
    for l in (2, 1, 0):
        Ws, Wn, _ = layers[l]
        dpre = dh * (hs[l + 1] > 0)
        grads += [dpre.sum(0), aggs[l].T @ dpre, hs[l].T @ dpre]
        dh = dpre @ Ws.T + back @ (dpre @ Wn.T)
    return {"logits": z, "loss": lg.mean()[None], "stats": torch.stack([L1, L2, m, lg], 1),
            "grads": torch.cat([v.reshape(-1) for v in grads[::-1]])}
