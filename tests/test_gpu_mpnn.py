"""GPU kernels of the learned warm start against the FP64 network oracle."""
import numpy as np
import pytest

from oracle import mpnn as ref
from gdi_synth import batch_union, erdos_renyi, random_geometric

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup(gdi):
    import torch
    from paper_1908_00210_gb300 import learn
    gs = [erdos_renyi(300, 0.03, 11), random_geometric(260, 0.12, 12), erdos_renyi(411, 0.015, 13, signed=False)]
    ids = np.array([5, 6, 7], dtype=np.uint32)
    b = learn.GraphBatch.from_graphs(gs, graph_ids=ids)
    gp, u = batch_union(gs)
    rng = np.random.default_rng(2)
    y = np.empty(gp[-1], dtype=np.int8)
    for g in range(len(gs)):
        n = gp[g + 1] - gp[g]
        y[gp[g]:gp[g + 1]] = rng.permutation(np.where(np.arange(n) < n // 2, 1, -1))
    model = learn.MPNN(seed=3, lam=0.2, feat_seed=12345, steps=3)
    return learn, torch, gs, ids, b, gp, u, y, model


@pytest.mark.parametrize("flags", [0, 1, 3])
def test_features_match_oracle(setup, flags):
    learn, torch, gs, ids, b, gp, u, y, model = setup
    m = learn.MPNN(seed=3, lam=0.2, feat_seed=12345, steps=3, feat_flags=flags)
    X = m.features(b).cpu().numpy()
    Xr = ref.features(gp, ids, u.row_ptr, u.col, 12345, 3, flags)
    assert np.max(np.abs(X - Xr)) < 1e-4


def test_forward_logits_within_1e2_of_fp64(setup):
    learn, torch, gs, ids, b, gp, u, y, model = setup
    Xr = ref.features(gp, ids, u.row_ptr, u.col, 12345, 3)
    X = torch.from_numpy(Xr.astype(np.float32)).cuda()
    z, _ = model.forward(b, X)
    P = ref.effective_params(model.params.cpu().numpy())
    zr, _ = ref.forward(P, u.row_ptr, u.col, Xr.astype(np.float32).astype(np.float64))
    err = np.max(np.abs(z.cpu().numpy() - zr))
    assert err < 1e-2, err
    assert err < 1e-3 * max(1.0, np.max(np.abs(zr)))   # float32 activations: far inside the bar


def test_gradients_match_oracle_backward(setup):
    learn, torch, gs, ids, b, gp, u, y, model = setup
    Xr = ref.features(gp, ids, u.row_ptr, u.col, 12345, 3).astype(np.float32)
    X = torch.from_numpy(Xr).cuda()
    z, cache = model.forward(b, X)
    loss, stats = model.loss_and_backward(b, torch.from_numpy(y).cuda(), z, cache)
    g = model.grads.cpu().numpy()
    P = ref.effective_params(model.params.cpu().numpy())
    zr, cr = ref.forward(P, u.row_ptr, u.col, Xr.astype(np.float64))
    Lr, dzr, _ = ref.loss(gp, zr, y, model.lam)
    gr = ref.flat_grads(ref.backward(P, u.row_ptr, u.col, cr, dzr))
    assert abs(float(loss.item()) - Lr) < 1e-4 * max(1.0, abs(Lr))
    scale = np.max(np.abs(gr))
    assert np.max(np.abs(g - gr)) < 2e-3 * scale, (np.max(np.abs(g - gr)), scale)


def test_adam_step_matches_oracle(setup):
    learn, torch, gs, ids, b, gp, u, y, model = setup
    m2 = learn.MPNN(seed=9, lr=1e-2)
    rng = np.random.default_rng(1)
    grad = rng.standard_normal(m2.P).astype(np.float32)
    p0 = m2.params.cpu().numpy().astype(np.float64)
    m2.grads.copy_(torch.from_numpy(grad))
    m2.adam()
    p1, mm, vv = ref.adam_step(p0, grad.astype(np.float64), np.zeros(m2.P), np.zeros(m2.P), 1e-2, 0.9, 0.999, 1e-8, 1)
    assert np.max(np.abs(m2.params.cpu().numpy() - p1)) < 1e-6
    bf = m2.params_bf16.cpu().numpy().view(np.uint16)
    assert np.array_equal(bf.astype(np.uint32) << 16,
                          ref.bf16_round(m2.params.cpu().numpy()).astype(np.float32).view(np.uint32))


def test_rounding_matches_oracle(gdi):
    import torch
    from paper_1908_00210_gb300 import learn
    rng = np.random.default_rng(7)
    sizes = [1, 2, 7, 300, 1001, 5000]
    gp = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    z = (rng.standard_normal(gp[-1]) + 0.1).astype(np.float32)
    z[10:20] = z[10]                                     # ties inside a graph
    s = torch.empty(gp[-1], dtype=torch.int8, device="cuda")
    d_gp = torch.from_numpy(gp).cuda()      # keep the device buffers alive until the kernel ran
    d_z = torch.from_numpy(z).cuda()
    rc = learn.lib().gdi_mpnn_round(len(sizes), d_gp.data_ptr(), max(sizes), d_z.data_ptr(), s.data_ptr(), None)
    assert rc == 0
    torch.cuda.synchronize()
    assert np.array_equal(s.cpu().numpy(), ref.round_balanced(gp, z))


def test_training_reduces_loss_and_prediction_anneals(setup, gdi):
    """A few Adam steps on annealer labels reduce the loss; the rounded prediction is exactly
    balanced and gdi_anneal accepts it as a device-side initial state."""
    learn, torch, gs, ids, b, gp, u, y, model = setup
    labels, best = learn.label_graphs(gs, sweeps=300, replicas=2, seed=3)
    yl = torch.from_numpy(labels).cuda()
    m = learn.MPNN(seed=4, lr=3e-3, lam=0.1)
    first = float(m.train_step(b, yl).item())
    for _ in range(60):
        last = float(m.train_step(b, yl).item())
    assert last < first
    s = m.predict_spins(b)
    sh = s.cpu().numpy()
    for g in range(len(gs)):
        assert abs(int(sh[gp[g]:gp[g + 1]].astype(np.int64).sum())) == (gp[g + 1] - gp[g]) % 2
    cut, spins, ms = learn.anneal_batch(gs, sweeps=50, t0=0.5, t1=0.05, seed=5, replicas=1, init=s)
    assert np.all(np.isfinite(cut)) and ms > 0


def test_shipped_settings_features_logits_gradients_vs_fp64(gdi):
    """The settings the warm start ships with: 16 graphs of the recipe (n in [1000, 5000], half
    Erdos-Renyi, half random geometric; held-out seeds), 256 lazy-walk diffusion steps of the noise
    channels.  GPU features (FP32 diffusion) against the FP64 oracle; logits from the GPU's own
    features within 1e-2 of the FP64 forward on the FP64 features; gradients of one batch."""
    import torch
    from paper_1908_00210_gb300 import learn
    gs = learn.make_graphs(16, 900000)
    ids = np.arange(900000, 900016, dtype=np.uint32)
    b = learn.GraphBatch.from_graphs(gs, graph_ids=ids)
    gp, u = batch_union(gs)
    model = learn.MPNN(seed=21, lam=0.1, feat_seed=0x9E3779B9, steps=256, feat_flags=1)
    X = model.features(b)
    Xr = ref.features(gp, ids, u.row_ptr, u.col, 0x9E3779B9, 256, ref.ALIGN)
    ferr = np.max(np.abs(X.cpu().numpy() - Xr))
    assert ferr < 1e-3, ferr
    z, cache = model.forward(b, X)
    P = ref.effective_params(model.params.cpu().numpy())
    zr, cr = ref.forward(P, u.row_ptr, u.col, Xr)
    zerr = np.max(np.abs(z.cpu().numpy() - zr))
    assert zerr < 1e-2, zerr
    rng = np.random.default_rng(3)
    y = np.empty(gp[-1], dtype=np.int8)
    for g in range(len(gs)):
        n = gp[g + 1] - gp[g]
        y[gp[g]:gp[g + 1]] = rng.permutation(np.where(np.arange(n) < n // 2, 1, -1))
    loss, _ = model.loss_and_backward(b, torch.from_numpy(y).cuda(), z, cache)
    Lr, dzr, _ = ref.loss(gp, zr, y, model.lam)
    gr = ref.flat_grads(ref.backward(P, u.row_ptr, u.col, cr, dzr))
    assert abs(float(loss.item()) - Lr) < 1e-4 * max(1.0, abs(Lr))
    g = model.grads.cpu().numpy()
    assert np.max(np.abs(g - gr)) < 2e-3 * np.max(np.abs(gr))


def test_trained_start_against_untrained_and_plain_annealer(gdi):
    """What the trained network gains, on held-out graphs of the recipe (256 training graphs with
    annealer labels, 32 held-out graphs, 8 seeds each): annealed from its rounded prediction at
    T0 = 0.5 for 25 sweeps it reaches the plain annealer's median cut (2000 sweeps from a random
    start at T0 = 3.0) on more graphs than the same network untrained, and on far more than the plain
    annealer does in 25 sweeps.  The rounded noise channel 0 alone -- the spectral input the network
    receives -- is evaluated beside them: at the recipe's full scale it reaches as many graphs as the
    trained network (the ablation in the learned-start profile)."""
    from paper_1908_00210_gb300 import learn
    tr = learn.make_graphs_parallel(256, 500_000, processes=8)
    te = learn.make_graphs_parallel(32, 900_000, processes=8)
    labels, _ = learn.label_graphs(tr, sweeps=2000)
    m = learn.MPNN(seed=0, lr=2e-3, lam=0.1, steps=256, feat_flags=1)
    ds = learn.Dataset(tr, labels, m)
    hist = learn.train_dataset(m, ds, epochs=30)
    assert hist[-1] < hist[0] - 0.02
    un = learn.MPNN(seed=0, lr=2e-3, lam=0.1, steps=256, feat_flags=1)
    starts = {"noise_channel0": ("spins", learn.channel_spins(un, te, 0), 0.5), "untrained": (un, 0.5),
              "trained": (m, 0.5)}
    res = learn.evaluate_many(starts, te, ladder=[25, 100])
    reached = {k: res[k]["reached"][25] for k in ("noise_channel0", "untrained", "trained", "random_T3.0")}
    print("reached at 25 sweeps:", reached)
    assert reached["trained"] > reached["untrained"]
    assert reached["trained"] >= 8 and reached["random_T3.0"] == 0
    assert reached["noise_channel0"] >= 8


def _ring_graph(n, extra, seed):
    """A ring with `extra` random chords and, past vertex n - 3, two isolated vertices and a leaf."""
    from gdi_synth.graphs import from_edges
    rng = np.random.default_rng(seed)
    m = n - 3
    u, v = np.arange(m), (np.arange(m) + 1) % m
    u = np.concatenate([u, rng.integers(0, m, extra), [0]])
    v = np.concatenate([v, rng.integers(0, m, extra), [n - 1]])
    return from_edges(n, u, v)


@pytest.mark.parametrize("d,shift", [(8, 0), (16, 0), (64, 0), (64, 1), (5, 0), (33, 0)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_aggregate_widths_and_alignments(gdi, d, shift, mode):
    """Every width the vector kernel takes, the same width off a 16-byte boundary, and other widths;
    rows of 0, 1 and more than 32 neighbours.  Sums of at most 70 float32 products: 1e-5 of the
    largest value."""
    import torch
    from paper_1908_00210_gb300 import learn
    g = _ring_graph(203, 900, d)
    hub = np.arange(1, 70)
    from gdi_synth.graphs import from_edges
    u, v, _ = g.edges()
    g = from_edges(g.n, np.concatenate([u, np.zeros(69, np.int64)]), np.concatenate([v, hub]))
    rng = np.random.default_rng(d + mode)
    x = rng.standard_normal((g.n, d)).astype(np.float32)
    y0 = rng.standard_normal((g.n, d)).astype(np.float32)
    buf = torch.empty(2 * (g.n * d + 4), device="cuda")
    X = buf[shift:shift + g.n * d]
    Y = buf[g.n * d + 4 - (g.n * d) % 4 + shift:][:g.n * d]
    rp, col = torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col).cuda()
    f = [ref.mean_aggregate, ref.mean_aggregate_T, ref.lazy_walk][mode](g.row_ptr, g.col, x.astype(np.float64))
    f = np.where(np.isfinite(f), f, 0.0)
    for acc in (0, 1):
        X.copy_(torch.from_numpy(x.ravel()))
        Y.copy_(torch.from_numpy(y0.ravel()))
        rc = learn.lib().gdi_mpnn_aggregate(g.n, rp.data_ptr(), col.data_ptr(), X.data_ptr(), d, Y.data_ptr(), mode,
                                            acc, None)
        assert rc == 0
        want = f + acc * y0
        got = Y.cpu().numpy().reshape(g.n, d)
        assert np.max(np.abs(got - want)) < 1e-5 * np.max(np.abs(want)), (acc, np.max(np.abs(got - want)))


@pytest.mark.parametrize("n", [1, 31, 33, 4865, 9801])
@pytest.mark.parametrize("din,dout,shift", [(64, 64, 0), (16, 64, 0), (64, 64, 1), (7, 64, 0), (64, 1, 0), (16, 5, 0),
                                            (33, 33, 0), (1, 1, 0)])
def test_wgrad_shapes(gdi, n, din, dout, shift):
    """Row counts around the tiles and the blocks' chunks, widths that fill the tile and not, operands
    off a 16-byte boundary; the result is added to what is there.  A float32 sum of n products of
    standard normals, summed in trees of depth about 40, is expected 6e-8 sqrt(40 n) off, 4.5 times that at
    the worst of 4,096: 1e-5 (1 + sqrt(n)) is some five times as much."""
    import torch
    from paper_1908_00210_gb300 import learn
    rng = np.random.default_rng(n + din + dout)
    a, b = rng.standard_normal((n, din)).astype(np.float32), rng.standard_normal((n, dout)).astype(np.float32)
    o0, c0 = rng.standard_normal((din, dout)).astype(np.float32), rng.standard_normal(dout).astype(np.float32)

    def dev(x):
        t = torch.empty(x.size + 4, device="cuda")[shift:shift + x.size]
        t.copy_(torch.from_numpy(x.ravel()))
        return t
    A, Bm, out, cs = dev(a), dev(b), dev(o0), dev(c0)
    assert learn.lib().gdi_mpnn_wgrad(n, A.data_ptr(), din, Bm.data_ptr(), dout, out.data_ptr(), cs.data_ptr(), None) == 0
    want = o0 + a.astype(np.float64).T @ b.astype(np.float64)
    tol = 1e-5 * (1 + np.sqrt(n))
    assert np.max(np.abs(out.cpu().numpy().reshape(din, dout) - want)) < tol
    assert np.max(np.abs(cs.cpu().numpy() - (c0 + b.astype(np.float64).sum(0)))) < tol


@pytest.mark.parametrize("steps", [1, 5, 6])
def test_features_one_launch_and_the_rest(gdi, steps):
    """Graphs at the edges of the one-launch walk: one vertex, isolated vertices, sizes around the 32-row
    slices, a hub whose degree exceeds the counting sort's bins, a graph too dense for the laid-out
    columns and one too large for a block (both walked by the grid-wide kernel), and a batch whose mean is too
    large for a block.  Features are float32 sums of at most 9,100 terms, scaled to unit RMS: 1e-4."""
    from gdi_synth.graphs import from_edges, star_graph
    from paper_1908_00210_gb300 import learn
    rng = np.random.default_rng(steps)
    dense = np.triu_indices(400, 1)
    keep = rng.random(dense[0].size) < 0.5
    small = [from_edges(1, np.zeros(0), np.zeros(0)), _ring_graph(31, 5, 1), _ring_graph(32, 9, 2), _ring_graph(33, 0, 3),
             star_graph(700), from_edges(400, dense[0][keep], dense[1][keep]), _ring_graph(2047, 9000, 4)]
    big = _ring_graph(9101, 3000, 5)
    for gs in (small, small + [big] + small[1:], [big, big]):
        gp, u = batch_union(gs)
        ids = np.arange(3, 3 + len(gs), dtype=np.uint32)
        b = learn.GraphBatch.from_graphs(gs, graph_ids=ids)
        m = learn.MPNN(seed=1, feat_seed=77, steps=steps)
        X = m.features(b).cpu().numpy()
        Xr = ref.features(gp, ids, u.row_ptr, u.col, 77, steps)
        for q in range(len(gs)):
            if gs[q].n == 1:
                continue                       # one vertex: centred to 0, scaled by 1e-12
            s = slice(gp[q], gp[q + 1])
            assert np.max(np.abs(X[s] - Xr[s])) < 1e-4, (q, np.max(np.abs(X[s] - Xr[s])))


@pytest.mark.parametrize("steps", [1, 4, 5, 32, 33])
@pytest.mark.parametrize("cut", [(0, 700, 1999, 2000), (0, 300, 300, 1500, 2000), (0, 9400, 9600), (0, 200, 9600)])
def test_features_of_graphs_with_columns_between_them(gdi, cut, steps):
    """graph_ptr cuts connected graphs, so columns lead from one to another: walked as one graph, as the
    definition says, with every piece small (an empty and a one-vertex one among them) and with one too large
    for a block.  Float32 sums of at most some 2,000 terms, scaled to unit RMS: 1e-4."""
    import ctypes as C
    import torch
    from paper_1908_00210_gb300 import learn
    g = _ring_graph(cut[-1], 4 * cut[-1], len(cut))
    gp = np.array(cut, dtype=np.int64)
    ids = np.arange(9, 9 + len(cut) - 1, dtype=np.uint32)
    dev = [torch.from_numpy(a).cuda() for a in (gp, ids.view(np.int32), g.row_ptr, g.col)]
    X, scratch = torch.empty(g.n, 16, device="cuda"), torch.empty(16 * g.n, device="cuda")
    for _ in range(2):
        rc = learn.lib().gdi_mpnn_features(g.n, len(ids), *[a.data_ptr() for a in dev], 77, steps, 0, X.data_ptr(),
                                           scratch.data_ptr(), C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        Xr = ref.features(gp, ids, g.row_ptr, g.col, 77, steps)
        got = X.cpu().numpy()
        for a, b in zip(gp[:-1], gp[1:]):
            if b - a > 1:                  # (one vertex: centred to 0, scaled by 1e-12)
                assert np.max(np.abs(got[a:b] - Xr[a:b])) < 1e-4, (a, b)


@pytest.mark.parametrize("big,deg,small", [(300_000, 4, 40), (12_000, 6, 1)])
def test_features_of_one_large_graph_among_small_ones(gdi, big, deg, small):
    """The walk of a batch whose large graph does not fit a block takes no longer than a launch per step over all
    its vertices (it took 1.3 to 2 times as long)."""
    import torch
    from gdi_synth import from_edges
    from paper_1908_00210_gb300 import learn
    rng = np.random.default_rng(big)

    def graph(n, d):
        u, v = rng.integers(0, n, (2, n * d // 2))
        e = np.unique(np.minimum(u, v)[u != v].astype(np.int64) * n + np.maximum(u, v)[u != v])
        return from_edges(n, e // n, e % n)
    b = learn.GraphBatch.from_graphs([graph(big, deg)] + [graph(1000, 6)] * small)
    m = learn.MPNN(seed=1, steps=256)
    r = torch.empty(2, b.N, 8, device="cuda")

    def one_launch_per_step():
        for s in range(m.steps):
            learn.lib().gdi_mpnn_aggregate(b.N, b.row_ptr.data_ptr(), b.col.data_ptr(), r[s & 1].data_ptr(), 8,
                                           r[1 - (s & 1)].data_ptr(), 2, 0, m._st())

    def ms(f):
        f()
        t = []
        for _ in range(3):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            f()
            e1.record()
            e1.synchronize()
            t.append(e0.elapsed_time(e1))
        return min(t)
    assert ms(lambda: m.features(b)) < 1.1 * ms(one_launch_per_step)


@pytest.mark.parametrize("steps", [1, 2, 3, 4, 5, 8, 31, 32, 33])
@pytest.mark.parametrize("n,count", [(90, 1), (300, 40), (2000, 1), (2000, 20)])
def test_features_of_few_steps(gdi, n, count, steps):
    """Step counts on both sides of the line between a launch per step and the one-launch walk, and of 32.
    Float32 sums of at most 30 terms a step, scaled to unit RMS: 1e-4."""
    from paper_1908_00210_gb300 import learn
    gs = [_ring_graph(n + 3 * (i % 5), 4 * n, i) for i in range(count)]
    gp, u = batch_union(gs)
    ids = np.arange(count, dtype=np.uint32)
    X = learn.MPNN(seed=1, feat_seed=5, steps=steps).features(learn.GraphBatch.from_graphs(gs, graph_ids=ids))
    assert np.max(np.abs(X.cpu().numpy() - ref.features(gp, ids, u.row_ptr, u.col, 5, steps))) < 1e-4
