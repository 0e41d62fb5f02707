"""The learned proposal's network kernels (BF16 tensor cores, FP32
accumulation) against the FP64 oracle network, and its use by the planner."""
import numpy as np
import pytest

from oracle import kpo
from oracle.kpo import Oracle
from paper_2409_06807_gb300 import workloads as W
from parity_util import compare_pass, state_scale

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2409_06807_gb300.build import build_planner
    build_planner()
    from paper_2409_06807_gb300 import mlp, planner
    return mlp, planner


def _bf16(a):
    """Round float32 values to bfloat16 (nearest even), as float64."""
    u = np.asarray(a, np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def _oracle_params(p):
    """The parameters the device computes with: BF16 weights, FP32 biases."""
    q = p.astype(np.float64).copy()
    W1, b1, W2, b2, W3, b3 = kpo.mlp_split(q)
    for Wm in (W1, W2, W3):
        Wm[...] = _bf16(Wm)
    return q


def _data(n, seed):
    rng = np.random.default_rng(seed)
    x = np.zeros((n, 32), np.float32)
    x[:, :20] = rng.normal(0, 1, (n, 20))
    t = rng.uniform(-0.95, 0.95, (n, 4)).astype(np.float32)
    return x, t


@pytest.mark.parametrize("n", [1, 31, 32, 33, 200])
def test_forward_matches_oracle(M, n):
    import torch
    mlp, _ = M
    p = mlp.init_params(3)
    _, _, _, _, _, b3 = mlp.split(p)
    b3[4:] = -1.0
    net = mlp.Mlp(p, max_batch=256)
    x, _ = _data(n, 4)
    out = net.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    ref = kpo.mlp_forward(_oracle_params(p), _bf16(x))
    np.testing.assert_allclose(out[:, :4], ref[:, :4], atol=2e-2)
    np.testing.assert_allclose(out[:, 4:], ref[:, 4:], atol=2e-2)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128, 152 * 128 + 1, 3 * 152 * 128 + 77])
def test_forward_tile_edges(M, n):
    """The tensor-core inference kernel at the edges of its 128-row tiles and
    of its one-tile-per-SM grid (one CTA walking several tiles), and through
    unaligned device pointers, against the same arithmetic in plain torch:
    BF16 operands, FP32 sums.  A sum in another order can round a hidden
    value to the neighbouring BF16 number (2^-8 of it): the output moves by
    one such step times an output weight (at most 0.1 sqrt(6 / 256)) times
    the hidden value (below 8 here), so 2e-3 bounds a few of them."""
    import torch
    mlp, planner = M
    net = mlp.Mlp(mlp.init_params(3), max_batch=n)
    x = torch.from_numpy(_data(n, n)[0]).cuda()
    out = net.forward(x)

    def rnd(v):
        return v.to(torch.bfloat16).double()

    W1, b1, W2, b2, W3, b3 = [torch.from_numpy(v.copy()).cuda() for v in
                              mlp.split(mlp.init_params(3))]
    h = rnd((rnd(x) @ rnd(W1).T + b1.double()).clamp(min=0))
    h = rnd((h @ rnd(W2).T + b2.double()).clamp(min=0))
    o = h @ rnd(W3).T + b3.double()
    ref = torch.cat([torch.tanh(o[:, :4]), o[:, 4:].clamp(-4, 1)], 1)
    assert float((out.double() - ref).abs().max()) <= 2e-3
    # 4-byte aligned input and output
    xb = torch.zeros(n * 32 + 1, device="cuda")
    ob = torch.zeros(n * 8 + 1, device="cuda")
    xb[1:] = x.reshape(-1)
    assert planner.lib().kp_mlp_forward(net._ctx, xb.data_ptr() + 4, n, ob.data_ptr() + 4) == 0
    torch.cuda.synchronize()
    assert torch.equal(ob[1:].view(n, 8), out)


@pytest.mark.parametrize("n", [1, 17, 127, 128, 129, 1000, 152 * 128 + 5])
def test_gradients_tile_edges(M, n):
    """The one-kernel forward and backward pass at the edges of its 128-row
    tiles, against the same arithmetic in plain torch: BF16 operands and
    activations, FP32 (here FP64) sums, the FP32 output gradient in the second
    layer's gradient.  FP32 sums give 1e-6; where a sum in another order rounds
    an activation to the neighbouring BF16 number (2^-8 of it, one of at least
    256 in its row), a block moves by at most 2^-8 / sqrt(256) of itself per
    row touched: 2.5e-4, and four of those bound the few that occur."""
    import torch
    mlp, _ = M
    p = mlp.init_params(5)
    net = mlp.Mlp(p, max_batch=n)
    x, t = [torch.from_numpy(v).cuda() for v in _data(n, n)]
    g, loss = net.gradients(x, t)

    def rnd(v):
        return v.to(torch.float32).to(torch.bfloat16).double()

    W1, b1, W2, b2, W3, b3 = [torch.from_numpy(v.copy()).cuda() for v in mlp.split(p)]
    W1, W2, W3, xb = rnd(W1), rnd(W2), rnd(W3), rnd(x)
    h1 = rnd((xb @ W1.T + b1.double()).clamp(min=0))
    h2 = rnd((h1 @ W2.T + b2.double()).clamp(min=0))
    o = h2 @ W3.T + b3.double()
    mu, raw = torch.tanh(o[:, :4]), o[:, 4:]
    ls = raw.clamp(-4, 1)
    z = (t.double() - mu) * torch.exp(-ls)
    inside = ((raw >= -4) & (raw <= 1)).double()
    d = torch.cat([-z * torch.exp(-ls) * (1 - mu * mu), (1 - z * z) * inside], 1) / n
    d2 = rnd((d @ W3) * (h2 > 0))
    d1 = rnd((d2 @ W2) * (h1 > 0))
    ref = (d1.T @ xb, d1.sum(0), d2.T @ h1, d2.sum(0), rnd(d).T @ h2, d.sum(0))
    assert abs(loss - float((ls + 0.5 * z * z).sum() / n)) <= 1e-5 * max(1.0, abs(loss))
    for got, want in zip(mlp.split(g), ref):
        want = want.cpu().numpy()
        assert np.linalg.norm(got - want) <= 1e-3 * np.linalg.norm(want)


def test_gradients_match_oracle(M):
    """Every parameter block's gradient against the FP64 oracle's
    backpropagation (relative L2 error, BF16 activations)."""
    import torch
    mlp, _ = M
    p = mlp.init_params(5)
    net = mlp.Mlp(p, max_batch=512)
    x, t = _data(500, 6)
    g, loss = net.gradients(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    ref_loss, ref = kpo.mlp_loss_grad(_oracle_params(p), _bf16(x), t.astype(np.float64))
    assert abs(loss - ref_loss) <= 2e-2 * abs(ref_loss) + 1e-3
    for blk_g, blk_r in zip(mlp.split(g), kpo.mlp_split(ref)):
        err = np.linalg.norm(blk_g - blk_r) / max(np.linalg.norm(blk_r), 1e-12)
        assert err < 3e-2, err


def test_training_lowers_the_loss(M):
    """Targets that depend on the features: Adam steps on the device lower
    the negative log-likelihood well below its starting value."""
    import torch
    mlp, _ = M
    rng = np.random.default_rng(9)
    x = np.zeros((8192, 32), np.float32)
    x[:, :20] = rng.normal(0, 1, (8192, 20))
    t = np.tanh(x[:, :4] * 0.7 + 0.05 * rng.normal(0, 1, (8192, 4))).astype(np.float32)
    net = mlp.Mlp(mlp.init_params(1), max_batch=1024)
    X, T = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    first = net.gradients(X[:1024], T[:1024])[1]
    hist = mlp.train(net, X, T, epochs=6, batch=1024, lr=2e-3)
    last = net.gradients(X[:1024], T[:1024])[1]
    assert last < first - 1.0, (first, hist, last)


@pytest.mark.parametrize("fso", [False, True])
def test_harvest_matches_oracle(M, fso):
    """Lock-step plain passes with the harvest on: the device collects the
    same pairs as the oracle (features within BF16 rounding, targets within
    float32 rounding), compared as sorted sets; with kd-tree regions the
    grid-neighbour features are zero on both sides."""
    import torch
    _, P = M
    w = W.c1(2).with_(fso=fso)
    g = P.Planner(w)
    o = Oracle(w)
    g.reset()
    o.reset()
    g.set_harvest(100000)
    o.set_harvest(100000)
    g.enable_log(w.t_e)
    for _ in range(3):
        _, ost, orec = o.iterate(records=True)
        gs = g.expand_step(1)[0]
        assert compare_pass(w, ost, orec, gs, g.read_log(ost["n_samples"])) == 0
    gf, gt = (a.cpu().numpy() for a in g.harvest())
    of, ot = o.harvest()
    assert len(gf) == len(of) > 0
    kg = np.lexsort(np.round(gt, 4).T[::-1])
    ko = np.lexsort(np.round(ot, 4).T[::-1])
    np.testing.assert_allclose(gt[kg], ot[ko], atol=1e-5)
    np.testing.assert_allclose(gf[kg], of[ko], atol=2e-2, rtol=1e-2)
    if fso:
        assert np.all(gf[:, 14:20] == 0.0) and np.any(gf[:, 13] > 0.0)


def test_learned_pass_matches_oracle(M):
    """One pass from the root with a network attached: samples whose
    selector picks the uniform draw match the oracle as in the plain
    planner; learned samples draw their controls within BF16 tolerance and
    their durations exactly (the uniform draw)."""
    import torch
    mlp, P = M
    w = W.c2(0, lambda_max=256)
    p = mlp.init_params(2)
    _, _, _, _, _, b3 = mlp.split(p)
    b3[4:] = -1.5
    net = mlp.Mlp(p, max_batch=64)
    g = P.Planner(w)
    g.attach_mlp(net, 0.5)
    o = Oracle(w)
    o.set_mlp(_oracle_params(p).astype(np.float32), 0.5)
    g.reset()
    o.reset()
    g.enable_log(4096)
    _, ost, orec = o.iterate(records=True)
    gs = g.expand_step(1)[0]
    grec = g.read_log(ost["n_samples"])
    assert gs["n_samples"] == ost["n_samples"] == 256
    key = [w.seed & 0xFFFFFFFF, w.seed >> 32]
    sel = np.array([kpo.philox4x32_10([0, 0, j, 1], key)[2] for j in range(256)])
    learned = sel < 2 ** 31
    assert 0.35 < learned.mean() < 0.65
    uni = ~learned
    assert np.array_equal(grec["k"][uni], orec["k"][uni])
    ok = (grec["flags"][uni] & 1) == (orec["flags"][uni] & 1)
    amb = orec["m_valid"][uni] < 1e-4
    assert np.all(ok | amb)
    # the duration is the uniform draw for learned samples too
    assert np.array_equal(grec["k"], orec["k"])


def test_learned_plan_revalidated(M):
    """A trained network on the Dubins forest: every returned trajectory
    is valid under the oracle's dense re-check."""
    import torch
    mlp, P = M
    feats, targs = mlp.harvest(W.c2, list(range(3)), 60000)
    net = mlp.Mlp(max_batch=4096)
    mlp.train(net, feats, targs, epochs=2, batch=4096, lr=2e-3)
    for seed in (50, 51):
        w = W.c2(seed)
        g = P.Planner(w)
        g.attach_mlp(net, 0.5)
        st, traj = g.plan(max_iters=200)
        if st != P.OK:
            continue
        o = Oracle(w)
        scale = state_scale(w)
        prev = w.x_init.astype(np.float64)
        for e in range(len(traj["steps"])):
            depth, x_end = o.dense_check(prev, traj["ctrls"][e].astype(np.float64),
                                         int(traj["steps"][e]), 100)
            assert depth <= 1e-4
            assert np.max(np.abs(x_end - traj["states"][e]) / scale) <= 1e-4
            prev = traj["states"][e].astype(np.float64)
        assert np.linalg.norm(prev[:3] - w.goal_c) <= float(w.goal_r) * (1 + 1e-6)


def test_device_epoch_matches_step_loop(M):
    """One epoch driven on the device (one launch for all its mini-batches)
    against the same mini-batches stepped from the host: equal mean loss and
    parameters up to the rounding of FP32 sums; later epochs keep lowering the
    loss."""
    import torch
    mlp, _ = M
    rng = np.random.default_rng(21)
    n = 512 * 6 + 100  # the ragged tail is skipped by both
    x = np.zeros((n, 32), np.float32)
    x[:, :20] = rng.normal(0, 1, (n, 20))
    t = np.tanh(x[:, :4] * 0.5 + 0.05 * rng.normal(0, 1, (n, 4))).astype(np.float32)
    X, T = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    perm = torch.from_numpy(rng.permutation(n).astype(np.int64)).cuda()
    p0 = mlp.init_params(8)
    a = mlp.Mlp(p0, max_batch=512)
    b = mlp.Mlp(p0, max_batch=512)
    loss_a = a.train_epoch(X, T, perm, 1e-3)
    losses = []
    for i in range(0, n - 512 + 1, 512):
        idx = perm[i:i + 512]
        losses.append(b.train_step(X.index_select(0, idx).contiguous(),
                                   T.index_select(0, idx).contiguous(), 1e-3, want_loss=True))
    assert abs(loss_a - np.mean(losses)) <= 1e-3 * abs(np.mean(losses)) + 1e-4
    pa, pb = a.params(), b.params()
    assert np.max(np.abs(pa - pb)) < 5e-3
    later = [a.train_epoch(X, T, perm, 1e-3) for _ in range(2)]
    assert later[-1] < loss_a


def test_gradients_match_oracle_large_ragged_batch(M):
    """A batch of 4133 rows (65 k tiles of the tensor-core weight-gradient
    GEMMs over several splits, a partial last row tile): every parameter
    block's gradient against the FP64 oracle."""
    import torch
    mlp, _ = M
    p = mlp.init_params(12)
    net = mlp.Mlp(p, max_batch=4200)
    x, t = _data(4133, 13)
    g, loss = net.gradients(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    ref_loss, ref = kpo.mlp_loss_grad(_oracle_params(p), _bf16(x), t.astype(np.float64))
    assert abs(loss - ref_loss) <= 2e-2 * abs(ref_loss) + 1e-3
    for blk_g, blk_r in zip(mlp.split(g), kpo.mlp_split(ref)):
        err = np.linalg.norm(blk_g - blk_r) / max(np.linalg.norm(blk_r), 1e-12)
        assert err < 3e-2, err


def _frontier_coverage(P, net, mix, seeds):
    """New sub-regions reached, samples and integrator steps of one pass
    over each oracle-grown frontier (3 passes of the Dubins forest), with
    the network attached at 'mix' (0: the uniform draw alone)."""
    from oracle.kpo import Oracle
    new = samples = steps = 0
    expand_ns = net_ns = 0
    for s in seeds:
        w = W.c2(s)
        src = Oracle(w)
        src.reset()
        for _ in range(3):
            src.iterate()
        t = src.export()
        t["state"] = t["state"].astype(np.float32)
        t["ctrl"] = t["ctrl"].astype(np.float32)
        g = P.Planner(w)
        g.attach_mlp(net if mix > 0 else None, mix)
        g.import_tree(t)
        before = int(g.export_tree()["visited"].sum())
        st = g.expand_step(1)[0]
        inf = g.info()
        new += int(g.export_tree()["visited"].sum()) - before
        samples += inf["n_samples"]
        steps += inf["n_steps"]
        expand_ns += st["phase_ns"][0] + st["phase_ns"][1]
        net_ns += st["phase_ns"][3] + st["phase_ns"][6]
        g.close()
    return new, samples, steps, expand_ns, net_ns


def test_learned_gain_and_its_break_even(M):
    """What the trained network gains over the method without it, on the
    same frontiers and the same random stream: a network trained on pairs
    harvested evenly from 200 plain forest runs (2,000 a layout) reaches
    more new sub-regions per sample than the uniform draw alone.  Whether
    that pays depends on the network phase each pass adds before the
    expand; the gain needed to break even is that phase's time over the
    expand's (measured here, on the same passes).  Both are printed for
    the record; the benchmark reports them on 1,000 held-out layouts."""
    mlp, P = M
    feats, targs = mlp.harvest(W.c2, list(range(200)), 400_000)
    assert 300_000 <= feats.shape[0] <= 400_000
    net = mlp.Mlp(max_batch=4096)
    hist = mlp.train(net, feats, targs, epochs=4, batch=4096, lr=1e-3)
    assert hist[-1] < hist[0]
    seeds = list(range(20_000, 20_008))
    n0, s0, k0, e0, _ = _frontier_coverage(P, net, 0.0, seeds)
    n1, s1, k1, e1, f1 = _frontier_coverage(P, net, 0.5, seeds)
    assert s0 == s1  # same frontiers, same keys
    gain = (n1 / s1) / (n0 / s0) - 1.0
    break_even = f1 / e1
    print(f"learned: {gain:+.3f} new sub-regions per sample, {(n1 / k1) / (n0 / k0) - 1:+.3f} per "
          f"integrator step; network phase / expand = {break_even:.3f}")
    assert gain > 0.01, gain


@pytest.mark.parametrize("extra,limit", [(400, 0), (900, 0), (3800, 0), (0, 60)])
def test_learned_plan_with_less_shared_memory(M, extra, limit):
    """The second layer's weights are staged in shared memory beside the
    obstacles where they fit: with boxes added inside an obstacle (which changes
    no verdict) there is no room for them, and a capped launch has blocks of one
    group of threads.  The result is the same bytes."""
    mlp, P = M
    net = mlp.Mlp(mlp.init_params(4), max_batch=64)
    w = W.c2(3, lambda_max=32)
    boxes = np.asarray(w.boxes, dtype=np.float32)
    lo, hi = boxes[0, :3], boxes[0, 3:]
    mid = np.concatenate([lo + 0.4 * (hi - lo), lo + 0.6 * (hi - lo)])
    out = []
    for n, lim in ((0, 0), (extra, limit)):
        g = P.Planner(w.with_(boxes=np.concatenate([boxes, np.tile(mid, (n, 1))]).astype(np.float32)))
        g.attach_mlp(net, 0.5)
        g.set_grid_limit(lim)
        st, traj = g.plan(max_iters=12)
        i = g.info()
        out.append((st, traj, [i[k] for k in ("n_nodes", "n_ve", "n_samples", "n_steps", "goal_node")]))
    (s0, t0, i0), (s1, t1, i1) = out
    assert s0 == s1 and i0 == i1 and i0[0] > 1000
    for k in t0 or {}:
        assert np.array_equal(t0[k], t1[k])


def test_contexts_of_different_shared_memory(M):
    """A context's launch does not depend on which context was configured last:
    one with the network's weights staged, one with many obstacles, one plain."""
    mlp, P = M
    net = mlp.Mlp(mlp.init_params(4), max_batch=64)
    w = W.c2(3, lambda_max=32)
    boxes = np.asarray(w.boxes, dtype=np.float32)
    many = np.concatenate([boxes, np.tile(boxes[:1], (2000, 1))]).astype(np.float32)
    a, b, c = P.Planner(w), P.Planner(w.with_(boxes=many)), P.Planner(w)
    a.attach_mlp(net, 0.5)
    b.attach_mlp(net, 0.5)
    first = [g.plan(max_iters=6) for g in (a, b, c)]
    for order in ((0, 1, 2), (2, 1, 0), (1, 2, 0)):
        gs = (a, b, c)
        for k in order:
            gs[k].set_obstacles(many if k == 1 else boxes)
        for k in (0, 1, 2):
            st, t = gs[k].plan(max_iters=6)
            assert st == first[k][0] and np.array_equal(t["steps"], first[k][1]["steps"])
    assert first[0][0] == first[1][0]


@pytest.mark.parametrize("n", [1, 129, 2 * 152 * 128 + 5])
def test_inference_that_gives_up_says_so(M, n):
    """Inference whose products never come (the test hook) ends after the wait
    limit: every row is NaN, not what the output held before, the next call
    that reports says KP_ERR_TIMEOUT, and setting the parameters clears it."""
    import time

    import torch
    mlp, planner = M
    p = mlp.init_params(3)
    net = mlp.Mlp(p, max_batch=n)
    x, t = [torch.from_numpy(v).cuda() for v in _data(n, n)]
    want = net.forward(x)
    out = torch.full((n, 8), 0.25, device="cuda")
    net.selftest_hold(50_000_000)  # 50 ms
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    assert planner.lib().kp_mlp_forward(net._ctx, x.data_ptr(), n, out.data_ptr()) == 0
    torch.cuda.synchronize()
    assert 0.04 < time.perf_counter() - t0 < 0.15
    net.selftest_hold(0)
    assert bool(torch.isnan(out).all())
    with pytest.raises(planner.KpError) as e:
        net.gradients(x, t)
    assert e.value.status == planner.ERR_TIMEOUT
    net.set_params(p)
    assert torch.equal(net.forward(x), want)
    net.gradients(x, t)


@pytest.mark.parametrize("n", [1, 129, 152 * 128 + 5])
@pytest.mark.parametrize("form", ["gradients", "epoch"])
def test_training_that_gives_up_ends_at_once(M, n, form):
    """A training launch whose wait expires (the test hook) ends with
    KP_ERR_TIMEOUT after one wait limit: blocks wait for what they have in
    flight and for nothing else, those without a tile and those of one that had
    finished its tiles included.  Setting the parameters clears the error."""
    import time

    import torch
    mlp, planner = M
    p = mlp.init_params(3)
    net = mlp.Mlp(p, max_batch=n)
    x, t = [torch.from_numpy(v).cuda() for v in _data(2 * n, n)]
    perm = torch.arange(2 * n, dtype=torch.int32, device="cuda")
    call = (lambda: net.gradients(x[:n], t[:n])) if form == "gradients" else \
        (lambda: net.train_epoch(x, t, perm))
    want = call()
    net.set_params(p)
    net.selftest_hold(100_000_000)  # 100 ms
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with pytest.raises(planner.KpError) as e:
        call()
    took = time.perf_counter() - t0
    assert e.value.status == planner.ERR_TIMEOUT and 0.09 < took < 0.2
    net.selftest_hold(0)
    net.set_params(p)
    got = call()
    if form == "gradients":
        assert np.array_equal(got[0], want[0]) and got[1] == want[1]
    else:
        assert got == want


@pytest.mark.parametrize("n", [40, 300])
def test_gradients_of_an_infinite_output_gradient(M, n):
    """A target so far off that the squared deviation overflows FP32: the
    gradient of that output is -inf, and what follows from it is infinite or NaN
    where FP32 arithmetic makes it so (every infinity in the second layer's
    gradient with its weight's sign), not NaN throughout."""
    import torch
    mlp, _ = M
    p = mlp.init_params(5)
    net = mlp.Mlp(p, max_batch=n)
    x, t = [torch.from_numpy(v).cuda() for v in _data(n, n)]
    t[7, 2] = 1e25
    g, loss = net.gradients(x, t)
    assert loss == np.inf

    def rnd(v):
        return v.to(torch.float32).to(torch.bfloat16).double()

    W1, b1, W2, b2, W3, b3 = [torch.from_numpy(v.copy()).cuda() for v in mlp.split(p)]
    W1, W2, W3, xb = rnd(W1), rnd(W2), rnd(W3), rnd(x)
    h1 = rnd((xb @ W1.T + b1.double()).clamp(min=0))
    h2 = rnd((h1 @ W2.T + b2.double()).clamp(min=0))
    o = (h2 @ W3.T + b3.double()).float()
    mu, ls = torch.tanh(o[:, :4]), o[:, 4:]
    assert float(ls.abs().max()) < 1
    z = (t - mu) * torch.exp(-ls)
    d = (torch.cat([-z * torch.exp(-ls) * (1 - mu * mu), 1 - z * z], 1) / n).double()
    assert int(torch.isinf(d).sum()) == 1
    # (no matrix product here: it may split the sums)
    d2 = torch.where(h2 > 0, (d[:, :, None] * W3[None]).sum(1), 0.0).float().to(torch.bfloat16).double()
    ref = dict(W2=(d2[:, :, None] * h1[:, None, :]).sum(0), b2=d2.sum(0),
               W3=(d[:, :, None] * h2[:, None, :]).sum(0), b3=d.sum(0))
    got = dict(zip(("W1", "b1", "W2", "b2", "W3", "b3"), mlp.split(g)))
    for k, want in ref.items():
        want = want.cpu().numpy()
        assert np.isinf(want).any(), k
        assert np.array_equal(np.isnan(got[k]), np.isnan(want)), k
        assert np.array_equal(np.isposinf(got[k]), np.isposinf(want)), k
        assert np.array_equal(np.isneginf(got[k]), np.isneginf(want)), k
