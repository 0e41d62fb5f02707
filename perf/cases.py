"""The measured cases: what a user of the planner has it do.

Every case goes through the public entry points: ``Planner`` (one query or a
fixed number of loop passes), ``kp_plan_static`` (the no-allocation form),
``Server`` (a batch of queries) and ``Mlp`` (the learned proposal's inference,
gradients and training).  Sizes are those of the repository's workloads, tests
and benchmark, and odd ones around them.

A planning query's result is a function of its inputs bit by bit, whatever the
launch shape, so these cases compare exactly.  The network's cases compare
within what BF16 operands with FP32 sums give.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2409_06807_gb300 import mlp as M
from paper_2409_06807_gb300 import planner as P
from paper_2409_06807_gb300 import serve as S
from paper_2409_06807_gb300 import workloads as W

SYSTEM = {"di": W.DI, "dubins": W.DUBINS, "quad": W.QUAD}


def _problem(kind, system, boxes, grid, sub, lambda_max, t_e, passes, **more):
    d = dict(kind=kind, system=system, boxes=boxes, gx=grid[0], gy=grid[1], gz=grid[2],
             sx=sub[0], sy=sub[1], sz=sub[2], lambda_max=lambda_max, t_e=t_e, passes=passes,
             speed_bins=1, heading=0, pitch=0, kdtree=False, replan=False, mix=0.0)
    d.update(more)
    return d


def listed():
    return [
        # inference on a few nodes: the smallest call, one launch
        dict(name="mlp_forward_small", kind="forward", rows=33),
        # inference on every node of a large frontier
        dict(name="mlp_forward_large", kind="forward", rows=262145),
        # the proposal's training: mini-batches of 4,096 rows, forward,
        # backward and optimiser step, as the training loop runs them
        dict(name="mlp_train_epoch", kind="train", batch=4096, steps=16),
        # a small query re-planned as the obstacles change: latency counts
        _problem("plan", "di", 16, (8, 8, 8), (4, 4, 4), 32, 65536, 400, replan=True,
                 name="di_replan"),
        # the same size through the entry that allocates nothing
        _problem("static", "di", 16, (8, 8, 8), (4, 4, 4), 32, 65536, 400, name="di_static"),
        # the benchmark's query: Dubins airplane in a forest
        _problem("plan", "dubins", 200, (16, 16, 16), (4, 4, 4), 64, 1 << 20, 400,
                 name="dubins_forest"),
        # regions over position, heading and pitch, with sizes that are no
        # power of two anywhere
        _problem("grow", "dubins", 137, (11, 13, 7), (3, 5, 2), 37, 300007, 20, heading=5, pitch=3,
                 name="dubins_ragged_state_grid"),
        # regions from the kd-tree over the obstacle faces
        _problem("plan", "dubins", 150, (1, 1, 1), (4, 4, 4), 64, 1 << 20, 100, kdtree=True,
                 name="dubins_kdtree"),
        # half of the controls from the network
        _problem("plan", "dubins", 200, (16, 16, 16), (4, 4, 4), 64, 1 << 20, 100, mix=0.5,
                 name="dubins_learned"),
        # a fixed number of passes with a large frontier: throughput counts
        _problem("grow", "dubins", 200, (16, 16, 16), (4, 4, 4), 64, 1 << 22, 30,
                 name="dubins_large_frontier"),
        # the largest query: quadrotor in a building
        _problem("plan", "quad", 1200, (16, 16, 16), (4, 4, 4), 128, 1 << 22, 400, speed_bins=4,
                 name="quad_building"),
        # a batch of mixed queries through the server
        dict(name="serving_batch", kind="serve", queries=48, team_blocks=32, box_lo=10,
             box_hi=1000, t_e_lo=16384, t_e_hi=1 << 20),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["forward", "gradients", "train", "di", "static", "dubins", "dubins",
                       "ragged", "kdtree", "learned", "quad", "serve"])
    if kind == "forward":
        return dict(kind=kind, rows=log(1, 262145))
    if kind == "gradients":
        return dict(kind=kind, rows=log(17, 32768))
    if kind == "train":
        return dict(kind=kind, batch=log(1000, 8192), steps=rng.randint(2, 16))
    if kind == "serve":
        return dict(kind=kind, queries=rng.randint(8, 48), team_blocks=rng.choice([8, 16, 24, 32]),
                    box_lo=10, box_hi=log(40, 1000), t_e_lo=16384, t_e_hi=log(40000, 1 << 20))
    if kind in ("di", "static"):
        g = rng.randint(5, 9)
        return _problem("plan" if kind == "di" else "static", "di", rng.randint(3, 48),
                        (g, g, rng.randint(5, 9)), (4, 4, rng.randint(3, 4)), rng.randint(16, 32),
                        log(20000, 65536), 400, replan=kind == "di" and rng.random() < 0.5)
    boxes = rng.randint(60, 220)
    if kind == "dubins":
        return _problem(rng.choice(["plan", "grow"]), "dubins", boxes,
                        (rng.randint(10, 18), rng.randint(10, 18), rng.randint(8, 16)), (4, 4, 4),
                        rng.randint(30, 64), log(100000, 1 << 22), rng.randint(12, 30),
                        replan=rng.random() < 0.3)
    if kind == "ragged":
        return _problem("grow", rng.choice(["di", "dubins"]), boxes,
                        (rng.randint(5, 13), rng.randint(5, 13), rng.randint(3, 9)),
                        (rng.randint(2, 5), rng.randint(2, 5), rng.randint(2, 3)),
                        rng.randint(11, 61), log(50000, 1000000), rng.randint(8, 24),
                        heading=rng.randint(2, 6), pitch=rng.randint(2, 4))
    if kind == "kdtree":
        return _problem("plan", "dubins", rng.randint(30, 180), (1, 1, 1),
                        (rng.randint(2, 5), rng.randint(2, 5), rng.randint(2, 4)),
                        rng.randint(30, 64), log(100000, 1 << 20), rng.randint(20, 60), kdtree=True)
    if kind == "learned":
        return _problem("plan", "dubins", boxes, (16, 16, 16), (4, 4, 4), rng.randint(30, 64),
                        log(100000, 1 << 20), rng.randint(12, 60),
                        mix=round(rng.uniform(0.2, 0.8), 2))
    tiles = rng.randint(6, 20)
    return _problem("plan", "quad", 3 * tiles * tiles, (16, 16, rng.randint(10, 16)), (4, 4, 4),
                    rng.randint(48, 128), log(200000, 1 << 22), rng.randint(10, 60),
                    speed_bins=rng.randint(1, 4))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _boxes(case, w, seed):
    if case["system"] == "di":
        return W.random_boxes(seed, case["boxes"], keep_clear=[
            (tuple(w.x_init[:3]), 0.02), ((0.9, 0.9, 0.9), 0.05)])
    if case["system"] == "dubins":
        return W.forest_boxes(seed, case["boxes"], keep_clear=[
            (tuple(w.x_init[:3]), 0.03), ((0.95, 0.95, 0.5), 0.05)])
    return W.building_boxes(seed, tiles=max(3, int(round(math.sqrt(case["boxes"] / 3)))))


def _workload(case, seed):
    w = {"di": W.c1, "dubins": W.c2, "quad": W.c3}[case["system"]](seed)
    w = w.with_(boxes=_boxes(case, w, seed), grid=(case["gx"], case["gy"], case["gz"]),
                sub=(case["sx"], case["sy"], case["sz"]), t_e=case["t_e"],
                lambda_max=case["lambda_max"], speed_bins=case["speed_bins"], fso=case["kdtree"])
    if case["heading"]:
        w = w.with_(state_grid=(0, 0, 0, case["heading"], case["pitch"]) + (0,) * 7)
    if case["kind"] == "grow":  # no goal: the passes run to their number
        w = w.with_(goal_c=np.full(3, 9.0, np.float32), goal_r=np.float32(0.0))
    return w


def _features(rows, seed):
    """Node features of the ranges the planner gives: states and goal offset
    in [-1, 1], coverage and free-volume shares, log counts, acceptance
    probabilities (most of them near the floor), zeros from 20 on."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.zeros((rows, 32), dtype=torch.float32, device="cuda")
    x[:, :9] = 2 * torch.rand((rows, 9), generator=g, device="cuda") - 1
    x[:, 9:11] = torch.rand((rows, 2), generator=g, device="cuda")
    x[:, 11:13] = 8 * torch.rand((rows, 2), generator=g, device="cuda")
    x[:, 13:20] = torch.rand((rows, 7), generator=g, device="cuda") ** 4
    t = 2 * torch.rand((rows, 4), generator=g, device="cuda") - 1
    return x, t


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradients"):
        x, t = _features(case["rows"], seed)
        return dict(case=case, net=M.Mlp(M.init_params(seed), max_batch=case["rows"]), x=x, t=t)
    if kind == "train":
        rows = case["batch"] * case["steps"]
        x, t = _features(rows, seed)
        g = torch.Generator(device="cpu").manual_seed(seed)
        perm = torch.randperm(rows, generator=g, dtype=torch.int32).cuda()
        return dict(case=case, net=M.Mlp(M.init_params(seed), max_batch=case["batch"]), x=x, t=t,
                    perm=perm)
    if kind == "serve":
        mix = W.serving_mix(case["queries"], seed=seed, t_e_range=(case["t_e_lo"], case["t_e_hi"]),
                            box_range=(case["box_lo"], case["box_hi"]))
        return dict(case=case, queries=[w for _, w in mix])
    w = _workload(case, seed)
    if kind == "static":
        return dict(case=case, w=w, structs=P.structs(w), goal=P.goal_struct(w),
                    boxes=np.ascontiguousarray(w.boxes), x=np.ascontiguousarray(w.x_init))
    pl = P.Planner(w)
    state = dict(case=case, w=w, pl=pl)
    if case["mix"] > 0.0:
        state["net"] = M.Mlp(M.init_params(seed), max_batch=64)
        pl.attach_mlp(state["net"], case["mix"])
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _rows(t, room=512):
    """A trajectory as one array of 'room' rows (state, control, steps; zeros
    after its end), so that every layout's result has the same shape."""
    n = len(t["steps"])
    a = np.zeros((room, 17), np.float32)
    a[:n, : t["states"].shape[1]] = t["states"]
    a[:n, 12: 12 + t["ctrls"].shape[1]] = t["ctrls"]
    a[:n, 16] = t["steps"]
    return a


def _static(s):
    f32p = C.POINTER(C.c_float)
    states, ctrls = np.zeros((4096, 12), np.float32), np.zeros((4096, 4), np.float32)
    steps = np.zeros(4096, np.int32)
    traj = P.Traj(4096, 0, states.ctypes.data_as(f32p), ctrls.ctypes.data_as(f32p),
                  steps.ctypes.data_as(C.POINTER(C.c_int32)))
    sysm, ws, prm = s["structs"]
    obs = P.Obstacles(s["boxes"].ctypes.data_as(f32p), len(s["boxes"]))
    budget = P.Budget(s["case"]["passes"], 0.0)
    st = P.lib().kp_plan_static(C.byref(sysm), C.byref(ws), C.byref(obs), C.byref(prm),
                                s["x"].ctypes.data_as(f32p), C.byref(s["goal"]), C.byref(budget),
                                C.byref(traj),
                                C.c_void_p(torch.cuda.current_stream().cuda_stream))
    if st not in (P.OK, P.NO_SOLUTION):
        raise P.KpError(st, "kp_plan_static")
    n = traj.n_edges
    return dict(status=st, rows=_rows(dict(states=states[:n], ctrls=ctrls[:n], steps=steps[:n])))


def _serve(s):
    case = s["case"]
    srv = S.Server(pool_bytes=6 << 30, team_blocks=case["team_blocks"], max_slots=64)
    ids = [srv.submit(w) for w in s["queries"]]
    done = {d["id"]: d for d in srv.drain()}
    rows = []
    for q in ids:
        st, t = srv.result(q)
        rows.append(_rows(t))
    srv.close()
    count = np.array([[done[q][k] for k in ("status", "n_edges", "iterations", "n_nodes", "samples")]
                      for q in ids], np.int64)
    return dict(counts=count, rows=np.concatenate(rows))


def _layers(p):
    return dict(zip(("W1", "b1", "W2", "b2", "W3", "b3"), M.split(p)))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "forward":
        return s["net"].forward(s["x"])
    if kind == "gradients":
        g, loss = s["net"].gradients(s["x"], s["t"])
        return dict(loss=loss, **_layers(g))
    if kind == "train":
        loss = s["net"].train_epoch(s["x"], s["t"], s["perm"], 1e-3)
        return dict(loss=loss, params=s["net"].params())
    if kind == "static":
        return _static(s)
    if kind == "serve":
        return _serve(s)
    pl = s["pl"]
    if case["replan"]:
        pl.set_obstacles(s["w"].boxes)
    else:
        # with several contexts in a program: the loop kernel's shared memory
        # limit is the one of the context configured last
        pl.set_grid_limit(0)
    if kind == "grow":
        pl.reset()
        stats = pl.expand_step(case["passes"])
        return np.array([[d[f] for f in P.STAT_FIELDS] for d in stats], np.int64)
    st, t = pl.plan(max_iters=case["passes"])
    i = pl.info()
    return dict(status=st, rows=_rows(t), counts=np.array(
        [i[k] for k in ("n_nodes", "n_ve", "iteration", "goal_node", "state", "n_samples",
                        "n_steps", "n_hull_checks")], np.int64))


# ---------------------------------------------------------------------------
# work, tolerance, exact
# ---------------------------------------------------------------------------

# lane operations: a sample's draw, binning and claim; an integrator step with
# its state-box test; a step's hull (the tests against boxes depend on the
# broad phase and are left out)
_OPS = {"di": (157, 18, 6), "dubins": (157, 127, 6), "quad": (173, 337, 6)}
# integrator steps of a served query's sample, by system
_STEPS = {W.DI: 4, W.DUBINS: 6, W.QUAD: 11}
_NAME = {v: k for k, v in SYSTEM.items()}
_NET_MACS = 32 * 256 + 256 * 256 + 256 * 8


def _node_bytes(system):
    d, n = (12, 4) if system == "quad" else (6, 3)
    return 4 * d + 4 * n + 4 + 1 + 4 + 4 + 1


def work(case):
    kind = case["kind"]
    n_params = M.num_params()
    if kind == "forward":
        return dict(bytes=case["rows"] * (32 + 8) * 4 + 4 * n_params, flops=2 * _NET_MACS * case["rows"])
    if kind in ("gradients", "train"):
        rows = case["rows"] if kind == "gradients" else case["batch"] * case["steps"]
        # forward, weight gradients, and the hidden layers' input gradients
        macs = 2 * _NET_MACS + 256 * 256 + 256 * 8
        return dict(bytes=rows * 36 * 4 + 8 * n_params * (1 if kind == "gradients" else 4),
                    flops=2 * macs * rows)
    if kind == "serve":
        # counted on one batch: samples drawn and nodes written
        s = prepare(case, 0)
        counts = run(s)["counts"]
        b = f = 0
        for w, row in zip(s["queries"], counts):
            a, step, hull = _OPS[_NAME[w.system]]
            f += int(row[4]) * (a + _STEPS[w.system] * (step + hull))
            b += int(row[3]) * _node_bytes(_NAME[w.system]) + len(w.boxes) * 24
        return dict(bytes=b, flops=f)
    # a query's samples, steps and nodes depend on the layout: counted on one
    s = prepare(dict(case, kind="plan" if kind == "static" else kind), 0)
    run(s)
    i = s["pl"].info()
    a, step, hull = _OPS[case["system"]]
    return dict(bytes=i["n_nodes"] * _node_bytes(case["system"]) + case["boxes"] * 24,
                flops=i["n_samples"] * a + i["n_steps"] * step + i["n_hull_checks"] * hull)


def tolerance(case):
    # four times what the present code differs by from the same arithmetic in
    # plain torch with the sums in another order (a sum in another order can
    # round a hidden value to the neighbouring BF16 number)
    if case["kind"] == "forward":
        return dict(rel=3.5e-4, max=4.5e-2)  # seen: 8.7e-5, 1.1e-2
    if case["kind"] == "gradients":
        return dict(rel=3e-4, max=1.4e-2)  # seen: 6.5e-5, 3.4e-3
    if case["kind"] == "train":
        # after a second epoch of 16 steps on the same state: Adam's first
        # steps turn a gradient's sign into a whole step (seen: 1e-3, 5e-2)
        return dict(rel=4e-3, max=0.2)
    return "exact"


def _net64(p, x):
    z1 = x @ p["W1"].T + p["b1"]
    h1 = z1.clamp(min=0)
    z2 = h1 @ p["W2"].T + p["b2"]
    h2 = z2.clamp(min=0)
    return h1, h2, h2 @ p["W3"].T + p["b3"]


def _grad64(p, x, t):
    """Loss and gradient of the batch-mean Gaussian negative log-likelihood."""
    m = x.shape[0]
    h1, h2, o = _net64(p, x)
    mu, raw = torch.tanh(o[:, :4]), o[:, 4:]
    ls = raw.clamp(-4.0, 1.0)
    z = (t - mu) * torch.exp(-ls)
    loss = (ls + 0.5 * z * z).sum() / m
    inside = ((raw >= -4.0) & (raw <= 1.0)).double()
    do = torch.cat([-z * torch.exp(-ls) * (1 - mu * mu), (1 - z * z) * inside], 1) / m
    d2 = (do @ p["W3"]) * (h2 > 0)
    d1 = (d2 @ p["W2"]) * (h1 > 0)
    g = dict(W1=d1.T @ x, b1=d1.sum(0), W2=d2.T @ h1, b2=d2.sum(0), W3=do.T @ h2, b3=do.sum(0))
    return loss, g


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("forward", "gradients", "train"):
        return None  # a tree's growth has no value apart from its own rounding
    rows = case["rows"] if kind != "train" else case["batch"] * case["steps"]
    x, t = _features(rows, seed)
    p = {k: torch.from_numpy(v.copy()).cuda().double()
         for k, v in _layers(M.init_params(seed)).items()}
    if kind == "forward":
        out = []
        for i in range(0, rows, 65536):
            o = _net64(p, x[i:i + 65536].double())[2]
            out.append(torch.cat([torch.tanh(o[:, :4]), o[:, 4:].clamp(-4.0, 1.0)], 1))
        return torch.cat(out)
    if kind == "gradients":
        loss, g = _grad64(p, x.double(), t.double())
        return dict(loss=float(loss), **g)
    g = torch.Generator(device="cpu").manual_seed(seed)
    perm = torch.randperm(rows, generator=g, dtype=torch.int32).cuda().long()
    m = {k: torch.zeros_like(v) for k, v in p.items()}
    v2 = {k: torch.zeros_like(v) for k, v in p.items()}
    total = 0.0
    for b in range(case["steps"]):
        idx = perm[b * case["batch"]:(b + 1) * case["batch"]]
        loss, gr = _grad64(p, x[idx].double(), t[idx].double())
        total += float(loss)
        for k in p:
            m[k] = 0.9 * m[k] + 0.1 * gr[k]
            v2[k] = 0.999 * v2[k] + 0.001 * gr[k] ** 2
            p[k] = p[k] - 1e-3 * (m[k] / (1 - 0.9 ** (b + 1))) / (
                torch.sqrt(v2[k] / (1 - 0.999 ** (b + 1))) + 1e-8)
    return dict(loss=total / case["steps"],
                params=torch.cat([p[k].reshape(-1) for k in ("W1", "b1", "W2", "b2", "W3", "b3")]))
