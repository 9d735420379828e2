"""Performance cases of the planner: what a program that uses it has it do.

Every case is one call chain through the public entry points of
``paper_2411_13507_gb300.plan`` and ``.refine`` on inputs drawn from a seed
with the distributions of the planner's own workloads (``synth.py``), drawn
here vectorised.  ``exact`` restates the results in 64 bits in plain torch and
numpy.  Kinds:

* ``query``   buildGraph and findPath of one environment
  (``build_edges_async``, ``search_async``), the graph and its path returned;
* ``search``  findPath of a few trips on a graph that is there;
* ``batch``   many queries of uneven size, prepared once, built and searched;
* ``cut``     the keep-out cut of a built graph against obstacles;
* ``replan``  a run of replanning ticks, host to host (``Replanner.tick``);
* ``planes``  closest points and separating planes of points and obstacles;
* ``mpc``     the MPC refinement's QP for a batch of problems;
* ``refine``  loss and gradients of Bezier segments (``refine_loss``).
"""
from __future__ import annotations

import heapq
from math import comb, factorial, log
from types import SimpleNamespace

import numpy as np
import torch

from paper_2411_13507_gb300 import plan as P
from paper_2411_13507_gb300 import refine as R

BOUNDS = {2: (2.0, 4.0), 3: (3.0, 6.0, 30.0)}  # per-axis bounds of the 2-D double and the 3-D triple integrator
MPC_DT, MPC_WIDTH = 0.1, 5.0
MPC_W = dict(Q=[1.0, 1.0, 0.1, 0.1], F=[0.5, 0.5, 0.05, 0.05], R=[0.05, 0.05], V=[2.0, 2.0, 2.0, 2.0])
TRIPS = 4  # searches of a pass on one graph
REFINE_RMAX, REFINE_DELTA = 12, 0.1


def listed():
    return [
        # the smallest whole query: the 2-D workload in FP64, launches and latency count
        dict(name="query_2d_f64", kind="query", m=2, p=5, arith="f64", N=512, K=16, nT=8, tighten=0.0, cost="state"),
        # the same size in the precision form (halves on the tensor cores)
        dict(name="query_2d_tf32", kind="query", m=2, p=5, arith="tf32", N=512, K=16, nT=8, tighten=0.0, cost="state"),
        # the planner's main workload: one large 3-D environment in FP32
        dict(name="query_3d_f32", kind="query", m=3, p=7, arith="f32", N=8192, K=64, nT=16, tighten=0.0, cost="state"),
        # an ordinary 3-D environment of odd size, degree 5, tracking margin, position-only cost
        dict(name="query_3d_ragged", kind="query", m=3, p=5, arith="f32", N=1531, K=23, nT=11, tighten=0.05, cost="pos"),
        # new starts and goals on the large graph: the search's latency
        dict(name="search_3d", kind="search", m=3, p=7, arith="f32", N=8192, K=64, nT=16, tighten=0.0, cost="state"),
        # many environments of uneven size at once (the largest case)
        dict(name="batch_3d", kind="batch", Q=256, n_lo=512, n_hi=16384, k_lo=8, k_hi=128, t_lo=8, t_hi=16),
        # obstacles moved: the keep-out cut of a graph of the paper's scale
        dict(name="cut_2d", kind="cut", N=5000, obst=500, nT=1, width=5.0),
        # the replanning loop as a robot's program runs it, from host to host
        dict(name="replan_2d", kind="replan", N=5000, obst=500, ticks=6, width=5.0),
        # closest points and separating planes, all pairs
        dict(name="planes_2d", kind="planes", m=2, arith="f32", N=5000, obst=500, width=5.0),
        # a batch of MPC problems (horizon 10) with the planes of the nearest obstacles
        dict(name="mpc_2d", kind="mpc", B=1024, H=10, obst=500),
        # trajectory refinement, forward and backward: a large batch ...
        dict(name="refine_3d", kind="refine", m=3, p=7, S=65536),
        # ... and a small odd one in 2-D
        dict(name="refine_2d_small", kind="refine", m=2, p=5, S=777),
    ]


def _log_int(rng, lo, hi):
    return int(round(np.exp(rng.uniform(log(lo), log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "search", "batch", "cut", "replan", "planes", "mpc", "refine"])
    if kind in ("query", "search"):
        m = rng.choice([2, 3])
        arith = rng.choice(["f64", "f32"] if kind == "search" or m == 3 else ["f64", "f32", "tf32", "bf16"])
        return dict(kind=kind, m=m, p=rng.choice([3, 5] if m == 2 else [5, 7]), arith=arith,
                    N=_log_int(rng, 64, 3000) if m == 2 else _log_int(rng, 300, 10000),
                    K=_log_int(rng, 4, 40) if m == 2 else _log_int(rng, 12, 128), nT=rng.randint(3, 16),
                    tighten=rng.choice([0.0, 0.0, 0.05]), cost=rng.choice(["state", "state", "pos"]))
    if kind == "batch":
        return dict(kind=kind, Q=_log_int(rng, 3, 96), n_lo=rng.choice([100, 512]), n_hi=_log_int(rng, 1000, 16384),
                    k_lo=8, k_hi=rng.randint(16, 128), t_lo=rng.randint(3, 8), t_hi=rng.randint(9, 16))
    if kind == "cut":
        return dict(kind=kind, N=_log_int(rng, 200, 5000), obst=_log_int(rng, 10, 700), nT=rng.randint(1, 3), width=5.0)
    if kind == "replan":
        return dict(kind=kind, N=_log_int(rng, 500, 5000), obst=_log_int(rng, 20, 500), ticks=rng.randint(3, 6), width=5.0)
    if kind == "planes":
        return dict(kind=kind, m=rng.choice([2, 3]), arith=rng.choice(["f32", "f64"]), N=_log_int(rng, 50, 8000),
                    obst=_log_int(rng, 5, 500), width=5.0)
    if kind == "mpc":
        return dict(kind=kind, B=_log_int(rng, 16, 2048), H=rng.randint(5, 16), obst=_log_int(rng, 50, 500))
    m = rng.choice([2, 3])
    return dict(kind=kind, m=m, p=5 if m == 2 else 7, S=_log_int(rng, 30, 100000))


# ---------------------------------------------------------------- inputs ----


def _f32(x):
    return np.asarray(x, dtype=np.float32).astype(np.float64)


def _polytopes(rng, m, K, domain, side, max_cuts, f32):
    """Axis boxes cut by up to max_cuts random planes that keep the box centre inside: CSR rows, and the boxes."""
    c = rng.uniform(domain[0], domain[1], (K, m))
    h = 0.5 * rng.uniform(side[0], side[1], (K, m))
    cuts = rng.integers(0, max_cuts + 1, K)
    nrm = rng.normal(size=(K, max_cuts, m))
    nrm /= np.linalg.norm(nrm, axis=2, keepdims=True)
    off_b = np.einsum("kca,ka->kc", nrm, c) + rng.uniform(0.2, 0.9, (K, max_cuts)) * np.einsum("kca,ka->kc", np.abs(nrm), h)
    eye = np.eye(m)
    box_A = np.stack([eye, -eye], 1).reshape(2 * m, m)
    box_b = np.stack([c + h, -(c - h)], 2).reshape(K, 2 * m)
    A = np.concatenate([np.broadcast_to(box_A, (K, 2 * m, m)), nrm], 1)
    b = np.concatenate([box_b, off_b], 1)
    keep = np.arange(2 * m + max_cuts)[None] < (2 * m + cuts)[:, None]
    if f32:
        A, b = _f32(A), _f32(b)
    off = np.concatenate([[0], np.cumsum(2 * m + cuts)]).astype(np.int32)
    padded = np.where(keep[..., None], A, 0.0), np.where(keep, b, 1.0)
    return off, A[keep], b[keep], padded, (c - h, c + h)


def _positions(rng, which, padded, boxes, f32):
    """Uniform points in the chosen polytopes, by rejection from their boxes."""
    lo, hi = boxes[0][which], boxes[1][which]
    A, b = padded[0][which], padded[1][which]
    x = np.zeros_like(lo)
    left = np.arange(len(which))
    while left.size:
        y = lo[left] + (hi[left] - lo[left]) * rng.random((left.size, lo.shape[1]))
        y = _f32(y) if f32 else y
        ok = np.all(np.einsum("nra,na->nr", A[left], y) <= b[left] - 1e-9, axis=1)
        x[left[ok]] = y[ok]
        left = left[~ok]
    return x


def _linked(rng, x, padded):
    """Two polytopes that a chain of overlaps (shared states) links, if the environment has any: where a trip starts and ends."""
    A, b = padded
    inside = np.all((x @ A.reshape(-1, A.shape[2]).T).reshape(len(x), *b.shape) <= b, axis=2).astype(np.float32)
    reach = np.minimum(inside.T @ inside, 1.0)
    for _ in range(int(np.ceil(np.log2(len(reach))))):
        reach = np.minimum(reach @ reach, 1.0)
    part = np.flatnonzero(reach[np.argmax(reach.sum(1))])
    return rng.choice(part if len(part) > 1 else len(reach), 2, replace=False)


def _model(m, p, tighten=0.0, cost="state"):
    return SimpleNamespace(m=m, gamma=m, degree=p, bounds=BOUNDS[m], tighten=tighten, cost_mode=cost, interior="elevate")


def _environment(rng, m, p, N, K, nT, f32, tighten=0.0, cost="state", trips=1):
    """One planning query in free polytopes: the 2-D or the 3-D workload at the given sizes."""
    domain, side, cuts = ((0.0, 10.0), (2.0, 5.0), 4) if m == 2 else ((0.0, 20.0), (2.0, 6.0), 6)
    off, A, b, padded, boxes = _polytopes(rng, m, K, domain, side, cuts, f32)
    x = np.zeros((N, m * m))
    x[:, :m] = _positions(rng, rng.integers(0, K, N), padded, boxes, f32)
    x[:, m:] = rng.uniform(-1.0, 1.0, (N, m * m - m))
    T = np.linspace(0.2, 2.0, nT) if m == 2 else np.sort(np.exp(rng.uniform(log(0.1), log(3.0), nT)))
    trips = [_positions(rng, _linked(rng, x[:1024, :m], padded), padded, boxes, f32) for _ in range(trips)]
    if f32:
        x, T = _f32(x), _f32(T)
    return SimpleNamespace(model=_model(m, p, tighten, cost), dtype="f32" if f32 else "f64", states=x, T=T, poly_off=off,
                           A=A, b=b, start_pos=trips[0][0], goal_pos=trips[0][1], trips=trips)


def _obstacles(rng, m, n, width):
    off, A, b, _, _ = _polytopes(rng, m, n, (0.0, width), (0.005 * width, 0.02 * width), 3, False)
    return SimpleNamespace(off=off, A=A, b=b)


def _keepout(rng, N, n_obst, nT, width):
    """The keep-out scene: one free box, curves of about half a second, small obstacles."""
    x = np.concatenate([rng.uniform(0.0, width, (N, 2)), rng.uniform(-1.0, 1.0, (N, 2))], 1)
    A = np.array([[1.0, 0.0], [-1.0, 0.0], [0.0, 1.0], [0.0, -1.0]])
    b = np.array([width, 0.0, width, 0.0])
    T = np.array([0.5, 0.4, 0.6])[:nT]
    ends = rng.uniform(0.1 * width, 0.9 * width, (2, 2))
    prob = SimpleNamespace(model=_model(2, 5), dtype="f64", states=x, T=np.sort(T), poly_off=np.array([0, 4], dtype=np.int32),
                           A=A, b=b, start_pos=ends[0], goal_pos=ends[1])
    return prob, _obstacles(rng, 2, n_obst, width)


def _ticks(rng, prob, obs, ticks):
    """Per tick: the obstacles after a random walk of 0.002 a tick, and a start that moves towards the goal."""
    got = []
    rows = np.diff(obs.off)
    b = obs.b
    for t in range(ticks):
        step = np.repeat(rng.normal(0.0, 0.002, (len(rows), 2)), rows, axis=0)
        b = b + np.sum(obs.A * step, axis=1)
        start = prob.start_pos + 0.02 * t * (prob.goal_pos - prob.start_pos)
        got.append((SimpleNamespace(off=obs.off, A=obs.A, b=b), start, prob.goal_pos))
    return got


def _batch(case, seed):
    """Queries of uneven size: the sizes go with the case, everything else with the seed."""
    Q = case["Q"]
    rng = np.random.default_rng(Q)
    Ns = np.floor(np.exp(rng.uniform(log(case["n_lo"]), log(case["n_hi"] + 1), Q))).astype(int)
    Ks = rng.integers(case["k_lo"], case["k_hi"] + 1, Q)
    Ts = rng.integers(case["t_lo"], case["t_hi"] + 1, Q)
    rng = np.random.default_rng(seed)
    return [_environment(rng, 3, 7, int(n), int(k), int(t), True) for n, k, t in zip(Ns, Ks, Ts)]


def _mpc_references(rng, B, H):
    """Samples of random cubics in time (positions, velocities) that stay in the inner 90% of the box."""
    t = (MPC_DT * np.arange(H + 1))[None, :, None]
    p0 = rng.uniform(0.1 * MPC_WIDTH, 0.9 * MPC_WIDTH, (B, 1, 2))
    d = rng.normal(size=(B, 1, 2))
    v0 = d / np.linalg.norm(d, axis=2, keepdims=True) * rng.uniform(0.2, 1.0, (B, 1, 1))
    a0, j0 = 0.5 * rng.normal(size=(B, 1, 2)), 0.5 * rng.normal(size=(B, 1, 2))
    pos = p0 + v0 * t + a0 * t ** 2 / 2 + j0 * t ** 3 / 6
    ref = np.concatenate([pos, v0 + a0 * t + j0 * t ** 2 / 2], 2)
    return ref[np.all((pos >= 0.05 * MPC_WIDTH) & (pos <= 0.95 * MPC_WIDTH), axis=(1, 2))]


def _segments(rng, S, m, p):
    """Segments around random lines, each in a polytope that holds its control polygon (float32 arrays)."""
    d = rng.normal(size=(S, 1, m))
    d /= np.linalg.norm(d, axis=2, keepdims=True)
    pts = rng.uniform(0.0, 20.0, (S, 1, m)) + (np.arange(p + 1) / p)[None, :, None] * rng.uniform(1.0, 4.0, (S, 1, 1)) * d
    pts[:, 1:p] += rng.normal(size=(S, p - 1, m))
    lo = pts.min(1) - rng.uniform(1.0, 3.0, (S, m))
    hi = pts.max(1) + rng.uniform(1.0, 3.0, (S, m))
    cuts = REFINE_RMAX - 2 * m if m == 3 else 4
    nrm = rng.normal(size=(S, cuts, m))
    nrm /= np.linalg.norm(nrm, axis=2, keepdims=True)
    ncut = rng.integers(0, cuts + 1, S)
    A = np.zeros((S, REFINE_RMAX, m))
    b = np.ones((S, REFINE_RMAX))
    for a in range(m):
        A[:, 2 * a, a], A[:, 2 * a + 1, a] = 1.0, -1.0
        b[:, 2 * a], b[:, 2 * a + 1] = hi[:, a], -lo[:, a]
    off = np.einsum("sla,sca->slc", pts, nrm).max(1) + rng.uniform(0.1, 1.0, (S, cuts))
    A[:, 2 * m:2 * m + cuts], b[:, 2 * m:2 * m + cuts] = nrm, off
    pad = np.arange(REFINE_RMAX)[None] >= (2 * m + ncut)[:, None]
    A[pad], b[pad] = 0.0, 1.0
    f = lambda a: a.astype(np.float32)
    return f(pts), f(rng.uniform(0.2, 2.0, S)), f(A), f(b), (2 * m + ncut).astype(np.int32), f(rng.uniform(0.5, 1.5, S))


# --------------------------------------------------------------- prepare ----


def _empty(pl, N, cap, need):
    """A graph with room for `cap` edges (or what is needed), zeros where no edge will be written."""
    g = pl.alloc_graph(N, max(int(cap), need))
    for a in (g.col, g.w, g.tidx, g.mask):
        a.zero_()
    return g


def _pairs(m, N, K):
    """Candidate pairs of an environment, on the high side: a state lies in its own polytope and, by volume, in
    about 9% (2-D) or 0.4% (3-D) of the others."""
    inside = 1.0 + (K - 1) * (0.086 if m == 2 else 0.004)
    return min(1.5 * K * (N * inside / K) ** 2, float(N) * N)


def _search_buffers(pl, N):
    out = pl.alloc_search(N)
    out["path"].zero_()
    return out


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _query_problem(case, seed):
    rng = np.random.default_rng(seed)
    f32 = case["m"] == 3 and case["arith"] == "f32"
    return _environment(rng, case["m"], case["p"], case["N"], case["K"], case["nT"], f32, case["tighten"], case["cost"], TRIPS)


def _prepare_query(case, seed):
    prob = _query_problem(case, seed)
    pl = P.Planner.for_problem(prob, arith=case["arith"])
    dp = P.to_device(prob, input=prob.dtype)
    graph = _empty(pl, dp.N, _pairs(case["m"], dp.N, case["K"]), pl.build_edges(dp).E)
    return SimpleNamespace(kind="query", pl=pl, dp=dp, graph=graph, out=_search_buffers(pl, dp.N))


def _prepare_search(case, seed):
    s = _prepare_query(case, seed)
    s.kind, s.trips = "search", _query_problem(case, seed).trips
    s.out = [_search_buffers(s.pl, s.dp.N) for _ in s.trips]
    s.graph = s.pl.build_edges(s.dp, s.graph)
    return s


def _prepare_batch(case, seed):
    probs = _batch(case, seed)
    pl = P.Planner.for_problem(probs[0])
    dps = [P.to_device(q, input="f32") for q in probs]
    sizes = [max(g.E, int(_pairs(3, dp.N, dp.K))) for g, dp in zip(pl.build_batched(dps), dps)]
    dev = dps[0].states.device

    def packed(counts, dtype):
        """One array for the whole batch, and every query's part of it (aligned parts, zeros between them)."""
        at = np.concatenate([[0], np.cumsum([-(-max(c, 1) // 64) * 64 for c in counts])])
        whole = torch.zeros(int(at[-1]), dtype=dtype, device=dev)
        return whole, [whole[int(a):int(a) + max(c, 1)] for a, c in zip(at, counts)]

    Ns = [dp.N for dp in dps]
    arrays = dict(row_off=packed([n + 1 for n in Ns], torch.int32), col=packed(sizes, torch.int32),
                  w=packed(sizes, torch.float32), tidx=packed(sizes, torch.uint8), mask=packed(sizes, torch.int32),
                  count=packed([1] * len(dps), torch.int64), path=packed(Ns, torch.int32),
                  path_len=packed([1] * len(dps), torch.int32), cost=packed([1] * len(dps), torch.float64),
                  status=packed([1] * len(dps), torch.int32))
    part = {k: v[1] for k, v in arrays.items()}
    graphs = [P.Graph(N=Ns[q], cap=max(1, sizes[q]), **{k: part[k][q] for k in ("row_off", "col", "w", "tidx", "mask", "count")})
              for q in range(len(dps))]
    outs = [{k: part[k][q] for k in ("path", "path_len", "cost", "status")} for q in range(len(dps))]
    pl.prepare_batched(dps, graphs)
    pl.prepare_search_batched(dps, graphs, outs)
    return SimpleNamespace(kind="batch", pl=pl, dps=dps, whole={k: v[0] for k, v in arrays.items()})


def _prepare_cut(case, seed):
    prob, obs = _keepout(np.random.default_rng(seed), case["N"], case["obst"], case["nT"], case["width"])
    pl = P.Planner.for_problem(prob)
    dp = P.to_device(prob)
    graph = pl.build_edges(dp)
    do = P.obstacles_to_device(obs)
    return SimpleNamespace(kind="cut", pl=pl, dp=dp, graph=graph, obst=do, out=_empty(pl, dp.N, 16 * dp.N, pl.cut_edges(dp, graph, do).E))


def _prepare_replan(case, seed):
    rng = np.random.default_rng(seed)
    prob, obs = _keepout(rng, case["N"], case["obst"], 1, case["width"])
    pl = P.Planner.for_problem(prob, stream=torch.cuda.Stream())
    dp = P.to_device(prob)
    torch.cuda.synchronize()
    graph = pl.build_edges(dp)
    ticks = _ticks(rng, prob, obs, case["ticks"])
    rp = P.Replanner(pl, dp, graph, n_max=case["obst"], rows_max=8)
    rp.capture(obs, prob.start_pos, prob.goal_pos)
    return SimpleNamespace(kind="replan", rp=rp, ticks=ticks)


def _prepare_planes(case, seed):
    rng = np.random.default_rng(seed)
    obs = _obstacles(rng, case["m"], case["obst"], case["width"])
    x = rng.uniform(0.0, case["width"], (case["N"], case["m"]))
    pl = P.Planner(case["m"], case["m"], 5, BOUNDS[case["m"]], arith=case["arith"], input=case["arith"])
    dt = torch.float32 if case["arith"] == "f32" else torch.float64
    return SimpleNamespace(kind="planes", pl=pl, points=torch.tensor(x, dtype=dt, device="cuda"),
                           obst=P.obstacles_to_device(obs, input=case["arith"]))


def _prepare_mpc(case, seed):
    rng = np.random.default_rng(seed)
    B, H = case["B"], case["H"]
    obs = P.obstacles_to_device(_obstacles(rng, 2, case["obst"], MPC_WIDTH))
    pl = P.Planner(2, 2, 5, BOUNDS[2], arith="f64", input="f64")
    kept, have = [], 0
    while have < B:  # references whose nodes keep 0.05 from every obstacle
        ref = torch.tensor(_mpc_references(rng, 8 * B, H), device="cuda")
        if ref.shape[0]:
            near = pl.obstacle_planes(ref[:, :, :2].reshape(-1, 2).contiguous(), obs, nearest_only=True)["nearest_dist"]
            kept.append(ref[near.view(-1, H + 1).min(1).values >= 0.05])
            have += kept[-1].shape[0]
    ref = torch.cat(kept)[:B].contiguous()
    planes = torch.empty((B, H, 3), dtype=torch.float32, device="cuda")
    pl.nearest_planes_async(ref[:, :H, :2].reshape(-1, 2).contiguous(), obs, planes.view(-1, 3))
    box = np.array([[1.0, 0.0], [-1.0, 0.0], [0.0, 1.0], [0.0, -1.0]])
    prm = pl.mpc_params(H, MPC_DT, MPC_W["Q"], MPC_W["F"], MPC_W["R"], MPC_W["V"], box, [MPC_WIDTH, 0.0, MPC_WIDTH, 0.0])
    return SimpleNamespace(kind="mpc", pl=pl, prm=prm, ref=ref, x0=ref[:, 0].contiguous(), planes=planes, out=pl.alloc_mpc(B, H))


def _prepare_refine(case, seed):
    arrays = _segments(np.random.default_rng(seed), case["S"], case["m"], case["p"])
    pts, T, A, b, nrows, up = (torch.tensor(a, device="cuda") for a in arrays)
    refiner = R.Refiner(case["m"], case["m"], case["p"], BOUNDS[case["m"]])
    return SimpleNamespace(kind="refine", refiner=refiner, P=pts.requires_grad_(), T=T.requires_grad_(), A=A, b=b, nrows=nrows, up=up)


# ------------------------------------------------------------------- run ----


def _edges(g):
    return dict(row_off=g.row_off, col=g.col, w=g.w, tidx=g.tidx, mask=g.mask, count=g.count)


def run(s):
    return globals()["_run_" + s.kind](s)


def _run_query(s):
    s.pl.build_edges_async(s.dp, s.graph)
    s.pl.search_async(s.dp, s.graph, s.dp.start_pos, s.dp.goal_pos, s.out)
    return dict(_edges(s.graph), **s.out)


def _run_search(s):
    for (start, goal), out in zip(s.trips, s.out):
        s.pl.search_async(s.dp, s.graph, start, goal, out)
    return s.out


def _run_batch(s):
    s.pl.build_batched_async()
    s.pl.search_batched_async()
    return s.whole


def _run_cut(s):
    s.pl.cut_edges_async(s.dp, s.graph, s.obst, s.out)
    return _edges(s.out)


def _run_replan(s):
    got = [s.rp.tick(*t) for t in s.ticks]
    path = np.full((len(got), s.rp.dp.N), -1, dtype=np.int32)
    for row, r in zip(path, got):
        row[:len(r["path"] or ())] = r["path"] or ()
    return dict(path=path, cost=np.array([r["cost"] for r in got]), edges=np.array([r["edges"] for r in got]))


def _run_planes(s):
    return s.pl.obstacle_planes(s.points, s.obst)


def _run_mpc(s):
    s.pl.mpc_qp_async(s.prm, s.x0, s.ref, s.planes, s.out)
    return s.out


def _run_refine(s):
    loss = R.refine_loss(s.P, s.T, s.A, s.b, s.nrows, s.refiner)
    dP, dT = torch.autograd.grad(loss, (s.P, s.T), s.up)
    return dict(loss=loss, dP=dP, dT=dT)


# ------------------------------------------------------------------ work ----


def _query_work(m, p, N, K, nT, w_bytes):
    """States and rows in, the graph out; the checks' operations with early exits.

    About 40% of the candidate pairs are edges.  A check needs about 33
    operations (m = 3) when it stops at the first violated row; the FP32 and
    FP64 forms count alike.
    """
    pairs = _pairs(m, N, K)
    edges = 0.4 * pairs
    size = 4 if w_bytes == 4 else 8
    return N * m * m * size + K * 3 * m * (m + 1) * size + N * 4 + edges * (9 + w_bytes), pairs * nT * (33 if m == 3 else 15), edges


def work(case):
    k = case["kind"]
    if k in ("query", "search"):
        nbytes, flops, edges = _query_work(case["m"], case["p"], case["N"], case["K"], case["nT"], 8 if case["arith"] == "f64" else 4)
        # every search: columns and weights once, distances
        search = (TRIPS if k == "search" else 1) * (edges * (12 if case["arith"] == "f64" else 8) + 16 * case["N"])
        return dict(bytes=search if k == "search" else nbytes + search, flops=2 * edges + (0 if k == "search" else flops))
    if k == "batch":
        got = [_query_work(3, 7, (case["n_lo"] * case["n_hi"]) ** 0.5 * f, (case["k_lo"] + case["k_hi"]) / 2,
                           (case["t_lo"] + case["t_hi"]) / 2, 4) for f in (0.25, 0.5, 1.0, 2.0, 4.0)]
        return dict(bytes=case["Q"] * sum(g[0] + 8 * g[2] for g in got) / 5, flops=case["Q"] * sum(g[1] for g in got) / 5)
    if k in ("cut", "replan"):
        edges = 45000.0 * (case["N"] / 5000.0) ** 2
        units = edges * case.get("nT", 1) * case.get("ticks", 1)
        # graph in, half of it out; a box test (about 8 operations) per curve and obstacle
        return dict(bytes=units * 17 * 1.5 + case["N"] * 36 + case["obst"] * 5.5 * 24, flops=8 * units * case["obst"])
    if k == "planes":
        pairs = float(case["N"]) * case["obst"]
        return dict(bytes=pairs * 4 * (2 * case["m"] + 2), flops=pairs * 40 * case["m"])
    if k == "mpc":
        B, H, nv = case["B"], case["H"], 2 * case["H"]
        # references, planes in, nodes and inputs out; gradient, unconstrained minimum and about four active-set steps
        return dict(bytes=B * (8.0 * (H + 1) * 4 * 2 + 8 * H * 4 + 12 * H), flops=B * (16.0 * (H + 1) * nv + 24.0 * nv * nv))
    S, m, p = case["S"], case["m"], case["p"]
    # points, duration, rows, upstream gradient in; loss and gradients out; about 40 operations a margin
    margins = 2 * m * sum(p - q + 1 for q in range(1, m + 1)) + (p - 1) * (3 * m)
    return dict(bytes=S * 4.0 * (2 * (p + 1) * m + 4 + REFINE_RMAX * (m + 1) + 1), flops=S * 40.0 * margins)


# ----------------------------------------------------------------- exact ----


def _maps(g, p, T):
    """Linear maps of xi = [x_i; x_j] (one axis): control points, hodograph rows by order, cost rows by derivative."""
    q = 2 * g - 1
    B = np.zeros((q + 1, 2 * g))
    for l in range(g):
        for k in range(l + 1):
            v = comb(l, k) * factorial(q - k) / factorial(q) * T ** k
            B[l, k], B[q - l, g + k] = v, (-1) ** k * v

    def elevate(a, b):
        return np.array([[comb(a, j) * comb(b - a, i - j) / comb(b, i) if 0 <= i - j <= b - a else 0.0 for j in range(a + 1)]
                         for i in range(b + 1)])

    D = elevate(q, p) @ B
    rows = [factorial(p) / factorial(p - k) * T ** -k * np.diff(D, n=k, axis=0) for k in range(g + 1)]
    cost = [np.diff(elevate(p - d, p) @ rows[d], axis=0) for d in range(g)]
    return D, rows[1:], cost


def _graph64(prob):
    """Edges of one query in 64 bits: source, column and weight of every edge, and (T, control points) by duration."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t64 = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=dev)
    md = prob.model
    m, g, p, N = md.m, md.gamma, md.degree, prob.states.shape[0]
    X = t64(prob.states).view(N, g, m)
    best = torch.full((N * N,), float("inf"), dtype=torch.float64, device=dev)
    maps = [_maps(g, p, float(T)) for T in prob.T]
    half = lambda M, x, s: torch.einsum("rc,ncm->nrm", t64(M)[:, s * g:(s + 1) * g], x)
    for k in range(len(prob.poly_off) - 1):
        r = slice(prob.poly_off[k], prob.poly_off[k + 1])
        A, b = t64(prob.A[r]), t64(prob.b[r]) - md.tighten
        ids = torch.nonzero((X[:, 0] @ A.T <= b).all(1)).flatten()
        n = len(ids)
        if n < 2:
            continue
        x = X[ids]
        chunk = max(1, 40_000_000 // (n * p * m))
        for D, H, C in maps:
            HL, HR = ([half(h, x, s) for h in H] for s in (0, 1))
            DL, DR = half(D, x, 0), half(D, x, 1)
            CC = np.concatenate(C if md.cost_mode == "state" else C[:1])
            CL, CR = half(CC, x, 0), half(CC, x, 1)
            for i0 in range(0, n, chunk):
                i1 = min(n, i0 + chunk)
                ok = torch.ones((i1 - i0, n), dtype=torch.bool, device=dev)
                for hl, hr, c in zip(HL, HR, md.bounds):
                    ok &= ((hl[i0:i1, None] + hr[None]).abs() <= c - md.tighten).all(-1).all(-1)
                ii, jj = torch.nonzero(ok, as_tuple=True)
                ii = ii + i0
                ii, jj = ii[ii != jj], jj[ii != jj]
                pts = DL[ii, 1:p] + DR[jj, 1:p]
                ok = (pts @ A.T <= b).all(-1).all(-1)
                ii, jj = ii[ok], jj[ok]
                d = (CL[ii] + CR[jj]).view(len(ii), len(CC) // p, p, m)
                at = ids[ii] * N + ids[jj]
                best[at] = torch.minimum(best[at], d.square().sum((1, 3)).sqrt().sum(1))
    at = torch.nonzero(torch.isfinite(best)).flatten()
    return at // N, at % N, best[at]


def _shortest64(prob, src, dst, w, start_pos, goal_pos):
    """Cost of the shortest path between the states nearest to two positions (Dijkstra)."""
    m = prob.model.m
    near = lambda x: int(np.argmin(np.sum((prob.states[:, :m] - x) ** 2, axis=1)))
    s, goal = near(start_pos), near(goal_pos)
    src, dst, w = (a.cpu().numpy() for a in (src, dst, w))
    row = np.searchsorted(src, np.arange(prob.states.shape[0] + 1)).tolist()
    dst, w = dst.tolist(), w.tolist()
    dist, heap = {s: 0.0}, [(0.0, s)]
    while heap:
        d, u = heapq.heappop(heap)
        if u == goal:
            return d
        if d > dist[u]:
            continue
        for e in range(row[u], row[u + 1]):
            nd = d + w[e]
            if nd < dist.get(dst[e], np.inf):
                dist[dst[e]] = nd
                heapq.heappush(heap, (nd, dst[e]))
    return float("inf")


def _vertices(obs):
    """Corners of 2-D obstacles [n][v][2], padded with the first one; rows padded with ones that no point violates."""
    n, rmax = len(obs.off) - 1, int(np.diff(obs.off).max())
    A, b = np.zeros((n, rmax, 2)), np.ones((n, rmax))
    V = np.zeros((n, rmax * (rmax - 1) // 2, 2))
    for o in range(n):
        a, c = obs.A[obs.off[o]:obs.off[o + 1]], obs.b[obs.off[o]:obs.off[o + 1]]
        A[o, :len(c)], b[o, :len(c)] = a, c
        i, j = np.triu_indices(len(c), 1)
        det = a[i, 0] * a[j, 1] - a[i, 1] * a[j, 0]
        ok = np.abs(det) > 1e-14
        i, j, det = i[ok], j[ok], det[ok]
        v = np.stack([c[i] * a[j, 1] - c[j] * a[i, 1], a[i, 0] * c[j] - a[j, 0] * c[i]], 1) / det[:, None]
        v = v[np.all(v @ a.T <= c + 1e-12, axis=1)]
        V[o] = v[0]
        V[o, :len(v)] = v
    return A, b, V


def _free64(pts, obs):
    """Whether the hull of each curve's control points [E][l][2] misses every obstacle: no obstacle without a separating axis."""
    dev = pts.device
    A, b, V = (torch.as_tensor(a, dtype=torch.float64, device=dev) for a in _vertices(obs))
    free = torch.ones(len(pts), dtype=torch.bool, device=dev)
    lo, hi = pts.min(1).values, pts.max(1).values
    vlo, vhi = V.min(1).values, V.max(1).values
    i, j = np.triu_indices(pts.shape[1], 1)
    for e0 in range(0, len(pts), 20000):
        meet = ((lo[e0:e0 + 20000, None] <= vhi) & (hi[e0:e0 + 20000, None] >= vlo)).all(-1)
        e, o = torch.nonzero(meet, as_tuple=True)
        e = e + e0
        Pe, Vo = pts[e], V[o]
        apart = ((Pe @ A[o].transpose(1, 2)).min(1).values > b[o]).any(1)
        d = Pe[:, i] - Pe[:, j]
        nrm = torch.stack([-d[..., 1], d[..., 0]], -1).transpose(1, 2)
        p, v = Pe @ nrm, Vo @ nrm
        apart |= ((p.min(1).values > v.max(1).values) | (p.max(1).values < v.min(1).values)).any(1)
        free[e[~apart]] = False
    return free


def _cut64(prob, obs, src, dst):
    """Weights of the curves left after the cut, infinite where none is (durations are all feasible or not by themselves)."""
    dev = src.device
    m, g, p = 2, 2, 5
    X = torch.as_tensor(prob.states, device=dev).view(-1, g, m)
    best = torch.full((len(src),), float("inf"), dtype=torch.float64, device=dev)
    for T in prob.T:
        D, H, C = _maps(g, p, float(T))
        both = lambda M: torch.einsum("rc,ecm->erm", torch.as_tensor(np.ascontiguousarray(M), device=dev), torch.cat([X[src], X[dst]], 1))
        ok = _free64(both(D), obs)
        for h, c in zip(H, prob.model.bounds):
            ok &= (both(h).abs() <= c).all(-1).all(-1)
        ok &= ((both(D) >= 0.0) & (both(D) <= prob.b[0])).all(-1).all(-1)
        cost = both(np.concatenate(C)).view(len(src), g, p, m).square().sum((1, 3)).sqrt().sum(1)
        best = torch.where(ok, torch.minimum(best, cost), best)
    return best


def _planes64(x, obs):
    """Projections of points onto every obstacle: faces and edge segments, the nearest one."""
    m, n, P_ = x.shape[1], len(obs.off) - 1, len(x)
    dev = x.device
    z = torch.empty((P_, n, m), dtype=torch.float64, device=dev)
    for o in range(n):
        a, c = (torch.as_tensor(v[obs.off[o]:obs.off[o + 1]], dtype=torch.float64, device=dev) for v in (obs.A, obs.b))
        R_ = len(c)
        s = x @ a.T - c
        cand, far = [], []
        if m == 3:
            q = x[:, None] - (s / a.square().sum(1))[..., None] * a
            cand.append(q)
            far.append(~((q @ a.T) <= c + 1e-12).all(-1))
            i, j = np.triu_indices(R_, 1)
            d = torch.linalg.cross(a[i], a[j])
            ok = d.square().sum(1) > 1e-20
            i, j, d = i[ok.cpu().numpy()], j[ok.cpu().numpy()], d[ok]
            M = torch.stack([a[i], a[j], d], 1)
            base = torch.linalg.solve(M, torch.stack([c[i], c[j], torch.zeros_like(c[i])], 1))
            on = torch.zeros((len(i), R_), dtype=torch.bool, device=dev)
            on[torch.arange(len(i)), i] = on[torch.arange(len(i)), j] = True
        else:
            d = torch.stack([-a[:, 1], a[:, 0]], 1)
            base = a * (c / a.square().sum(1))[:, None]
            on = torch.eye(R_, dtype=torch.bool, device=dev)
        d = d / d.norm(dim=1, keepdim=True)
        slope, room = d @ a.T, c - base @ a.T
        flat = on | (slope.abs() < 1e-14)
        at = room / torch.where(flat, 1.0, slope)
        hi = torch.where(~flat & (slope > 0), at, float("inf")).min(1).values
        lo = torch.where(~flat & (slope < 0), at, -float("inf")).max(1).values
        none = (lo > hi) | ((slope.abs() < 1e-14) & ~on & (room < 0)).any(1)
        base, d, lo, hi = base[~none], d[~none], lo[~none], hi[~none]
        t = ((x[:, None] - base) * d).sum(-1).clamp(lo, hi)
        cand.append(base + t[..., None] * d)
        far.append(torch.zeros(t.shape, dtype=torch.bool, device=dev))
        q, far = torch.cat(cand, 1), torch.cat(far, 1)
        k = (q - x[:, None]).square().sum(-1).masked_fill(far, float("inf")).argmin(1)
        z[:, o] = torch.where((s <= 0).all(1)[:, None], x, q[torch.arange(P_), k])
    v = x[:, None] - z
    dist = v.norm(dim=2)
    h = torch.where(dist[..., None] > 0, v / dist.clamp(min=1e-300)[..., None], 0.0)
    return z, torch.cat([h, (h * z).sum(2, keepdim=True)], 2), dist


def _refine64(arrays, m, p):
    """The refinement's loss and gradients: relaxed log-barrier of every margin and the snap energy."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    pts, T, A, b, nrows, up = (torch.as_tensor(a, device=dev) for a in arrays)
    pts, T, A, b, up = (a.double() for a in (pts, T, A, b, up))
    pts.requires_grad_()
    T.requires_grad_()
    d = REFINE_DELTA
    phi = lambda x: torch.where(x >= d, -torch.log(x.clamp(min=d)), -log(d) + 0.5 * ((x - 2 * d) / d) ** 2 - 0.5)
    loss = 0.0
    for k, c in enumerate(BOUNDS[m], 1):
        Q = factorial(p) / factorial(p - k) * T[:, None, None] ** -k * torch.diff(pts, n=k, dim=1)
        loss = loss + phi(c - Q).sum((1, 2)) + phi(c + Q).sum((1, 2))
    live = torch.arange(REFINE_RMAX, device=dev)[None] < nrows[:, None]
    margin = b[:, None] - pts[:, 1:p] @ A.transpose(1, 2)
    loss = loss + torch.where(live[:, None], phi(margin), 0.0).sum((1, 2))
    q = p - 4
    G = torch.tensor([[comb(q, j) * comb(q, l) / ((2 * q + 1) * comb(2 * q, j + l)) for l in range(q + 1)] for j in range(q + 1)],
                     dtype=torch.float64, device=dev)
    d4 = torch.diff(pts, n=4, dim=1)
    loss = loss + (factorial(p) / factorial(q)) ** 2 * T ** -7 * torch.einsum("jl,sja,sla->s", G, d4, d4)
    dP, dT = torch.autograd.grad(loss, (pts, T), up)
    return dict(loss=loss.detach(), dP=dP, dT=dT)


def _padded(w, cap):
    return torch.cat([w, torch.zeros(max(0, int(cap) - len(w)), dtype=w.dtype, device=w.device)])


def exact(case, seed):
    k = case["kind"]
    none = dict(row_off=None, col=None, tidx=None, mask=None, count=None)
    if k in ("query", "search"):
        prob = _query_problem(case, seed)
        src, dst, w = _graph64(prob)
        trips = prob.trips if k == "search" else prob.trips[:1]
        cost = [torch.tensor([_shortest64(prob, src, dst, w, *t)], dtype=torch.float64) for t in trips]
        found = [dict(path=None, path_len=None, cost=c) for c in cost]
        return found if k == "search" else dict(none, w=_padded(w, _pairs(case["m"], case["N"], case["K"])), **found[0])
    if k == "cut":
        prob, obs = _keepout(np.random.default_rng(seed), case["N"], case["obst"], case["nT"], case["width"])
        src, dst, _ = _graph64(prob)
        w = _cut64(prob, obs, src, dst)
        return dict(none, w=_padded(w[torch.isfinite(w)], 16 * case["N"]))
    if k == "replan":
        rng = np.random.default_rng(seed)
        prob, obs = _keepout(rng, case["N"], case["obst"], 1, case["width"])
        src, dst, _ = _graph64(prob)
        cost = []
        for o, start, goal in _ticks(rng, prob, obs, case["ticks"]):
            w = _cut64(prob, o, src, dst)
            left = torch.isfinite(w)
            cost.append(_shortest64(prob, src[left], dst[left], w[left], start, goal))
        return dict(path=None, cost=np.array(cost), edges=None)
    if k == "planes":
        rng = np.random.default_rng(seed)
        obs = _obstacles(rng, case["m"], case["obst"], case["width"])
        x = rng.uniform(0.0, case["width"], (case["N"], case["m"]))
        if case["arith"] == "f32":
            x, obs = _f32(x), SimpleNamespace(off=obs.off, A=_f32(obs.A), b=_f32(obs.b))
        z, plane, dist = _planes64(torch.as_tensor(x, device="cuda" if torch.cuda.is_available() else "cpu"), obs)
        return dict(closest=z, plane=plane, dist=dist, nearest=None, nearest_dist=dist.min(1).values)
    if k == "refine":
        return _refine64(_segments(np.random.default_rng(seed), case["S"], case["m"], case["p"]), case["m"], case["p"])
    return None  # batch: minutes in 64 bits; mpc: a plain active-set solver takes seconds a problem
