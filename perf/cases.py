"""What a user of this framework has it do, as cases that can be timed and whose
outputs can be compared: edge validation batches (collision checks on their
own), whole plans, batches of plans, and the proposal network's inference and
training, each through the public entry points of paper_2609_30533_gb300.stp
and .proposal.

A case is a dict of plain values: "kind" says which entry point, the rest are
its sizes and options. listed() holds the fixed ones, draw() gives more of the
same ranges. prepare() makes what a program has in hand before the call, run()
is one pass, exact() the 64-bit value of what run() returns where it has one,
work() the bytes and operations that a pass cannot do without.

The robots and obstacle fields have the shapes of the repository's workloads:
a point robot among discs, a UR5e with 32 link spheres and a seeded 7-DoF arm
with 48 link spheres, both among moving spheres.
"""
import math

import numpy as np
import torch

from paper_2609_30533_gb300 import proposal, stp

# UR5e standard DH rows (a, alpha, d, theta_offset): Universal Robots' published table.
UR5E_DH = np.array([
    [0.0, math.pi / 2, 0.1625, 0.0],
    [-0.425, 0.0, 0.0, 0.0],
    [-0.3922, 0.0, 0.0, 0.0],
    [0.0, math.pi / 2, 0.1333, 0.0],
    [0.0, -math.pi / 2, 0.0997, 0.0],
    [0.0, 0.0, 0.0996, 0.0],
])
DOF = {"disc2d": 2, "ur5e": 6, "arm7": 7}
SPHERES = {"disc2d": 1, "ur5e": 32, "arm7": 48}
RES = 0.01  # edge check resolution of every workload
PATH_ROWS = 1024  # states of the trajectory buffer that a plan's path is copied into


# ---------------------------------------------------------------------------
# Cases.
# ---------------------------------------------------------------------------
def listed():
    return [
        # A controller or local planner checks a handful of candidate motions: latency counts.
        dict(name="edges-ur5e-61", kind="edges", robot="ur5e", n=61, obs=16, precision=0, mode="verdict",
             host=False),
        # Roadmap-sized validation of random steps (the repository's collision benchmark).
        dict(name="edges-ur5e-1m", kind="edges", robot="ur5e", n=1 << 20, obs=16, precision=0, mode="verdict",
             host=False),
        # Clearances of candidate motions for trajectory scoring, obstacles of different radii.
        dict(name="edges-arm7-clearance", kind="edges", robot="arm7", n=9973, obs=64, precision=0,
             mode="clearance", host=False),
        # Re-validation of a set of motions in double precision.
        dict(name="edges-arm7-f64", kind="edges", robot="arm7", n=2003, obs=64, precision=1, mode="verdict",
             host=False),
        # Motions of a mobile robot held in host arrays: copies in, verdicts and counts out.
        dict(name="edges-disc2d-host", kind="edges", robot="disc2d", n=30011, obs=8, precision=0, mode="verdict",
             host=True),
        # One query of a small mobile robot, few workers, many short iterations (interval root).
        dict(name="plan-disc2d", kind="plan", robot="disc2d", obs=8, horizon=20.0, variant=0, roots=4, workers=64,
             iters=256, learned=0),
        # One query of a 6-DoF arm (the repository's headline plan: root recycling, 32 iterations).
        dict(name="plan-ur5e", kind="plan", robot="ur5e", obs=16, horizon=15.0, variant=1, roots=8, workers=1024,
             iters=32, learned=0),
        # The widest iteration: 7-DoF arm, 64 obstacles, interval root.
        dict(name="plan-arm7", kind="plan", robot="arm7", obs=64, horizon=60.0, variant=0, roots=16, workers=4096,
             iters=16, learned=0),
        # Many queries of uneven robots and obstacle counts planned together (training-data generation).
        dict(name="batch-mixed-96", kind="batch", n=96, workers=256, iters=32, steps_form=True),
        # Proposals for a large set of queries resident on the device.
        dict(name="mlp-forward-64k", kind="forward", n=65536, host=False),
        # The training loop as proposal.train runs it: host minibatches of 128, validation at the end.
        dict(name="mlp-train-128", kind="loop", samples=512, batch=128, steps=25),
        # Large-batch training steps on device-resident samples.
        dict(name="mlp-train-64k", kind="steps", batch=65536, steps=4),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges; sizes spread over their logarithm."""
    kind = rng.choice(["edges", "edges", "edges", "plan", "plan", "batch", "forward", "loop", "steps"])
    if kind == "edges":
        robot = rng.choice(["disc2d", "ur5e", "arm7"])
        precision = 1 if rng.random() < 0.2 else 0
        mode = rng.choice(["verdict", "verdict", "clearance", "full"])
        most = {"disc2d": 1 << 20, "ur5e": 1 << 18, "arm7": 1 << 15}[robot]
        if mode != "verdict":
            most //= 8
        if precision:
            most //= 16
        obs = rng.randint(4, 32) if robot == "disc2d" else rng.randint(4, 128)
        host = rng.random() < 0.3
        return dict(kind=kind, robot=robot, n=_logint(rng, 61, most), obs=obs, precision=precision, mode=mode,
                    host=host)
    if kind == "plan":
        robot = rng.choice(["disc2d", "ur5e", "arm7"])
        most = {"disc2d": 1024, "ur5e": 2048, "arm7": 4096}[robot]
        obs = rng.randint(4, 32) if robot == "disc2d" else rng.randint(4, 96)
        return dict(kind=kind, robot=robot, obs=obs, horizon=round(rng.uniform(10.0, 60.0), 3),
                    variant=rng.choice([0, 1, 2]), roots=_logint(rng, 2, 64), workers=_logint(rng, 32, most),
                    iters=_logint(rng, 4, 128 if robot == "disc2d" else 16), learned=1 if rng.random() < 0.25 else 0)
    if kind == "batch":
        return dict(kind=kind, n=_logint(rng, 6, 96), workers=rng.choice([64, 128, 200, 256]),
                    iters=_logint(rng, 4, 32), steps_form=rng.random() < 0.7)
    if kind == "forward":
        return dict(kind=kind, n=_logint(rng, 1, 65536), host=rng.random() < 0.4)
    if kind == "loop":
        return dict(kind=kind, samples=_logint(rng, 100, 4000), batch=_logint(rng, 16, 512), steps=rng.randint(5, 25))
    return dict(kind="steps", batch=_logint(rng, 100, 65536), steps=rng.randint(1, 4))


# ---------------------------------------------------------------------------
# Problems.
# ---------------------------------------------------------------------------
def _sphere_layout(dh, n, radius):
    """Link spheres at equal arc length along each link's DH polyline, shared among links by |a| + |d|."""
    dof = len(dh)
    length = np.maximum(np.abs(dh[:, 0]) + np.abs(dh[:, 2]), 1e-6)
    share = length / length.sum() * (n - dof)
    count = 1 + np.floor(share).astype(int)
    for j in np.argsort(-(share - np.floor(share)), kind="stable")[:n - count.sum()]:
        count[j] += 1
    out = []
    for j in range(dof):
        a, alpha, d, _ = dh[j]
        p = [np.array([-a, -d * math.sin(alpha), -d * math.cos(alpha)]), np.array([-a, 0.0, 0.0]), np.zeros(3)]
        first, second = np.linalg.norm(p[1] - p[0]), np.linalg.norm(p[2] - p[1])
        for m in range(count[j]):
            s = (m + 0.5) / count[j] * (first + second)
            if s <= first and first > 0:
                c = p[0] + (p[1] - p[0]) * (s / first)
            else:
                c = p[1] + (p[2] - p[1]) * ((s - first) / second if second > 0 else 0.0)
            out.append([j + 1, c[0], c[1], c[2], radius])
    return np.array(out)


def _paths(rng, n_obs, n_way, half, H):
    """Obstacle waypoints in a cube, legs at one speed of at most 0.5 m/s over [0, H]."""
    pts = rng.uniform(-half, half, size=(n_obs, n_way, 3))
    total = np.linalg.norm(np.diff(pts, axis=1), axis=2).sum(1)
    shrink = np.minimum(1.0, 0.5 * H / np.maximum(total, 1e-12) * 0.999)
    pts = pts[:, :1] + (pts - pts[:, :1]) * shrink[:, None, None]
    legs = np.linalg.norm(np.diff(pts, axis=1), axis=2)
    way = np.zeros((n_obs, n_way, 4))
    way[:, 1:, 0] = np.cumsum(legs, 1) / legs.sum(1, keepdims=True) * H
    way[:, :, 1:] = pts
    return way


def _world(robot, obs, H, rng):
    """Keyword arguments of stp.Problem for a robot and its obstacles (no start, goal or planner settings)."""
    if robot == "disc2d":
        pos = rng.uniform(0.15, 0.85, size=(obs, 2))
        vel = rng.uniform(-0.1, 0.1, size=(obs, 2))
        way = np.zeros((obs, 2, 4))
        way[:, 0, 1:3] = pos
        way[:, 1, 0] = H
        way[:, 1, 1:3] = pos + H * vel
        return dict(dof=2, arm=False, dh=None, q_lo=np.zeros(2), q_hi=np.ones(2), spheres=np.zeros((1, 5)), v_max=0.5,
                    obs_radius=np.full(obs, 0.05), obs_way=way)
    if robot == "ur5e":
        dh, spheres, way = UR5E_DH, _sphere_layout(UR5E_DH, 32, 0.05), _paths(rng, obs, 4, 0.6, H)
        radius = np.full(obs, 0.06)
    else:
        dh = np.zeros((7, 4))
        dh[:, 1] = [math.pi / 2 if j % 2 == 0 else -math.pi / 2 for j in range(7)]
        dh[:, 2] = rng.uniform(0.1, 0.4, size=7)
        spheres, way = _sphere_layout(dh, 48, 0.04), _paths(rng, obs, 8, 1.0, H)
        radius = rng.uniform(0.04, 0.1, size=obs)
    d = len(dh)
    return dict(dof=d, arm=True, dh=dh, q_lo=np.full(d, -math.pi), q_hi=np.full(d, math.pi), spheres=spheres,
                v_max=math.pi / 2, obs_radius=radius, obs_way=way)


def _query(world, H, rng):
    """Start (free at time 0) and goal (free at some time) of a query, or None where the obstacles leave none
    (one of them at the arm's base); uniform candidates for the arms."""
    d = world["dof"]
    if not world["arm"]:
        return np.full(2, 0.05), np.full(2, 0.95)
    cand = rng.uniform(-math.pi, math.pi, size=(2, 64, d))
    P = stp.Problem(**world, q_start=cand[0, 0], q_goal=cand[1, 0], t_max=H, max_iters=1, ext_per_iter=32, env_dt=H)
    start = P.check_edges(cand[0], np.zeros(64), cand[0], np.zeros(64))[0]
    times = np.linspace(0.2 * H, 0.9 * H, 4)
    goals, at = np.repeat(cand[1], 4, axis=0), np.tile(times, 64)
    goal = P.check_edges(goals, at, goals, at)[0].reshape(64, 4).any(1)
    P.close()
    if not start.any() or not goal.any():
        return None
    return cand[0, int(np.argmax(start))], cand[1, int(np.argmax(goal))]


def _settings(robot, H):
    return dict(eta=0.1 if robot == "disc2d" else 0.5, edge_res=RES, env_dt=0.02, p_new=0.05, p_guided=0.95, t_max=H)


def _edges(case, seed):
    """World and space-time edges (float64 numpy) of an "edges" case: a step of the workload's range from a
    uniform state in a uniform direction (components that would leave the box are reflected) at full speed."""
    rng = np.random.default_rng([seed, 1])
    robot, n, H = case["robot"], case["n"], {"disc2d": 20.0, "ur5e": 15.0, "arm7": 60.0}[case["robot"]]
    world = _world(robot, case["obs"], H, rng)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dev = dict(device="cuda", dtype=torch.float64)
    lo, hi = torch.tensor(world["q_lo"], **dev), torch.tensor(world["q_hi"], **dev)
    d = world["dof"]
    qa = lo + torch.rand(n, d, generator=gen, **dev) * (hi - lo)
    step = torch.randn(n, d, generator=gen, **dev)
    step *= _settings(robot, H)["eta"] / step.norm(dim=1, keepdim=True)
    out = (qa + step > hi) | (qa + step < lo)
    qb = torch.clamp(qa + torch.where(out, -step, step), lo, hi)
    dur = (qb - qa).norm(dim=1) / world["v_max"]
    ta = torch.rand(n, generator=gen, **dev) * (H - dur)
    real = torch.float64 if case["precision"] else torch.float32
    return world, H, [x.to(real).contiguous() for x in (qa, ta, qb, ta + dur)]


_STREAM = []


def _stream():
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def _problem(case, seed):
    rng = np.random.default_rng([seed, 2])
    robot, H = case["robot"], case["horizon"]
    query = None
    while query is None:
        world = _world(robot, case["obs"], H, rng)
        query = _query(world, H, rng)
    qs, qg = query
    return stp.Problem(**world, q_start=qs, q_goal=qg, variant=case["variant"], n_roots=case["roots"],
                       ext_per_iter=case["workers"], max_iters=case["iters"], seed=seed, learned=case["learned"],
                       **_settings(robot, H))


def _samples(n, seed, device):
    """Features and targets as the pipeline collects them: 26 features in use, paths near the straight line."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.zeros(n, stp.MLP_IN, device="cuda")
    X[:, :26] = torch.rand(n, 26, generator=gen, device="cuda") * 2 - 1
    T = torch.zeros(n, stp.MLP_NTGT, device="cuda")
    T[:, 0] = 0.1 + 0.8 * torch.rand(n, generator=gen, device="cuda")
    T[:, 1:129] = (torch.rand(n, 128, generator=gen, device="cuda") - 0.5) * 0.4
    T[:, 129] = 7
    return (X, T) if device else (X.cpu().numpy(), T.cpu().numpy())


# ---------------------------------------------------------------------------
# prepare / run.
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=dict(case))
    if kind == "edges":
        world, H, edges = _edges(case, seed)
        q = 0.5 * (world["q_lo"] + world["q_hi"])
        s["P"] = stp.Problem(**world, q_start=q, q_goal=q + 0.25, max_iters=1, ext_per_iter=32,
                             precision=case["precision"], **dict(_settings(case["robot"], H), env_dt=H))
        if case["host"]:
            s["edges"] = [x.cpu().numpy() for x in edges]
        else:
            # The caller's buffers; every problem of the program on its one stream.
            s["edges"] = edges
            s["P"].set_stream(_stream().cuda_stream)
            s["verdict"] = torch.zeros(case["n"], dtype=torch.uint8, device="cuda")
            s["clearance"] = torch.zeros(case["n"], dtype=edges[0].dtype, device="cuda")
    elif kind == "plan":
        s["P"] = _problem(case, seed)
        if case["learned"]:
            net = stp.Mlp(1)
            net.set_params(proposal.init_params(seed))
            proposal.install(net, [s["P"]])
            net.close()
    elif kind == "batch":
        rng = np.random.default_rng([seed, 3])
        s["problems"] = []
        for i in range(case["n"]):
            one = dict(robot=("disc2d", "ur5e", "arm7")[i % 3], horizon=float(rng.uniform(10.0, 60.0)),
                       obs=int(rng.integers(4, 129)), variant=(0, 1, 1)[i % 3], roots=(4, 8, 16)[i % 3],
                       workers=case["workers"], iters=case["iters"], learned=0)
            if one["robot"] == "disc2d":
                one["obs"] = min(one["obs"], 32)
            s["problems"].append(_problem(one, seed * 1000 + i))
        # The pipeline's launch shape for per-step batches; the work queue with its defaults.
        s["batch"] = stp.Batch(s["problems"], nn_ctas=4, validate_ctas=8, launch_mode=stp.STP_LAUNCH_STEPS) \
            if case["steps_form"] else stp.Batch(s["problems"])
    elif kind == "forward":
        X, _ = _samples(case["n"], seed, not case["host"])
        s["net"], s["X"] = stp.Mlp(case["n"]), X
        s["net"].set_params(proposal.init_params(seed))
        if not case["host"]:
            s["Y"] = torch.zeros(case["n"], stp.MLP_OUT, device="cuda")
    elif kind == "loop":
        s["X"], s["T"] = _samples(case["samples"], seed, False)
        s["net"], s["start"] = stp.Mlp(case["batch"]), proposal.init_params(seed)
        s["net"].set_params(s["start"])
        s["seed"] = seed
    else:
        s["X"], s["T"] = _samples(case["batch"] * case["steps"], seed, True)
        s["net"] = stp.Mlp(case["batch"])
        s["net"].set_params(proposal.init_params(seed))
    torch.cuda.synchronize()
    return s


_COUNTS = ("iterations", "first_solution_iter", "nodes", "edges_validated", "bridges_validated", "root_checks",
           "nn_evals", "nn_nodes", "bridge_evals", "bridge_nodes")


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "edges":
        qa, ta, qb, tb = s["edges"]
        clear, early = case["mode"] == "clearance", case["mode"] != "full"
        if case["host"]:
            v, c, n = s["P"].check_edges(qa, ta, qb, tb, clearance=clear, early_exit=early, n_checks=True)
            return {"verdict": v, "clearance": c, "checks": n}
        s["P"].check_edges_device(qa.data_ptr(), ta.data_ptr(), qb.data_ptr(), tb.data_ptr(), case["n"],
                                  s["verdict"].data_ptr(), s["clearance"].data_ptr() if clear else None,
                                  early_exit=early)
        return {"verdict": s["verdict"], "clearance": s["clearance"] if clear else None}
    if kind == "plan":
        o = s["P"].plan()
        # The path in the planner's own precision, in the program's fixed trajectory buffer.
        path = np.zeros((PATH_ROWS, o.path.shape[1]), dtype=np.float32)
        path[:len(o.path)] = o.path[:PATH_ROWS]
        return {"status": o.status, "U": o.U, "C": o.C, "path": path, "states": len(o.path),
                "counts": np.array([o.stats[k] for k in _COUNTS])}
    if kind == "batch":
        _, stats = s["batch"].plan()
        return {"U": np.array([x["U"] for x in stats], dtype=np.float32),
                "C": np.array([x["C"] for x in stats], dtype=np.float32),
                "counts": np.array([[x[k] for k in _COUNTS] for x in stats])}
    if kind == "forward":
        if case["host"]:
            return s["net"].forward(s["X"])
        s["net"].forward_device(case["n"], s["X"].data_ptr(), s["Y"].data_ptr())
        return s["Y"]
    if kind == "loop":
        # Training from the program's initial parameters with the loop's own split, minibatches and validation.
        s["net"].set_params(s["start"])
        log = proposal.train(s["net"], s["X"], s["T"], case["steps"], case["batch"], 3e-4, seed=s["seed"],
                             eval_every=case["steps"])
        return {"losses": np.array(log.losses, dtype=np.float32), "validation": np.array([v for _, v in log.val], np.float32),
                "params": s["net"].get_params()}
    B = case["batch"]
    losses = [s["net"].train_step_device(B, s["X"][k * B:].data_ptr(), s["T"][k * B:].data_ptr(), 3e-4)
              for k in range(case["steps"])]
    return {"losses": np.array(losses, dtype=np.float32), "params": s["net"].get_params()}


# ---------------------------------------------------------------------------
# 64-bit values.
# ---------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "edges":
        return _exact_clearance(case, seed) if case["mode"] == "clearance" else None
    if kind == "forward":
        X, _ = _samples(case["n"], seed, True)
        return _network(_layers(proposal.init_params(seed)), X.double())[0].cpu().numpy()
    if kind == "steps":
        X, T = _samples(case["batch"] * case["steps"], seed, True)
        net, B = _Trainer(proposal.init_params(seed)), case["batch"]
        losses = [net.step(X[k * B:(k + 1) * B], T[k * B:(k + 1) * B]) for k in range(case["steps"])]
        return {"losses": np.array(losses), "params": net.flat()}
    if kind == "loop":
        # proposal.train's split, minibatches and choice of the best parameters.
        X, T = (torch.as_tensor(x, device="cuda") for x in _samples(case["samples"], seed, False))
        rng, n = np.random.default_rng(seed), case["samples"]
        perm = rng.permutation(n)
        nv = int(round(0.15 * n)) if n >= 8 else 0
        vi, ti = perm[:nv], perm[nv:]
        net = _Trainer(proposal.init_params(seed))
        first = net.flat()
        val, losses = [net.loss(X[vi], T[vi])], []
        for _ in range(case["steps"]):
            idx = ti[rng.integers(0, len(ti), size=min(case["batch"], len(ti)))]
            losses.append(net.step(X[idx], T[idx]))
        val.append(net.loss(X[vi], T[vi]))
        return {"losses": np.array(losses), "validation": np.array(val),
                "params": net.flat() if val[1] < val[0] else first}
    return None  # a randomised search: its decisions are compared as they are


def _exact_clearance(case, seed):
    world, _, edges = _edges(case, seed)
    qa, ta, qb, tb = (x.double() for x in edges)
    dev = dict(device="cuda", dtype=torch.float64)
    D = (qb - qa).norm(dim=1)
    L = torch.maximum(D, world["v_max"] * (tb - ta).abs())
    count = torch.clamp(torch.ceil(L / RES - 1e-3), min=1).long()
    way = torch.tensor(world["obs_way"], **dev)
    radius = torch.tensor(world["obs_radius"], **dev)
    spheres = torch.tensor(world["spheres"], **dev)
    out = torch.full((case["n"],), math.inf, **dev)
    points = 20000000 // (len(spheres) * len(radius))
    edge = torch.repeat_interleave(torch.arange(case["n"], device="cuda"), count)
    first = torch.cumsum(count, 0) - count
    for i in range(0, len(edge), points):
        e = edge[i:i + points]
        f = (torch.arange(i, i + len(e), device="cuda") - first[e] + 1).double() / count[e]
        q, t = qa[e] + f[:, None] * (qb[e] - qa[e]), ta[e] + f * (tb[e] - ta[e])
        # Obstacles: piecewise linear, held outside their waypoints.
        tc = torch.minimum(torch.maximum(t[:, None], way[None, :, 0, 0]), way[None, :, -1, 0])
        k = (way[None, :, 1:-1, 0] <= tc[:, :, None]).sum(2)
        m = torch.arange(len(radius), device="cuda")[None]
        w0, w1 = way[m, k], way[m, k + 1]
        o = w0[..., 1:] + ((tc - w0[..., 0]) / (w1[..., 0] - w0[..., 0]))[..., None] * (w1[..., 1:] - w0[..., 1:])
        c = _centres(world, spheres, q)
        gap = (c[:, :, None] - o[:, None]).norm(dim=3) - spheres[None, :, 4, None] - radius
        out.scatter_reduce_(0, e, gap.flatten(1).amin(1), "amin")
    return {"verdict": None, "clearance": out.cpu().numpy(), "checks": None}


def _centres(world, spheres, q):
    """Sphere centres of configurations q [n][dof] (standard DH forward kinematics)."""
    if not world["arm"]:
        p = torch.zeros(len(q), 1, 3, device="cuda", dtype=torch.float64)
        p[:, 0, :2] = q
        return p + spheres[None, :, 1:4]
    F = torch.eye(4, device="cuda", dtype=torch.float64).repeat(len(q), 1, 1)
    local = torch.cat([spheres[:, 1:4], torch.ones_like(spheres[:, :1])], 1)
    frame = spheres[:, 0].long().tolist()
    out = [None] * len(spheres)
    for j in range(world["dof"] + 1):
        if j > 0:
            a, alpha, d, off = world["dh"][j - 1]
            c, s = torch.cos(q[:, j - 1] + off), torch.sin(q[:, j - 1] + off)
            ca, sa, z = math.cos(alpha), math.sin(alpha), torch.zeros_like(c)
            A = torch.stack([c, -s * ca, s * sa, a * c, s, c * ca, -c * sa, a * s, z, z + sa, z + ca, z + d,
                             z, z, z, z + 1], 1).view(-1, 4, 4)
            F = F @ A
        for i, f in enumerate(frame):
            if f == j:
                out[i] = (F[:, :3] @ local[i])
    return torch.stack(out, 1)


_SHAPES = ((256, 32), (256,), (256, 256), (256,), (256, 256), (256,), (160, 256), (160,))


def _layers(flat):
    out, o = [], 0
    for shape in _SHAPES:
        n = math.prod(shape)
        out.append(torch.tensor(flat[o:o + n], device="cuda", dtype=torch.float64).view(shape))
        o += n
    return out


def _network(p, x):
    for k in range(4):
        x = x @ p[2 * k].T + p[2 * k + 1]
        if k < 3:
            x = torch.relu(x)
    return x, p


class _Trainer:
    """The network, its loss and Adam in 64 bits."""

    def __init__(self, flat):
        self.p = [x.requires_grad_() for x in _layers(flat)]
        self.m, self.v, self.k = [torch.zeros_like(x) for x in self.p], [torch.zeros_like(x) for x in self.p], 0

    def _loss(self, X, T):
        y, T = _network(self.p, X.double())[0], T.double()
        a, mu, s = y[:, :8], y[:, 8:16], torch.clamp(y[:, 16:24], -7, 2)
        z = (T[:, :1] - mu) / torch.exp(s)
        nll = -torch.logsumexp(torch.log_softmax(a, 1) - 0.5 * z * z - s - 0.5 * math.log(2 * math.pi), 1)
        use = torch.arange(8, device="cuda")[None] < T[:, 129:130]
        use[:, 7] = True
        err = (y[:, 24:152] - T[:, 1:129]).view(-1, 16, 8) * use[:, None]
        return (nll + (err * err).sum((1, 2)) / (16 * use.sum(1))).mean()

    def loss(self, X, T):
        with torch.no_grad():
            return float(self._loss(X, T))

    def step(self, X, T):
        loss = self._loss(X, T)
        grads = torch.autograd.grad(loss, self.p)
        self.k += 1
        with torch.no_grad():
            for i, (w, g) in enumerate(zip(self.p, grads)):
                if i >= 6:
                    g[152:] = 0
                self.m[i] = 0.9 * self.m[i] + 0.1 * g
                self.v[i] = 0.999 * self.v[i] + 0.001 * g * g
                w -= 3e-4 * (self.m[i] / (1 - 0.9 ** self.k)) / ((self.v[i] / (1 - 0.999 ** self.k)).sqrt() + 1e-8)
        return float(loss.detach())

    def flat(self):
        return torch.cat([x.detach().reshape(-1) for x in self.p]).cpu().numpy()


# ---------------------------------------------------------------------------
# Work that a pass cannot do without.
# ---------------------------------------------------------------------------
def _point_flops(robot, obs):
    """One check point: pair tests of 8 operations, sphere transforms, forward kinematics, interpolation."""
    S, d = SPHERES[robot], DOF[robot]
    return 8.0 * S * obs + (18.0 * S + 60.0 * d if robot != "disc2d" else 2.0 * S) + 9.0 * obs


def work(case):
    kind = case["kind"]
    if kind == "edges":
        # Every edge read, its results written, and at least one check point of it evaluated.
        real = 8 if case["precision"] else 4
        extra = (real if case["mode"] == "clearance" else 0) + (4 if case["host"] else 0)
        n = case["n"]
        return {"bytes": float(n * (2 * (DOF[case["robot"]] + 1) * real + 1 + extra)),
                "flops": n * _point_flops(case["robot"], case["obs"])}
    if kind == "plan":
        # Every worker's extension: at least one check point evaluated, its node written.
        n = case["workers"] * case["iters"]
        return {"bytes": 32.0 * n, "flops": n * _point_flops(case["robot"], case["obs"])}
    if kind == "batch":
        n = case["workers"] * case["iters"] * case["n"] / 3
        return {"bytes": 96.0 * n,
                "flops": n * (_point_flops("disc2d", 18) + _point_flops("ur5e", 66) + _point_flops("arm7", 66))}
    macs = 256 * 32 + 2 * 256 * 256 + 160 * 256
    if kind == "forward":
        n = case["n"]
        return {"bytes": 4.0 * (n * (32 + 160) + stp.MLP_NPARAM), "flops": 2.0 * n * macs}
    # Training: samples read, parameters and both moments read and written.
    per = 4.0 * (case["batch"] * (32 + 130) + 6 * stp.MLP_NPARAM)
    return {"bytes": per * case["steps"],
            "flops": 2.0 * case["batch"] * case["steps"] * (macs + 2 * macs - 256 * 32)}
