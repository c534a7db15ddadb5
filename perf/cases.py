"""Workloads of the flight-plan scheduler, as its users run them.

Every case is one call (or one short sequence of calls) of the Python API that mirrors the
C ABI: a separation check of a filed trajectory, a request planned on its own, batches,
departure candidates, co-simulation, the lookahead window, a serving burst, and the learned
proposal's training gradient and rollouts. Airspaces, known plans and requests have the
shapes of scenarios.py (C1, C2, C3, C4, E1); the known plans are made by one vectorised
generator here, so that a table of 100 000 plans is ready in well under a second.

Calls that admit plans start from the same table each time: the plan table is restored to
its snapshot first (fmdp_restore), as a what-if run over a live table does. The results of
the scheduler do not depend on timing; the number of speculative re-plans does, and is not
returned.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2008_03518_gb300 import scenarios as S
from paper_2008_03518_gb300.fmdp import MLP_PARAMS, Scheduler

WINDOW = 4096
WELLS = [(t, 300.0 + 10.0 * t, 1000.0, 0.97) for t in (-5.0, 0.0, 5.0, 10.0, 15.0)]
LAYERS = ((128, 256), (256, 256), (256, 256), (256, 256), (256, 25))


def listed():
    return [
        # an external plan checked against a small airport's traffic: the smallest call
        dict(name="check_200", kind="check", area="small", plans=200, samples=311),
        # the same check against a metropolitan table of short hops
        dict(name="check_100k", kind="check", area="hops", plans=100000, samples=1791),
        # one request planned, checked and admitted while its user waits
        dict(name="request_3k", kind="request", area="metro", plans=3000),
        # a day's requests: known plans loaded from host memory, then planned first come, first
        # served through speculative batches (the end-to-end benchmark)
        dict(name="day_3k", kind="day", area="metro", plans=3000, requests=1000),
        # a dense table and requests of uneven horizon, most of them independent
        dict(name="batch_20k", kind="batch", area="metro", plans=20000, requests=512),
        # restricted volumes and the sum of penalties, a crowded small airspace
        dict(name="restricted_200", kind="restricted", area="small", plans=200, requests=48, wells=12),
        # a burst of arrivals served against the largest table
        dict(name="serve_100k", kind="serve", area="hops", plans=100000, requests=512),
        # each request's departure chosen among eight minutes
        dict(name="departures_3k", kind="departures", area="metro", plans=3000, requests=64, delays=8),
        # the paper's own fidelity: 0.1 s steps, ten sub-steps ahead
        dict(name="lookahead_60", kind="lookahead", area="fine", plans=60, requests=4, window=10),
        # aircraft of one batch that see one another while they plan
        dict(name="cosim_3k", kind="cosim", area="metro", plans=3000, requests=128),
        # loss and gradient of the proposal network on one training batch
        dict(name="gradient_2048", kind="gradient", rows=2048),
        # proposals of the network and FastMDP's plans, side by side
        dict(name="proposals_20k", kind="proposals", area="metro", plans=20000, requests=256),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["check", "check", "request", "day", "batch", "batch", "restricted", "serve", "departures",
                       "lookahead", "cosim", "gradient", "proposals"])
    if kind == "check":
        area = rng.choice(["small", "metro", "hops"])
        plans = log_int(50, {"small": 1000, "metro": 20000, "hops": 100000}[area])
        return dict(kind=kind, area=area, plans=plans, samples=log_int(40, 1800))
    if kind == "request":
        return dict(kind=kind, area="metro", plans=log_int(200, 20000))
    if kind == "day":
        return dict(kind=kind, area="metro", plans=log_int(200, 3000), requests=log_int(16, 700))
    if kind == "batch":
        return dict(kind=kind, area="metro", plans=log_int(1000, 20000), requests=log_int(16, 512))
    if kind == "restricted":
        return dict(kind=kind, area="small", plans=log_int(50, 400), requests=log_int(4, 64), wells=log_int(2, 40))
    if kind == "serve":
        return dict(kind=kind, area="hops", plans=log_int(2000, 100000), requests=log_int(32, 512))
    if kind == "departures":
        return dict(kind=kind, area="metro", plans=log_int(200, 3000), requests=log_int(4, 64), delays=rng.randint(2, 8))
    if kind == "lookahead":
        return dict(kind=kind, area="fine", plans=log_int(10, 150), requests=rng.randint(1, 4), window=rng.randint(2, 16))
    if kind == "cosim":
        return dict(kind=kind, area="metro", plans=log_int(200, 3000), requests=log_int(4, 128))
    if kind == "gradient":
        return dict(kind=kind, rows=log_int(32, 8192))
    return dict(kind=kind, area="metro", plans=log_int(1000, 20000), requests=log_int(16, 256))


# ------------------------------------------------------------------ inputs


def airspace(area):
    """The fixed part of a scenario: box, step, actions, terrain (as scenarios.py has them)."""
    if area == "small":
        return SimpleNamespace(box=(0.0, 0.0, 0.0, 10000.0, 10000.0, 500.0), dt=1.0, heightmap=None, clearance=0.0,
                               actions=S.action_grid((-2.0, 0.0, 2.0)), window=2048)
    if area == "fine":
        return SimpleNamespace(box=(0.0, 0.0, 0.0, 4000.0, 4000.0, 500.0), dt=0.1, heightmap=None, clearance=0.0,
                               actions=S.action_grid((-2.0, 0.0, 2.0)), window=WINDOW)
    return SimpleNamespace(box=(0.0, 0.0, 0.0, 30000.0, 30000.0, 1000.0), dt=1.0, heightmap=S.fractal_heightmap(102),
                           clearance=60.0, actions=S.action_grid((-4.0, -2.0, 0.0, 2.0, 4.0)), window=WINDOW)


def cell_top(air, x, y):
    """Highest heightmap node of the grid cell of each point."""
    hm, box = air.heightmap, air.box
    ix = np.clip(((x - box[0]) / (box[3] - box[0]) * (hm.shape[1] - 1)).astype(np.int64), 0, hm.shape[1] - 2)
    iy = np.clip(((y - box[1]) / (box[4] - box[1]) * (hm.shape[0] - 1)).astype(np.int64), 0, hm.shape[0] - 2)
    return np.maximum(np.maximum(hm[iy, ix], hm[iy, ix + 1]), np.maximum(hm[iy + 1, ix], hm[iy + 1, ix + 1]))


def routes(rng, area, air, n):
    """Way points [n][K + 1][3], legs used, speed and departure step of n known plans."""
    box = air.box
    speed = rng.uniform(20.0, 40.0, n)
    if area in ("small", "fine"):  # straight flights between uniform points
        zlo, zhi = (50.0, 450.0) if area == "small" else (100.0, 400.0)
        pts = np.stack([rng.uniform(box[0], box[3], (n, 2)), rng.uniform(box[1], box[4], (n, 2)),
                        rng.uniform(zlo, zhi, (n, 2))], axis=2)
        return pts, np.ones(n, dtype=np.int64), speed, rng.integers(0, 601, n)
    lo, hi, near, far, late = (3, 6, 3000.0, 9000.0, 1800) if area == "metro" else (1, 2, 2000.0, 6000.0, 3000)
    x, y = rng.uniform(box[0], box[3], n), rng.uniform(box[1], box[4], n)
    pts = np.zeros((n, hi + 1, 3))
    for i in range(hi + 1):
        if i:
            turn, leg = rng.uniform(0.0, 2.0 * np.pi, n), rng.uniform(near, far, n)
            x, y = x + leg * np.cos(turn), y + leg * np.sin(turn)
            x = np.clip(np.where(x < box[0], 2 * box[0] - x, np.where(x > box[3], 2 * box[3] - x, x)), box[0], box[3])
            y = np.clip(np.where(y < box[1], 2 * box[1] - y, np.where(y > box[4], 2 * box[4] - y, y)), box[1], box[4])
        pts[:, i, 0], pts[:, i, 1] = x, y
        pts[:, i, 2] = np.minimum(cell_top(air, x, y) + rng.uniform(60.0, 600.0, n), box[5] - 1.0)
    return pts, rng.integers(lo, hi + 1, n), speed, rng.integers(0, late + 1, n)


def fly(pts, legs, speed, dt):
    """Samples every speed x dt metres along each route, ending at its end: (counts, xyz fp32)."""
    P = torch.as_tensor(pts, device="cuda")
    legs, step = torch.as_tensor(legs, device="cuda"), torch.as_tensor(speed * dt, device="cuda")
    n, K = P.shape[0], P.shape[1] - 1
    seg = P[:, 1:] - P[:, :-1]
    length = seg.square().sum(2).sqrt() * (torch.arange(K, device="cuda")[None] < legs[:, None])
    cum = torch.cat([torch.zeros(n, 1, device="cuda", dtype=torch.float64), length.cumsum(1)], 1)
    full = torch.floor(cum[:, -1] / step).to(torch.int64)
    count = full + 1 + ((cum[:, -1] - full * step) > 1e-9)
    of = torch.repeat_interleave(torch.arange(n, device="cuda"), count)
    k = torch.arange(of.numel(), device="cuda") - (count.cumsum(0) - count)[of]
    s = torch.minimum(k * step[of], cum[of, -1])
    leg = torch.zeros_like(of)
    for i in range(1, K):
        leg += (s >= cum[of, i]) & (i < legs[of])
    frac = (s - cum[of, leg]) / length[of, leg].clamp_min(1e-300)
    xyz = P[of, leg] + seg[of, leg] * frac[:, None]
    return count.to(torch.int32).cpu().numpy(), xyz.float().cpu().numpy()


def traffic(rng, case, air):
    """Known plans in the packed form of the API: first steps, sample counts, samples."""
    pts, legs, speed, t0 = routes(rng, case["area"], air, case["plans"])
    counts, xyz = fly(pts, legs, speed, air.dt)
    return np.minimum(t0, air.window - counts).astype(np.int64), counts, xyz


def requests(rng, case, air):
    kind, n = case["kind"], case.get("requests", 1)
    if kind == "lookahead":
        return S.make_requests(rng, air.box, n, zlo=100.0, zhi=400.0, tlo=0, thi=600, horizon=3000)
    if kind == "restricted":  # flights that leave the centre towards all sides within half a minute
        req = S.make_requests(rng, air.box, n, zlo=150.0, zhi=350.0, tlo=0, thi=30, horizon=900)
        for o, g in (("ox", "gx"), ("oy", "gy")):
            req[o] = 5000.0 + (req[o] - 5000.0) * 0.3
            req[g] = 5000.0 + (req[g] - 5000.0) * 0.85
        return req
    common = dict(hm=air.heightmap, zspan=(60.0, 500.0), tlo=0, thi=1800)
    if kind in ("batch", "proposals"):
        return S.make_requests(rng, air.box, n, horizon_range=(60, 1800), reach_frac=0.8, **common)
    return S.make_requests(rng, air.box, n, horizon=1800, **common)


def network(rng):
    """Parameters of a proposal network that steers for the goal (as a trained one does), with
    noise on every weight."""
    unit = lambda i: np.sqrt(2.0 / i)  # noqa: E731
    W = [rng.normal(0.0, 0.08 * unit(i), (i, o)) for i, o in LAYERS]
    b = [rng.normal(0.0, 0.01, o) for _, o in LAYERS]
    for j, (f, sign) in enumerate([(6, 1.0), (6, -1.0), (7, 1.0), (7, -1.0), (4, 1.0), (4, -1.0)]):
        W[0][f, j] += sign  # bearing of the goal (cos, sin) and its height, both signs
        for l in (1, 2, 3):
            W[l][j, j] += 1.0
    for a, (turn, climb) in enumerate(S.action_grid((-4.0, -2.0, 0.0, 2.0, 4.0))):
        c, s = math.cos(math.radians(turn)), math.sin(math.radians(turn))
        for j, w in enumerate((30.0 * c, -30.0 * c, 30.0 * s, -30.0 * s, climb, -climb)):
            W[4][j, a] += w
        b[4][a] -= 0.1 * climb * climb
    flat = np.concatenate([np.concatenate([w.ravel(), v]) for w, v in zip(W, b)]).astype(np.float32)
    assert flat.size == MLP_PARAMS
    return flat


def training_rows(rng, n):
    """Feature rows as collected ones look (own terms; a third of the sectors hold a plan), in bf16
    values, and the actions taken."""
    X = np.zeros((n, 128), dtype=np.float32)
    X[:, :8] = rng.uniform(-1.0, 1.0, (n, 8))
    held = rng.uniform(size=(n, 20, 1)) < 0.33
    X[:, 8:] = (held * rng.normal(0.0, 0.4, (n, 20, 6))).reshape(n, 120)
    return torch.from_numpy(X).bfloat16().float().numpy(), rng.integers(0, 25, n).astype(np.uint8)


def filed_trajectory(rng, case, air):
    """A trajectory of the given number of samples along a straight line that turns once."""
    box, n = air.box, case["samples"]
    m = np.array([0.25 * (box[3] - box[0]), 0.25 * (box[4] - box[1])])
    a, b, c = (rng.uniform(box[:2] + m, np.array(box[3:5]) - m) for _ in range(3))
    t = np.linspace(0.0, 2.0, n)[:, None]
    xy = np.where(t < 1.0, a + (b - a) * t, b + (c - b) * (t - 1.0))
    z = rng.uniform(150.0, 400.0) + 20.0 * np.sin(np.linspace(0.0, 6.0, n))
    return int(rng.integers(0, 120)), np.concatenate([xy, z[:, None]], axis=1).astype(np.float32)


def inputs(case, seed):
    """Everything a case is made of, as plain arrays."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "gradient":
        return SimpleNamespace(params=network(rng), rows=training_rows(rng, case["rows"]))
    air = airspace(case["area"])
    d = SimpleNamespace(air=air, plans=traffic(rng, case, air))
    if case["kind"] == "check":
        d.filed = filed_trajectory(rng, case, air)
        return d
    if case["kind"] == "serve":
        d.requests = S.serving_requests(air, np.zeros(case["requests"]), seed, time_scale=60.0, sim_start=600)
        return d
    d.requests = requests(rng, case, air)
    if case["kind"] == "restricted":  # x, y, z, radius, magnitude, decay
        n, box = case["wells"], air.box
        d.statics = np.stack([rng.uniform(box[0], box[3], n), rng.uniform(box[1], box[4], n), rng.uniform(0.0, 300.0, n),
                              rng.uniform(150.0, 500.0, n), rng.uniform(300.0, 900.0, n), np.full(n, 0.98)], axis=1)
    if case["kind"] == "proposals":
        d.params = network(rng)
    return d


# ------------------------------------------------------------------ the calls


def prepare(case, seed):
    d = inputs(case, seed)
    st = SimpleNamespace(kind=case["kind"], case=case)
    if case["kind"] == "gradient":  # the network's own context: no traffic
        air = airspace("small")
        st.s = Scheduler(air.box, air.dt, 0.99, S.action_grid((-4.0, -2.0, 0.0, 2.0, 4.0)), (150.0, 30.0),
                         n_slices_window=64, max_slots=64)
        st.s.learned_set_params(d.params)
        st.X, st.y = d.rows
        return st
    air = d.air
    extra = {}
    if case["kind"] == "restricted":
        extra = dict(static_wells=d.statics, combine=1)
    if case["kind"] == "lookahead":
        extra = dict(lookahead_W=case["window"])
    st.s = Scheduler(air.box, air.dt, 0.99, air.actions, (150.0, 30.0), n_slices_window=air.window,
                     max_slots=case["plans"] + 2 * case.get("requests", 1) + 128, heightmap=air.heightmap,
                     clearance=air.clearance, **extra)
    t0s, counts, xyz = d.plans
    if case["kind"] == "day":  # the user's plan database, in pinned host memory
        st.plans = [torch.from_numpy(a).pin_memory() for a in (t0s, counts, xyz)]
    else:
        st.s.add_plans_packed(t0s, counts, xyz)
    if case["kind"] == "check":
        st.t0, st.xyz = d.filed
        return st
    st.requests = d.requests
    if case["kind"] == "proposals":
        st.s.learned_set_params(d.params)
    elif case["kind"] != "day":
        st.s.snapshot()
    return st


def columns(results, horizon=1800):
    """Results of a scheduling call as arrays (without what depends on timing: re-plans); the
    trajectories of all requests in one array each for samples and actions, zero past their ends."""
    out = {k: np.array([r[k] for r in results], dtype=np.int64)
           for k in ("verdict", "n_points", "plan_id", "first_conflict_step", "first_terrain_step", "near_ties")}
    out.update({k: np.array([r[k] for r in results]) for k in ("min_sep_h", "min_sep_v")})
    out["xyz"] = np.zeros((len(results), horizon + 1, 3), dtype=np.float32)
    out["actions"] = np.zeros((len(results), horizon), dtype=np.uint8)
    for xyz, actions, r in zip(out["xyz"], out["actions"], results):
        xyz[: len(r["xyz"])] = r["xyz"]
        actions[: len(r["actions"])] = r["actions"]
    return out


def run(st):
    s, kind = st.s, st.kind
    if kind == "check":
        return s.sep_check(st.t0, st.xyz)
    if kind == "gradient":
        loss, grad = s.learned_loss_grad(st.X, st.y)
        return {"loss": loss, "gradient": grad}
    if kind == "proposals":
        report, accepted, steps_p, steps_f = s.learned_evaluate(st.requests)
        return {"accepted": accepted, "steps_proposed": steps_p, "steps_fastmdp": steps_f,
                "captured": report["proposals_captured"], "mean_gap": report["mean_gap"]}
    if kind == "day":
        s.clear()
        s.add_plans_packed(*(t.numpy() for t in st.plans))
        out = columns(s.schedule_batch(st.requests))
        del out["plan_id"]  # ids go on counting over the table's life
        return out
    s.restore()
    if kind == "request":
        return columns([s.schedule(st.requests[0])])
    if kind == "serve":
        arrivals = np.zeros(len(st.requests))
        results, _, _ = s.serve(st.requests, arrivals, time_scale=60.0, max_in_flight=256, sim_start_step=600)
        return columns(results)
    if kind == "departures":
        results, chosen, verdicts = s.schedule_departures(st.requests, [60 * d for d in range(st.case["delays"])],
                                                          batched=True)
        return dict(columns(results), chosen=chosen, verdicts=verdicts)
    if kind == "lookahead":
        return columns(s.schedule_many(st.requests), 3000)
    if kind == "cosim":
        return columns(s.schedule_cosim(st.requests))
    return columns(s.schedule_batch(st.requests))


# ------------------------------------------------------------------ what a pass cannot do without

SAMPLES = {"small": 170.0, "metro": 880.0, "hops": 200.0, "fine": 700.0}  # mean samples of a known plan
STEPS = {"small": 130.0, "metro": 500.0, "hops": 320.0, "fine": 650.0}    # mean steps of a planned request
SPAN = {"small": 750.0, "metro": 2700.0, "hops": 3200.0, "fine": 1300.0}  # steps the known plans cover


def work(case):
    """Known samples of the rows a call reads, each once (12 bytes), its inputs and its results; per
    rollout step and action some 60 operations of goal term and terrain, and per near plan sample five
    wells of 10 operations for each action. Restoring a table moves its samples once more."""
    kind = case["kind"]
    if kind == "gradient":
        rows, flops = case["rows"], sum(i * o for i, o in LAYERS)
        return {"bytes": rows * 128 * 4.0 + 2 * 4.0 * MLP_PARAMS, "flops": 2.0 * rows * (3 * flops - 128 * 256)}
    area, plans = case["area"], case["plans"]
    samples = plans * SAMPLES[area]
    if kind == "check":
        pairs = samples / SPAN[area] * min(case["samples"], SPAN[area])
        return {"bytes": 12.0 * (pairs + case["samples"]), "flops": 10.0 * pairs}
    steps = STEPS[area] * case["requests"] if "requests" in case else STEPS[area]
    steps *= case.get("delays", 1) * (2.0 if kind in ("lookahead", "proposals") else 1.0)
    acts = 15 if area in ("small", "fine") else 25
    air = {"small": 10.0, "metro": 30.0, "hops": 30.0, "fine": 4.0}[area]
    near = samples / SPAN[area] * min(1.0, 1.2 / (air * air))  # samples whose wells reach, per step
    sub = case.get("window", 1)
    flops = steps * sub * acts * (60.0 + 50.0 * near)
    rows = 1.0 if kind != "request" else STEPS[area] / SPAN[area]
    return {"bytes": 12.0 * samples * (rows + (0.0 if kind == "proposals" else 2.0)) + 25.0 * steps, "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits, by plain numpy


def terrain(air, x, y):
    hm, box = air.heightmap.astype(np.float64), air.box
    fx = (x - box[0]) / (box[3] - box[0]) * (hm.shape[1] - 1)
    fy = (y - box[1]) / (box[4] - box[1]) * (hm.shape[0] - 1)
    ix = np.clip(np.floor(fx).astype(np.int64), 0, hm.shape[1] - 2)
    iy = np.clip(np.floor(fy).astype(np.int64), 0, hm.shape[0] - 2)
    ax, ay = fx - ix, fy - iy
    return (1 - ay) * ((1 - ax) * hm[iy, ix] + ax * hm[iy, ix + 1]) + ay * ((1 - ax) * hm[iy + 1, ix] + ax * hm[iy + 1, ix + 1])


def exact_check(air, plans, t0, path):
    """Conflicts and least separations of one trajectory against every known sample of its steps."""
    t0s, counts, xyz = plans
    at = np.repeat(t0s - (np.cumsum(counts) - counts), counts) + np.arange(len(xyz)) - t0  # index into the trajectory
    held = (at >= 0) & (at < len(path))
    at, d = at[held], path.astype(np.float64)[at[held]] - xyz[held].astype(np.float64)
    h, v = np.hypot(d[:, 0], d[:, 1]), np.abs(d[:, 2])
    both = (h < 150.0) & (v < 30.0)
    low = np.flatnonzero(path[:, 2] < terrain(air, path[:, 0].astype(float), path[:, 1].astype(float))) if air.heightmap is not None else []
    return {"first_conflict_step": int(at[both].min()) if both.any() else -1, "first_terrain_step": int(low[0]) if len(low) else -1,
            "conflicts": int(both.sum()), "min_sep_h": float(h[v < 30.0].min(initial=math.inf)),
            "min_sep_v": float(v[h < 150.0].min(initial=math.inf))}


def exact_request(air, plans, r):
    """One request flown by the greedy rule, every value in 64 bits, then checked."""
    t0s, counts, xyz = plans
    step_of = np.repeat(t0s - (np.cumsum(counts) - counts), counts) + np.arange(len(xyz))
    last = np.zeros(len(xyz), dtype=bool)
    last[np.cumsum(counts) - 1] = True
    order = np.argsort(step_of, kind="stable")
    first = np.searchsorted(step_of[order], np.arange(WINDOW + 2))
    s, goal = np.array([r["ox"], r["oy"], r["oz"]]), np.array([r["gx"], r["gy"], r["gz"]])
    step, bearing, h = float(r["speed"]), math.atan2(goal[1] - s[1], goal[0] - s[0]), 0
    path, acts, verdict = [s], [], 3
    if ((goal - s) ** 2).sum() <= step * step:
        verdict = 0
    while verdict == 3 and len(acts) < r["horizon"]:
        turn = [h + round(a / 15.0) for a, _ in air.actions]
        move = np.array([(step * math.cos(bearing + math.radians(15.0 * k)), step * math.sin(bearing + math.radians(15.0 * k)), c)
                         for k, (_, c) in zip(turn, air.actions)])
        nxt = s + move
        T = int(r["depart"]) + len(acts) + 1
        i = order[first[T]:first[T + 1]] if T <= WINDOW else order[:0]
        p = xyz[i].astype(np.float64)
        near = ((p - s) ** 2).sum(1) < 1500.0 ** 2
        i, p = i[near], p[near]
        vel = np.where(last[i][:, None], 0.0, xyz[np.minimum(i + 1, len(xyz) - 1)].astype(np.float64) - p)
        worst = np.zeros(len(move))
        for tau, R, mag, decay in WELLS:
            d = np.sqrt(((nxt[:, None] - (p + tau * vel)[None]) ** 2).sum(2))
            worst = np.maximum(worst, np.where(d < R, mag * decay ** d, 0.0).max(1, initial=0.0))
        c = nxt[:, 2] - terrain(air, nxt[:, 0], nxt[:, 1])
        q = 200.0 * 0.99 ** np.sqrt(((goal - nxt) ** 2).sum(1)) - worst - np.where(c < air.clearance, 1000.0 - c, 0.0)
        inside = ((nxt >= air.box[:3]) & (nxt <= air.box[3:])).all(1)
        if not inside.any():
            verdict = 4
            break
        a = int(np.argmax(np.where(inside, q, -np.inf)))
        s, h = nxt[a], turn[a]
        path.append(s)
        acts.append(a)
        if ((goal - s) ** 2).sum() <= step * step:
            verdict = 0
    path = np.array(path)
    chk = exact_check(air, plans, int(r["depart"]), path)
    flown = np.zeros((1, r["horizon"] + 1, 3))
    flown[0, :len(path)] = path
    return {"verdict": None, "n_points": None, "plan_id": None, "first_conflict_step": None, "first_terrain_step": None,
            "near_ties": None, "min_sep_h": np.array([chk["min_sep_h"]]), "min_sep_v": np.array([chk["min_sep_v"]]),
            "xyz": flown, "actions": None}


def exact_gradient(params, X, y):
    W, b, o = [], [], 0
    for i, k in LAYERS:
        W.append(params[o:o + i * k].reshape(i, k).astype(np.float64))
        b.append(params[o + i * k:o + i * k + k].astype(np.float64))
        o += i * k + k
    H = [X.astype(np.float64)]
    for l in range(4):
        H.append(np.maximum(H[-1] @ W[l] + b[l], 0.0))
    z = H[4] @ W[4] + b[4]
    z -= z.max(1, keepdims=True)
    p = np.exp(z) / np.exp(z).sum(1, keepdims=True)
    loss = -np.log(p[np.arange(len(y)), y]).mean()
    p[np.arange(len(y)), y] -= 1.0
    dz, parts = p / len(y), []
    for l in range(4, -1, -1):
        parts = [(H[l].T @ dz).ravel(), dz.sum(0)] + parts
        if l:
            dz = (dz @ W[l].T) * (H[l] > 0.0)
    return {"loss": float(loss), "gradient": np.concatenate(parts)}


def exact(case, seed):
    """In 64 bits: checks, one planned request and the gradient. A sequence of requests flown in plain
    numpy takes minutes, so those cases have none."""
    if case["kind"] not in ("check", "request", "gradient"):
        return None
    d = inputs(case, seed)
    if case["kind"] == "gradient":
        return exact_gradient(d.params, *d.rows)
    if case["kind"] == "check":
        return exact_check(d.air, d.plans, *d.filed)
    return exact_request(d.air, d.plans, d.requests[0])
