"""The workloads this planner's speed is measured on.

Each case is one call a planning program makes: an iteration from host arrays (the control loop
of one vehicle), an iteration on device tensors (a planner that lives beside other GPU work), a
submission of many uneven plans, or a burst of requests to the serving engine.  The scenes are
those of ``scenarios.py`` (lane lengths and spacings, obstacles of three circles, the paper's
costs), placed in a map frame: the lane starts somewhere and points somewhere, as a road does,
unless the case plans in the lane's own frame.  The warm start is a smooth manoeuvre, as an
earlier iteration leaves it.
"""
import math

import numpy as np
import torch

import paper_2308_01654_gb300 as mp

DEV = "cuda"


def listed():
    base = dict(call="plan", K=1024, T=50, dt=0.05, lane="straight", aligned=False, n_ref=200, n_obs=1,
                motion="static", bf16=False, rate=False, to_go=False, vertex=False, contact=False, tuned=False,
                plans=1)
    cases = [
        # one vehicle's control cycle at the smallest useful size, a planner used as constructed
        dict(base, name="cycle_1k"),
        # the paper's own setting: 2560 samples of 16 steps of 0.25 s, steering-rate model, speed cap
        dict(base, name="paper_rate_model", K=2560, T=16, dt=0.25, lane="curved", n_ref=600, n_obs=2, rate=True),
        # receding horizon on a winding lane in traffic with a per-step forecast of every obstacle
        dict(base, name="cycle_8k_forecast", K=8192, T=100, lane="curved", n_ref=1000, n_obs=8, motion="table",
             tuned=True),
        # odd sizes, nearest-vertex lane keeping and contact-only safety, obstacles at constant velocity
        dict(base, name="cycle_odd_vertex", K=3001, T=77, lane="curved", n_ref=481, n_obs=11, motion="moving",
             vertex=True, contact=True),
        # the same loop on device tensors, moving traffic on a straight road, a planner used as constructed
        dict(base, name="device_8k_moving", call="device", K=8192, T=100, n_ref=1000, n_obs=8, motion="moving"),
        # per-step cost-to-go weights
        dict(base, name="device_16k_to_go", call="device", K=16384, T=64, lane="curved", n_ref=1000, n_obs=8,
             to_go=True, tuned=True),
        # the planner's full-size iteration, in the lane's frame
        dict(base, name="device_64k", call="device", K=65536, T=200, dt=0.025, aligned=True, n_ref=2000, n_obs=64,
             tuned=True),
        # the same size with bfloat16 noise, on a road of any heading
        dict(base, name="device_64k_bf16", call="device", K=65536, T=200, dt=0.025, n_ref=2000, n_obs=64, bf16=True,
             tuned=True),
        # the most samples one plan is asked for, on a winding road: more noise than the cache holds
        dict(base, name="device_256k_curved", call="device", K=262144, T=100, lane="curved", n_ref=1000, n_obs=32,
             tuned=True),
        # a fleet's uneven plans in one submission
        dict(base, name="batch_256", call="batch", n_ref=1000, plans=256, tuned=True),
        # a small depot's submission, bfloat16 noise, launch shape as constructed
        dict(base, name="batch_12_bf16", call="batch", n_ref=1000, plans=12, bf16=True),
        # a burst of vehicles that ask the server for a plan at the same time
        dict(base, name="serve_burst_32", call="serve", n_ref=1000, plans=32, tuned=True),
    ]
    return cases


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    c = dict(call=rng.choice(["plan", "plan", "device", "device", "device", "batch", "serve"]), dt=0.05,
             lane=rng.choice(["straight", "curved"]), aligned=rng.random() < 0.25, bf16=rng.random() < 0.3,
             rate=False, to_go=False, vertex=False, contact=False, tuned=rng.random() < 0.6, plans=1)
    if c["call"] in ("batch", "serve"):
        # the plans' sizes (_scenes): K 2^10 .. 2^14, T 30 .. 150, 0 .. 32 obstacles, lanes of both kinds
        c.update(K=1024, T=50, n_obs=1, motion="static", lane="straight", aligned=False, n_ref=1000,
                 plans=_log_int(rng, 4, 200 if c["call"] == "batch" else 64))
        return c
    c["K"] = _log_int(rng, 512, 16384) if c["call"] == "plan" else _log_int(rng, 2048, 262144)
    c["T"] = _log_int(rng, 12, 256)
    while c["K"] * c["T"] > 65536 * 200:
        c["T"] = max(12, c["T"] // 2)
    c["n_ref"] = _log_int(rng, 100, 2000)
    c["n_obs"] = rng.choice([0, 1, 2, 5, 8, 13, 32, 64])
    c["motion"] = rng.choice(["static", "static", "moving", "table"])
    c["dt"] = 0.025 if c["T"] > 120 else 0.05
    form = rng.random()
    if form < 0.12:
        c.update(rate=True, dt=0.25, T=min(c["T"], 24))
    elif form < 0.22 and c["K"] * c["T"] <= 2_000_000:
        c["to_go"] = True
    elif form < 0.3:
        c["vertex"] = True
    if rng.random() < 0.1:
        c["contact"] = True
    return c


# ---------------------------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------------------------

def _params(K, T, dt, seed, session, rate, lam=None):
    sa, sd = (0.85, 0.05) if rate else (0.5, 0.05)
    lam = (150.0 if rate else 1.0) if lam is None else lam
    p = dict(K=K, T=T, dt=dt, wheelbase=2.7, sigma=[sa, sd], u_min=[-3.0, -0.5], u_max=[3.0, 0.5], lam=lam,
             gamma=1.0, R=[lam / (sa * sa), lam / (sd * sd)], w_dist=15.0, w_target=7.0, w_yaw=120.0, w_speed=5.0,
             w_safe=25.0, w_terminal=0.0, v_ref=30.0 / 3.6, v_max=math.inf, d_safe_c=0.0, d_safe_0=0.5,
             collision_only=0, n_ego=3, ego_offset=[0.0, 1.35, 2.7], ego_radius=[1.1, 1.1, 1.1], ref_mode=0,
             sg_enable=1, shift=0, noise_bf16=0, seed=seed, session=session, model=0, cost_to_go=0)
    if rate:
        p.update(model=1, u_min=[-2.5, -0.11], u_max=[1.1, 0.11], d_safe_c=1.36, d_safe_0=11.0, v_max=30.0 / 3.6)
    return p


def _lane(kind, n, spacing):
    xs = spacing * np.arange(n, dtype=np.float64)
    return np.stack([xs, 3.0 * np.sin(2.0 * np.pi * xs / 80.0) if kind == "curved" else np.zeros(n)], axis=1)


def _obstacles(rng, ref, n_obs, x_hi, lateral, moving):
    """Car-like objects of three circles along the lane's tangent (rows x, y, r, vx, vy)."""
    rows = []
    for j in range(n_obs):
        x, lat, r = rng.uniform(8.0, x_hi), rng.uniform(-lateral, lateral), rng.uniform(0.8, 1.2)
        i = int(np.clip(np.searchsorted(ref[:, 0], x) - 1, 0, len(ref) - 2))
        d = (ref[i + 1] - ref[i]) / np.linalg.norm(ref[i + 1] - ref[i])
        p = ref[i] + (x - ref[i, 0]) / max(ref[i + 1, 0] - ref[i, 0], 1e-9) * (ref[i + 1] - ref[i])
        speed = rng.uniform(0.0, 10.0) if moving and j % 2 else 0.0
        for o in (-1.5, 0.0, 1.5):
            q = p + lat * np.array([-d[1], d[0]]) + o * d
            rows.append([q[0], q[1], r, speed * d[0], speed * d[1]])
    return np.asarray(rows, dtype=np.float64).reshape(-1, 5)


def _forecast(circles, T, dt):
    s = (np.arange(T, dtype=np.float64) + 1.0) * dt
    return np.ascontiguousarray(np.stack([circles[None, :, 0] + circles[None, :, 3] * s[:, None],
                                          circles[None, :, 1] + circles[None, :, 4] * s[:, None]], axis=2))


def _place(rng, sc, aligned):
    """The scene in the map: turned and moved as a road lies (rows of points, velocities, yaw)."""
    if aligned:
        return sc
    a, o = rng.uniform(-math.pi, math.pi), rng.uniform(-400.0, 400.0, 2)
    R = np.array([[math.cos(a), math.sin(a)], [-math.sin(a), math.cos(a)]])
    sc["ref"] = sc["ref"] @ R + o
    sc["circles"] = np.concatenate([sc["circles"][:, :2] @ R + o, sc["circles"][:, 2:3], sc["circles"][:, 3:] @ R],
                                   axis=1)
    sc["x0"][:2] = sc["x0"][:2] @ R + o
    sc["x0"][2] += a
    return sc


def _scene(rng, p, lane, n_ref, n_obs, motion, aligned):
    """One plan's inputs as numpy arrays (binary64)."""
    spacing = 0.1 if n_ref >= 1500 else 0.5
    ref = _lane(lane, n_ref, spacing)
    x_hi = max(20.0, min(300.0, ref[-1, 0]))
    lateral = 5.0 if n_obs > 32 else 3.0
    yaw0 = math.atan2(ref[1, 1] - ref[0, 1], ref[1, 0] - ref[0, 0])
    v0 = 7.0 if p["model"] == 1 else rng.uniform(5.0, 10.0)
    x0 = np.array([0.0, rng.uniform(-0.5, 0.5), yaw0, v0] + ([0.0] if p["model"] == 1 else []))
    sc = dict(params=p, x0=x0, ref=ref, circles=_obstacles(rng, ref, n_obs, x_hi, lateral, motion != "static"))
    sc = _place(rng, sc, aligned)
    sc["centres"] = _forecast(sc["circles"], p["T"], p["dt"]) if motion == "table" and n_obs else None
    t = np.arange(p["T"]) * p["dt"]
    f, g = rng.uniform(0.5, 2.0, 2)
    steer = 0.02 if p["model"] == 1 else 0.03
    sc["U"] = np.stack([0.4 * np.sin(f * t), steer * np.sin(g * t + 0.5)], axis=1)
    for k in ("x0", "ref", "circles"):
        sc[k] = np.ascontiguousarray(sc[k])
    return sc


def _scenes(case, seed):
    rng = np.random.Generator(np.random.PCG64([int(seed), 2308]))
    if case["call"] in ("batch", "serve"):
        # the plans' sizes belong to the case, their scenes to the seed
        sizes = np.random.Generator(np.random.PCG64([case["plans"], 2308]))
        out = []
        for i in range(case["plans"]):
            p = _params(1 << int(sizes.integers(10, 15)), int(sizes.integers(30, 151)), 0.05, int(seed), i, False)
            p.update(noise_bf16=int(case["bf16"]), shift=int(case["call"] == "serve"))
            out.append(_scene(rng, p, "curved" if i % 2 else "straight", case["n_ref"], int(sizes.integers(0, 33)),
                              "static", False))
        return out
    p = _params(case["K"], case["T"], case["dt"], int(seed), 0, case["rate"])
    p.update(noise_bf16=int(case["bf16"]), cost_to_go=int(case["to_go"]), ref_mode=int(case["vertex"]),
             collision_only=int(case["contact"]), shift=int(case["call"] == "plan"))
    return [_scene(rng, p, case["lane"], case["n_ref"], case["n_obs"], case["motion"], case["aligned"])]


# ---------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------

_STREAM = []


def _stream():
    """The program's compute stream: its planners queue on it one after another."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def prepare(case, seed):
    scenes = _scenes(case, seed)
    if case["call"] in ("plan", "device"):
        sc = scenes[0]
        stream = _stream().cuda_stream if case["call"] == "device" else None
        pl = mp.Planner(sc["params"], stream=stream)
        if case["tuned"]:
            pl.autotune(sc["x0"], sc["ref"], sc["circles"], sc["centres"])
        pl.set_controls(sc["U"], 0)
        st = dict(call=case["call"], planner=pl, scene=sc)
        if case["call"] == "device":
            dev = (lambda a: None if a is None else torch.tensor(a, dtype=torch.float64, device=DEV))
            T, nx = case["T"], 5 if case["rate"] else 4
            st.update(x0=dev(sc["x0"]), ref=dev(sc["ref"]), circles=dev(sc["circles"]), centres=dev(sc["centres"]),
                      u=torch.empty((T, 2), dtype=torch.float64, device=DEV),
                      x=torch.empty((T + 1, nx), dtype=torch.float64, device=DEV))
            torch.cuda.synchronize()        # the inputs are there before the planner's stream reads them
        return st
    n = len(scenes)
    caps = dict(max_samples=sum(s["params"]["K"] for s in scenes),
                max_rollout_steps=sum(s["params"]["K"] * s["params"]["T"] for s in scenes),
                max_T=max(s["params"]["T"] for s in scenes), max_ref=case["n_ref"],
                max_circ=max(max(len(s["circles"]) for s in scenes), 1), noise_bf16=int(case["bf16"]))
    if case["call"] == "batch":
        bp = mp.BatchPlanner(max_slots=n, max_batch=n, pipelines=2, **caps)
        plans = [mp.BatchPlan(s["params"], i, s["x0"], s["ref"], s["circles"], s["centres"])
                 for i, s in enumerate(scenes)]
        if case["tuned"]:
            bp.autotune(plans)
        for i, s in enumerate(scenes):
            bp.set_controls(i, s["U"], 0)
        return dict(call="batch", engine=bp, plans=plans, reqs=bp.requests(plans))
    srv = mp.Server(max_sessions=n, max_batch=256, pipelines=3, **caps)
    cparams = [mp.make_params(s["params"]) for s in scenes]
    if case["tuned"]:
        mid = sorted(range(n), key=lambda i: scenes[i]["params"]["K"] * scenes[i]["params"]["T"])[n // 2]
        s = scenes[mid]
        srv.autotune(cparams[mid], s["x0"], s["ref"], s["circles"], min(8, n))
    for i, s in enumerate(scenes):
        srv.set_controls(i, s["U"], 0)
    return dict(call="serve", server=srv, scenes=scenes, cparams=cparams)


def run(state):
    if state["call"] == "plan":
        sc = state["scene"]
        u, x, info = state["planner"].plan(sc["x0"], sc["ref"], sc["circles"], sc["centres"])
        return dict(u=u, x=x, argmin=info["argmin"], n_finite=info["n_finite"], s_min=info["s_min"],
                    eta=info["eta"])
    if state["call"] == "device":
        state["planner"].plan_device(state["x0"], state["ref"], state["circles"], state["centres"], state["u"],
                                     state["x"])
        return dict(u=state["u"], x=state["x"])
    if state["call"] == "batch":
        state["engine"].plan(state["plans"], state["reqs"])
        return dict(u=np.concatenate([p.u for p in state["plans"]]),
                    x=np.concatenate([p.x for p in state["plans"]]))
    srv, n = state["server"], len(state["scenes"])
    for i, (s, cp) in enumerate(zip(state["scenes"], state["cparams"])):
        srv.enqueue(cp, i, s["x0"], s["ref"], s["circles"] if len(s["circles"]) else None)
    got = []
    while len(got) < n:
        got += srv.poll(n, wait_ms=1000, with_outputs=True)
    got.sort(key=lambda r: r["session"])
    if any(r["status"] for r in got):
        raise RuntimeError("a served plan failed")
    return dict(u=np.concatenate([r["u"] for r in got]), x=np.concatenate([r["x"] for r in got]))


def work(case):
    """Bytes: each plan's inputs and results once, in binary64.  Operations of a rollout-step: 150
    for its noise, dynamics and costs, 13 for the distance to the one closest segment and 17 for
    the one closest obstacle circle."""
    flops = nbytes = 0.0
    for s in _scenes(case, 0):
        p = s["params"]
        K, T, nc = p["K"], p["T"], len(s["circles"])
        flops += float(K) * T * (150.0 + 13.0 + (17.0 if nc else 0.0))
        nbytes += 8.0 * (4 + 2 * len(s["ref"]) + 5 * nc + (2 * T * nc if s["centres"] is not None else 0) +
                         4 * T + 2 * T + 4 * (T + 1))
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------------
# the same iteration in binary64, straight from its definition
# ---------------------------------------------------------------------------------------------

def _philox(c, k):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    M = 0xFFFFFFFF
    c0, c1, c2, c3 = c
    k0, k1 = k
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57          # wraps modulo 2^64: the same bits
        c0, c1, c2, c3 = (p1 >> 32) & M ^ c1 ^ k0, p1 & M, (p0 >> 32) & M ^ c3 ^ k1, p0 & M
    return c0, c1, c2, c3


def _round_bf16(z):
    b = z.contiguous().view(torch.int64)
    b = (b + 0x0FFFFFFFFFFF + ((b >> 45) & 1)) & ~0x1FFFFFFFFFFF
    return b.view(torch.float64)


def _exact_noise(p):
    K, T = p["K"], p["T"]
    j = torch.arange((T + 1) // 2, device=DEV, dtype=torch.int64)[:, None]
    k = torch.arange(K, device=DEV, dtype=torch.int64)[None, :]
    zero = torch.zeros((j.shape[0], K), device=DEV, dtype=torch.int64)
    w = _philox((j + zero, k + zero, zero, zero + p["session"]), (p["seed"] & 0xFFFFFFFF, p["seed"] >> 32))
    u = [((x >> 8) | 1).double() * 2.0 ** -24 for x in w]
    z = torch.empty((2 * j.shape[0], K, 2), device=DEV, dtype=torch.float64)
    for h in (0, 1):
        r = torch.sqrt(-2.0 * torch.log(u[2 * h]))
        z[h::2, :, 0] = r * torch.cos(2.0 * math.pi * u[2 * h + 1])
        z[h::2, :, 1] = r * torch.sin(2.0 * math.pi * u[2 * h + 1])
    z = z[:T]
    return _round_bf16(z) if p["noise_bf16"] else z


def _exact_reference(px, py, ref, vertex):
    """Squared distance to the lane and the lane's heading there, for flat arrays of points."""
    seg = ref[1:] - ref[:-1]
    head = torch.atan2(seg[:, 1], seg[:, 0])
    d2, idx = torch.empty_like(px), torch.empty(px.shape, dtype=torch.int64, device=DEV)
    step = max(1, (1 << 27) // ref.shape[0])
    for a in range(0, px.shape[0], step):
        x, y = px[a:a + step, None], py[a:a + step, None]
        if vertex:
            d = (x - ref[None, :, 0]).square_().add_((y - ref[None, :, 1]).square_())
        else:
            dx, dy = x - ref[None, :-1, 0], y - ref[None, :-1, 1]
            l2 = seg.square().sum(1)
            tau = (dx * (seg[:, 0] / l2)).add_(dy * (seg[:, 1] / l2)).clamp_(0.0, 1.0)
            d = dx.addcmul_(tau, seg[None, :, 0], value=-1.0).square_()
            d.add_(dy.addcmul_(tau, seg[None, :, 1], value=-1.0).square_())
        d2[a:a + step], idx[a:a + step] = d.min(dim=1)
    return d2, head[idx.clamp(max=head.shape[0] - 1)]


def _exact_costs(sc):
    """Step costs [T][K] and the applied perturbations [T][K][2]."""
    p = sc["params"]
    K, T, dt, L = p["K"], p["T"], p["dt"], p["wheelbase"]
    f = (lambda a: torch.tensor(a, dtype=torch.float64, device=DEV))
    U, ref, circ = f(sc["U"]), f(sc["ref"]), f(sc["circles"])
    eps = _exact_noise(p) * f(p["sigma"])
    v_app = torch.minimum(torch.maximum(U[:, None, :] + eps, f(p["u_min"])), f(p["u_max"]))
    eps = v_app - U[:, None, :]
    R = f(p["R"])
    alpha = (p["gamma"] - 1.0) / (2.0 * p["gamma"])
    cost = ((1.0 + alpha) * (eps * (R * U)[:, None, :]).sum(2)).add_((0.5 * (R * U * U).sum(1))[:, None])
    # trajectories
    st = [torch.full((K,), float(s), dtype=torch.float64, device=DEV) for s in sc["x0"]]
    tr = torch.empty((4, T, K), dtype=torch.float64, device=DEV)
    for t in range(T):
        x, y, th, v = st[:4]
        a = v_app[t, :, 0]
        if math.isfinite(p["v_max"]):
            a = torch.clamp(torch.minimum(a, (p["v_max"] - v) / dt), min=p["u_min"][0])
        steer = st[4] if p["model"] == 1 else v_app[t, :, 1]
        new = [x + v * torch.cos(th) * dt, y + v * torch.sin(th) * dt, th + v * torch.tan(steer) / L * dt, v + a * dt]
        if p["model"] == 1:
            new.append(st[4] + v_app[t, :, 1] * dt)
        st = new
        for i in range(4):
            tr[i, t] = st[i]
    X, Y, TH, V = tr
    del v_app
    goal = ref[-1]
    d_goal = (X - goal[0]).square() + (Y - goal[1]).square()
    first = torch.full((1, K), float((sc["x0"][0] - sc["ref"][-1, 0]) ** 2 + (sc["x0"][1] - sc["ref"][-1, 1]) ** 2),
                       dtype=torch.float64, device=DEV)
    q = p["w_target"] * (d_goal > torch.cat([first, d_goal[:-1]])).double()
    q += p["w_speed"] * (V - p["v_ref"]).square()
    d2, head = _exact_reference(X.reshape(-1), Y.reshape(-1), ref, p["ref_mode"] == 1)
    q += p["w_dist"] * d2.view(T, K)
    dyaw = TH - head.view(T, K)
    q += p["w_yaw"] * (dyaw - 2.0 * math.pi * torch.round(dyaw / (2.0 * math.pi))).square()
    if circ.shape[0]:
        cen = f(sc["centres"]) if sc["centres"] is not None else f(_forecast(sc["circles"], T, dt))
        gap = torch.full((T, K), math.inf, dtype=torch.float64, device=DEV)
        for e in range(p["n_ego"]):
            ex, ey = X + p["ego_offset"][e] * torch.cos(TH), Y + p["ego_offset"][e] * torch.sin(TH)
            for c in range(circ.shape[0]):
                d = torch.hypot(ex - cen[:, c, 0:1], ey - cen[:, c, 1:2]).sub_(circ[c, 2] + p["ego_radius"][e])
                torch.minimum(gap, d, out=gap)
        safe = (p["d_safe_c"] * V + p["d_safe_0"] - gap).clamp_(min=0.0).square_()
        if p["collision_only"]:
            safe[gap > 0.0] = 0.0
        q += p["w_safe"] * safe
    return cost + q, eps


def _exact_plan(sc):
    p = sc["params"]
    T, dt, lam = p["T"], p["dt"], p["lam"]
    cost, eps = _exact_costs(sc)
    S = cost.sum(0)
    s_min, arg = S.min(0)
    w = torch.exp(-(S - s_min) / lam)
    eta = w.sum()
    if p["cost_to_go"]:
        to_go = cost.flip(0).cumsum(0).flip(0)
        wt = torch.exp(-(to_go - to_go.min(dim=1, keepdim=True).values) / lam)
        du = (wt[:, :, None] * eps).sum(1) / wt.sum(1)[:, None]
        eta = wt[0].sum()
    else:
        du = (w[None, :, None] * eps).sum(1) / eta
    lo, hi = np.array(p["u_min"]), np.array(p["u_max"])
    u = np.clip(sc["U"] + du.cpu().numpy(), lo, hi)
    at = np.clip(np.arange(T)[:, None] + np.arange(-2, 3)[None, :], 0, T - 1)
    u = np.clip((u[at] * np.array([-3.0, 12.0, 17.0, 12.0, -3.0])[None, :, None]).sum(1) / 35.0, lo, hi)
    x = np.empty((T + 1, len(sc["x0"])))
    x[0] = sc["x0"]
    for t in range(T):
        px, py, th, v = x[t, :4]
        a = u[t, 0]
        if math.isfinite(p["v_max"]):
            a = max(min(a, (p["v_max"] - v) / dt), p["u_min"][0])
        steer = x[t, 4] if p["model"] == 1 else u[t, 1]
        x[t + 1, :4] = [px + v * math.cos(th) * dt, py + v * math.sin(th) * dt,
                        th + v * math.tan(steer) / p["wheelbase"] * dt, v + a * dt]
        if p["model"] == 1:
            x[t + 1, 4] = x[t, 4] + u[t, 1] * dt
    return dict(u=u, x=x, argmin=int(arg), n_finite=int(torch.isfinite(S).sum()), s_min=float(s_min), eta=float(eta))


def exact(case, seed):
    got = [_exact_plan(sc) for sc in _scenes(case, seed)]
    if case["call"] == "plan":
        return got[0]
    if case["call"] == "device":
        return dict(u=got[0]["u"], x=got[0]["x"])
    return dict(u=np.concatenate([g["u"] for g in got]), x=np.concatenate([g["x"] for g in got]))
