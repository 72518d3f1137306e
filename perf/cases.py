"""Timed workloads of the framework's public entry points.

Every case is a plain dict; ``prepare`` builds what a program holds before
the call (inputs in device memory, a context or a network), ``run`` is one
pass through the entry points, ``exact`` the same results in 64 bits from
plain torch.  Sizes come from the package's workloads (synth.py, bench.py):
lanes of 2-200 vehicles up to 20,000 lanes of 100, horizons of 20-1,000 steps
of 0.1 s, checkpoint intervals 8 (the default) and 50, batches of uneven
scenarios, the initializer's 8,192-row batches, the filtering (6,101
trajectories) and reconstruction (21,750 trajectories) sets and the lane
geometry pipeline.
"""
import math

import numpy as np
import torch

from paper_2412_16750_gb300 import api, synth

DT = float(np.float32(0.1))
A_MIN = -10.0
GAP_FLOOR = 0.1
MAX_VEHICLE_STEPS = 2_000_000_000


def listed():
    return [
        # the smallest scene: one loss and gradient of 10 lanes x 100 vehicles, bound by latency and launches
        dict(name="small_loss_grad", kind="loss_grad", lanes=10, lo=100, hi=100, K=100, stride=1, ckpt=8),
        # a whole short fit of the same scene, the call that a user makes for one road section
        dict(name="small_fit", kind="fit", lanes=10, lo=100, hi=100, K=100, stride=1, ckpt=8, iters=50),
        # a city-sized scene of uneven lanes, observed every third step
        dict(name="ragged_loss_grad", kind="loss_grad", lanes=10_000, lo=2, hi=200, K=301, stride=3, ckpt=8),
        # the paper's scale: Adam iterations of 2 million vehicles over 1,000 steps, checkpoints every 50
        dict(name="paper_fit", kind="fit", lanes=20_000, lo=100, hi=100, K=1000, stride=1, ckpt=50, iters=2),
        # the differentiable simulator inside a user's own torch program: autograd through the trajectory
        dict(name="autograd", kind="autograd", lanes=2000, lo=100, hi=100, K=100, ckpt=8),
        # prediction after a fit: positions and speeds of a long rollout
        dict(name="rollout", kind="rollout", lanes=5000, lo=100, hi=100, K=1000),
        # independent uneven scenarios in one call, observed every tenth step
        dict(name="batch_loss_grad", kind="batch", scen=256, stride=10),
        # the learned initial guess of a 200,000-vehicle scene: features and inference
        dict(name="initial_guess", kind="guess", lanes=2000, lo=100, hi=100),
        # one training batch of the initializer: loss and gradient
        dict(name="train_batch", kind="train", batch=8192),
        # filtering of densely observed trajectories (0.1 s), Adam iterations
        dict(name="filtering_fit", kind="recon", n=6101, t_lo=30.0, t_hi=90.0, dense=True, dt=0.1, iters=20),
        # reconstruction of sparsely observed trajectories (1 s steps, up to 20 minutes), Adam iterations
        dict(name="reconstruction_fit", kind="recon", n=21750, t_lo=120.0, t_hi=1200.0, dense=False, dt=1.0, iters=10),
        # the training-free prediction pipeline: lanes, projection, a short-horizon fit, rollout, back-projection
        dict(name="predict_rollout", kind="predict", scen=2000, iters=500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["loss_grad", "loss_grad", "fit", "fit", "autograd", "rollout", "batch", "guess", "train", "recon",
                       "recon", "predict"])
    if kind == "batch":
        return dict(kind=kind, scen=_log(rng, 4, 1024), stride=rng.choice([1, 5, 10]))
    if kind == "train":
        return dict(kind=kind, batch=_log(rng, 500, 8192))
    if kind == "recon":
        if rng.random() < 0.5:
            return dict(kind=kind, n=_log(rng, 100, 12000), t_lo=30.0, t_hi=90.0, dense=True, dt=0.1, iters=rng.randint(5, 20))
        return dict(kind=kind, n=_log(rng, 100, 21750), t_lo=120.0, t_hi=float(rng.randint(300, 1200)), dense=False,
                    dt=1.0, iters=rng.randint(3, 10))
    if kind == "predict":
        return dict(kind=kind, scen=_log(rng, 20, 4000), iters=rng.choice([100, 200, 500]))
    even = rng.random() < 0.5
    per = rng.randint(20, 180)
    c = dict(kind=kind, lanes=_log(rng, 4, 20_000), lo=per if even else 2, hi=per if even else rng.randint(64, 200))
    if kind == "guess":
        return c
    c["K"] = _log(rng, 40, 1000)
    if kind != "rollout":
        c["ckpt"] = rng.choice([8, 8, 8, 50])
    if kind in ("loss_grad", "fit"):
        c["stride"] = rng.choice([1, 1, 2, 5, 10])
    if kind == "fit":
        c["iters"] = rng.randint(2, 8)
    most = MAX_VEHICLE_STEPS // (4 if kind in ("rollout", "autograd") else 1)
    c["lanes"] = max(4, min(c["lanes"], int(most / (c["K"] * c.get("iters", 1) * _mean(c)))))
    return c


# ---- inputs ---------------------------------------------------------------------


def _mean(c):
    return 0.5 * (c["lo"] + c["hi"])


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo


def _scene(counts, g):
    """Lanes head first with the given vehicle counts: bumper gaps U[20, 40] m, speeds U[10, 30] m/s and the
    parameter ranges of synth.TRUE_RANGES."""
    counts = torch.as_tensor(counts, device="cuda", dtype=torch.int64)
    off = torch.cat([counts.new_zeros(1), counts.cumsum(0)])
    N = int(off[-1])
    head = torch.zeros(N, dtype=torch.bool, device="cuda")
    head[off[:-1][counts > 0]] = True
    length = torch.full((N,), synth.LENGTH, device="cuda")
    back = torch.where(head, torch.zeros((), device="cuda"), _uniform(g, N, *synth.GAP_RANGE) + synth.LENGTH).double()
    at = back.cumsum(0)
    first = torch.repeat_interleave(off[:-1], counts)
    p0 = (at[first] - at).float()
    v0 = _uniform(g, N, *synth.SPEED_RANGE)
    truth = torch.stack([_uniform(g, N, lo, hi) for lo, hi in synth.TRUE_RANGES] + [torch.full((N,), synth.DELTA, device="cuda")])
    return dict(off=off.int(), N=N, head=head, length=length, p0=p0, v0=v0, truth=truth)


def _counts(c):
    """Vehicles per lane; array shapes depend on the case alone, values on the seed."""
    g = torch.Generator().manual_seed(c["lanes"] + c["hi"])
    return torch.randint(c["lo"], c["hi"] + 1, (c["lanes"],), generator=g)


def _plain(N):
    return torch.tensor(synth.PLAIN_INIT, device="cuda")[:, None].repeat(1, N).contiguous()


def _near(truth, g):
    """Parameters on the way to a solution: the true ones times U[0.85, 1.15]."""
    th = truth * _uniform(g, truth.shape, 0.85, 1.15)
    th[5] = synth.DELTA
    return th.contiguous()


def _targets(sc, K, stride, g):
    """Noisy observations (K // stride, N) of the true trajectory (float32 torch)."""
    n = K // stride
    y = torch.empty((n, sc["N"]), device="cuda")
    y.normal_(0.0, synth.NOISE_STD, generator=g)
    p, v = sc["p0"], sc["v0"]
    for k in range(1, n * stride + 1):
        p, v = _step(p, v, sc["truth"], sc["head"], sc["length"], DT)
        if k % stride == 0:
            y[k // stride - 1] += p
    return y


def prepare(case, seed):
    return dict(globals()["_prepare_" + case["kind"]](case, seed), case=case)


def _prepare_sim(case, seed):
    g = _gen(seed)
    sc = _scene(_counts(case), g)
    sc["scene"] = api.Scene.from_lane_off(sc["off"], sc["length"])
    sc["ctx"] = api.Context(ckpt_interval=case.get("ckpt", 8))
    return sc, g


def _prepare_loss_grad(case, seed):
    sc, g = _prepare_sim(case, seed)
    return dict(sc, theta=_near(sc["truth"], g), y=_targets(sc, case["K"], case["stride"], g))


def _prepare_fit(case, seed):
    sc, g = _prepare_sim(case, seed)
    return dict(sc, theta=_plain(sc["N"]), y=_targets(sc, case["K"], case["stride"], g))


def _prepare_autograd(case, seed):
    sc, g = _prepare_sim(case, seed)
    w = torch.empty((case["K"] + 1, sc["N"]), device="cuda")
    w.normal_(0.0, 1.0, generator=g)
    theta, p0, v0 = (x.clone().requires_grad_(True) for x in (_near(sc["truth"], g), sc["p0"], sc["v0"]))
    return dict(sc, theta=theta, p0=p0, v0=v0, w=w)


def _prepare_rollout(case, seed):
    sc, g = _prepare_sim(case, seed)
    return dict(sc, theta=_near(sc["truth"], g))


def _prepare_batch(case, seed):
    lanes, K, counts = synth.config2_tables(case["scen"], np.random.default_rng(case["scen"]))
    scen_off = synth.lane_offsets(lanes)
    g = _gen(seed)
    sc = _scene(np.concatenate(counts), g)
    stride = case["stride"]
    batch = api.Batch(scen_off, K, np.full(len(K), DT), np.full(len(K), stride), sc["off"].cpu().numpy(), sc["length"])
    full = _targets(sc, int(K.max()), stride, g)
    y = torch.cat([full[: K[s] // stride, batch.veh_off[s]:batch.veh_off[s + 1]].reshape(-1) for s in range(len(K))])
    return dict(sc, batch=batch, full=full, y=y, theta=_near(sc["truth"], g), ctx=api.Context())


def _prepare_guess(case, seed):
    sc, g = _prepare_sim(case, seed)
    net = api.Mlp(8192, synth.mlp_init(seed))
    return dict(sc, y=_targets(sc, 20, 1, g), net=net, w=torch.as_tensor(synth.mlp_init(seed), device="cuda"))


def _prepare_train(case, seed):
    g = _gen(seed)
    B = case["batch"]
    sc = _scene([100] * -(-B // 100), g)
    X = _features(sc, _targets(sc, 20, 1, g))[:B].to(torch.bfloat16).contiguous()
    lo, hi = (torch.tensor(b, device="cuda") for b in (api.BOX_LO, api.BOX_HI))
    labels = ((sc["truth"][:5].T - lo) / (hi - lo))[:B].contiguous()
    w = synth.mlp_init(seed)
    return dict(net=api.Mlp(B, w), X=X, labels=labels, w=torch.as_tensor(w, device="cuda"))


def _prepare_recon(case, seed):
    """Observed positions of smooth speed profiles (the recipe of synth.recon_observations), longest first."""
    n = case["n"]
    g = _gen(n)
    T = torch.sort(_uniform(g, n, case["t_lo"], case["t_hi"]).double(), descending=True).values
    if case["dense"]:
        t = torch.arange(int(case["t_hi"] / 0.1) + 2, device="cuda", dtype=torch.float64)[None, :].repeat(n, 1) * 0.1
    else:
        e = torch.empty((n, int(case["t_hi"]) + 1), device="cuda", dtype=torch.float64).exponential_(1.0, generator=g)
        t = torch.cat([torch.zeros((n, 1), device="cuda", dtype=torch.float64), (1.0 + e).cumsum(1)], 1)
    keep = t <= T[:, None]
    off = torch.cat([torch.zeros(1, device="cuda", dtype=torch.int64), keep.sum(1).cumsum(0)]).int()
    t = t.float().double()
    g = _gen(seed)
    vm = _uniform(g, n, 8.0, 25.0).double()
    A1, A2 = vm * _uniform(g, n, 0.0, 0.3), vm * _uniform(g, n, 0.0, 0.2)
    w1, w2 = 2 * math.pi / _uniform(g, n, 60.0, 300.0).double(), 2 * math.pi / _uniform(g, n, 15.0, 60.0).double()
    f1, f2 = (_uniform(g, n, 0.0, 2 * math.pi).double() for _ in range(2))
    p = _uniform(g, n, 0.0, 1000.0).double()[:, None] + vm[:, None] * t
    for A, w, f in ((A1, w1, f1), (A2, w2, f2)):
        p = p - (A / w)[:, None] * (torch.cos(w[:, None] * t + f[:, None]) - torch.cos(f)[:, None])
    p = p + torch.empty_like(p).normal_(0.0, 0.3 if case["dense"] else 1.0, generator=g)
    rec = api.Recon(off, t[keep].float(), p[keep].float(), float(np.float32(case["dt"])), ctx=api.Context())
    return dict(rec=rec, init=rec.init_vars(), t=t[keep].float(), p=p[keep].float(), off=off)


def _agents(c):
    """Agents kept of c["scen"] scenarios of 17.5 +- 8 agents, so that their number depends on the case alone."""
    return int(17.5 * c["scen"] - 32 * math.sqrt(c["scen"]))


def _prepare_predict(case, seed):
    s = synth.prediction_scenes(case["scen"], np.random.default_rng(seed))

    def dev(x, dtype=torch.float32):
        return torch.as_tensor(np.ascontiguousarray(x), dtype=dtype, device="cuda")

    ctx = api.Context()
    lanes = api.Lanes(dev(s["pt_off"], torch.int32), dev(s["px"]), dev(s["py"]), ctx=ctx)
    h, n = s["n_hist"], _agents(case)
    return dict(lanes=lanes, x=dev(s["x"][:h, :n]), y=dev(s["y"][:h, :n]), lo=dev(s["lane_lo"][:n], torch.int32),
                hi=dev(s["lane_hi"][:n], torch.int32), dt=s["dt"], n_fut=s["n_fut"], ctx=ctx)


# ---- one pass ---------------------------------------------------------------------


def run(state):
    return globals()["_run_" + state["case"]["kind"]](state, state["case"])


def _run_loss_grad(s, c):
    loss, g, gp, gv = api.loss_grad(s["theta"], s["p0"], s["v0"], s["scene"], c["K"], DT, s["y"], c["stride"], ctx=s["ctx"])
    return dict(loss=loss, theta=g, p0=gp, v0=gv)


def _run_fit(s, c):
    theta = s["theta"].clone()
    hist = api.fit(theta, s["p0"], s["v0"], s["scene"], c["K"], DT, s["y"], c["stride"], c["iters"], ctx=s["ctx"])
    return dict(theta=theta, loss=hist)


def _run_autograd(s, c):
    traj = api.IdmFunction.apply(s["theta"], s["p0"], s["v0"], s["scene"], c["K"], DT, A_MIN, s["ctx"])
    g, gp, gv = torch.autograd.grad(traj, (s["theta"], s["p0"], s["v0"]), s["w"])
    return dict(traj=traj.detach(), theta=g, p0=gp, v0=gv)


def _run_rollout(s, c):
    P, V = api.simulate(s["theta"], s["p0"], s["v0"], s["scene"], c["K"], DT, want_speed=True, ctx=s["ctx"])
    return dict(positions=P, speeds=V)


def _run_batch(s, c):
    scen, total, g, gp, gv = api.batch_loss_grad(s["theta"], s["p0"], s["v0"], s["batch"], s["y"], ctx=s["ctx"])
    return dict(scenarios=scen, loss=total, theta=g, p0=gp, v0=gv)


def _run_guess(s, c):
    X = api.mlp_features(s["scene"], s["p0"], s["v0"], 20, DT, s["y"])
    theta = torch.empty((6, s["N"]), device="cuda")
    theta[5] = synth.DELTA
    return dict(features=X, theta=s["net"].predict_params(X, theta))


def _run_train(s, c):
    loss, grad = s["net"].loss_grad(s["X"], s["labels"])
    return dict(loss=loss, grad=grad)


def _run_recon(s, c):
    theta, dp, dv = (x.clone() for x in s["init"])
    hist = s["rec"].fit(theta, dp, dv, c["iters"])
    return dict(theta=theta, dp=dp, dv=dv, loss=hist)


def _run_predict(s, c):
    r = api.predict_rollout(s["lanes"], s["x"], s["y"], s["lo"], s["hi"], s["dt"], s["n_fut"], c["iters"], ctx=s["ctx"])
    return {k: r[k] for k in ("perm", "lane", "theta", "loss", "s_hist", "x", "y")}


# ---- work ---------------------------------------------------------------------------
# Operations of one vehicle-step: the forward step 35 and the loss, recompute-free reverse step and gradient sums 110
# (special functions counted once each); of one GELU 20.


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        steps = c["scen"] * 32.5 * 101 * 275
        return dict(bytes=4 * steps / c["stride"] + 100 * c["scen"] * 32.5 * 101, flops=145 * steps)
    if kind == "train":
        return dict(bytes=c["batch"] * 180 + 8 * 153605, flops=c["batch"] * 876032.0)
    if kind == "recon":
        steps = c["n"] * 0.5 * (c["t_lo"] + c["t_hi"]) / c["dt"]
        obs = steps if c["dense"] else 0.5 * steps
        # observations, dp and dv in and out, once: an iteration's state need not leave the chip in principle
        return dict(bytes=8 * obs + 16 * steps, flops=150 * steps * c["iters"])
    if kind == "predict":
        agents = _agents(c)
        return dict(bytes=agents * (11 * 12 + 80 * 8 + 60), flops=agents * (145 * 10 * c["iters"] + 35 * 80 + 11 * 150 * 13 + 750 * 13))
    N = c["lanes"] * _mean(c)
    if kind == "guess":
        return dict(bytes=N * (80 + 160 + 24), flops=N * (2 * 152832.0 + 3 * 256 * 20))
    steps = N * c["K"]
    if kind == "rollout":
        return dict(bytes=8 * steps + 36 * N, flops=35 * steps)
    if kind == "autograd":
        return dict(bytes=8 * steps + 70 * N, flops=145 * steps)
    it = c.get("iters", 1)
    return dict(bytes=4 * steps / c["stride"] * it + 70 * N, flops=145 * steps * it)


# ---- 64-bit references --------------------------------------------------------------


def _softplus(x):
    return torch.logaddexp(x, torch.zeros((), dtype=x.dtype, device=x.device))


def _accel(v, gap, dv, th, dt, head=None):
    v0, T, s0, am, b, delta = th
    z = _softplus(s0 + v * T + v * dv / (2 * torch.sqrt(am * b))) / gap.clamp(min=GAP_FLOOR)
    if head is not None:
        z = torch.where(head, torch.zeros((), dtype=z.dtype, device=z.device), z)
    a = am * (1 - (v / v0) ** delta - z * z)
    lb = torch.where(-v / dt > A_MIN, -v / dt, torch.full((), A_MIN, dtype=v.dtype, device=v.device))
    return lb + _softplus(a - lb)


def _ahead(x):
    return torch.cat([x[:1], x[:-1]])


def _step(p, v, th, head, length, dt):
    gap = torch.where(head, torch.full((), 100.0, dtype=p.dtype, device=p.device), _ahead(p) - p - _ahead(length))
    return p + dt * v, v + dt * _accel(v, gap, v - _ahead(v), th, dt, head)


def _forward64(s, theta, K):
    th, head, length = theta.detach().double(), s["head"], s["length"].double()
    P = torch.empty((K + 1, s["N"]), device="cuda", dtype=torch.float64)
    V = torch.empty_like(P)
    P[0], V[0] = s["p0"].detach(), s["v0"].detach()
    for k in range(K):
        P[k + 1], V[k + 1] = _step(P[k], V[k], th, head, length, DT)
    return P, V


def _reverse64(s, theta, P, V, seed_of):
    """Gradients of theta, p0, v0 from dL/dP[k] = seed_of(k) (None where zero)."""
    K, th, length = P.shape[0] - 1, theta.detach().double(), s["length"].double()
    gth, lp, lv = torch.zeros_like(th), torch.zeros_like(P[0]), torch.zeros_like(P[0])
    for k in range(K, -1, -1):
        q = seed_of(k)
        if q is not None:
            lp = lp + q
        if k == 0:
            break
        with torch.enable_grad():
            p, v, t = (x.detach().requires_grad_(True) for x in (P[k - 1], V[k - 1], th))
            lp, lv, gt = torch.autograd.grad(_step(p, v, t, s["head"], length, DT), (p, v, t), (lp, lv))
        gth += gt
    return gth, lp, lv


def _loss_grad64(s, theta, K, stride):
    P, V = _forward64(s, theta, K)
    n = K // stride
    r = P[stride::stride][:n] - s["y"]
    g = _reverse64(s, theta, P, V, lambda k: 2.0 / n * r[k // stride - 1] if k >= 1 and k % stride == 0 else None)
    return r.square().sum() / n, g


def _adam(x, g, m, v, t, lr):
    m.mul_(0.9).add_(0.1 * g)
    v.mul_(0.999).add_(0.001 * g * g)
    x.sub_(lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8))


def exact(case, seed):
    f = globals().get("_exact_" + case["kind"])
    if f is None:
        return None
    if "lanes" in case and "K" in case and _mean(case) * case["lanes"] * case["K"] * case.get("iters", 1) > 2.2e9:
        return None
    if "K" in case and case["K"] * case.get("iters", 1) > 6000:
        return None
    with torch.no_grad():
        return f(prepare(case, seed), case)


def _exact_loss_grad(s, c):
    loss, g = _loss_grad64(s, s["theta"], c["K"], c["stride"])
    return dict(loss=loss, theta=g[0], p0=g[1], v0=g[2])


def _exact_fit(s, c):
    if _mean(c) * c["lanes"] * c["K"] * c["iters"] > 2e9:
        return None
    th = s["theta"].double()
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    lo, hi = (torch.tensor(b, device="cuda", dtype=torch.float64)[:, None] for b in (api.BOX_LO, api.BOX_HI))
    hist = []
    for it in range(c["iters"]):
        loss, g = _loss_grad64(s, th, c["K"], c["stride"])
        hist.append(loss)
        lr = 0.1 + (0.01 - 0.1) * it / (c["iters"] - 1) if c["iters"] > 1 else 0.1
        _adam(th[:5], g[0][:5], m[:5], v[:5], it + 1, lr)
        th[:5] = torch.minimum(torch.maximum(th[:5], lo), hi)
    return dict(theta=th, loss=torch.stack(hist))


def _exact_autograd(s, c):
    P, V = _forward64(s, s["theta"], c["K"])
    g = _reverse64(s, s["theta"], P, V, lambda k: s["w"][k].double())
    return dict(traj=P, theta=g[0], p0=g[1], v0=g[2])


def _exact_rollout(s, c):
    P, V = _forward64(s, s["theta"], c["K"])
    return dict(positions=P, speeds=V)


def _exact_batch(s, c):
    b, stride = s["batch"], c["stride"]
    K = int(b.K.max())
    nv = np.diff(b.veh_off)
    per = torch.as_tensor(np.repeat(b.K, nv), device="cuda")
    n = (per // stride).double()
    P, V = _forward64(s, s["theta"], K)
    k_of = torch.arange(1, K // stride + 1, device="cuda")[:, None] * stride
    r = torch.where(k_of <= per, P[stride::stride][:K // stride] - s["full"], 0.0)
    g = _reverse64(s, s["theta"], P, V, lambda k: 2.0 / n * r[k // stride - 1] if k >= 1 and k % stride == 0 else None)
    scen_of = torch.as_tensor(np.repeat(np.arange(len(b.K)), nv), device="cuda")
    scen = torch.zeros(len(b.K), device="cuda", dtype=torch.float64).index_add_(0, scen_of, r.square().sum(0) / n)
    return dict(scenarios=scen, loss=scen.sum(), theta=g[0], p0=g[1], v0=g[2])


def _features(s, y):
    """Feature rows in 64 bits from 20 observations of every vehicle and its leader."""
    obs = torch.cat([s["p0"][None], y[:20]]).double()
    v = torch.cat([s["v0"][None].double(), (obs[2:21] - obs[0:19]) / (2 * DT)]) / 30.0
    lead = torch.stack([_ahead(o) for o in obs[:20]])
    x_e, x_l = (obs[:20] - obs[0]) / 100.0, (lead - obs[0]) / 100.0
    v_l = torch.stack([_ahead(o) for o in v])
    return torch.cat([x_e, v, torch.where(s["head"], x_e + 2.0, x_l), torch.where(s["head"], v, v_l)]).T


def _layers(w):
    at, out = 0, []
    for fan_in, fan_out in synth.MLP_SIZES:
        out.append((w[at:at + fan_in * fan_out].view(fan_out, fan_in), w[at + fan_in * fan_out:at + fan_in * fan_out + fan_out]))
        at += fan_in * fan_out + fan_out
    return out


def _net64(w, X):
    h = X
    for q, (W, b) in enumerate(_layers(w)):
        h = torch.nn.functional.linear(h, W, b)
        h = torch.nn.functional.gelu(h) if q < 3 else torch.sigmoid(h)
    return h


def _exact_guess(s, c):
    X = _features(s, s["y"])
    lo, hi = (torch.tensor(b, device="cuda", dtype=torch.float64)[:, None] for b in (api.BOX_LO, api.BOX_HI))
    out = _net64(s["w"].double(), X).T
    return dict(features=X, theta=torch.cat([lo + (hi - lo) * out, torch.full((1, s["N"]), synth.DELTA, device="cuda")]))


def _exact_train(s, c):
    with torch.enable_grad():
        w = s["w"].double().requires_grad_(True)
        loss = (_net64(w, s["X"].double()) - s["labels"].double()).square().mean()
        grad, = torch.autograd.grad(loss, w)
    return dict(loss=loss.detach(), grad=grad)


def _exact_recon(s, c):
    rec = s["rec"]
    K, n, dt = rec.k_max, rec.N, rec.dt
    if K * c["iters"] > 20000:
        return None
    Ki = rec.K[:n].long()
    live = torch.arange(K, device="cuda")[:, None] < Ki
    obs_k, of = rec.obs_k[:rec.n_obs].long(), torch.repeat_interleave(torch.arange(n, device="cuda"), s["off"].diff().long())
    use = obs_k > 0
    at, y = obs_k[use] * n + of[use], s["p"].double()[use]
    th, dp, dv = s["init"][0].double(), s["init"][1][:, :n].double(), s["init"][2][:, :n].double()
    moments = [(torch.zeros_like(x), torch.zeros_like(x)) for x in (th, dp, dv)]
    lo, hi = (torch.tensor(b, device="cuda", dtype=torch.float64)[:, None] for b in (api.RECON_BOX_LO, api.RECON_BOX_HI))
    hist = []
    for it in range(c["iters"]):
        P = torch.empty((K + 1, n), device="cuda", dtype=torch.float64)
        V = torch.empty_like(P)
        P[0], V[0] = rec.p_init[:n], rec.v_init[:n]
        for k in range(K):
            P[k + 1] = torch.where(live[k], P[k] + dt * V[k], P[k])
            V[k + 1] = torch.where(live[k], V[k] + dt * _accel(V[k], dp[k], dv[k], th, dt), V[k])
        r = P.view(-1)[at] - y
        hist.append(r.abs().sum())
        seed = torch.zeros((K + 1) * n, device="cuda", dtype=torch.float64).index_add_(0, at, torch.sign(r)).view(K + 1, n)
        with torch.enable_grad():
            t, d, e, v = (x.detach().requires_grad_(True) for x in (th, dp, dv, V[:K]))
            a = _accel(v, d, e, t, dt)
            Av, = torch.autograd.grad(a.sum(), v, retain_graph=True)
            lp, lv, mu = torch.zeros_like(P[0]), torch.zeros_like(P[0]), torch.zeros_like(dp)
            for k in range(K - 1, -1, -1):
                lp = lp + seed[k + 1]
                mu[k] = torch.where(live[k], dt * lv, 0.0)
                lv = torch.where(live[k], lv + dt * lp + mu[k] * Av[k], lv)
            g = torch.autograd.grad((mu * a).sum(), (t, d, e))
        lr = 0.1 + (0.01 - 0.1) * it / (c["iters"] - 1) if c["iters"] > 1 else 0.1
        for q, (x, gx) in enumerate(zip((th, dp, dv), g)):
            rows = slice(0, 5) if q == 0 else slice(None)
            x0 = x.clone()
            _adam(x[rows], gx[rows], moments[q][0][rows], moments[q][1][rows], it + 1, lr)
            if q > 0:
                x.copy_(torch.where(live, x, x0))
        th[:5] = torch.minimum(torch.maximum(th[:5], lo), hi)
    full = [x.double().clone() for x in s["init"][1:]]
    full[0][:, :n], full[1][:, :n] = dp, dv
    return dict(theta=th, dp=full[0], dv=full[1], loss=torch.stack(hist))
