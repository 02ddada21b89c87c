"""The work a user of this framework has it do, as timed cases.

Each case is one pass through the public binding (`paper_1906_02318_gb300.mpmi`): a control
tick from device or host buffers, a screened tick, a batch of served sessions, a training
gradient of the screener, or a model fit.  Sizes are those of the benchmark, the tests and the
serving mix (N log-uniform in 1k..64k, H in 20..100), up to a million candidates.

Persistent host ticks are not among them: their kernel stays resident between calls, so a
device-wide wait after a pass would time its idle limit.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1906_02318_gb300 import mpmi

# ---------------------------------------------------------------- plants and their data
# Cart-pole (100 Hz) and dynamic bicycle (60 Hz), float64, semi-implicit Euler.
LO = {"bot": np.array([-1.0]), "car": np.array([-0.4, -1.0])}
HI = {"bot": np.array([1.0]), "car": np.array([0.4, 1.0])}
BOX = {"bot": np.array([[-0.6, 0.6], [-2.0, 2.0], [-2.5, 2.5], [-2.0, 2.0]]),
       "car": np.array([[-100.0, 100.0], [-100.0, 100.0], [-np.pi, np.pi], [0.0, 30.0],
                        [-3.0, 3.0], [-1.5, 1.5]])}
SAFE = {"bot": (np.array([-0.5, -np.inf, -2.0, -np.inf]), np.array([0.5, np.inf, 2.0, np.inf])),
        "car": (np.full(6, -np.inf), np.array([np.inf, np.inf, np.inf, 25.0, np.inf, np.inf]))}
HELD = {"bot": (4, 11), "car": (6, 7, 30, 31)}  # lifted features that depend on the input alone
HALF_WIDTH = 4.0
SIGMA = np.array([0.005, 0.02, 0.005, 0.02])    # per-step noise of the balance bot
LIVE = 0.7    # share of the N H prediction steps that run before a violation, typically


def _cartpole(x, u):
    th, thd, pos, vel = x.T
    force, s, c = 10.0 * u[:, 0], np.sin(x[:, 0]), np.cos(x[:, 0])
    tmp = (force + 0.05 * thd * thd * s) / 1.1
    acc = (9.8 * s - c * tmp) / (0.5 * (4.0 / 3.0 - 0.1 * c * c / 1.1))
    thd2, vel2 = thd + 0.01 * acc, vel + 0.01 * (tmp - 0.05 * acc * c / 1.1)
    return np.stack([th + 0.01 * thd2, thd2, pos + 0.01 * vel2, vel2], axis=1)


def _bicycle(x, u):
    px, py, psi, vx, vy, om = x.T
    delta, acc, dt = u[:, 0], u[:, 1], 1.0 / 60.0
    v = np.maximum(vx, 1.0)
    ff = 8.0e4 * (delta - np.arctan2(vy + 1.2 * om, v))
    fr = -8.0e4 * np.arctan2(vy - 1.4 * om, v)
    vx2 = vx + dt * ((5000.0 * acc - ff * np.sin(delta)) / 1500.0 + vy * om)
    vy2 = vy + dt * ((ff * np.cos(delta) + fr) / 1500.0 - vx * om)
    om2 = om + dt * (1.2 * ff * np.cos(delta) - 1.4 * fr) / 2250.0
    psi2 = psi + dt * om2
    c, s = np.cos(psi2), np.sin(psi2)
    return np.stack([px + dt * (vx2 * c - vy2 * s), py + dt * (vx2 * s + vy2 * c), psi2, vx2,
                     vy2, om2], axis=1)


def _transitions(plant, rng, m):
    """One-step transitions (x, u, x_next), states and inputs uniform over their boxes."""
    x = rng.uniform(BOX[plant][:, 0], BOX[plant][:, 1], size=(m, len(BOX[plant])))
    u = rng.uniform(LO[plant], HI[plant], size=(m, len(LO[plant])))
    return x, u, (_cartpole if plant == "bot" else _bicycle)(x, u)


def _lift(plant, x, u):
    one = np.ones(len(x))
    if plant == "bot":
        th, thd, pos, vel = x.T
        a, s, c = u[:, 0], np.sin(th), np.cos(th)
        return np.stack([th, thd, pos, vel, a, s, c, thd * thd, thd * a, thd * thd * s, a * c,
                         one], axis=1)
    px, py, psi, vx, vy, om = x.T
    d, a, s, c = u[:, 0], u[:, 1], np.sin(psi), np.cos(psi)
    return np.stack([px, py, psi, vx, vy, om, d, a, s, c, vx * c, vx * s, vy * c, vy * s, om * vx,
                     om * vy, vx * vx, vy * vy, om * om, d * vx, d * vy, d * om, a * vx, d * c,
                     d * s, a * c, a * s, om * c, om * s, vx * vy, d * d, one], axis=1)


def _least_squares(plant, x, u, xn):
    """K and the relative residual of the least-squares fit, in 64 bits."""
    X, Y = _lift(plant, x, u), _lift(plant, xn, u)
    K = np.linalg.lstsq(X, Y, rcond=None)[0].T.copy()
    for j in HELD[plant]:
        K[j] = 0.0
        K[j, j] = 1.0
    return K, float(np.linalg.norm(X @ K.T - Y) / np.linalg.norm(Y))


def _track(rng):
    """A closed road: 12 control points, periodic Catmull-Rom, 384 segments."""
    ang = (np.arange(12) + 0.1 * rng.uniform(-1.0, 1.0, 12)) * (2.0 * np.pi / 12)
    rad = 60.0 * rng.uniform(0.7, 1.3, 12)
    p = np.stack([rad * np.cos(ang), rad * np.sin(ang)], axis=1)
    s = (np.arange(32) / 32.0)[:, None]
    out = []
    for i in range(12):
        a, b, c, d = (p[(i + k) % 12] for k in (-1, 0, 1, 2))
        out.append(0.5 * (2 * b + s * (c - a) + s * s * (2 * a - 5 * b + 4 * c - d)
                          + s ** 3 * (-a + 3 * b - 3 * c + d)))
    return np.concatenate(out)


def _states(plant, rng, count, track):
    """States and user inputs as a controller's closed loop visits them."""
    if plant == "bot":
        w = np.array([0.2, 0.6, 1.0, 0.8])
        x = rng.uniform(-w, w, size=(count, 4))
    else:
        i = rng.integers(0, len(track), count)
        d = track[(i + 1) % len(track)] - track[i]
        psi = np.arctan2(d[:, 1], d[:, 0])
        off = rng.uniform(-2.0, 2.0, count)
        x = np.stack([track[i, 0] - off * np.sin(psi), track[i, 1] + off * np.cos(psi),
                      psi + rng.uniform(-0.15, 0.15, count), rng.uniform(6.0, 16.0, count),
                      rng.uniform(-0.3, 0.3, count), rng.uniform(-0.3, 0.3, count)], axis=1)
    u = np.clip(rng.normal(0.0, 0.4, size=(count, len(LO[plant]))), -1.0, 1.0)
    u = LO[plant] + 0.5 * (u + 1.0) * (HI[plant] - LO[plant])
    return x, u.astype(np.float32).astype(np.float64)


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest tick: one balance-bot decision, 1024 candidates, 20 steps ahead
        dict(name="bot_1k", kind="tick", plant="bot", n=1024, h=20),
        # the 100 Hz closed loop at the size of the benchmark, from host buffers
        dict(name="bot_host_16k", kind="host", plant="bot", n=16384, h=50),
        # 10,000 candidates with the method's per-step Gaussian noise
        dict(name="bot_noise_10k", kind="tick", plant="bot", n=10000, h=50, noise=True),
        # a million candidates, every slot's time to violation and cost kept (an offline study)
        dict(name="bot_1m", kind="tick", plant="bot", n=1048576, h=50, per_slot=True),
        # the 60 Hz race car in its closed loop
        dict(name="car_16k", kind="tick", plant="car", n=16384, h=60),
        # the race car at the screener's size with every slot's label kept (training data)
        dict(name="car_64k", kind="tick", plant="car", n=65536, h=60, per_slot=True),
        # the same prediction on the tensor cores
        dict(name="car_tensor_64k", kind="tick", plant="car", n=65536, h=60, rollout="tensor"),
        # the factorised prediction, an odd number of candidates and a long horizon
        dict(name="car_factored_30k", kind="tick", plant="car", n=30001, h=100,
             rollout="factored"),
        # a tick that the trained network screens first
        dict(name="car_screened_64k", kind="screened", n=65536, h=60, tau=0.95),
        # forward and backward of the screener on one training minibatch
        dict(name="train_8k", kind="train", batch=8192),
        # both plants' sessions served together, one batch each
        dict(name="serve_48", kind="serve", sessions=48),
        # the model of a new plant: 20,000 race-car transitions
        dict(name="fit_car_20k", kind="fit", plant="car", m=20000),
    ]


def draw(rng: random.Random):
    size = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    kind = rng.choice(["tick", "tick", "tick", "tick", "host", "screened", "train", "serve", "fit"])
    plant = rng.choice(["bot", "car"])
    if kind == "host":
        return dict(kind=kind, plant=plant, n=size(1000, 65536), h=rng.randint(20, 100))
    if kind == "screened":
        # without the network (tau 0) a sixteenth of the slots in cost order, as the benchmark does
        return dict(kind=kind, n=size(4000, 65536), h=rng.randint(40, 80),
                    tau=rng.choice([0.0, 0.9, 0.95]))
    if kind == "train":
        return dict(kind=kind, batch=size(200, 16384))
    if kind == "serve":
        return dict(kind=kind, sessions=size(2, 48))
    if kind == "fit":
        return dict(kind=kind, plant=plant, m=size(500, 20000))
    c = dict(kind=kind, plant=plant, n=size(500, 1048576 if plant == "bot" else 131072),
             h=rng.randint(20, 100), per_slot=rng.random() < 0.5)
    option = rng.choice(["", "", "noise" if plant == "bot" else "tensor", "factored", "no_user"])
    if option == "noise":
        c["noise"] = True
        c["n"] = min(c["n"], 100000)
    elif option == "no_user":
        c["user"] = False
    elif option:
        c["rollout"] = option
    if plant == "bot" and not option and rng.random() < 0.3:
        c["sampler"] = "grid"
    return c


# ---------------------------------------------------------------- what a program holds
_shared = {}


def _context():
    if "ctx" not in _shared:
        _shared["ctx"] = mpmi.Context(0)
    return _shared["ctx"]


class State:
    """Handles and buffers of one case; closed in the order that the library asks for."""

    def __init__(self, case):
        self.case, self.tick = case, 0
        self.sessions, self.servers, self.screeners, self.models = [], [], [], []

    def __del__(self):
        for s in self.sessions:
            s.close()
        for s in self.servers + self.screeners + self.models:
            s.free()


def _model(st, plant, rng, track):
    """A fitted operator as a saved model holds it, with its safety set."""
    K = _least_squares(plant, *_transitions(plant, rng, 5000))[0]
    m = mpmi.model_from_operator(_context(), plant, K.astype(np.float32).astype(np.float64))
    st.models.append(m)
    mpmi.set_safety_set(m, *SAFE[plant], track=track, half_width=HALF_WIDTH)
    return m


def _dev(a):
    return torch.tensor(a, dtype=torch.float64, device="cuda")


def _weights(rng):
    f32 = lambda s, shape: rng.normal(0.0, s, shape).astype(np.float32)  # noqa: E731
    return dict(W1=f32(math.sqrt(2 / 12), (128, 12)), b1=f32(0.05, 128),
                W2=f32(math.sqrt(2 / 128), (128, 128)), b2=f32(0.05, 128),
                w3=f32(math.sqrt(1 / 128), 128), b3=f32(0.05, ()))


def _network(P, f):
    gelu = lambda z: torch.nn.functional.gelu(z, approximate="tanh")  # noqa: E731
    h = gelu(f @ P["W1"].T + P["b1"])
    return torch.sigmoid(gelu(h @ P["W2"].T + P["b2"]) @ P["w3"] + P["b3"])


def _trained(rng, f, y, steps=240, batch=4096):
    """Weights of a screener trained on (features, ttv / H), in 64 bits."""
    P = {k: torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=True)
         for k, v in _weights(rng).items()}
    opt = torch.optim.Adam(P.values(), lr=3e-3)
    f, y = f.double(), y.double()
    for _ in range(steps):
        i = torch.from_numpy(rng.integers(0, len(f), batch)).cuda()
        opt.zero_grad()
        (_network(P, f[i]) - y[i]).square().mean().backward()
        opt.step()
    return {k: v.detach().cpu().numpy() for k, v in P.items()}


def _labels(st, model, scr, rng, track, n, h, ticks):
    """Screener inputs and ttv / H of every slot of `ticks` ticks."""
    s = mpmi.Session(_context(), model, n, h, LO["car"], HI["car"], seed=int(rng.integers(1 << 30)))
    st.sessions.append(s)
    x, u = _states("car", rng, ticks, track)
    f = torch.empty((ticks, n + 1, 12), device="cuda")
    ttv = torch.empty((ticks, n + 1), dtype=torch.int32, device="cuda")
    res = torch.zeros(mpmi.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    for t in range(ticks):
        xd, ud = _dev(x[t]), _dev(u[t])
        scr.features(s, xd, ud, f[t], tick=t)
        mpmi.evaluate_candidates_device(s, xd, ud, res, tick=t, ttv_dev=ttv[t])
    torch.cuda.synchronize()
    return f.reshape(-1, 12), (ttv.float() / h).reshape(-1)


def _requests(rng, sessions):
    """(plant, N, H, seed) of the serving mix: half balance bots, half race cars."""
    return [("bot" if i % 2 == 0 else "car", int(round(math.exp(rng.uniform(math.log(1024), math.log(65536))))),
             int(rng.integers(20, 101)), int(rng.integers(1 << 30))) for i in range(sessions)]


def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _train_data(case, seed):
    """Weights, minibatch and targets of a training step: ten inputs that a tick's slots share
    (a minibatch mixes the slots of many ticks) and the candidate's two."""
    rng, b = _rng(seed), case["batch"]
    w = _weights(rng)
    ticks = np.concatenate([rng.uniform(-0.6, 0.6, (64, 2)), rng.uniform(0.95, 1.0, (64, 1)),
                            rng.uniform(0.2, 0.8, (64, 1)), rng.normal(0.0, 0.2, (64, 6))], axis=1)
    f = np.concatenate([ticks[rng.integers(0, 64, b)], rng.uniform(-1.0, 1.0, (b, 2))], axis=1)
    y = np.where(rng.random(b) < 0.5, 1.0, rng.integers(5, 60, b) / 60.0)
    return w, f.astype(np.float32), y.astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    st = State(case)
    rng = _rng(seed)
    if kind == "fit":
        st.data = _transitions(case["plant"], rng, case["m"])
        _context()
        return st
    if kind == "train":
        w, f, y = _train_data(case, seed)
        model = _model(st, "car", rng, _track(rng))
        st.scr = mpmi.Screener(_context(), model, w, max_batch=case["batch"], max_slots=1024)
        st.screeners.append(st.scr)
        st.f, st.y = torch.from_numpy(f).cuda(), torch.from_numpy(y).cuda()
        st.grad = torch.zeros(mpmi.SCREENER_PARAMS, device="cuda")
        st.loss = torch.zeros(1, device="cuda")
        return st
    if kind == "serve":
        st.ids, st.x, st.u, st.srv = {}, {}, {}, {}
        req = _requests(rng, case["sessions"])
        for plant in ("bot", "car"):
            track = _track(rng) if plant == "car" else None
            mine = [r for r in req if r[0] == plant]
            srv = mpmi.Server(_context(), _model(st, plant, rng, track), max(1, len(mine)))
            st.servers.append(srv)
            st.srv[plant] = srv
            st.ids[plant] = [srv.admit(n, h, LO[plant], HI[plant], seed=s) for _, n, h, s in mine]
            st.x[plant], st.u[plant] = _states(plant, rng, len(mine), track)
        return st
    plant, n, h = case.get("plant", "car"), case["n"], case["h"]
    # the sampler's key comes first, so that exact() knows it
    key = int(rng.integers(1 << 30))
    track = _track(rng) if plant == "car" else None
    x, u = _states(plant, rng, 1, track)
    model = _model(st, plant, rng, track)
    st.s = mpmi.Session(_context(), model, n, h, LO[plant], HI[plant],
                        include_user=case.get("user", True), sampler=case.get("sampler", "uniform"),
                        seed=key)
    st.sessions.append(st.s)
    if kind == "host":
        st.x, st.u = x[0], u[0]
        return st
    st.x, st.u = _dev(x[0]), _dev(u[0])
    st.res = torch.zeros(mpmi.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    if kind == "screened":
        st.scr = mpmi.Screener(_context(), model, _weights(rng), max_batch=1, max_slots=n + 1)
        st.screeners.append(st.scr)
        st.scr.set_weights(_trained(rng, *_labels(st, model, st.scr, rng, track, 2047, h, 32)))
        return st
    st.ttv = st.cost = None
    if case.get("per_slot"):
        st.ttv = torch.zeros(st.s.n_slots, dtype=torch.int32, device="cuda")
        st.cost = torch.zeros(st.s.n_slots, device="cuda")
    if case.get("noise"):
        st.s.set_noise(SIGMA)
    if "rollout" in case:
        st.s.set_rollout(case["rollout"])
    return st


# ---------------------------------------------------------------- one pass
def run(st):
    kind, t = st.case["kind"], st.tick
    st.tick += 1  # every call is the next tick: new candidates
    if kind == "tick":
        mpmi.evaluate_candidates_device(st.s, st.x, st.u, st.res, tick=t, ttv_dev=st.ttv,
                                        cost_dev=st.cost)
        return [st.res] if st.ttv is None else [st.res, st.ttv, st.cost]
    if kind == "host":
        mpmi.evaluate_candidates(st.s, st.x, st.u, tick=t)
        return mpmi.select_input(st.s)
    if kind == "screened":
        tau = st.case["tau"]
        mpmi.evaluate_screened(st.s, st.scr, st.x, st.u, st.res, tau=tau, m=16, tick=t,
                               k=1 if tau > 0 else st.case["n"] // 16)
        return [st.res]
    if kind == "train":
        st.scr.gradients(st.f, st.y, st.grad, st.loss)
        return [st.grad, st.loss]
    if kind == "serve":
        for plant, srv in st.srv.items():
            srv.submit(st.ids[plant], st.x[plant], st.u[plant], [t] * len(st.ids[plant]))
            srv.launch()
        out = {}
        for plant, srv in st.srv.items():
            got = sorted(srv.collect(), key=lambda g: g[0]) if st.ids[plant] else []
            out[plant] = {k: np.array([r[k] for _, r in got])
                          for k in ("u_r", "index", "status", "n_safe", "executed_steps")}
        return out
    model, residual = mpmi.fit_model(_context(), st.case["plant"], *st.data)
    K = model.get_operator()
    model.free()
    return [K, residual]


# ---------------------------------------------------------------- the least work of a pass
def _tick_flops(plant, n, h):
    # the held features keep their values over the horizon: the other rows and columns remain
    return LIVE * n * h * 2 * (10 * 10 if plant == "bot" else 28 * 28)


def work(case):
    kind = case["kind"]
    if kind == "fit":
        nx, n = (4, 12) if case["plant"] == "bot" else (6, 32)
        nu, m = len(LO[case["plant"]]), case["m"]
        # read the transitions; triangularise n columns and carry n right-hand sides
        return dict(bytes=8 * m * (2 * nx + nu), flops=6.0 * m * n * n)
    if kind == "train":
        b = case["batch"]
        return dict(bytes=4 * (b * 13 + 2 * mpmi.SCREENER_PARAMS),
                    flops=2.0 * b * (12 * 128 + 128 * 128 + 128) * 3)
    if kind == "serve":
        # the mix's mean candidate count is that of the log-uniform law; both halves' horizons
        # average 60
        n, s = (65536 - 1024) / math.log(64), case["sessions"]
        flops = (s - s // 2) * _tick_flops("bot", n, 60) + (s // 2) * _tick_flops("car", n, 60)
        return dict(bytes=s * 400.0, flops=flops)
    plant, n, h = case.get("plant", "car"), case["n"], case["h"]
    fixed = 4 * 144 + 176 if plant == "bot" else 4 * 1024 + 38800 + 176
    if kind == "screened":
        # every slot's cost (and its score: a 12-128-128-1 network), then a few of the rollouts
        net = 2.0 * (12 * 128 + 128 * 128 + 128) * n if case["tau"] > 0 else 0.0
        return dict(bytes=fixed + (73220 if case["tau"] > 0 else 0),
                    flops=6.0 * n + net + 0.05 * _tick_flops("car", n, h))
    if case.get("rollout") == "factored":
        # three read-outs (position and speed) of four products each per step
        reads, held = (2, 2) if plant == "bot" else (3, 4)
        return dict(bytes=fixed + 8.0 * n * bool(case.get("per_slot")),
                    flops=LIVE * n * h * 2 * reads * held)
    return dict(bytes=fixed + 8.0 * n * bool(case.get("per_slot")), flops=_tick_flops(plant, n, h))


# ---------------------------------------------------------------- in 64 bits
def _philox(count, key):
    """Philox4x32-10 words of counters (i, 0, 0, 0), i < count: the first tick's candidates."""
    c = [np.arange(count, dtype=np.uint64)] + [np.zeros(count, dtype=np.uint64) for _ in range(3)]
    low, k0, k1 = np.uint64(0xFFFFFFFF), key & 0xFFFFFFFF, key >> 32
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & low,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def exact(case, seed):
    """Costs, gradients and operators; a decision (a slot, a step count) has no 64-bit value
    of its own."""
    kind = case["kind"]
    if kind == "fit":
        return list(_least_squares(case["plant"], *_transitions(case["plant"], _rng(seed), case["m"])))
    if kind == "train":
        w, f, y = _train_data(case, seed)
        P = {k: torch.tensor(v, dtype=torch.float64, requires_grad=True) for k, v in w.items()}
        loss = (_network(P, torch.from_numpy(f).double()) - torch.from_numpy(y).double()).square().mean()
        loss.backward()
        return [torch.cat([P[k].grad.reshape(-1) for k in ("W1", "b1", "W2", "b2", "w3", "b3")]),
                loss.detach().reshape(1)]
    if kind != "tick" or not case.get("per_slot"):
        return None
    plant, n = case["plant"], case["n"]
    rng = _rng(seed)
    key = int(rng.integers(1 << 30))
    u = _states(plant, rng, 1, _track(rng) if plant == "car" else None)[1][0]
    lo, w = LO[plant].astype(np.float32), (HI[plant] - LO[plant]).astype(np.float32)
    if case.get("sampler") == "grid":
        xi = ((np.arange(n) + 0.5) * 2.0 / n - 1.0).astype(np.float32)[:, None]
    else:  # candidates are 32-bit numbers by definition
        words = _philox(n, key)
        xi = np.stack([lo[j] + w[j] * ((words[j] >> np.uint64(8)).astype(np.float32) * np.float32(2.0 ** -24))
                       for j in range(len(lo))], axis=1)
    cost = np.square(xi.astype(np.float64) - u).sum(axis=1)
    if case.get("user", True):
        cost = np.concatenate([[0.0], cost])
    return [None, None, cost]
