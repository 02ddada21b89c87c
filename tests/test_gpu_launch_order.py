"""Launches that may start before the previous kernel on the stream ends still read what
it wrote: inputs updated between ticks, results chained from tick to tick, several
streams, and graph replays."""
import numpy as np
import pytest

from workloads import data

from parity import bot_env, car_env, gpu_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_02318_gb300 import build, mpmi
    build.build()
    ctx = mpmi.Context(0)
    envs = dict(bot=bot_env(), car=car_env())
    return mpmi, ctx, {k: (e, gpu_model(mpmi, ctx, e)) for k, e in envs.items()}


def _case(lib, ctx, envs, which, N, rollout):
    import torch
    env, model = envs[which]
    s = lib.Session(ctx, model, N, 40, env.lo, env.hi, seed=3)
    s.set_rollout(rollout)
    x = (np.array([0.05, 0.1, 0.2, -0.1]) if which == "bot"
         else data.car_start_state(env.track, vx=12.0))
    u = data.to_f32_exact(data.user_input_once(2, env.lo, env.hi))
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    return s, dev(x), dev(u)


CASES = [("bot", 900, "full"), ("bot", 70000, "full"), ("bot", 3000, "factored"),
         ("car", 900, "full"), ("car", 16384, "full"), ("car", 66000, "full"),
         ("car", 5000, "tensor"), ("car", 5000, "factored")]


def _step(lib, s, x, u, res, t):
    """One tick, then a torch kernel that moves the state by the tick's own result."""
    lib.evaluate_candidates_device(s, x, u, res, tick=t)
    u_r = res[:8 * s.nu].view(dtype=x.dtype)
    x[1:1 + s.nu] += 0.01 * u_r


@pytest.mark.parametrize("which,N,rollout", CASES)
def test_back_to_back_ticks_see_each_other(setup, which, N, rollout):
    import torch
    lib, ctx, envs = setup
    out = []
    for wait in (True, False):
        s, x, u = _case(lib, ctx, envs, which, N, rollout)
        res = torch.zeros((30, lib.RESULT_BYTES), dtype=torch.uint8, device="cuda")
        for t in range(30):
            _step(lib, s, x, u, res[t], t)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        out.append((res.cpu().numpy(), x.cpu().numpy()))
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("which,N,rollout", CASES)
def test_captured_ticks_replay(setup, which, N, rollout):
    import torch
    lib, ctx, envs = setup
    s, x, u = _case(lib, ctx, envs, which, N, rollout)
    x0 = x.clone()
    res = torch.zeros((4, lib.RESULT_BYTES), dtype=torch.uint8, device="cuda")

    def run():
        x.copy_(x0)
        for t in range(4):
            _step(lib, s, x, u, res[t], t)

    run()
    torch.cuda.synchronize()
    want = res.cpu().numpy().copy()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        run()
    for _ in range(3):
        res.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(res.cpu().numpy(), want)
    s.close()


def test_host_ticks_alternate_streams(setup):
    """A host tick is ordered behind the last one's kernel whichever stream it takes."""
    import torch
    lib, ctx, envs = setup
    env, model = envs["bot"]
    streams = [torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()]
    out = []
    for pick in (lambda t: 0, lambda t: t % 3, lambda t: (t // 2) % 3):
        s = lib.Session(ctx, model, 4096, 40, env.lo, env.hi, seed=8)
        got = []
        for t in range(40):
            lib.evaluate_candidates(s, [0.05, 0.01 * t, 0.0, 0.0], [0.3], tick=t,
                                    stream=streams[pick(t)])
            r = lib.select_input(s)
            got.append((r["index"], r["n_safe"], r["executed_steps"], float(r["u_r"][0])))
        s.close()
        out.append(got)
    assert out[0] == out[1] == out[2]


def test_training_steps_back_to_back(setup):
    """Training steps with nothing between them but the kernel that gathers the next
    minibatch: the losses and weights of the same steps with a wait after each."""
    import torch
    lib, ctx, envs = setup
    model = envs["car"][1]
    rng = np.random.default_rng(12)
    bank = torch.tensor(rng.uniform(-1, 1, (20000, 12)), dtype=torch.float32, device="cuda")
    target = torch.tensor(rng.uniform(0, 1, 20000), dtype=torch.float32, device="cuda")
    sizes = [256, 17, 4096, 8192, 2500] * 10
    pick = [torch.tensor(rng.integers(0, 20000, b), device="cuda") for b in sizes]
    out = []
    for wait in (True, False):
        scr = lib.Screener(ctx, model, data.screener_init(7), max_batch=8192, max_slots=64)
        loss = torch.zeros(len(sizes), device="cuda")
        grad = torch.zeros((len(sizes), lib.SCREENER_PARAMS), device="cuda")
        f, y = torch.empty((8192, 12), device="cuda"), torch.empty(8192, device="cuda")
        scr.train_step(bank[:64], target[:64], loss[:1])  # all buffers and code are in place
        torch.cuda.synchronize()
        for t, i in enumerate(pick):
            torch.index_select(bank, 0, i, out=f[:len(i)])
            torch.index_select(target, 0, i, out=y[:len(i)])
            if t % 3 == 2:
                scr.gradients(f[:len(i)], y[:len(i)], grad[t], loss[t:t + 1])
            scr.train_step(f[:len(i)], y[:len(i)], loss[t:t + 1], lr=1e-2)
            scr.train_step(f[:len(i)], y[:len(i)], loss[t:t + 1], lr=1e-2)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        w = lib.pack_weights(scr.get_weights())
        out.append((loss.cpu().numpy(), grad.cpu().numpy(), w))
        scr.free()
    assert np.all(np.isfinite(out[0][0])) and len(set(out[0][0])) > 40
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("rollout", ["full", "tensor", "factored"])
def test_screened_ticks_back_to_back(setup, rollout):
    """Screened ticks in cost order and with the network, some falling back to the full
    evaluation, between training steps (the network's weights change under way) and on
    states that a kernel on the stream writes: the same ticks with a wait after each."""
    import torch
    lib, ctx, envs = setup
    env, model = envs["car"]
    N, T = 3000, 36
    rng = np.random.default_rng(21)
    x0 = data.car_start_state(env.track, vx=12.0)
    bank = x0 + rng.uniform(-1, 1, (T, 6)) * [1.5, 1.5, 0.2, 4, 0.3, 0.3]
    bank[::5, :2] += 40.0  # off the road: every kept slot is unsafe
    bank = torch.tensor(bank, device="cuda")
    u = torch.tensor(data.to_f32_exact(data.user_input_once(2, env.lo, env.hi)), device="cuda")
    f = torch.tensor(rng.uniform(-1, 1, (512, 12)), dtype=torch.float32, device="cuda")
    y = torch.tensor(rng.uniform(0, 1, 512), dtype=torch.float32, device="cuda")
    idx = [torch.tensor([t], device="cuda") for t in range(T)]
    w = {k: np.asarray(v).copy() for k, v in data.screener_init(7).items()}
    w["w3"] = (4.0 * w["w3"]).astype(np.float32)  # spread the scores
    out = []
    for wait in (True, False):
        scr = lib.Screener(ctx, model, w, max_batch=512, max_slots=N + 1)
        s = lib.Session(ctx, model, N, 40, env.lo, env.hi, seed=3)
        s.set_rollout(rollout)
        x = torch.zeros((1, 6), dtype=torch.float64, device="cuda")
        loss = torch.zeros(T, device="cuda")
        res = torch.zeros((T, lib.RESULT_BYTES), dtype=torch.uint8, device="cuda")
        lst = torch.full((T, N + 1), -1, dtype=torch.int32, device="cuda")
        cnt = torch.zeros((T, 1), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        for t in range(T):
            torch.index_select(bank, 0, idx[t], out=x)
            tau, k = [(0.0, 150), (0.5, 1), (0.9, 1)][t % 3]
            lists = dict(list_dev=lst[t], n_list_dev=cnt[t]) if t % 4 == 3 else {}
            lib.evaluate_screened(s, scr, x[0], u, res[t], k=k, tau=tau, m=16, tick=t, **lists)
            if t % 6 == 5:
                scr.train_step(f, y, loss[t:t + 1], lr=1e-2)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        kept = [sorted(row[:n].tolist()) for row, n in zip(lst.cpu().numpy(), cnt.cpu().numpy()[:, 0])]
        out.append((res.cpu().numpy(), loss.cpu().numpy(), kept))
        s.close()
        scr.free()
    flags = [lib.result_from_bytes(torch.from_numpy(r), 2)["flags"] for r in out[0][0]]
    assert any(g & 2 for g in flags) and any(not g & 2 for g in flags)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2] and any(out[0][2])
