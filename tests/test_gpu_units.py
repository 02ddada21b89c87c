"""Ticks over sorted units (one lane per candidate, many candidates) against the same
ticks in a shape that never sorts, bit for bit in every per-slot output."""
import numpy as np
import pytest

from workloads import data

from parity import bot_env, car_env, gpu_model, run_gpu

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


def _same(a, b):
    assert np.array_equal(a["ttv"], b["ttv"]) and np.array_equal(a["cost"], b["cost"],
                                                                equal_nan=True)
    for k in ("index", "status", "n_safe", "ttv", "executed_steps", "n_slots"):
        assert a["result"][k] == b["result"][k]
    assert np.array_equal(a["result"]["u_r"], b["result"]["u_r"])


# one tile per warp (race car), several tiles per warp, two units per block (a unit
# holds 8192 slots: more than 152 x 8192 of them), ragged ends; with and without u_h,
# the grid sampler, per-step noise, two candidates per thread
@pytest.mark.parametrize("which,N,H,kw", [
    ("car", 20001, 60, {}), ("car", 38911, 30, {}), ("car", 38912, 60, {}),
    ("car", 65536, 60, {}), ("car", 150001, 30, {"include_user": False}),
    ("car", 130321, 25, {"sampler": "grid"}), ("car", 140000, 20, {"noise": True}),
    ("bot", 62500, 50, {}), ("bot", 70001, 50, {"include_user": False}),
    ("bot", 131072, 100, {"sampler": "grid"}), ("bot", 100003, 30, {"noise": True}),
    ("bot", 100003, 30, {"cands": 2}), ("bot", 1300001, 20, {})])
def test_sorted_units_change_no_result(setup, which, N, H, kw):
    lib, ctx, envs = setup
    env, model = envs[which]
    kw = dict(kw)
    noise, cands = kw.pop("noise", False), kw.pop("cands", 0)
    x_t = (np.array([0.1, 0.3, -0.5, 0.4]) if which == "bot" else
           data.car_start_state(env.track, vx=13.0) + np.array([1.0, -0.5, 0.05, 0, 0, 0]))
    u_h = data.to_f32_exact(data.user_input_once(5, env.lo, env.hi))
    out = []
    for shape in (dict(cands=cands, lanes=1 if cands else 0), dict(lanes=2)):
        s = lib.Session(ctx, model, N, H, env.lo, env.hi, seed=9, **kw, **shape)
        if noise:
            s.set_noise([0.002] * env.spec.lo.size)
        out.append([run_gpu(lib, s, x_t, u_h, tick=t) for t in (0, 1 << 33)])
        s.close()
    for a, b in zip(*out):
        _same(a, b)


@pytest.mark.parametrize("which", ["bot", "car"])
def test_caller_samples_outside_the_box(setup, which):
    """Caller samples may lie anywhere: outside the box, infinite, NaN."""
    import torch
    lib, ctx, envs = setup
    env, model = envs[which]
    N = 140003
    rng = np.random.default_rng(3)
    c = rng.uniform(3 * env.lo, 3 * env.hi, size=(N, len(env.lo))).astype(np.float32)
    c[::97, 0], c[5::101, 0], c[7::103, 0] = np.nan, np.inf, -np.inf
    cd = torch.tensor(c, device="cuda")
    x_t = np.zeros(4) if which == "bot" else data.car_start_state(env.track, vx=13.0)
    u_h = data.to_f32_exact(data.user_input_once(6, env.lo, env.hi))
    out = []
    for lanes in (0, 2):
        s = lib.Session(ctx, model, N, 20, env.lo, env.hi, sampler="external", lanes=lanes)
        out.append(run_gpu(lib, s, x_t, u_h, candidates=cd))
        s.close()
    _same(*out)


@pytest.mark.parametrize("which,sizes", [
    ("car", [(60001, 30), (40000, 60), (0, 25), (5000, 100), (33333, 20)]),
    ("bot", [(65536, 50), (65535, 20), (1, 60), (64, 50), (65000, 100), (50001, 35), (33, 90)])])
def test_served_units_equal_the_tick_alone(setup, which, sizes):
    """A batch large enough to be served as sorted units: every session's result is that
    of its tick alone, over two batches (other states, other candidates)."""
    import torch
    lib, ctx, envs = setup
    env, model = envs[which]
    srv = lib.Server(ctx, model, 8)
    slots = [srv.admit(n, h, env.lo, env.hi, seed=50 + i, stream_id=i)
             for i, (n, h) in enumerate(sizes)]
    rng = np.random.default_rng(4)
    for batch in range(2):
        x = (rng.uniform([-0.2, -0.6, -1, -0.8], [0.2, 0.6, 1, 0.8], (len(sizes), 4))
             if which == "bot" else data.car_start_state(env.track, vx=12.0)
             + rng.uniform(-1, 1, (len(sizes), 6)) * [2, 2, 0.1, 4, 0.3, 0.3])
        u = data.to_f32_exact(rng.uniform(env.lo, env.hi, (len(sizes), len(env.lo))))
        ticks = [1000 * batch + i for i in range(len(sizes))]
        srv.submit(slots, x, u, ticks)
        srv.launch()
        got = dict(srv.collect())
        for i, (n, h) in enumerate(sizes):
            s = lib.Session(ctx, model, n, h, env.lo, env.hi, seed=50 + i, stream_id=i, lanes=2)
            want = run_gpu(lib, s, x[i], u[i], tick=ticks[i])["result"]
            s.close()
            for k in ("index", "status", "n_safe", "ttv", "cost", "executed_steps", "n_slots"):
                assert got[slots[i]][k] == want[k], (i, k)
            assert np.array_equal(got[slots[i]]["u_r"], want["u_r"])
    srv.free()


def test_served_large_batch_equals_the_tick_alone(setup):
    """A batch past the size at which an untuned race-car server takes two candidates
    per thread (1,200 slots per SM): ragged ends, one-slot and long-horizon sessions."""
    sizes = [(131071, 30), (64000, 60), (0, 25), (30011, 100), (33, 20), (65, 40)]
    test_served_units_equal_the_tick_alone(setup, "car", sizes)


@pytest.mark.parametrize("which,N", [("bot", 140005), ("car", 65537), ("car", 20003)])
def test_samples_in_order(setup, which, N):
    """Caller samples ordered by the first input, sorted units and the factorised
    rollout's chunks against the two-lane shape."""
    import torch
    lib, ctx, envs = setup
    env, model = envs[which]
    c = np.random.default_rng(8).uniform(env.lo, env.hi, (N, len(env.lo))).astype(np.float32)
    cd = torch.tensor(c[np.argsort(c[:, 0])], device="cuda")
    x_t = np.array([0.1, 0.2, 0, 0]) if which == "bot" else data.car_start_state(env.track, vx=13.0)
    u_h = data.to_f32_exact(data.user_input_once(7, env.lo, env.hi))
    out = []
    for lanes in (0, 2):
        s = lib.Session(ctx, model, N, 40, env.lo, env.hi, sampler="external", lanes=lanes)
        out.append(run_gpu(lib, s, x_t, u_h, candidates=cd))
        if lanes == 0:  # the same prediction up to its rounding: nearly all steps agree
            s.set_rollout("factored")
            f = run_gpu(lib, s, x_t, u_h, candidates=cd)
        s.close()
    _same(*out)
    assert np.mean(f["ttv"] != out[0]["ttv"]) < 1e-3
    assert np.array_equal(f["cost"], out[0]["cost"])


@pytest.mark.parametrize("which,sizes", [
    ("car", [(3001, 30), (0, 60), (33, 25)]), ("car", [(9001, 60), (4096, 25), (257, 100)]),
    ("car", [(40001, 30), (9999, 60), (1, 20)]), ("bot", [(2001, 50), (0, 20), (77, 100)])])
def test_served_small_batches_equal_the_tick_alone(setup, which, sizes):
    """Batches of the sizes at which an untuned server takes several lanes per candidate."""
    test_served_units_equal_the_tick_alone(setup, which, sizes)


def test_tensor_rollout_one_or_several_tiles_per_cta(setup):
    """Either side of the size at which the tensor-core rollout's CTAs take more than one
    tile (another kernel instance): the candidates both ticks share agree bit for bit."""
    import torch
    lib, ctx, envs = setup
    env, model = envs["car"]
    tiles = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    x_t = data.car_start_state(env.track, vx=14.0) + np.array([0.5, -0.5, 0.1, 0, 0, 0])
    u_h = data.to_f32_exact(data.user_input_once(9, env.lo, env.hi))
    out = []
    for n_slots in (128 * tiles, 128 * tiles + 1):
        s = lib.Session(ctx, model, n_slots - 1, 60, env.lo, env.hi, seed=11)
        s.set_rollout("tensor")
        out.append(run_gpu(lib, s, x_t, u_h, tick=3))
        s.close()
    n = 128 * tiles
    assert np.array_equal(out[0]["ttv"], out[1]["ttv"][:n])
    assert np.array_equal(out[0]["cost"], out[1]["cost"][:n])
    assert 0 < out[0]["result"]["n_safe"] < n
