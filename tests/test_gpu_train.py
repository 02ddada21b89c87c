"""The training kernel's tiles: gradients at batches around the tile sizes and the
block count against the float64 chain rule, and the same bits on every run."""
import numpy as np
import pytest

from oracle import screener as osc
from workloads import data

from parity import car_env, gpu_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_02318_gb300 import build, mpmi
    build.build()
    ctx = mpmi.Context(0)
    return mpmi, ctx, gpu_model(mpmi, ctx, car_env())


# tiles of 16 samples up to 16 per SM (152 SMs: 2432), 32 up to 4864, then 64; more
# tiles than blocks past 64 per SM (9728).  exact: max_batch = the batch, which
# bounds the blocks to one per 32 samples
@pytest.mark.parametrize("B, exact", [(1, True), (15, True), (16, False), (17, True), (33, True),
                                      (250, True), (250, False), (2433, False), (4864, True),
                                      (4865, False), (8192, False), (9729, False), (20011, True)])
def test_gradients_around_the_tiles(setup, B, exact):
    import torch
    lib, ctx, model = setup
    w = data.screener_init(7)
    rng = np.random.default_rng(B)
    f = data.to_f32_exact(rng.uniform(-1, 1, (B, 12)))
    t = data.to_f32_exact(rng.uniform(0, 1, B))
    scr = lib.Screener(ctx, model, w, max_batch=B if exact else 24000, max_slots=64)
    fd = torch.tensor(f, dtype=torch.float32, device="cuda")
    td = torch.tensor(t, dtype=torch.float32, device="cuda")
    out = []
    for _ in range(2):
        g = torch.full((lib.SCREENER_PARAMS,), float("nan"), device="cuda")
        loss = torch.full((1,), float("nan"), device="cuda")
        scr.gradients(fd, td, g, loss)
        torch.cuda.synchronize()
        out.append((g.cpu().numpy(), float(loss.item())))
    scr.free()
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    cache = osc.forward(w, f)
    ref = osc.backward(w, cache, t)
    got = lib.unpack_weights(out[0][0])
    assert out[0][1] == pytest.approx(osc.loss(cache["y"], t), rel=1e-5)
    for k in ref:
        # float32 sums of products: the error of each is a few hundred roundings
        # (2^-24) of the largest entry's terms
        scale = float(np.max(np.abs(ref[k])))
        assert np.max(np.abs(np.asarray(got[k]) - ref[k])) <= 1e-4 * scale + 1e-9, k


def test_step_whose_staging_runs_out_keeps_the_weights(setup):
    """A training step whose weights never arrive in shared memory (test hook): after the
    bounded wait the loss is NaN, the weights and Adam's moments are untouched, and the
    following steps are those of a screener that never saw it."""
    import torch
    lib, ctx, model = setup
    rng = np.random.default_rng(5)
    f = torch.tensor(rng.uniform(-1, 1, (40, 12)), dtype=torch.float32, device="cuda")
    y = torch.tensor(rng.uniform(0, 1, 40), dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, device="cuda")
    out = []
    for fail in (False, True):
        scr = lib.Screener(ctx, model, data.screener_init(7), max_batch=64, max_slots=64)
        losses = []
        for t in range(3):
            if fail and t == 1:
                before = lib.pack_weights(scr.get_weights())
                scr.withhold_staging(True)
                scr.train_step(f, y, loss, lr=1e-2)
                assert np.isnan(float(loss.item()))
                g = torch.zeros(lib.SCREENER_PARAMS, device="cuda")
                scr.gradients(f, y, g, loss)
                assert np.isnan(float(loss.item())) and bool(torch.isnan(g).any())
                scr.withhold_staging(False)
                assert np.array_equal(lib.pack_weights(scr.get_weights()), before)
            scr.train_step(f, y, loss, lr=1e-2)
            losses.append(float(loss.item()))
        out.append((losses, lib.pack_weights(scr.get_weights())))
        scr.free()
    # the step counter of Adam's bias correction has moved on by the failed step
    assert out[0][0][:2] == out[1][0][:2]
    assert np.all(np.isfinite(out[1][1])) and np.max(np.abs(out[0][1] - out[1][1])) < 2e-2


def test_every_smallest_tile_has_a_record(setup):
    """A screener made for its minibatch can give each tile of 16 samples a block of its
    own: the records (seen in the memory in use) grow by one per 16 samples."""
    lib, ctx, model = setup
    used = []
    for max_batch in (16, 160, 161):
        before = ctx.lib.mpmi_memory_in_use(ctx.handle)
        scr = lib.Screener(ctx, model, data.screener_init(7), max_batch=max_batch, max_slots=64)
        used.append(ctx.lib.mpmi_memory_in_use(ctx.handle) - before)
        scr.free()
    record = 4 * (lib.SCREENER_PARAMS + 1)  # the gradient and the loss
    assert used[1] - used[0] >= 9 * record and used[2] - used[1] >= record


def test_a_short_budget_takes_fewer_records(setup):
    """A memory budget that has no room for a record per tile still takes the screener, with
    fewer records (its blocks loop over tiles), down to one; its gradients meet the same
    bound.  Below that it is refused."""
    import torch
    lib, _, _ = setup
    record = 4 * (lib.SCREENER_PARAMS + 4)  # the gradient, the loss, padding, the flag
    free = lib.Context(0)
    model = gpu_model(lib, free, car_env())
    base = free.memory_in_use()
    scr = lib.Screener(free, model, data.screener_init(7), max_batch=320, max_slots=64)
    whole = free.memory_in_use() - base  # twenty records
    scr.free()
    model.free()
    rng = np.random.default_rng(6)
    w = data.screener_init(7)
    f = data.to_f32_exact(rng.uniform(-1, 1, (320, 12)))
    t = data.to_f32_exact(rng.uniform(0, 1, 320))
    cache = osc.forward(w, f)
    ref = osc.backward(w, cache, t)
    fd = torch.tensor(f, dtype=torch.float32, device="cuda")
    td = torch.tensor(t, dtype=torch.float32, device="cuda")
    for fewer in (0, 10, 19):
        ctx = lib.Context(0, base + whole - fewer * record)
        model = gpu_model(lib, ctx, car_env())
        scr = lib.Screener(ctx, model, w, max_batch=320, max_slots=64)
        assert ctx.memory_in_use() <= base + whole - fewer * record
        g, loss = torch.zeros(lib.SCREENER_PARAMS, device="cuda"), torch.zeros(1, device="cuda")
        scr.gradients(fd, td, g, loss)
        got = lib.unpack_weights(g.cpu().numpy())
        assert float(loss.item()) == pytest.approx(osc.loss(cache["y"], t), rel=1e-5)
        for k in ref:
            scale = float(np.max(np.abs(ref[k])))
            assert np.max(np.abs(np.asarray(got[k]) - ref[k])) <= 1e-4 * scale + 1e-9, k
        scr.free()
        model.free()
    ctx = lib.Context(0, base + whole - 20 * record)
    model = gpu_model(lib, ctx, car_env())
    with pytest.raises(lib.MpmiError):
        lib.Screener(ctx, model, w, max_batch=320, max_slots=64)
    model.free()
