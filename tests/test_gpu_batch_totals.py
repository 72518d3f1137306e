"""A batch of more scenarios than the lane packing of one scene has chunks, past
one fold window of the gradient sums: every segment has totals of its own.  The
same lanes as one scene give the same gradients, bit for bit (a vehicle's sums
depend on its own steps and the fold windows only)."""
import numpy as np
import pytest

from paper_2412_16750_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DT = float(np.float32(0.1))


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16750_gb300 import api as _api
    return _api


@pytest.mark.parametrize("shape", [(0, 0), (4, 4), (8, 8)])
def test_more_scenarios_than_chunks(api, shape):
    S, K = 2500, 264
    rng = np.random.default_rng(7)
    counts = rng.integers(1, 6, size=S)
    sc = synth.make_scene(counts, rng)
    N = int(sc["lane_off"][-1])
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    args = dev(sc["theta_true"]), dev(sc["p_init"]), dev(sc["v_init"])
    y = api.simulate(*args, scene, K, DT)[8::8].contiguous() + dev(rng.normal(0, 1.0, size=(K // 8, N)))
    batch = api.Batch(np.arange(S + 1), np.full(S, K), np.full(S, DT, np.float32), np.full(S, 8), sc["lane_off"],
                      sc["length"])
    lo = sc["lane_off"]
    yb = torch.cat([y[:, int(lo[s]):int(lo[s + 1])].reshape(-1) for s in range(S)])
    ctx = api.Context(vpt=shape[0], warps_per_segment=shape[1])
    ref = api.loss_grad(*args, scene, K, DT, y, 8, ctx=api.Context(vpt=4, warps_per_segment=4))[1:]
    got = api.batch_loss_grad(*args, batch, yb, ctx=ctx)[2:]
    ctx.check_status()
    for a, b in zip(got, ref):
        assert torch.equal(a, b)


def test_malformed_offsets_past_the_window_are_flagged(api):
    """Offsets that go back and forth make more segments than lanes of so few
    vehicles can: the call flags them and leaves the context usable."""
    L, K = 4000, 264
    rng = np.random.default_rng(8)
    sc = synth.make_scene([1, 2], rng)
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    args = dev(sc["theta_true"]), dev(sc["p_init"]), dev(sc["v_init"])
    y = torch.zeros((K, 3), device="cuda")
    bad = api.Scene.from_lane_off(dev(np.arange(L + 1) % 2, torch.int32), dev(sc["length"]))
    good = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    ctx = api.Context(vpt=4, warps_per_segment=4)
    ref = api.loss_grad(*args, good, K, DT, y, 1, ctx=ctx)
    ctx.check_status()
    api.loss_grad(*args, bad, K, DT, y, 1, ctx=ctx)
    with pytest.raises(Exception, match="lane"):
        ctx.check_status()
    for a, b in zip(api.loss_grad(*args, good, K, DT, y, 1, ctx=ctx), ref):
        assert torch.equal(a, b)
    ctx.check_status()
