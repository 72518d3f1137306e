"""Horizons of up to two intervals that 2 vehicles per thread run as one (its tape
holds 16 steps): gradients, dense seeds and fits equal those of 4 vehicles per
thread, which keep the interval, bit for bit; the loss keeps the sums of the
interval's segments."""
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


@pytest.mark.parametrize("K,C", [(2, 1), (9, 8), (10, 5), (15, 8), (16, 8), (16, 15), (17, 9)])
@pytest.mark.parametrize("counts,stride", [((64, 3, 1, 60), 1), ((33, 0, 17, 5, 64, 2), 2)])
def test_one_run_equals_two(api, K, C, counts, stride):
    rng = np.random.default_rng(K + C)
    sc = synth.make_scene(counts, rng)
    N, n_obs = int(sc["lane_off"][-1]), K // stride
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    args = dev(sc["theta_true"]), dev(sc["p_init"]), dev(sc["v_init"]), scene, K, DT
    y = api.simulate(*args)[stride::stride][:n_obs].contiguous() + dev(rng.normal(0, 2.0, size=(n_obs, N)))
    gP, gV = dev(rng.normal(size=(K + 1, N))), dev(rng.normal(size=(K + 1, N)))
    ref = None
    for shape in ((4, 4), (2, 1), (2, 2), (2, 8)):
        ctx = api.Context(vpt=shape[0], warps_per_segment=shape[1], ckpt_interval=C)
        loss, *out = api.loss_grad(*args, y, stride, ctx=ctx)
        out += list(api.backward(*args, gP, gV, ctx=ctx))
        for mode in ("graph", "single"):
            ctx.set_fit_mode(mode)
            w = dev(synth.plain_init(N))
            api.fit(w, *args[1:], y, stride, 3, ctx=ctx)
            out.append(w)
        ctx.check_status()
        if ref is None:
            ref, ref_loss = out, loss.item()
        assert abs(loss.item() - ref_loss) <= 1e-6 * ref_loss
        for a, b in zip(out, ref):
            assert torch.equal(a, b), shape
