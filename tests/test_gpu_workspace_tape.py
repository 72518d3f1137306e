"""Intervals deeper than the adjoint's tape under a workspace cap: room for the
checkpoints and `rows` sub-checkpoint rows (20 bytes per vehicle each), fewer than
the tape that runs best without a cap asks for.  The call then takes a deeper tape
with fewer groups per SM; the gradients keep their bits.  The rows are what the
tapes held in shared memory alone needed."""
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


@pytest.mark.parametrize("shape,C,rows,dense", [
    ((4, 4), 10, 0, False),
    ((4, 4), 50, 4, False),
    ((4, 1), 20, 1, False),
    ((2, 8), 17, 0, False),
    ((2, 8), 34, 1, False),
    ((2, 4), 17, 0, True),
    ((4, 4), 12, 0, True),
    ((4, 2), 11, 0, True),
    ((8, 4), 9, 0, True),
])
def test_capped_call_runs_with_a_deeper_tape(api, shape, C, rows, dense):
    rng = np.random.default_rng(C)
    sc = synth.make_scene((100,) * 40, rng)
    N, K = 4000, C
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    args = dev(sc["theta_true"]), dev(sc["p_init"]), dev(sc["v_init"]), scene, K, DT
    y = dev(np.stack([sc["p_init"] + 0.1 * (k + 1) * sc["v_init"] for k in range(K)]))
    gP = dev(rng.normal(size=(K + 1, N)))
    res = []
    # initial gaps and one checkpoint: 24 bytes per vehicle; a few KB of lane tables
    for cap in (0, 24 * N + 20 * N * rows + 16384):
        ctx = api.Context(cap, *shape, ckpt_interval=C)
        out = api.backward(*args, gP, ctx=ctx) if dense else api.loss_grad(*args, y, 1, ctx=ctx)[1:]
        ctx.check_status()
        res.append(out)
    for a, b in zip(*res):
        assert torch.equal(a, b)


def test_no_room_at_all_is_refused(api):
    sc = synth.make_scene((100,) * 40, np.random.default_rng(0))
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    args = dev(sc["theta_true"]), dev(sc["p_init"]), dev(sc["v_init"]), scene, 64, DT
    ctx = api.Context(24 * 4000 + 16384, 4, 4, ckpt_interval=64)
    with pytest.raises(Exception, match="workspace"):
        api.loss_grad(*args, torch.zeros((64, 4000), device="cuda"), 1, ctx=ctx)
