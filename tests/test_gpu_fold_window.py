"""Horizons around one fold window of the gradient sums (256 steps) at checkpoint
intervals that do not divide it: 251-256 steps at interval 50 are six checkpoint
segments, one more than a window holds, and yet within the window, so that no
totals exist.  Within it a gradient does not depend on the interval, bit for bit,
so each is compared with the one at interval 8, which divides the window and which
the parity tests compare with the FP64 oracle."""
import numpy as np
import pytest

import oracle
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


def dev(x, t=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")


@pytest.mark.parametrize("K,C", [(250, 50), (251, 50), (256, 50), (253, 9), (256, 3), (256, 64)])
def test_gradients_and_fits(api, K, C):
    rng = np.random.default_rng(K + C)
    counts = (64, 3, 1, 60, 0, 41)
    sc = synth.make_scene(counts, rng)
    N = int(sc["lane_off"][-1])
    th = synth.f32(sc["theta_true"] * np.r_[rng.uniform(0.9, 1.1, size=(5, N)), np.ones((1, N))])
    P, _ = oracle.forward(sc["lane_off"], sc["length"], th, sc["p_init"], sc["v_init"], K, DT)
    Y = synth.f32(P[1:] + rng.normal(0, 2.0, size=(K, N)))
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    state = dev(sc["p_init"]), dev(sc["v_init"])
    y = dev(Y)
    gP = dev(synth.f32(rng.normal(size=(K + 1, N))))
    batch = api.Batch([0, 3, 6], [K, K], [0.1, 0.1], [1, 1], sc["lane_off"], sc["length"])
    n0 = int(sc["lane_off"][3])
    yb = torch.cat([y[:, :n0].reshape(-1), y[:, n0:].reshape(-1)])

    def outputs(shape, interval):
        ctx = api.Context(vpt=shape[0], warps_per_segment=shape[1], ckpt_interval=interval)
        out = list(api.loss_grad(dev(th), *state, scene, K, DT, y, 1, ctx=ctx)[1:])
        out += list(api.backward(dev(th), *state, scene, K, DT, gP, ctx=ctx))
        out += list(api.batch_loss_grad(dev(th), *state, batch, yb, ctx=ctx)[2:])
        for mode in ("graph", "single"):
            ctx.set_fit_mode(mode)
            w = dev(synth.plain_init(N))
            api.fit(w, *state, scene, K, DT, y, 1, 2, ctx=ctx)
            out.append(w)
        w = dev(synth.plain_init(N))
        api.batch_fit(w, *state, batch, yb, 2, ctx=ctx)
        ctx.check_status()
        return out + [w]

    for shape in ((0, 0), (2, 1), (4, 4), (8, 4)):
        got, ref = outputs(shape, C), outputs(shape, 8)
        for a, b in zip(got, ref):
            assert torch.equal(a, b), shape
