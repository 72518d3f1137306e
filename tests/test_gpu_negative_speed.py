"""Gradients of scenes whose vehicles start with a negative speed (accepted, and
non-negative after one step): with delta = 4 the delta gradient takes r^4 ln r
as 0 for r <= 0, as the oracle and the CPU backend do.  With speeds of -0.9 to -0.2
m/s, targets v0 of 1-2 m/s and steps of 1 s the first step would otherwise carry
most of the delta gradient.  The parity tests' bar applies (1e-4 relative per
parameter)."""
import numpy as np
import pytest

import oracle
from paper_2412_16750_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DT = 1.0


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16750_gb300 import api as _api
    return _api


@pytest.mark.parametrize("counts,K,shape", [
    ((3, 1, 30, 7), 1, (0, 0)),
    ((3, 1, 30, 7), 6, (0, 0)),
    ((3, 1, 30, 7), 12, (4, 4)),
    ((33, 64, 2), 6, (2, 8)),
    ((33, 64, 2), 6, (8, 1)),
])
def test_delta_gradient_after_a_negative_start(api, counts, K, shape):
    rng = np.random.default_rng(sum(counts) + K)
    sc = synth.make_scene(counts, rng)
    N = int(sc["lane_off"][-1])
    th = sc["theta_true"].copy()
    th[0] = rng.uniform(1.0, 2.0, size=N)
    th = synth.f32(th)
    v0 = synth.f32(np.where(rng.random(N) < 0.7, -1.0, 1.0) * rng.uniform(0.2, 0.9, size=N))
    assert (v0 < 0).any()
    P, V = oracle.forward(sc["lane_off"], sc["length"], th, sc["p_init"], v0, K, DT)
    assert np.isfinite(P).all()
    Y = synth.f32(P[1:] + rng.normal(0, 2.0, size=(K, N)))
    gV = synth.f32(rng.normal(size=(K + 1, N)))
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    ctx = api.Context(vpt=shape[0], warps_per_segment=shape[1])
    args = dev(th), dev(sc["p_init"]), dev(v0), scene, K, DT
    _, seed = oracle.mse_seed(P, Y, 1)
    for got, q, gv in ((api.loss_grad(*args, dev(Y), 1, ctx=ctx)[1], seed, None),
                       (api.backward(*args, dev(seed), dev(gV), ctx=ctx)[0], seed, gV)):
        ctx.check_status()
        ref, _, _ = oracle.adjoint(sc["lane_off"], sc["length"], th, K, DT, P, V, q, gv)
        for r in range(6):
            d = np.linalg.norm(got[r].double().cpu().numpy() - ref[r])
            assert d <= 1e-4 * np.linalg.norm(ref[r]) + 1e-12, r
