"""The adjoint's tape (speeds, seeds and one coefficient in shared memory, the
others in tensor memory) over its depths: checkpoint intervals shallower and
deeper than the tape, with and without tape blocks, every kernel shape, rows
that allow 16-byte copies (vehicles a multiple of four) and rows that do not,
observed every step and sparsely, dense seeds of positions and speeds.

A vehicle's gradient is the same sum in the same order whatever the shape and
the interval (the horizon stays within one fold window of the sums), so all of
them have to agree bit for bit; against the FP64 oracle the parity tests' bars
apply (1e-4 relative per parameter)."""
import numpy as np
import pytest

import oracle
from paper_2412_16750_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DT = float(np.float32(0.1))
SHAPES = ((0, 0), (2, 1), (2, 4), (2, 8), (4, 1), (4, 2), (4, 4), (4, 8), (8, 1), (8, 4), (8, 8))
INTERVALS = (1, 2, 3, 8, 9, 16, 17, 40, 64)


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16750_gb300 import api as _api
    return _api


def dev(x, t=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")


@pytest.mark.parametrize("counts,K,stride", [
    ((64, 3, 1, 60), 41, 1),        # 128 vehicles: aligned rows
    ((33, 0, 17, 5, 64, 2), 41, 3),  # 121: unaligned
    ((1,), 1, 1),
    ((63, 64), 8, 9),               # nothing observed
    ((30,) * 11, 17, 17),           # one observation, at the last step
])
def test_gradient_bits_over_shapes_and_intervals(api, counts, K, stride):
    rng = np.random.default_rng(sum(counts) + K)
    sc = synth.make_scene(counts, rng)
    N, n_obs = int(sc["lane_off"][-1]), K // stride
    th = synth.f32(sc["theta_true"] * np.r_[rng.uniform(0.9, 1.1, size=(5, N)), np.ones((1, N))])
    P, V = oracle.forward(sc["lane_off"], sc["length"], th, sc["p_init"], sc["v_init"], K, DT)
    Y = synth.f32(P[stride::stride][:n_obs] + rng.normal(0, 2.0, size=(n_obs, N)))
    gP = synth.f32(rng.normal(size=(K + 1, N)))
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    args = dev(th), dev(sc["p_init"]), dev(sc["v_init"]), scene, K, DT
    y, wP, wV = dev(Y), dev(gP), dev(rng.normal(size=(K + 1, N)))
    ref = None
    for shape in SHAPES:
        for C in INTERVALS if shape in ((0, 0), (4, 4), (2, 8)) else (8, 17):
            ctx = api.Context(vpt=shape[0], warps_per_segment=shape[1], ckpt_interval=C)
            loss, *out = api.loss_grad(*args, y if n_obs else None, stride, ctx=ctx)
            out += list(api.backward(*args, wP, ctx=ctx)) + list(api.backward(*args, wP, wV, ctx=ctx))
            ctx.check_status()
            if ref is None:
                ref, ref_loss = out, loss.item()
            assert abs(loss.item() - ref_loss) <= 1e-6 * ref_loss
            for a, b in zip(out, ref):
                assert torch.equal(a, b), (shape, C)
    L, seed = oracle.mse_seed(P, Y, stride) if n_obs else (0.0, np.zeros_like(P))
    assert abs(ref_loss - L) <= 1e-5 * abs(L)
    for got, q in ((ref[0], seed), (ref[3], gP)):
        g_ref, _, _ = oracle.adjoint(sc["lane_off"], sc["length"], th, K, DT, P, V, q)
        for r in range(6):
            scale = np.linalg.norm(g_ref[r])
            assert np.linalg.norm(got[r].double().cpu().numpy() - g_ref[r]) <= 1e-4 * scale + 1e-12


# the horizon is one interval: 20 bytes of checkpoint and 4 of initial gap per
# vehicle and a few KB of lane tables, but no room for a sub-checkpoint (20
# more), so the tape has to hold the interval whole
@pytest.mark.parametrize("shape,C", [((4, 4), 9), ((4, 1), 10), ((2, 4), 17), ((2, 8), 17), ((4, 2), 31)])
def test_interval_deeper_than_the_tape_without_room(api, shape, C):
    rng = np.random.default_rng(C)
    sc = synth.make_scene((100,) * 40, rng)
    N = 4000
    th = synth.f32(sc["theta_true"])
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    y = dev(np.stack([sc["p_init"] + 0.1 * (k + 1) * sc["v_init"] for k in range(C)]))
    res = []
    for cap in (0, 24 * N + 16384):
        ctx = api.Context(cap, *shape, ckpt_interval=C)
        res.append(api.loss_grad(dev(th), dev(sc["p_init"]), dev(sc["v_init"]), scene, C, DT, y, 1, ctx=ctx))
        ctx.check_status()
    (loss, *out), (loss_tight, *out_tight) = res
    assert abs(loss.item() - loss_tight.item()) <= 1e-6 * loss.item()
    for a, b in zip(out, out_tight):
        assert torch.equal(a, b)
