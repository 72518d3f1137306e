"""Packing of scenes with many lanes: few vehicles in them (the search for the
first lane that no longer fits a segment must not walk all empty lanes from each
one), more lanes than one block or the whole cluster stages, a lane longer than
a segment.
Against the FP64 oracle (positions within 1e-3 m, the parity tests' bar), and
timed beside a scene with as many lanes that all hold a vehicle, which has the
same offsets to stage and as many segments at least."""
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


def sparse(lanes, at, n):
    c = np.zeros(lanes, np.int64)
    c[at] = n
    return c


def dev(x, t=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")


def scene_args(api, counts):
    sc = synth.make_scene(counts, np.random.default_rng(1))
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    return sc, (dev(sc["theta_true"]), dev(sc["p_init"]), dev(sc["v_init"]), scene)


@pytest.mark.parametrize("counts", [
    sparse(30000, slice(0, None, 1000), 2),
    sparse(32768, slice(32767, None), 64),
    sparse(32768, slice(0, 1), 1),
    sparse(32769, slice(16000, 16400), 3),
    sparse(4096, slice(5, None, 41), 64),        # prepared in one launch
    sparse(20000, slice(0, 18), 1),              # empty lanes to the end after one more than a linear search
    sparse(20000, slice(3, None, 17), 5),
    np.full(5000, 20),                           # fewer chunks than blocks
    np.r_[np.full(4200, 1), np.full(100, 64)],
    sparse(262144, slice(9, None, 61), 4),       # the most lanes that the cluster stages
    sparse(300000, slice(7, None, 97), 3),       # more
], ids=lambda c: "%dx%d" % (len(c), c.sum()))
def test_mostly_empty_lanes(api, counts):
    sc, args = scene_args(api, counts)
    K, N = 5, int(sc["lane_off"][-1])
    P, V = oracle.forward(sc["lane_off"], sc["length"], sc["theta_true"], sc["p_init"], sc["v_init"], K, DT)
    y = P[1:] + np.random.default_rng(2).normal(0, 1.0, size=(K, N))
    L, seed = oracle.mse_seed(P, synth.f32(y), 1)
    g_ref, _, _ = oracle.adjoint(sc["lane_off"], sc["length"], sc["theta_true"], K, DT, P, V, seed)
    for shape in ((0, 0), (2, 1), (4, 4)):
        ctx = api.Context(vpt=shape[0], warps_per_segment=shape[1])
        traj = api.simulate(*args, K, DT, ctx=ctx)
        loss, g, _, _ = api.loss_grad(*args, K, DT, dev(synth.f32(y)), 1, ctx=ctx)
        ctx.check_status()
        assert float(np.abs(traj.double().cpu().numpy() - P).max()) <= 1e-3
        assert abs(loss.item() - L) <= 1e-5 * L
        for r in range(6):
            assert np.linalg.norm(g[r].double().cpu().numpy() - g_ref[r]) <= 1e-4 * np.linalg.norm(g_ref[r]) + 1e-12


@pytest.mark.parametrize("lanes,at", [(100, 57), (5000, 4999), (5000, 2000)])
def test_lane_longer_than_a_segment_is_flagged(api, lanes, at):
    counts = np.full(lanes, 20)
    counts[at] = 65
    sc, args = scene_args(api, counts)
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]), max_lane=64)
    ctx = api.Context(vpt=2, warps_per_segment=1)
    api.simulate(*args[:3], scene, 3, DT, ctx=ctx)
    with pytest.raises(Exception, match="lane"):
        ctx.check_status()


@pytest.mark.parametrize("lanes", [4096, 30000])
def test_empty_lanes_cost_no_more_than_full_ones(api, lanes):
    def us(counts):
        _, args = scene_args(api, counts)
        N = int(counts.sum())
        y = torch.zeros((1, N), device="cuda")
        ctx = api.Context(vpt=4, warps_per_segment=4)
        run = lambda: api.loss_grad(*args, 1, DT, y, 1, ctx=ctx)  # noqa: E731
        for _ in range(3):
            run()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for _ in range(20):
            torch.cuda.synchronize()
            a.record()
            for _ in range(4):
                run()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 4 * 1e3)
        return best

    full, empty = us(np.ones(lanes, np.int64)), us(sparse(lanes, slice(0, None, 1000), 2))
    assert empty <= 1.3 * full, (empty, full)
