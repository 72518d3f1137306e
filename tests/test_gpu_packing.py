"""Packing of lanes into segments (launch_build_segments): scenes on each side
of its rules -- lanes that fit one wave, mean lanes under and over 16 vehicles,
more lanes than the staged offsets hold, a last chunk of a few lanes, empty
and single-vehicle lanes, lanes of a whole segment.

With delta = 4 everywhere a vehicle's trajectory and gradient do not depend on
the segment it lands in, so every kernel shape has to give the same bits; a
vehicle that the packing lost or doubled would differ.  A few lanes are also
compared with the FP64 oracle (positions within 1e-3 m, the parity tests'
bar)."""
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


def counts(kind, rng):
    if kind == "one wave":
        return rng.integers(0, 65, size=200)
    if kind == "even":
        return np.full(1601, 64)                      # 1,600 + a last lane alone
    if kind == "uneven":
        return np.r_[rng.integers(0, 65, size=3000), 0, 0, 1]
    if kind == "short":
        return rng.integers(0, 7, size=6000)
    if kind == "whole segments":
        return np.r_[np.full(400, 64), np.full(50, 0), np.full(400, 33)]
    if kind == "unstaged short":
        return rng.integers(0, 4, size=40000)
    return np.r_[rng.integers(10, 30, size=33000), 64]  # "unstaged"


@pytest.mark.parametrize("kind", ["one wave", "even", "uneven", "short", "whole segments", "unstaged short", "unstaged"])
def test_every_shape_gives_the_same_vehicles(api, kind):
    rng = np.random.default_rng(len(kind))
    n = counts(kind, rng)
    sc = synth.make_scene(n, rng)
    N, K, s = int(sc["lane_off"][-1]), 6, 2
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    th, p0, v0 = dev(sc["theta_true"]), dev(sc["p_init"]), dev(sc["v_init"])
    y = dev(sc["p_init"] + rng.normal(10.0, 5.0, size=(K // s, N)))
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    ref = None
    for shape in ((0, 0), (2, 1), (2, 8), (4, 1), (4, 4), (8, 2)):
        ctx = api.Context(vpt=shape[0], warps_per_segment=shape[1])
        out = [api.simulate(th, p0, v0, scene, K, DT, ctx=ctx)]
        loss, g, gp, gv = api.loss_grad(th, p0, v0, scene, K, DT, y, s, ctx=ctx)
        out += [g, gp, gv]
        ctx.check_status()
        if ref is None:
            ref, ref_loss = out, loss.item()
        for a, b in zip(out, ref):
            assert torch.equal(a, b), shape
        assert abs(loss.item() - ref_loss) <= 1e-6 * ref_loss
    lo = sc["lane_off"]
    for l in [0, len(n) // 2, len(n) - 1]:
        a, e = int(lo[l]), int(lo[l + 1])
        if a == e:
            continue
        P, _ = oracle.forward(np.array([0, e - a], np.int32), sc["length"][a:e], sc["theta_true"][:, a:e],
                              sc["p_init"][a:e], sc["v_init"][a:e], K, DT)
        assert float(np.abs(ref[0][:, a:e].double().cpu().numpy() - P).max()) <= 1e-3
