"""A fit's result does not depend on the slot mapping that the launch picks
(interleaved, or consecutive for a scene's horizons of 256 steps and more with 4
vehicles per thread), on the kernel shape or on the launch form: up to one fold
window of the gradient sums (256 steps) a vehicle's gradient is the same sum in
the same order, so the fitted parameters agree bit for bit.  Beyond it the sums
fold by checkpoint interval, which all runs share here."""
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


@pytest.mark.parametrize("K,C", [(255, 8), (256, 8), (257, 8), (256, 50), (300, 9)])
@pytest.mark.parametrize("counts", [(64, 3, 1, 60), (33, 0, 17, 5, 64, 2)])
def test_same_fit_over_mappings_shapes_and_forms(api, counts, K, C):
    rng = np.random.default_rng(K + C)
    sc = synth.make_scene(counts, rng)
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    scene = api.Scene.from_lane_off(dev(sc["lane_off"], torch.int32), dev(sc["length"]))
    p0, v0 = dev(sc["p_init"]), dev(sc["v_init"])
    P = api.simulate(dev(sc["theta_true"]), p0, v0, scene, K, DT)
    y = P[5::5].contiguous() + dev(rng.normal(0, 1.0, size=(K // 5, scene.n_vehicles)))
    ref = None
    for shape in ((2, 1), (2, 8), (4, 1), (4, 4), (4, 8), (8, 1), (8, 8)):
        for mode in ("graph", "single"):
            ctx = api.Context(vpt=shape[0], warps_per_segment=shape[1], ckpt_interval=C)
            ctx.set_fit_mode(mode)
            th = dev(synth.plain_init(scene.n_vehicles))
            hist = api.fit(th, p0, v0, scene, K, DT, y, 5, 3, ctx=ctx)
            ctx.check_status()
            if ref is None:
                ref, ref_hist = th, hist
            assert torch.equal(th, ref), (shape, mode)
            torch.testing.assert_close(hist, ref_hist, rtol=1e-6, atol=0)
