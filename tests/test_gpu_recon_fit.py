"""The reconstruction fit's warp-specialized kernel at the edges of its
pipeline: horizons around the chunk of 16 steps, lone and partial warps of
trajectories, row strides with and without 16-byte row copies, several
observations per step, a delta other than 4, and enough trajectories for the
kernel with more blocks per SM.  Against the FP64 oracle, with the tolerances
of the fit's parity test (test_gpu_recon.py): observed positions lie metres
away from every iterate, so that no residual's sign is ambiguous."""
import numpy as np
import pytest

from oracle import recon as R
from paper_2412_16750_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = (1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 65, 100)


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16750_gb300 import api as _api
    return _api


def cuda(x, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dtype, device="cuda")


def scene(n, edges, per_step, dt):
    """Trajectory i observed per_step times a step up to step edges[i mod len]
    (longest first), 15-25 m ahead of or behind a 12 m/s motion."""
    rng = np.random.default_rng(n + per_step)
    K = np.sort(np.array([edges[i % len(edges)] for i in range(n)]))[::-1]
    ts, ps, counts = [], [], []
    for i in range(n):
        t = np.arange(0, K[i] * per_step + 1) * (dt / per_step)
        p = 100.0 + 12.0 * t + rng.choice([-1.0, 1.0]) * rng.uniform(15.0, 25.0, size=len(t))
        p[:2] = 100.0 + 12.0 * t[:2]
        ts.append(t)
        ps.append(p)
        counts.append(len(t))
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    return off, synth.f32(np.concatenate(ts)), synth.f32(np.concatenate(ps))


@pytest.mark.parametrize("n,edges,per_step,pad,delta", [
    (1, (1,), 1, None, 4.0),
    (1, (17,), 1, 0, 4.0),
    (14, EDGES, 1, None, 4.0),
    (33, EDGES, 1, 0, 4.0),
    (45, EDGES, 3, None, 4.0),
    (31, EDGES, 9, 1, 3.5),
    (9800, (1, 15, 16, 17, 33), 1, None, 4.0),
])
def test_fit_edges(api, n, edges, per_step, pad, delta):
    dt = float(np.float32(0.5))
    off, t, p = scene(n, edges, per_step, dt)
    obs_k = R.nearest_steps(t, dt)
    K = R.horizons(off, obs_k)
    # the steps right after the start, where the trajectory has not left its
    # first observation, carry no observation away from it: drop them
    keep = (obs_k == 0) | (obs_k >= 1) & (np.abs(p - (100.0 + 12.0 * t)) > 1.0)
    tr = np.repeat(np.arange(n), np.diff(off))
    keep[off[1:] - 1] = True
    p = np.where(keep & (obs_k >= 1) & (np.abs(p - (100.0 + 12.0 * t)) <= 1.0), p + 20.0, p)
    first = np.zeros(len(t), bool)
    first[off[:-1]] = True
    keep |= first
    off = np.concatenate([[0], np.cumsum(np.bincount(tr[keep], minlength=n))]).astype(np.int32)
    t, p, obs_k = t[keep], p[keep], obs_k[keep]
    K = R.horizons(off, obs_k)
    k_max = int(K.max())
    p0 = np.full(n, 100.0)
    v0 = np.full(n, 12.0)
    th = synth.f32(np.array(api.RECON_INIT)[:, None].repeat(n, 1))
    th[5] = delta
    dp, dv = np.full((k_max, n), 10.0), np.zeros((k_max, n))
    n_iter, lo, hi = 3, api.RECON_BOX_LO, api.RECON_BOX_HI
    th_r, dp_r, dv_r, hist_r = R.fit(K, dp, dv, th, p0, v0, dt, off, obs_k, p, n_iter, 0.1, 0.01, lo, hi, -10.0)
    rec = api.Recon(cuda(off, torch.int32), cuda(t), cuda(p), dt, ld=None if pad is None else n + pad)
    rec.p_init.copy_(cuda(p0))
    rec.v_init.copy_(cuda(v0))
    assert rec.k_max == k_max
    th_g, dp_g, dv_g = cuda(th), cuda(dp), cuda(dv)
    hist = rec.fit(th_g, dp_g, dv_g, n_iter, 0.1, 0.01, lo, hi)
    rec.ctx.check_status()
    np.testing.assert_allclose(hist.cpu().numpy(), hist_r, rtol=1e-5)
    np.testing.assert_allclose(th_g.double().cpu().numpy(), th_r, rtol=1e-4, atol=1e-5)
    np.testing.assert_allclose(dp_g.double().cpu().numpy(), dp_r, rtol=0, atol=1e-3)
    np.testing.assert_allclose(dv_g.double().cpu().numpy(), dv_r, rtol=0, atol=1e-3)
