"""The initializer's features divide by 100 m and 30 m/s as CUDA's own division
does: bit for bit the bf16 rows that the same FP32 expressions give with a / b
on the device (torch divides one tensor by another that way), for ordinary
values and for signed zeros, subnormal, huge, infinite and undefined ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PREFIX = 20
SPECIAL = [0.0, -0.0, 1e-45, -1e-45, 1.4e-39, -2.3e-38, 1.2e-37, -9e-31, 3.3e-30, 1e36, -3.4e38, np.inf, -np.inf, np.nan]

# divided by 100 or 30: midway between subnormals whose roundings differ in bf16
TIES = [float(t) for t in np.array([0x0095FFCE, 0x012EFFE7, 0x002CFFF1, 0x0068FFF1, 0x00A4FFF1],
                                   np.uint32).view(np.float32)]


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16750_gb300 import api as _api
    return _api


def values(kind, shape, rng):
    if kind == "ordinary":
        return rng.normal(0.0, 300.0, size=shape).astype(np.float32)
    if kind == "exponents":
        m = np.ldexp(rng.uniform(-2.0, 2.0, size=shape), rng.integers(-149, 127, size=shape))
        return m.astype(np.float32)
    if kind == "subnormal":  # integer multiples of the smallest: quotients that are ties among them
        return rng.integers(-2**22, 2**22, size=shape).astype(np.int32).astype(np.float32) * np.float32(2.0**-149)
    x = np.array(SPECIAL + TIES, dtype=np.float32)
    return rng.choice(np.r_[x, -x], size=shape)


@pytest.mark.parametrize("kind", ["ordinary", "exponents", "subnormal", "special"])
@pytest.mark.parametrize("origin", [0.0, -0.0, 731.25])
def test_rows_equal_true_division(api, kind, origin):
    rng = np.random.default_rng(len(kind))
    counts = rng.integers(1, 9, size=700)
    off = np.r_[0, np.cumsum(counts)].astype(np.int32)
    N, dt, s = int(off[-1]), float(np.float32(0.1)), 2
    cuda = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    y0 = cuda(np.full(N, origin, np.float32))
    v = cuda(values(kind, N, rng))
    y = cuda(values(kind, (PREFIX, N), rng))
    scene = api.Scene.from_lane_off(cuda(off), torch.full((N,), 5.0, device="cuda"))
    got = api.mlp_features(scene, y0, v, PREFIX * s, dt, y, s)
    obs = torch.cat([y0[None], y])
    inv = np.float32(1.0) / (np.float32(2.0) * np.float32(s) * np.float32(dt))
    hundred, thirty = torch.full((1, 1), 100.0, device="cuda"), torch.full((1, 1), 30.0, device="cuda")
    head = torch.zeros(N, dtype=torch.bool, device="cuda")
    head[cuda(off[:-1].astype(np.int64))] = True
    x = (obs[:PREFIX] - y0) / hundred                                     # own positions
    sp = torch.cat([v[None], (obs[2:] - obs[:PREFIX - 1]) * torch.full((1, 1), float(inv), device="cuda")]) / thirty
    xl = torch.where(head, x + 2.0, (torch.roll(obs[:PREFIX], 1, 1) - y0) / hundred)   # the leader's
    spl = torch.where(head, sp, torch.roll(sp, 1, 1))
    ref = torch.cat([x, sp, xl, spl]).T.contiguous().bfloat16()
    nan = ref.isnan()
    assert torch.equal(got.isnan(), nan)
    same = (got.view(torch.int16) == ref.view(torch.int16)) | nan
    assert bool(same.all()), (int((~same).sum()), got[~same][:4], ref[~same][:4])


def test_first_vehicle_has_no_vehicle_before_it(api):
    """Offsets that do not start at 0 (malformed) leave vehicle 0 in no lane: its
    rows are those of a lane head, and nothing in front of the arrays is read."""
    rng = np.random.default_rng(0)
    cuda = lambda x: torch.as_tensor(np.asarray(x, np.float32), device="cuda")  # noqa: E731
    args = cuda(rng.normal(0, 100, 5)), cuda(rng.normal(20, 3, 5)), 20, 0.1, cuda(rng.normal(0, 100, (PREFIX, 5)))
    rows = [api.mlp_features(api.Scene.from_lane_off(torch.tensor(off, dtype=torch.int32), torch.full((5,), 5.0)), *args)
            for off in ([0, 1, 5], [1, 3, 5])]
    assert torch.equal(rows[0][0], rows[1][0])
