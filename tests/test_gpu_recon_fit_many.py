"""The reconstruction fit with more than two blocks of trajectories per SM, which
runs the kernel with the shallower copies: the edges of its pipeline (see
test_gpu_recon_fit.py) with the number of trajectories taken from the device,
horizons up to 100 steps, unaligned rows, several observations per step, and a
delta other than 4."""
import pytest

import test_gpu_recon_fit as fit

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

api = fit.api


@pytest.mark.parametrize("edges,per_step,pad,delta", [
    ((100, 1, 15, 16, 17, 33, 64), 1, None, 4.0),
    ((100, 2, 31, 48, 65), 3, 1, 3.5),
])
def test_fit_with_three_blocks_per_sm(api, edges, per_step, pad, delta):
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    fit.test_fit_edges(api, 64 * n_sm + 33, edges, per_step, pad, delta)
