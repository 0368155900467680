"""An initial step below the FP32 pass's time unit of 2^-53 (f32_step.cuh): the step doubles from there
on, so the pass finishes its paths as it does with the default h0, in both FP32 kernels (N = 10:
20,000 paths by four lanes each, 50,000 by one thread each)."""
import numpy as np
import pytest

from gpu_common import nphc
from paper_1104_5497_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,count", [(5, 256), (8, 16384), (10, 20000), (10, 50000)])
@pytest.mark.parametrize("h0", [1e-17, 1e-25])
def test_tiny_first_step(N, count, h0):
    import torch
    N_ = nphc()
    g = I.draw_pair_normals(np.random.default_rng(N), N)
    system = N_.System(N, 0.9, N_.xy_couplings(N, 0.9, g, 0.1))
    ended = []
    for h in (0.0, h0):
        opts = N_.options_default(gamma=I.draw_gamma(np.random.default_rng(N)))
        opts.h0 = h or opts.h0
        ep = N_.DeviceEndpoints.empty(system.n, (np.arange(count, dtype=np.int64) * 7919) % system.npaths)
        ws = torch.empty(system.workspace_size(count), dtype=torch.uint8, device="cuda")
        N_.track(system, opts, N_.PREC_MIXED, ep, ws)
        st = ep.tensors["status"].cpu().numpy()
        ended.append(np.isin(st, [N_.PATH_REACHED, N_.PATH_DIVERGED]))
    # another step sequence: a path in a hundred may be handed off in one of the two only
    assert ended[0].mean() > 0.8
    assert np.count_nonzero(ended[0] != ended[1]) <= count // 100 + 1
