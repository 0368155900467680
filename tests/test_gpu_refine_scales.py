"""Refinement at couplings of any size (sums on exponent-chosen grids, gsum in nphc_internal.cuh):
J times a power of two has the same stationary points and scales the gradient rows exactly, so
Newton's iterates are the same bit for bit, from 2^-400 to 2^400.  Points with large and small
components, real and non-real."""
import numpy as np
import pytest

from gpu_common import nphc
from paper_1104_5497_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [3, 6, 9, 13])
def test_refined_points_do_not_depend_on_the_scale_of_j(N):
    import torch
    N_ = nphc()
    g = I.draw_pair_normals(np.random.default_rng(N), N)
    J = N_.xy_couplings(N, 1.0, g, 0.1)
    opts = N_.options_default(gamma=I.draw_gamma(np.random.default_rng(N)))
    count = min(4 ** (N - 1), 500)
    system = N_.System(N, J=J)
    ep = N_.DeviceEndpoints.empty(system.n, np.arange(count) * (system.npaths // count))
    ws = torch.empty(system.workspace_size(count), dtype=torch.uint8, device="cuda")
    N_.track(system, opts, N_.PREC_MIXED, ep, ws)
    torch.cuda.synchronize()
    reached = ep.tensors["status"] == N_.PATH_REACHED
    assert bool(reached.any())
    start = {k: v.clone() for k, v in ep.tensors.items()}
    z = {}
    for k in (-400, -40, 0, 40, 400):
        for name, v in ep.tensors.items():
            v.copy_(start[name])
        N_.refine_certify(N_.System(N, J=np.ldexp(J, k)), opts, ep)
        torch.cuda.synchronize()
        z[k] = torch.cat([ep.tensors["z_re"], ep.tensors["z_im"]])[:, reached].clone()
    for k, v in z.items():
        assert bool((v == z[0]).all()), k
    assert bool((z[0] != torch.cat([start["z_re"], start["z_im"]])[:, reached]).any())
