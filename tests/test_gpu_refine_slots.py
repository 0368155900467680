"""The refinement kernel's slots (xy_refine_group.cuh): an endpoint's outcome is the same, bit
for bit, whether its slot has held other endpoints before (one launch over all paths, in either
order) or it is the only one of its slot (launches of 256, fewer than there are warps).  Slots
change hands at all four lanes' different speeds, so the launches are repeated."""
import numpy as np
import pytest

from gpu_common import nphc
from paper_1104_5497_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,count", [(6, 1024), (7, 4096), (8, 16384), (9, 16384), (10, 16384), (11, 8192)])
def test_slots_do_not_mix_endpoints(N, count):
    import torch
    N_ = nphc()
    g = I.draw_pair_normals(np.random.default_rng(70 + N), N)
    system = N_.System(N, 0.8, N_.xy_couplings(N, 0.8, g, 0.1))
    opts = N_.options_default(gamma=I.draw_gamma(np.random.default_rng(N)))
    ep = N_.DeviceEndpoints.empty(system.n, np.arange(count) * (system.npaths // count))
    ws = torch.empty(system.workspace_size(count), dtype=torch.uint8, device="cuda")
    N_.track(system, opts, N_.PREC_MIXED, ep, ws)
    torch.cuda.synchronize()
    start = {k: v.clone() for k, v in ep.tensors.items()}

    def refined(lists):
        for k, v in ep.tensors.items():
            v.copy_(start[k])
        for l in lists:
            if l is None:
                N_.refine_certify(system, opts, ep)
            else:
                l = torch.tensor(l, dtype=torch.int32, device="cuda")
                N_.refine_certify(system, opts, ep, l, torch.tensor([l.numel()], dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        return {k: v.clone() for k, v in ep.tensors.items()}

    alone = refined([list(range(i, min(i + 256, count))) for i in range(0, count, 256)])
    for turn in range(6):
        got = refined([None] if turn % 2 == 0 else [list(range(count - 1, -1, -1))])
        for k in ("z_re", "z_im", "cls", "alpha", "beta", "gamma", "resid"):
            a, b = alone[k], got[k]
            same = (a == b) | (a.isnan() & b.isnan()) if a.is_floating_point() else a == b
            assert bool(same.all()), (turn, k, torch.nonzero(~same)[:4].tolist())
