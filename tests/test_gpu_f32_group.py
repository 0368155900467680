"""The FP32 pass with four lanes per path (xy_track_group.cuh) at the edges of its layout:
every ring size (rows that do not fill the lanes, N = 3 .. 13) and path counts around one
path, one warp (8 paths) and one block (32), through a step-by-step run (FP32 pass, FP64
continuation of the hand-offs, refinement and certification) against the oracle, path by
path.  The endpoints of both are Newton-refined in FP64, so the tolerance is that of the
other parity tests: 1e-10 relative to 1 + |z|."""
import numpy as np
import pytest

import oracle as O
from gpu_common import nphc
from paper_1104_5497_gb300 import inputs as I

pytestmark = pytest.mark.gpu
CERT = (2, 3, 4)   # real, non-real, undecided (the oracle's numbers too)


def run_paths(N_, system, gamma, paths, use_list):
    import torch
    opts = N_.options_default(gamma=gamma)
    ep = N_.DeviceEndpoints.empty(system.n, paths)
    ws = torch.empty(system.workspace_size(ep.count), dtype=torch.uint8, device="cuda")
    if use_list:   # the same paths through a work list, in reverse order
        lst = torch.arange(ep.count - 1, -1, -1, dtype=torch.int32, device="cuda")
        N_.track(system, opts, N_.PREC_MIXED, ep, ws, lst, torch.tensor([ep.count], dtype=torch.int32, device="cuda"))
    else:
        N_.track(system, opts, N_.PREC_MIXED, ep, ws)
    st = ep.tensors["status"]
    todo = torch.nonzero((st == N_.PATH_HANDOFF) | (st == N_.PATH_HANDOFF_COND)).flatten().to(torch.int32)
    fp32 = {k: v.clone() for k, v in ep.tensors.items()}
    if todo.numel():
        n = torch.tensor([todo.numel()], dtype=torch.int32, device="cuda")
        N_.track(system, opts, N_.PREC_FP64, ep, ws, todo, n, resume=True)
    N_.refine_certify(system, opts, ep)
    torch.cuda.synchronize()
    z = (ep.tensors["z_re"] + 1j * ep.tensors["z_im"]).cpu().numpy().T
    return ep.tensors["cls"].cpu().numpy(), z, fp32


@pytest.mark.parametrize("N", range(3, 14))
@pytest.mark.parametrize("count", [1, 9, 37])
def test_few_paths_match_the_oracle(N, count):
    N_ = nphc()
    count = min(count, 4 ** (N - 1))
    g = I.draw_pair_normals(np.random.default_rng(40 + N), N)
    gamma = I.draw_gamma(np.random.default_rng(N))
    system = N_.System(N, 1.1, N_.xy_couplings(N, 1.1, g, 0.1))
    first = (4 ** (N - 1) - count) // 3
    cls, z, a = run_paths(N_, system, gamma, np.arange(first, first + count), False)
    ref = O.solve_system(O.xy_terms(N, O.couplings(N, 1.1, g, 0.1)), gamma, path0=first, npaths=count)
    cert, ref_cert = np.isin(cls, CERT), np.isin(ref["cls"], CERT + (5,))
    assert np.array_equal(cert, ref_cert)
    kept = cert & (ref["cls"] != 5)   # the oracle has deduplicated
    assert np.array_equal(cls[kept], ref["cls"][kept])
    if cert.any():
        err = np.abs(z[cert] - ref["z"][cert]).max(axis=1)
        assert np.all(err <= 1e-10 * (1 + np.abs(ref["z"][cert]).max(axis=1)))
    # a path's arithmetic does not depend on the paths it shares a warp with
    _, _, b = run_paths(N_, system, gamma, np.arange(first, first + count), True)
    for k in ("z_re", "z_im", "t", "h", "status", "steps", "solves", "newton"):
        assert bool((a[k] == b[k]).all()), k
