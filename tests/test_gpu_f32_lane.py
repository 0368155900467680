"""The FP32 pass with one path per thread (xy_track_lane.cuh), which launches with several waves of
paths take (xy_inst.cu), against the four-lane kernel that fewer paths take.  Both follow the same
paths with different roundings and both are Newton-refined in FP64, so endpoints agree to 1e-10
relative to 1 + |z|; a path that passes very close to another may end on that one's endpoint
instead: one in a thousand is allowed."""
import numpy as np
import pytest

from gpu_common import assert_same_point_sets, certified_set, nphc
from paper_1104_5497_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def endpoints(N_, system, gamma, paths):
    import torch
    opts = N_.options_default(gamma=gamma)
    ep = N_.DeviceEndpoints.empty(system.n, paths)
    ws = torch.empty(system.workspace_size(ep.count), dtype=torch.uint8, device="cuda")
    N_.track(system, opts, N_.PREC_MIXED, ep, ws)
    st = ep.tensors["status"]
    todo = torch.nonzero((st == N_.PATH_HANDOFF) | (st == N_.PATH_HANDOFF_COND)).flatten().to(torch.int32)
    if todo.numel():
        n = torch.tensor([todo.numel()], dtype=torch.int32, device="cuda")
        N_.track(system, opts, N_.PREC_FP64, ep, ws, todo, n, resume=True)
    N_.refine_certify(system, opts, ep)
    torch.cuda.synchronize()
    return (ep.tensors["z_re"] + 1j * ep.tensors["z_im"]).cpu().numpy().T, ep.tensors["cls"].cpu().numpy()


# odd and even M, with and without a column of its own for the second right-hand side; the larger
# rings: blocks of the four-lane kernel that decide together against warps that decide alone
@pytest.mark.parametrize("N,count", [(10, 40001), (11, 70001), (11, 190001), (12, 80001), (13, 180001)])
def test_many_paths_match_few(N, count):
    N_ = nphc()
    g = I.draw_pair_normals(np.random.default_rng(60 + N), N)
    gamma = I.draw_gamma(np.random.default_rng(N))
    system = N_.System(N, 0.9, N_.xy_couplings(N, 0.9, g, 0.1))
    paths = (np.arange(count, dtype=np.int64) * 7919) % system.npaths
    some = np.arange(0, count, count // 2000)
    za, ca = endpoints(N_, system, gamma, paths)
    zb, cb = endpoints(N_, system, gamma, paths[some])
    za, ca = za[some], ca[some]
    both = np.isin(ca, (2, 3)) & np.isin(cb, (2, 3))
    err = np.abs(za[both] - zb[both]).max(axis=1) / (1 + np.abs(zb[both]).max(axis=1))
    assert both.sum() > 0
    assert np.count_nonzero(ca != cb) <= len(some) // 1000
    assert np.count_nonzero(err > 1e-10) <= len(some) // 1000


@pytest.mark.parametrize("N,count", [(5, 600), (6, 128), (7, 40), (8, 12), (9, 6)])
def test_large_batches_match_single_solves(N, count):
    N_ = nphc()
    some = I.disordered_batch(2, 90 + N, n_lo=N, n_hi=N)
    inst = [some[i % 2] for i in range(count)]
    systems = [N_.System(N, i.sigma, N_.xy_couplings(N, i.sigma, i.g, i.eps)) for i in inst]
    opts = [N_.options_default(gamma=i.gamma) for i in inst]
    batch = N_.Batch(systems)
    batch.solve(opts)
    for k in (0, count - 1):
        a, b = batch.result(k), N_.solve(systems[k], opts[k])
        for key in ("paths", "real", "nonreal"):
            assert a.counts()[key] == b.counts()[key], (k, key)
        ea, eb = a.endpoints(), b.endpoints()
        assert_same_point_sets(certified_set(ea["z"], ea["cls"], [N_.END_REAL, N_.END_NONREAL]),
                               certified_set(eb["z"], eb["cls"], [N_.END_REAL, N_.END_NONREAL]))
