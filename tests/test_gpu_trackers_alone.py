"""The ring's trackers by themselves, before any other stage can repair what they leave: the FP32
kernels' hand-off share and their endpoints as they come, the four-lane FP64 kernel on whole passes
and on long lists of hand-offs, against the kernel that fewer paths take."""
import numpy as np
import pytest

from gpu_common import nphc
from paper_1104_5497_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def ring(N_, N):
    g = I.draw_pair_normals(np.random.default_rng(60 + N), N)
    return (N_.System(N, 0.9, N_.xy_couplings(N, 0.9, g, 0.1)),
            N_.options_default(gamma=I.draw_gamma(np.random.default_rng(N))))


def track(N_, system, opts, prec, paths):
    import torch
    ep = N_.DeviceEndpoints.empty(system.n, np.asarray(paths, dtype=np.int64))
    ws = torch.empty(system.workspace_size(ep.count), dtype=torch.uint8, device="cuda")
    N_.track(system, opts, prec, ep, ws)
    torch.cuda.synchronize()
    return ep, ws


def points(ep):
    t = ep.tensors
    return (t["z_re"] + 1j * t["z_im"]).cpu().numpy().T, t["status"].cpu().numpy()


def relative(za, zb):
    return np.linalg.norm(za - zb, axis=1) / (1 + np.linalg.norm(zb, axis=1))


@pytest.mark.parametrize("N,many", [(9, 65536), (10, 50001), (11, 20001), (12, 20001), (13, 20001)])
def test_fp32_pass_alone(N, many):
    """A converged FP32 point's last correction is at most eps_fp32 (1 + ||z||), so two passes of
    different rounding end within 2 eps_fp32 of each other; at most a path in a hundred takes another
    decision somewhere (a hand-off, a neighbouring path).  At most a fifth is handed off (N = 13: 10%)."""
    N_ = nphc()
    system, opts = ring(N_, N)
    paths = (np.arange(many, dtype=np.int64) * 7919) % system.npaths
    some = np.arange(0, many, many // 3000)
    za, sa = points(track(N_, system, opts, N_.PREC_MIXED, paths)[0])
    zb, sb = points(track(N_, system, opts, N_.PREC_MIXED, paths[some])[0])
    handed = np.isin(sa, [N_.PATH_HANDOFF, N_.PATH_HANDOFF_COND])
    assert handed.mean() <= 0.2
    assert np.isin(sa, [N_.PATH_REACHED, N_.PATH_DIVERGED])[~handed].all()
    assert np.count_nonzero(sa[some] != sb) <= len(some) // 100
    both = (sa[some] == N_.PATH_REACHED) & (sb == N_.PATH_REACHED)
    assert both.sum() > len(some) // 20
    assert np.count_nonzero(relative(za[some][both], zb[both]) > 2 * opts.eps_fp32) <= len(some) // 100


@pytest.mark.parametrize("N", [9, 11, 12, 13])
def test_fp64_pass_alone(N):
    """6,200 paths by four lanes each, 3,100 of them by a warp each: FP64 endpoints within 2 eps_fp64."""
    N_ = nphc()
    system, opts = ring(N_, N)
    opts.precision = N_.PREC_FP64
    paths = (np.arange(6200, dtype=np.int64) * 7919) % system.npaths
    za, sa = points(track(N_, system, opts, N_.PREC_FP64, paths)[0])
    zb, sb = points(track(N_, system, opts, N_.PREC_FP64, paths[::2])[0])
    za, sa = za[::2], sa[::2]
    assert np.count_nonzero(sa != sb) <= len(sb) // 100
    both = (sa == N_.PATH_REACHED) & (sb == N_.PATH_REACHED)
    assert both.sum() > len(sb) // 20
    assert np.count_nonzero(relative(za[both], zb[both]) > 2 * opts.eps_fp64) <= len(sb) // 100


@pytest.mark.parametrize("N,count", [(11, 40001), (12, 40001)])
def test_long_lists_of_hand_offs(N, count):
    """More hand-offs than 32 per scheduler (a condition limit of 30 hands off most paths on their
    way): four lanes each, against a warp each (threads_per_path 32)."""
    import torch
    N_ = nphc()
    system, opts = ring(N_, N)
    opts.kappa_fp32 = 30.0
    ep, ws = track(N_, system, opts, N_.PREC_MIXED, (np.arange(count, dtype=np.int64) * 7919) % system.npaths)
    st = ep.tensors["status"]
    todo = torch.nonzero((st == N_.PATH_HANDOFF) | (st == N_.PATH_HANDOFF_COND)).flatten().to(torch.int32)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert todo.numel() >= 32 * 4 * sms
    n = torch.tensor([todo.numel()], dtype=torch.int32, device="cuda")
    saved = {k: v.clone() for k, v in ep.tensors.items()}
    ends = []
    for per in (0, 32):
        for k, v in saved.items():
            ep.tensors[k].copy_(v)
        opts.threads_per_path = per
        N_.track(system, opts, N_.PREC_FP64, ep, ws, todo, n, resume=True)
        torch.cuda.synchronize()
        z, s = points(ep)
        ends.append((z[todo.cpu().numpy()], s[todo.cpu().numpy()], s))
    (za, sa, alla), (zb, sb, allb) = ends
    others = np.ones(count, bool)
    others[todo.cpu().numpy()] = False
    assert np.array_equal(alla[others], saved["status"].cpu().numpy()[others])
    assert not np.isin(sa, [N_.PATH_HANDOFF, N_.PATH_HANDOFF_COND]).any()
    assert np.count_nonzero(sa != sb) <= len(sb) // 100
    both = (sa == N_.PATH_REACHED) & (sb == N_.PATH_REACHED)
    assert both.sum() >= 1000
    assert np.count_nonzero(relative(za[both], zb[both]) > 2 * opts.eps_fp64) <= len(sb) // 100
