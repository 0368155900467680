"""Far endpoints (some |Re z_i| or |Im z_i| >= 65,536 at the default refine_eps): whether such a
solution certifies depends on the rounding of the FP32 pass and of the refinement, so each keeps
one order of operations (xy_track.cuh, xy_refine_far.cuh) whatever the launch."""
import os

import numpy as np
import pytest

from gpu_common import nphc
from paper_1104_5497_gb300 import inputs as I

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "far_endpoints.txt")
FAR = 2.0 ** 16


def ring(N_, N, seed):
    """sigma ~ U[0.5, 3], gamma and one normal per pair from the seed; J = d^-sigma (1 + 0.1 g)."""
    rng = np.random.default_rng(seed)
    sigma = float(rng.uniform(0.5, 3.0))
    gamma = I.draw_gamma(rng)
    g = I.draw_pair_normals(rng, N)
    i = np.arange(N)
    d = np.abs(i[:, None] - i[None, :])
    d = np.minimum(d, N - d)
    J = np.where(d > 0, np.maximum(d, 1).astype(float) ** -sigma, 0.0)
    return N_.System(N, J=J * (1.0 + 0.1 * g)), N_.options_default(gamma=gamma)


def track(N_, system, opts, paths):
    import torch
    ep = N_.DeviceEndpoints.empty(system.n, np.asarray(paths, dtype=np.int64))
    ws = torch.empty(system.workspace_size(ep.count), dtype=torch.uint8, device="cuda")
    N_.track(system, opts, N_.PREC_MIXED, ep, ws)
    torch.cuda.synchronize()
    return ep


def refine(N_, system, opts, ep):
    import torch
    N_.refine_certify(system, opts, ep)
    torch.cuda.synchronize()
    return ep


def far_entries(N_, ep):
    t = ep.tensors
    size = np.maximum(t["z_re"].abs().amax(0).cpu().numpy(), t["z_im"].abs().amax(0).cpu().numpy())
    return np.nonzero((t["status"].cpu().numpy() == N_.PATH_REACHED) & (size >= FAR))[0]


def columns(ep, at, keys):
    return {k: ep.tensors[k].cpu().numpy()[..., at] for k in keys}


def test_classes_of_known_far_endpoints():
    N_ = nphc()
    rows = np.loadtxt(GOLDEN, dtype=np.int64)
    wrong = []
    for N, seed in sorted({(int(r[0]), int(r[1])) for r in rows}):
        mine = rows[(rows[:, 0] == N) & (rows[:, 1] == seed)]
        system, opts = ring(N_, N, seed)
        ep = refine(N_, system, opts, track(N_, system, opts, mine[:, 2]))
        got = ep.tensors["cls"].cpu().numpy()
        wrong += [(*r, int(c)) for r, c in zip(mine.tolist(), got) if c != r[3]]
    assert not wrong


# N = 9: the four-lane kernel in either launch; N = 10: the per-thread kernel over the whole ring,
# the four-lane kernel over its far paths alone; N = 12 (a part of the ring): a large FP64 share
@pytest.mark.parametrize("N,count", [(9, 65536), (10, 262144), (12, 60001)])
def test_far_endpoints_do_not_depend_on_their_company(N, count):
    import torch
    N_ = nphc()
    system, opts = ring(N_, N, 1000 + N)
    paths = (np.arange(count, dtype=np.int64) * 7919) % system.npaths
    all_ = track(N_, system, opts, paths)
    far = far_entries(N_, all_)
    assert len(far) >= 8
    few = track(N_, system, opts, paths[far])
    for k in ("z_re", "z_im", "t", "h", "status"):
        a, b = columns(all_, far, [k])[k], few.tensors[k].cpu().numpy()
        assert np.array_equal(a, b), k
    refine(N_, system, opts, all_)
    refine(N_, system, opts, few)
    one = track(N_, system, opts, paths[far[:12]])
    for i in range(one.count):   # refined one at a time
        N_.refine_certify(system, opts, one, torch.tensor([i], dtype=torch.int32, device="cuda"),
                          torch.tensor([1], dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    for k in ("z_re", "z_im", "cls", "alpha", "beta", "gamma", "resid"):
        a, b, c = columns(all_, far, [k])[k], few.tensors[k].cpu().numpy(), one.tensors[k].cpu().numpy()
        assert np.array_equal(a, b), k
        assert np.array_equal(a[..., :c.shape[-1]], c), k


def test_far_list_follows_the_refinement_tolerance():
    """The line moves with refine_eps (2^9 at 1e-10), and no tolerance means no far endpoints."""
    N_ = nphc()
    system, opts = ring(N_, 9, 1009)
    paths = np.arange(system.npaths)
    base = track(N_, system, opts, paths).tensors["solves"].cpu().numpy()
    opts.refine_eps = 1e-10
    more = track(N_, system, opts, paths).tensors["solves"].cpu().numpy()
    opts.refine_eps = 0.0
    none = track(N_, system, opts, paths).tensors["solves"].cpu().numpy()
    assert base.sum() > none.sum() and more.sum() > base.sum()
    assert (base >= none).all() and (more >= base).all()


@pytest.mark.parametrize("N,count", [(8, 16384), (11, 300001), (12, 300001), (13, 300001)])
def test_short_and_long_lists_agree_bit_for_bit(N, count):
    """Far paths are tracked by a warp each, or by a thread each when there are 64 or more for every
    scheduler.  With the line at 2^-4 every path that reaches t = 1 is far: the whole launch takes
    the per-thread kernel (not at N = 8, where both are short lists), a tenth of it the other."""
    import torch
    N_ = nphc()
    system, opts = ring(N_, N, 2000 + N)
    opts.refine_eps = 0.01
    paths = (np.arange(count, dtype=np.int64) * 7919) % system.npaths
    all_ = track(N_, system, opts, paths)
    reached = int((all_.tensors["status"] == N_.PATH_REACHED).sum())
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert N == 8 or reached >= 64 * 4 * sms
    some = np.arange(0, count, 10)
    few = track(N_, system, opts, paths[some])
    assert (few.tensors["status"] == N_.PATH_REACHED).sum() < 64 * 4 * sms
    same = all_.tensors["status"].cpu().numpy()[some] == few.tensors["status"].cpu().numpy()
    assert same.mean() > 0.999   # (two FP32 kernels may run before: another path may be handed off)
    at = same & (few.tensors["status"].cpu().numpy() == N_.PATH_REACHED)
    assert at.sum() > 100
    for k in ("z_re", "z_im", "t", "h", "steps"):
        a, b = columns(all_, some, [k])[k], few.tensors[k].cpu().numpy()
        if k == "steps" and N < 12:
            continue   # counts of the pass before, of either kernel, included
        assert np.array_equal(a[..., at], b[..., at]), k


def test_batches_match_single_solves_at_far_endpoints():
    """Rings of three sizes, two or more of each: a group's far paths are listed and tracked together."""
    N_ = nphc()
    rings = [ring(N_, N, seed) for N, seed in ((9, 1009), (8, 1017), (9, 1340), (8, 1034), (9, 1323), (6, 7))]
    systems, opts = [r[0] for r in rings], [r[1] for r in rings]
    opts[2].refine_eps = 2e-14   # a line of its own
    batch = N_.Batch(systems)
    far = 0
    for flags in (0, N_.BATCH_GRAPH, N_.BATCH_GRAPH):   # eager, captured, replayed
        batch.solve(opts, flags)
        for k in range(len(rings)):
            a, b = batch.result(k).endpoints(), N_.solve(systems[k], opts[k]).endpoints()
            at = (b["status"] == N_.PATH_REACHED) & (np.maximum(abs(b["z"].real), abs(b["z"].imag)).max(axis=1) >= FAR)
            far += int(at.sum())
            assert np.array_equal(a["status"][at], b["status"][at])
            assert np.array_equal(a["cls"][at], b["cls"][at]) and np.array_equal(a["z"][at], b["z"][at])
            assert [a["cls"].tolist().count(c) for c in range(7)] == [b["cls"].tolist().count(c) for c in range(7)]
    assert far >= 60
