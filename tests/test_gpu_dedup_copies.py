"""Deduplication of solutions with many copies (a pair whose entries are both listed and whose higher
path is marked is not compared again), of none, and of entry counts off the fill kernel's 16-byte
words: the lowest path of every solution keeps its class, every entry of a solution reached twice
is listed once."""
import numpy as np
import pytest

from gpu_common import nphc
from paper_1104_5497_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copies", [1, 2, 3, 201])
@pytest.mark.parametrize("take", [1, 7, 19])
def test_copies_of_certified_solutions(copies, take):
    import torch
    N_ = nphc()
    inst = I.ring_random_sigma(7, 3)
    system = N_.System(7, inst.sigma)
    opts = N_.options_default(gamma=inst.gamma)
    res = N_.solve(system, opts)
    e = res.endpoints()
    pick = np.flatnonzero(np.isin(e["cls"], [N_.END_REAL, N_.END_NONREAL]))[:take]
    assert len(pick) == take
    who = np.random.default_rng(copies).permutation(np.repeat(np.arange(take), copies))
    ep = N_.DeviceEndpoints.empty(system.n, np.random.default_rng(1).permutation(len(who)) + 5)
    z = e["z"][pick[who]].T
    ep.tensors["z_re"].copy_(torch.as_tensor(z.real.copy()))
    ep.tensors["z_im"].copy_(torch.as_tensor(z.imag.copy()))
    ep.tensors["status"].fill_(N_.PATH_REACHED)
    N_.refine_certify(system, opts, ep)
    before = ep.tensors["cls"].cpu().numpy()
    assert np.isin(before, [N_.END_REAL, N_.END_NONREAL]).all()
    ws = torch.empty(system.workspace_size(ep.count), dtype=torch.uint8, device="cuda")
    dup, n = torch.zeros(len(who), dtype=torch.int32, device="cuda"), torch.full((1,), 9, dtype=torch.int32, device="cuda")
    N_.dedup(system, opts, ep, ws, dup, n)
    torch.cuda.synchronize()
    after, path = ep.tensors["cls"].cpu().numpy(), ep.tensors["path"].cpu().numpy()
    for s in range(take):
        mine = np.flatnonzero(who == s)
        low = mine[path[mine].argmin()]
        assert after[low] == before[low]
        assert (after[mine[mine != low]] == N_.END_DUPLICATE).all()
    listed = np.sort(dup.cpu().numpy()[:int(n)])
    assert np.array_equal(listed, np.arange(len(who)) if copies > 1 else [])
