"""Classification when couplings differ by hundreds of orders: a rotation between two equal diagonal
entries whose coupling's square underflows (or overflows), in the midst of ordinary ones."""
import numpy as np
import pytest

from gpu_common import nphc

pytestmark = pytest.mark.gpu


def hessian(J, theta):
    th = np.append(theta, 0.0)
    C = J * np.cos(th[:, None] - th[None, :])
    np.fill_diagonal(C, 0.0)
    return (np.diag(C.sum(1)) - C)[:-1, :-1]


@pytest.mark.parametrize("N", [4, 5, 8, 9, 13])
@pytest.mark.parametrize("tiny", [1e-170, 1e-300, 5e-324, 1e-12, 0.0])
def test_tiny_coupling_between_equal_sites(N, tiny):
    """All couplings 1/2, the pinned site's 1, but for `tiny` between pairs of free sites (every pair in
    turn); at theta = 0 and at a collinear point with half of the sites turned round."""
    import torch
    N_ = nphc()
    M = N - 1
    for a in range(M):
        for b in range(a + 1, M):
            J = np.full((N, N), 0.5)
            J[M, :] = J[:, M] = 1.0
            J[a, b] = J[b, a] = tiny
            np.fill_diagonal(J, 0.0)
            system = N_.System(N, J=J)
            ep = N_.DeviceEndpoints.empty(system.n, np.arange(2))
            t = ep.tensors
            theta = np.zeros((2, M))
            theta[1, ::2] = np.pi
            x = torch.as_tensor(np.where(theta == 0, 1.0, -1.0).T.copy(), device="cuda")
            t["z_re"][:M].copy_(x)
            t["z_re"][M:].zero_()
            t["z_im"].zero_()
            t["cls"].fill_(N_.END_REAL)
            f64 = dict(dtype=torch.float64, device="cuda")
            th, index = torch.zeros(M, 2, **f64), torch.zeros(2, dtype=torch.int32, device="cuda")
            energy, least, logdet = (torch.zeros(2, **f64) for _ in range(3))
            N_.classify(system, ep, th, index, energy, least, logdet)
            for k in range(2):
                w = np.linalg.eigvalsh(hessian(J, theta[k]))
                size = np.abs(w).max()
                if np.abs(w).min() < 1e-10 * size:   # a singular Hessian: no sign to compare
                    continue
                assert int(index[k]) == int((w < 0).sum()), (a, b, k)
                # Jacobi and LAPACK: each within a few M eps of the largest eigenvalue
                assert abs(float(least[k]) - np.abs(w).min()) <= 1e-13 * size
                assert abs(float(logdet[k]) - np.log(np.abs(w)).sum()) <= 1e-13 * size * (1 / np.abs(w)).sum()


@pytest.mark.parametrize("scale", [1.0, 1e-100, 1e-150, 1e-158, 1e-161, 1e-170, 1e150, 1e160])
def test_angles_of_scaled_points(scale):
    """theta, V and the index depend on a point's angles only, whatever its size (x^2 + y^2 subnormal, zero
    or infinite among them): V within a few ulp of the sum's terms (36 pairs, each at most 2)."""
    import torch
    N_ = nphc()
    N, M, n = 9, 8, 5
    rng = np.random.default_rng(4)
    J = rng.standard_normal((N, N))
    J = np.triu(J, 1) + np.triu(J, 1).T
    system = N_.System(N, J=J)
    angle = rng.uniform(-np.pi, np.pi, (n, M))
    ep = N_.DeviceEndpoints.empty(system.n, np.arange(n))
    t = ep.tensors
    t["z_re"].copy_(torch.as_tensor(scale * np.concatenate([np.cos(angle), np.sin(angle)], 1).T.copy(), device="cuda"))
    t["z_im"].zero_()
    t["cls"].fill_(N_.END_REAL)
    f64 = dict(dtype=torch.float64, device="cuda")
    th, index = torch.zeros(M, n, **f64), torch.zeros(n, dtype=torch.int32, device="cuda")
    energy, least, logdet = (torch.zeros(n, **f64) for _ in range(3))
    N_.classify(system, ep, th, index, energy, least, logdet)
    for k in range(n):
        full = np.append(th[:, k].cpu().numpy(), 0.0)
        V = 0.5 * (J * (1 - np.cos(full[:, None] - full[None, :]))).sum()
        assert abs(float(energy[k]) - V) <= 1e-14 * np.abs(J).sum()
        assert int(index[k]) == int((np.linalg.eigvalsh(hessian(J, full[:-1])) < 0).sum())
