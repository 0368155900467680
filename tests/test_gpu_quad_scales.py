"""The compensated residual of a generic quadratic system (quad_warp.cuh) when its variables and
equations differ by many orders: refine_certify without Newton steps (refine_iters = 0) returns
||P(z)||_inf at the given point, compared with rational arithmetic.  One equation is evaluated near
a cancellation, every other one vanishes exactly.

Tolerance: 2^-51 of the value (rounding, modulus) and 2^-82 of the equation's largest term: its sum
of T = 11 terms takes 4 T roundings a part of at most 4 T ulp of the low word, 2^-106 of a grid
that is up to 2^11 times the largest term (about 2^22 in all, doubled twice for the products')."""
from fractions import Fraction

import numpy as np
import pytest

from gpu_common import nphc

pytestmark = pytest.mark.gpu


def parts(c, a, b):
    """c a b for complex doubles, exactly."""
    (ar, ai), (br, bi), (cr, ci) = (((Fraction(v.real), Fraction(v.imag))) for v in (a, b, c))
    mr, mi = ar * br - ai * bi, ar * bi + ai * br
    return cr * mr - ci * mi, cr * mi + ci * mr


def check(N_, z, terms, k):
    """Equation k: the terms (c, a, b) (-1: 1); equation i != k: z_i - fixed value."""
    import torch
    n = len(z)
    w = lambda i: complex(1.0) if i < 0 else complex(z[i])
    eq, va, vb, co = [], [], [], []
    for i in range(n):
        if i != k:
            eq += [i, i]
            va += [i, -1]
            vb += [-1, -1]
            co += [1.0, -z[i]]
    re = im = Fraction(0)
    most = 0.0
    for c, a, b in terms:
        eq.append(k)
        va.append(a)
        vb.append(b)
        co.append(c)
        r, i = parts(complex(c), w(a), w(b))
        re, im = re + r, im + i
        most = max(most, abs(complex(c)) * abs(w(a)) * abs(w(b)))
    want = float(np.hypot(float(re), float(im)))
    system = N_.System.quadratic(n, np.array(eq), np.array(va), np.array(vb), np.array(co, dtype=complex))
    opts = N_.options_default(gamma=1j, precision=N_.PREC_FP64)
    opts.refine_iters = 0
    ep = N_.DeviceEndpoints.empty(n, np.arange(1))
    zt = torch.as_tensor(np.asarray(z, dtype=complex), device="cuda")
    ep.tensors["z_re"].copy_(zt.real[:, None])
    ep.tensors["z_im"].copy_(zt.imag[:, None])
    ep.tensors["status"].fill_(N_.PATH_REACHED)
    N_.refine_certify(system, opts, ep)
    got = float(ep.tensors["resid"].cpu()[0])
    assert abs(got - want) <= 2.0 ** -51 * want + 2.0 ** -82 * most, (got, want, most)


@pytest.mark.parametrize("big", [2.0 ** 10, 2.0 ** 24, 9e7, 2.0 ** 60])
@pytest.mark.parametrize("step", [0, 1, 7])
def test_small_variable_beside_a_large_one(big, step):
    """z^2 - 2 z + (1 - 2^-30) at and next to its root 1 + 2^-15."""
    N_ = nphc()
    z = 1.0 + 2.0 ** -15 + step * 2.0 ** -52
    check(N_, [big, z], [(1.0, 1, 1), (-2.0, 1, -1), (1.0 - 2.0 ** -30, -1, -1)], 1)
    check(N_, [z, big, -big], [(1.0, 0, 0), (-2.0, 0, -1), (1.0 - 2.0 ** -30, -1, -1)], 0)


@pytest.mark.parametrize("n", [2, 3, 5, 8, 11, 12])
def test_unequal_scales(n):
    """Ten random terms in variables of 1e-9 .. 1e9 with coefficients that make them alike up to a
    factor of 1e6, and the constant that cancels them to its own rounding."""
    N_ = nphc()
    for seed in range(4):
        rng = np.random.default_rng(100 * n + seed)
        cpx = lambda size: complex(size * rng.standard_normal(), size * rng.standard_normal())
        z = [cpx(10.0 ** rng.uniform(-9, 9)) for _ in range(n)]
        terms = []
        for _ in range(10):
            a, b = int(rng.integers(0, n)), int(rng.integers(-1, n))
            size = abs(z[a]) * (abs(z[b]) if b >= 0 else 1.0)
            terms.append((cpx(10.0 ** rng.uniform(-6, 0) / size), a, b))
        re = im = Fraction(0)
        for c, a, b in terms:
            r, i = parts(c, z[a], z[b] if b >= 0 else complex(1.0))
            re, im = re + r, im + i
        terms.append((complex(-float(re), -float(im)), -1, -1))
        check(N_, z, terms, int(rng.integers(0, n)))
