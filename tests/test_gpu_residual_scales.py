"""The FP64 kernels' compensated residuals of the XY ring (warp_residual, g64_residual, rg_row) row by
row against rational arithmetic, when couplings and coordinates of different sites differ by many
orders.

Tolerance of a row: 2^-52 of its value (rounded once) and 2^-85 of the largest product in it.  A
row's sum U takes at most 4 x 13 roundings a part in its low word, each at most 4 x 13 ulp of
2^(k - 106), 2^k up to 2^7 times the largest term: 2^(12 + 7 - 106) of it = 2^-87; the products with
the site's own coordinates and with gamma (1 - t) or t add a factor of at most four."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from gpu_common import nphc

pytestmark = pytest.mark.gpu

SOURCE = """
#include "xy_refine_group.cuh"
#include "xy_track_group64.cuh"
// block b: point b; J [N * N], z [2 M] and out [2 M] complex per point; par (t, 1 - t, gamma)
template <int M, int KIND>
__global__ void k(const double *J, const double *par, const cx<double> *z, cx<double> *out) {
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ double Jw[NPHC_MAXN * NPHC_JSTRIDE], Jg[M * (M + 1)], jj[M];
    const int lane = threadIdx.x, g = lane >> 3, pth = lane & 7;
    for (int i = lane; i < NPHC_MAXN * NPHC_JSTRIDE; i += 32) {
        const int r = i / NPHC_JSTRIDE, c = i % NPHC_JSTRIDE;
        Jw[i] = r <= M && c <= M ? J[r * (M + 1) + c] : 0.0;
    }
    for (int i = lane; i < M * (M + 1); i += 32) Jg[i] = J[i];
    __syncwarp();
    z += blockIdx.x * 2 * M;
    out += blockIdx.x * 2 * M;
    const double s = par[0], omt = par[1];
    const cx<double> gam = {par[2], par[3]};
    cx<double> *const sm = reinterpret_cast<cx<double> *>(raw);
    if (KIND < 2) {   // W1 = -H at ZC, (x, y) or (p, q)
        const WarpPath<M> P{sm, lane};
        for (int i = lane; i < 2 * M; i += 32) P.at(WarpLayout<M>::ZC, i) = z[i];
        __syncwarp();
        warp_residual<M, KIND == 1>(P, Jw, s, omt, gam);
        for (int i = lane; i < 2 * M; i += 32) out[i] = P.at(WarpLayout<M>::W1, i);
    } else if (KIND == 2) {   // -H's rows, (p, q)
        const G64Path<M> G{sm + pth, Jg, g, 0xffffffffu};
        for (int i = g; i < 2 * M; i += 4) G.at(G64Layout<M>::PQ, i) = z[i];
        __syncwarp();
        for (int j = g; j < M; j += 4) {
            cx<double> up, uq, rf, rg;
            g64_residual<M>(G, j, s, EFT<double>::mul(omt, gam.re), EFT<double>::mul(omt, gam.im), up, uq, rf, rg);
            out[j] = rf;
            out[M + j] = rg;
        }
    } else {   // P's rows, (x, y)
        const RGPath<M> G{sm + pth, Jg, jj, g, 0xffffffffu};
        for (int i = g; i < 2 * M; i += 4) G.at(RGLayout<M>::Z, i) = z[i];
        __syncwarp();
        for (int j = g; j < M; j += 4) {
            cx<double> f, gg, u, w;
            rg_row<M>(G, j, f, gg, u, w);
            out[j] = cx<double>{-f.re, -f.im};
            out[M + j] = cx<double>{-gg.re, -gg.im};
        }
    }
}
template <int M, int KIND>
int launch(const double *J, const double *par, const void *z, void *out, int n) {
    const int smem = KIND < 2 ? (int)warp_track_smem_per_warp<M>() : KIND == 2 ? (int)g64_smem_per_block<M>()
                                                                              : (int)rg_smem_per_block<M>();
    cudaFuncSetAttribute(k<M, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    k<M, KIND><<<n, 32, smem>>>(J, par, (const cx<double> *)z, (cx<double> *)out);
    return (int)cudaDeviceSynchronize();
}
template <int M>
int by_kind(int kind, const double *J, const double *par, const void *z, void *out, int n) {
    return kind == 0 ? launch<M, 0>(J, par, z, out, n) : kind == 1 ? launch<M, 1>(J, par, z, out, n)
         : kind == 2 ? launch<M, 2>(J, par, z, out, n) : launch<M, 3>(J, par, z, out, n);
}
extern "C" int run(int M, int kind, const double *J, const double *par, const void *z, void *out, int n) {
    return M == 4 ? by_kind<4>(kind, J, par, z, out, n) : M == 9 ? by_kind<9>(kind, J, par, z, out, n)
                                                                 : by_kind<12>(kind, J, par, z, out, n);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    nphc()
    from paper_1104_5497_gb300 import build as B
    d = tmp_path_factory.mktemp("residual")
    src, so = d / "residual.cu", d / "residual.so"
    src.write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", str(src), "-o", str(so)], check=True)
    f = ctypes.CDLL(os.fspath(so)).run
    f.argtypes = [ctypes.c_int] * 2 + [ctypes.c_void_p] * 4 + [ctypes.c_int]
    return f


class Cx:
    """A complex rational and the size of the largest product it was summed from."""

    def __init__(self, re, im=0, size=None):
        self.re, self.im = Fraction(re), Fraction(im)
        self.size = max(abs(float(self.re)), abs(float(self.im))) if size is None else size

    def __add__(self, o):
        return Cx(self.re + o.re, self.im + o.im, max(self.size, o.size))

    def __sub__(self, o):
        return Cx(self.re - o.re, self.im - o.im, max(self.size, o.size))

    def __mul__(self, o):
        return Cx(self.re * o.re - self.im * o.im, self.re * o.im + self.im * o.re, self.size * o.size)


def rows(J, z, light_cone, t, gr, gi):
    """H's rows f_1 .. f_M, g_1 .. g_M (t and the products gamma (1 - t) as given) at (x, y) or (p, q)."""
    M = len(z) // 2
    a, b = [Cx(v.real, v.imag) for v in z[:M]], [Cx(v.real, v.imag) for v in z[M:]]
    one, half, quarter = Cx(1), Cx(Fraction(1, 2)), Cx(Fraction(1, 4))
    t, g, i = Cx(t), Cx(gr, gi), Cx(0, 1)
    f, c = [], []
    for k in range(M):
        u = w = Cx(0)
        for l in range(M):
            u, w = u + Cx(J[k, l]) * a[l], w + Cx(J[k, l]) * b[l]
        u = u + Cx(J[k, M])
        if light_cone:
            w = w + Cx(J[k, M])
            p, q = a[k], b[k]
            s, d = p * q * half, (p * p + q * q) * quarter
            X, Y, F, G = s + d - one, s - d - one, i * half * (q * u - p * w), p * q - one
        else:
            x, y = a[k], b[k]
            X, Y, F, G = x * x - one, y * y - one, y * u - x * w, x * x + y * y - one
        f.append(g * X + t * F)
        c.append(g * Y + t * G)
    return f + c


@pytest.mark.parametrize("M", [4, 9, 12])
@pytest.mark.parametrize("kind", [0, 1, 2, 3])   # warp (x, y), warp (p, q), four lanes (p, q), refinement
@pytest.mark.parametrize("t", [0.3, 1.0 - 2.0 ** -40, 1.0])
def test_rows_at_unequal_scales(run, M, kind, t):
    import torch
    t = 1.0 if kind == 3 else t
    for seed in range(3):
        rng = np.random.default_rng(1000 * M + 10 * kind + seed)
        n, weak = 8, 10.0 ** rng.uniform(-12, 0, M + 1)
        J = weak[:, None] * weak[None, :] * rng.standard_normal((M + 1, M + 1))
        J = np.triu(J, 1) + np.triu(J, 1).T
        # p from 1e-7 to 1e7, q its reciprocal up to 1e-9; (x, y) from them
        p = 10.0 ** rng.uniform(-7, 7, (n, M)) * np.exp(2j * np.pi * rng.random((n, M)))
        q = (1 + 1e-9 * rng.standard_normal((n, M))) / p
        z = np.concatenate([p, q] if kind in (1, 2) else [(p + q) / 2, (p - q) / 2j], 1)
        gam = np.exp(2j * np.pi * rng.random())
        omt = 1.0 - t
        par = np.array([t, omt, gam.real, gam.imag])
        dev = lambda v: torch.as_tensor(np.ascontiguousarray(v), device="cuda")
        Jd, pd, zd = dev(J), dev(par), dev(z)
        out = torch.empty_like(zd)
        assert run(M, kind, Jd.data_ptr(), pd.data_ptr(), zd.data_ptr(), out.data_ptr(), n) == 0
        got = out.cpu().numpy()
        for e in range(n):
            want = rows(J, z[e], kind in (1, 2), t, omt * gam.real, omt * gam.imag)
            for r, w in enumerate(want):
                for have, exact in ((got[e, r].real, -w.re), (got[e, r].imag, -w.im)):
                    err = abs(float(Fraction(float(have)) - exact))
                    bound = 2.0 ** -52 * abs(float(exact)) + 2.0 ** -85 * w.size
                    assert err <= bound, (seed, e, r, err, bound)
