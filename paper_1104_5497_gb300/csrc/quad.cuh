// quad.cuh -- a generic square system of quadratics, P_i(z) = sum_t c_t w(a_t) w(b_t)
// with w(-1) = 1 (a term list), tracked along the same total-degree gamma-trick homotopy
//   H(z, t) = gamma (1 - t) Q(z) + t P(z),  Q_i = z_i^2 - 1,
// from the 2^n start points z in {+1, -1}^n (section "Numerical Polynomial Homotopy
// Continuation Method", including its one-variable example x^2 - 5 from x^2 - 1), in
// FP64, then refined, certified (alpha-theory) and deduplicated like the XY ring.
//
// Tracking, refinement and certification run with one path per warp (quad_warp.cuh).  This
// file is the Cauchy endgame's policy, one path per thread: the terms are sorted by equation
// on the host (row offsets in QSys.row) and live in device memory owned by the system; every
// thread reads them in the same order (broadcast loads).  The Jacobian is dense: H_z is built
// in the per-thread shared matrix and factored by the augmented Householder QR (aug_qr_solve).
#pragma once

#include "cauchy.cuh"
#include "quad_warp.cuh"

// Policy of cauchy_body: FP64, one dense NV x NV Jacobian per thread.
template <int NVT>
struct QuadProblem {
    using R = double;
    using Sys = QSys;
    static constexpr int BLOCK = 32;
    static constexpr int NV = NVT;
    static constexpr int MD = NVT;

    template <class V>
    static __device__ __forceinline__ cx<double> w(const V &z, int a) {
        return a < 0 ? cx<double>{1.0, 0.0} : z.get(a);
    }

    // -H(z, t) with exact products and double-double sums, rounded once (as for the XY ring)
    static __device__ __forceinline__ void residual(const Sys &S, const SVec<double, BLOCK> &pt,
                                                    double s, double omt,
                                                    const SVec<double, BLOCK> &out, bool wr) {
        residual_g(S, pt, s, omt, cx<double>{S.gre, S.gim}, out, wr);
    }

    template <class Out2>
    static __device__ __forceinline__ bool solve(const Sys &S, const SMat<NV, double, BLOCK> &A,
                                                 const SVec<double, BLOCK> &pt, double s,
                                                 double omt, bool two_rhs,
                                                 const SVec<double, BLOCK> &res,
                                                 const SVec<double, BLOCK> &out1, const Out2 &out2,
                                                 bool wr) {
        return solve_g(S, A, pt, s, omt, cx<double>{S.gre, S.gim}, two_rhs, res, out1, out2, wr);
    }

    // the same with an explicit gamma (the Cauchy endgame's real-t equivalent at a complex t)
    static __device__ __forceinline__ void residual_g(const Sys &S, const SVec<double, BLOCK> &pt,
                                                      double s, double omt, cx<double> gam,
                                                      const SVec<double, BLOCK> &out, bool wr) {
        using E = EFT<double>;
        const ext<double> zero = {0.0, 0.0};
        const double g1r = E::mul(omt, gam.re), g1i = E::mul(omt, gam.im);
#pragma unroll 1
        for (int i = 0; i < NV; i++) {
            ext<double> pr = zero, pi = zero;
#pragma unroll 1
            for (int t = S.row[i]; t < S.row[i + 1]; t++) {
                const QTerm T = S.terms[t];
                const cx<double> wa = w(pt, T.a), wb = w(pt, T.b);
                ext<double> mr = zero, mi = zero;   // wa * wb
                ext_acc(mr, wa.re, wb.re);
                ext_acc(mr, -wa.im, wb.im);
                ext_acc(mi, wa.re, wb.im);
                ext_acc(mi, wa.im, wb.re);
                ext_acc_ext(pr, T.cre, mr);
                ext_acc_ext(pr, -T.cim, mi);
                ext_acc_ext(pi, T.cre, mi);
                ext_acc_ext(pi, T.cim, mr);
            }
            const cx<double> zi = pt.get(i);
            ext<double> qr = {-1.0, 0.0}, qi = zero;   // z_i^2 - 1
            ext_acc(qr, zi.re, zi.re);
            ext_acc(qr, -zi.im, zi.im);
            ext_acc(qi, 2.0 * zi.re, zi.im);
            ext<double> hr = zero, hi = zero;
            ext_acc_ext(hr, g1r, qr);
            ext_acc_ext(hr, -g1i, qi);
            ext_acc_ext(hr, s, pr);
            ext_acc_ext(hi, g1r, qi);
            ext_acc_ext(hi, g1i, qr);
            ext_acc_ext(hi, s, pi);
            if (wr) out.set(i, cx<double>{-ext_val(hr), -ext_val(hi)});
        }
    }

    // H_z d = r: r = -H_t (two_rhs false) or r1 = res and r2 = -H_t (two_rhs true)
    template <class Out2>
    static __device__ __forceinline__ bool solve_g(const Sys &S, const SMat<NV, double, BLOCK> &A,
                                                   const SVec<double, BLOCK> &pt, double s,
                                                   double omt, cx<double> gam, bool two_rhs,
                                                   const SVec<double, BLOCK> &res,
                                                   const SVec<double, BLOCK> &out1,
                                                   const Out2 &out2, bool wr) {
        const cx<double> g2 = cscale(2.0 * omt, gam);
#pragma unroll 1
        for (int c = 0; c < NV; c++)
#pragma unroll 1
            for (int i = 0; i < NV; i++) A.set(i, c, cx<double>{0.0, 0.0});
#pragma unroll 1
        for (int i = 0; i < NV; i++) {
            const cx<double> zi = pt.get(i);
            A.set(i, i, cmul(g2, zi));
            cx<double> p = cx<double>{0.0, 0.0};
#pragma unroll 1
            for (int t = S.row[i]; t < S.row[i + 1]; t++) {
                const QTerm T = S.terms[t];
                const cx<double> c = cx<double>{T.cre, T.cim};
                const cx<double> wa = w(pt, T.a), wb = w(pt, T.b);
                p = cadd(p, cmul(c, cmul(wa, wb)));
                if (T.a >= 0) A.set(i, T.a, cadd(A.get(i, T.a), cscale(s, cmul(c, wb))));
                if (T.b >= 0) A.set(i, T.b, cadd(A.get(i, T.b), cscale(s, cmul(c, wa))));
            }
            // -H_t = gamma Q - P
            const cx<double> z2 = cmul(zi, zi);
            const cx<double> mht = csub(cmul(gam, cx<double>{z2.re - 1.0, z2.im}), p);
            A.set(i, NV, two_rhs ? res.get(i) : mht);
            if (two_rhs) A.set(i, NV + 1, mht);
        }
        const bool ok = aug_qr_solve<NV, double, BLOCK>(A, two_rhs);
        double chk = 0.0;
#pragma unroll 1
        for (int i = 0; i < NV; i++) {
            const cx<double> d0 = A.get(i, NV);
            chk += cabs2(d0);
            if (two_rhs) {
                const cx<double> d1 = A.get(i, NV + 1);
                chk += cabs2(d1);
                if (wr) out2.set(i, d1);
            }
            if (wr) out1.set(i, d0);
        }
        return ok && isfinite(chk);
    }
};

template <int NV>
__global__ void __launch_bounds__(32)
    quad_cauchy_kernel(const __grid_constant__ QSys S, const __grid_constant__ EGCtl C,
                       const EPView ep, const WorkList wl, int32_t *cyc, int32_t *egst) {
    cauchy_body<QuadProblem<NV>>(S, C, ep, wl, cyc, egst);
}
