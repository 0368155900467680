// xy_refine_far.cuh -- refinement and certification of the XY ring's far endpoints, one warp per
// endpoint (the method and its formulas: xy_endgame.cuh).
//
// The certificate is taken at the first iterate whose Newton correction is at most
// refine_eps (1 + ||z||).  At ||z|| ~ 1e6 that tolerance, the corrections' rounding and the certificate's
// bound lie within a factor of a hundred of each other, so whether such an endpoint certifies depends
// on the rounding of every operation, and another operation order certifies others: of
// 77,000 certified endpoints of N = 13 samples 13 had another class by the four-lane kernel
// (xy_refine_group.cuh), from the same starting points.  So the far endpoints keep one fixed order
// of operations, the one their classes have always been decided with: P in double-double sums,
// Householder QR with stored reflectors, ||DP^-1||_F column by column.  The line is far_exponent
// (nphc_internal.cuh): 0.1% of the endpoints of a ring lie beyond it.
//
// Every sum runs in that order whatever the lanes; they share out what is independent: sites,
// matrix entries, columns under a reflector, right-hand sides.  Bound by the FP64 pipe (67 cycles a
// warp instruction): some 4,000 of them per evaluation at M = 12.
#pragma once

#include "xy_endgame.cuh"

// Working set of one endpoint, in complex doubles.
template <int M>
struct FarLayout {
    static constexpr int TQ = 0;                // conj(tau) of the reflectors
    static constexpr int AH = TQ + M;           // frame a^
    static constexpr int BH = AH + M;           // frame b^
    static constexpr int IV = BH + M;           // iv (real part)
    static constexpr int AD = IV + M;           // d f_j / d c_j
    static constexpr int BD = AD + M;           // d f_j / d s_j
    static constexpr int Z = BD + M;            // c_1..c_M, s_1..s_M
    static constexpr int D = Z + 2 * M;         // -P, then the Newton correction
    static constexpr int S = D + 2 * M;         // M x M, column-major; its QR
    static constexpr int B = S + M * M;         // M right-hand sides
    static constexpr int TOTAL = B + M * M;
};

// Double-double sums, renormalised after every operation.
struct dd {
    double hi, lo;
};
__device__ __forceinline__ dd dd_two_prod(double a, double b) {
    const double p = __dmul_rn(a, b);
    return dd{p, __fma_rn(a, b, -p)};
}
__device__ __forceinline__ dd dd_add(dd a, dd b) {
    const double s = __dadd_rn(a.hi, b.hi);
    const double bb = __dsub_rn(s, a.hi);
    const double e = __dadd_rn(__dsub_rn(a.hi, __dsub_rn(s, bb)), __dsub_rn(b.hi, bb));
    const double lo = __dadd_rn(e, __dadd_rn(a.lo, b.lo));
    const double hi = __dadd_rn(s, lo);
    return dd{hi, __dsub_rn(lo, __dsub_rn(hi, s))};
}
__device__ __forceinline__ dd dd_mul_d(dd a, double b) {   // b a double
    const dd p = dd_two_prod(a.hi, b);
    const double lo = __fma_rn(a.lo, b, p.lo);
    const double hi = __dadd_rn(p.hi, lo);
    return dd{hi, __dsub_rn(lo, __dsub_rn(hi, p.hi))};
}
__device__ __forceinline__ double dd_val(dd a) { return __dadd_rn(a.hi, a.lo); }

__device__ __forceinline__ double far_max(double v) {   // over the warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <int M>
struct FarPath {
    using L = FarLayout<M>;
    cx<double> *f;      // working set, in shared memory
    const double *J;    // J[k * (M + 1) + l], l = M the pinned site
    int lane;
    __device__ __forceinline__ cx<double> &at(int off, int i) const { return f[off + i]; }
    __device__ __forceinline__ cx<double> &S(int i, int c) const { return f[L::S + c * M + i]; }

    // -P(z) into D; returns ||P||_inf
    __device__ double minus_p() const {
        double res = 0.0;
        if (lane < M) {
            const int k = lane;
            const double *Jk = J + k * (M + 1);
            dd ur = {Jk[M], 0.0}, ui = {0.0, 0.0}, wr = {0.0, 0.0}, wi = {0.0, 0.0};
#pragma unroll 1
            for (int l = 0; l < M; l++) {   // J_kk = 0 adds exact zeros
                const cx<double> xl = at(L::Z, l), yl = at(L::Z, M + l);
                ur = dd_add(ur, dd_two_prod(Jk[l], xl.re));
                ui = dd_add(ui, dd_two_prod(Jk[l], xl.im));
                wr = dd_add(wr, dd_two_prod(Jk[l], yl.re));
                wi = dd_add(wi, dd_two_prod(Jk[l], yl.im));
            }
            const cx<double> x = at(L::Z, k), y = at(L::Z, M + k);
            const dd fr = dd_add(dd_add(dd_mul_d(ur, y.re), dd_mul_d(ui, -y.im)),   // f = y u - x w
                                 dd_add(dd_mul_d(wr, -x.re), dd_mul_d(wi, x.im)));
            const dd fi = dd_add(dd_add(dd_mul_d(ui, y.re), dd_mul_d(ur, y.im)),
                                 dd_add(dd_mul_d(wi, -x.re), dd_mul_d(wr, -x.im)));
            dd gr = dd_add(dd_add(dd_two_prod(x.re, x.re), dd_two_prod(-x.im, x.im)),
                           dd_add(dd_two_prod(y.re, y.re), dd_two_prod(-y.im, y.im)));
            gr = dd_add(gr, dd{-1.0, 0.0});                                         // g = x^2 + y^2 - 1
            const dd gi = dd_add(dd_two_prod(2.0 * x.re, x.im), dd_two_prod(2.0 * y.re, y.im));
            const cx<double> fk = {dd_val(fr), dd_val(fi)}, gk = {dd_val(gr), dd_val(gi)};
            res = fmax(sqrt(cabs2(fk)), sqrt(cabs2(gk)));
            at(L::D, k) = cx<double>{-fk.re, -fk.im};
            at(L::D, M + k) = cx<double>{-gk.re, -gk.im};
        }
        __syncwarp();
        return far_max(res);
    }

    // C_kj, the q_j-coefficient of gradient row k in the frame
    __device__ __forceinline__ cx<double> C(int k, int j) const {
        const cx<double> ah = at(L::AH, j), bh = at(L::BH, j);
        if (k == j) return cadd(cmulc(ah, at(L::AD, j)), cmulc(bh, at(L::BD, j)));
        return cscale(J[k * (M + 1) + j], csub(cmulc(ah, at(L::Z, M + k)), cmulc(bh, at(L::Z, k))));
    }

    // Frames, diagonal Jacobian entries, S and its Householder QR: R above a real diagonal, the
    // reflectors (1, v) below it, conj(tau) in TQ.  False when S is singular.
    __device__ bool factor() const {
        if (lane < M) {
            const int j = lane;
            const double *Jj = J + j * (M + 1);
            cx<double> u = {Jj[M], 0.0}, w = {0.0, 0.0};
#pragma unroll 1
            for (int l = 0; l < M; l++) {
                const cx<double> xl = at(L::Z, l), yl = at(L::Z, M + l);
                u.re += Jj[l] * xl.re;
                u.im += Jj[l] * xl.im;
                w.re += Jj[l] * yl.re;
                w.im += Jj[l] * yl.im;
            }
            at(L::AD, j) = cx<double>{-w.re, -w.im};
            at(L::BD, j) = u;
            const cx<double> a = cscale(2.0, at(L::Z, j)), b = cscale(2.0, at(L::Z, M + j));
            const double iv = rsqrt(cabs2(a) + cabs2(b));
            at(L::IV, j) = cx<double>{iv, 0.0};
            at(L::AH, j) = cscale(iv, a);
            at(L::BH, j) = cscale(iv, b);
        }
        __syncwarp();
#pragma unroll 1
        for (int e = lane; e < M * M; e += 32) {
            const int j = e / M, k = e % M;
            const cx<double> ah = at(L::AH, j), bh = at(L::BH, j);
            S(k, j) = k == j ? csub(cmul(at(L::AD, j), bh), cmul(at(L::BD, j), ah))
                             : cscale(J[k * (M + 1) + j], cadd(cmul(at(L::Z, M + k), bh), cmul(at(L::Z, k), ah)));
        }
        __syncwarp();
        bool ok = true;
#pragma unroll 1
        for (int k = 0; k < M; k++) {
            const cx<double> al = S(k, k);
            double xn2 = 0.0;
#pragma unroll 1
            for (int i = k + 1; i < M; i++) xn2 += cabs2(S(i, k));
            const double an = sqrt(cabs2(al) + xn2);
            ok = ok && an > 0.0;
            const double beta = al.re >= 0.0 ? -an : an;
            const cx<double> tauc = cx<double>{(beta - al.re) / beta, al.im / beta};
            const cx<double> sc = crecip(cx<double>{al.re - beta, al.im});
            __syncwarp();
            if (lane > k && lane < M) S(lane, k) = cmul(S(lane, k), sc);
            if (lane == k) {
                S(k, k) = cx<double>{beta, 0.0};
                at(L::TQ, k) = tauc;
            }
            __syncwarp();
            if (lane > k && lane < M) {
                const int c = lane;
                cx<double> wv = S(k, c);
#pragma unroll 1
                for (int i = k + 1; i < M; i++) wv = cadd(wv, cmulc(S(i, k), S(i, c)));
                wv = cmul(tauc, wv);
                S(k, c) = csub(S(k, c), wv);
#pragma unroll 1
                for (int i = k + 1; i < M; i++) S(i, c) = csub(S(i, c), cmul(S(i, k), wv));
            }
            __syncwarp();
        }
        return ok;
    }

    // b <- R^-1 Q^H b by one lane; returns ||b||^2 afterwards
    __device__ double schur_solve(cx<double> *b) const {
#pragma unroll 1
        for (int k = 0; k < M; k++) {
            cx<double> wv = b[k];
#pragma unroll 1
            for (int i = k + 1; i < M; i++) wv = cadd(wv, cmulc(S(i, k), b[i]));
            wv = cmul(at(L::TQ, k), wv);
            b[k] = csub(b[k], wv);
#pragma unroll 1
            for (int i = k + 1; i < M; i++) b[i] = csub(b[i], cmul(S(i, k), wv));
        }
        double n2 = 0.0;
#pragma unroll 1
        for (int k = M - 1; k >= 0; k--) {
            cx<double> acc = b[k];
#pragma unroll 1
            for (int c = k + 1; c < M; c++) acc = csub(acc, cmul(S(k, c), b[c]));
            acc = cscale(1.0 / S(k, k).re, acc);
            b[k] = acc;
            n2 += cabs2(acc);
        }
        return n2;
    }

    // D <- DP^-1 D after factor; returns ||D||^2
    __device__ double solve() const {
        cx<double> *const d = f + L::D;
        if (lane < M) d[M + lane] = cscale(at(L::IV, lane).re, d[M + lane]);
        __syncwarp();
        if (lane < M) {
            cx<double> acc = d[lane];
#pragma unroll 1
            for (int j = 0; j < M; j++) acc = csub(acc, cmul(C(lane, j), d[M + j]));
            d[lane] = acc;
        }
        __syncwarp();
        if (lane == 0) schur_solve(d);
        __syncwarp();
        if (lane < M) {
            const cx<double> ah = at(L::AH, lane), bh = at(L::BH, lane), q = d[M + lane], s = d[lane];
            const cx<double> dx = cadd(cmulc(ah, q), cmul(bh, s)), dy = csub(cmulc(bh, q), cmul(ah, s));
            d[lane] = dx;
            d[M + lane] = dy;
        }
        __syncwarp();
        double n2 = 0.0;
#pragma unroll 1
        for (int j = 0; j < M; j++) n2 += cabs2(d[j]) + cabs2(d[M + j]);
        return n2;
    }

    // ||DP^-1||_F after factor
    __device__ double inv_fro() const {
        double s = 0.0;
#pragma unroll 1
        for (int j = 0; j < M; j++) s += at(L::IV, j).re * at(L::IV, j).re;
        // columns of S^-1 and of S^-1 C D^-1, one on each lane
#pragma unroll 1
        for (int h = 0; h < 2; h++) {
            double n2 = 0.0;
            if (lane < M) {
                cx<double> *const b = f + L::B + lane * M;
#pragma unroll 1
                for (int k = 0; k < M; k++)
                    b[k] = h == 0 ? cx<double>{k == lane ? 1.0 : 0.0, 0.0} : cscale(at(L::IV, lane).re, C(k, lane));
                n2 = schur_solve(b);
            }
#pragma unroll 1
            for (int j = 0; j < M; j++) s += __shfl_sync(0xffffffffu, n2, j);
        }
        __syncwarp();
        return sqrt(s);
    }

    // ||DP||_F after factor
    __device__ double jac_fro() const {
        double s = 0.0;
#pragma unroll 1
        for (int k = 0; k < M; k++) {
            const double xy = cabs2(at(L::Z, k)) + cabs2(at(L::Z, M + k));
            double jj = 0.0;
#pragma unroll 1
            for (int j = 0; j < M; j++) jj += J[k * (M + 1) + j] * J[k * (M + 1) + j];
            s += jj * xy + cabs2(at(L::AD, k)) + cabs2(at(L::BD, k)) + 4.0 * xy;
        }
        return sqrt(s);
    }

    __device__ double z_norm2() const {
        double s = 0.0;
#pragma unroll 1
        for (int k = 0; k < 2 * M; k++) s += cabs2(at(L::Z, k));
        return s;
    }
    __device__ __forceinline__ double z_max() const {
        return far_max(lane < 2 * M ? sqrt(cabs2(at(L::Z, lane))) : 0.0);
    }

    // ||DP^-1||_F from a factorisation made at Z with ||DP^-1 P|| = dn; whether the point may certify
    __device__ bool certify(const XYSys &sys, double dn, double &inv) const {
        const double fro = jac_fro(), zi = z_max();
        inv = inv_fro();
        return isfinite(dn) && isfinite(inv) && fro * inv <= sys.kappa_sing * fmax(1.0, zi * zi);
    }
    __device__ bool evaluate_and_certify(const XYSys &sys, double &beta, double &inv, double &res) const {
        res = minus_p();
        if (!factor()) return false;
        beta = sqrt(solve());
        return certify(sys, beta, inv);
    }
};

// Refinement, certification and the real test of entry e, which reached t = 1; the whole warp, its
// control flow uniform.
template <int M>
__device__ __noinline__ void far_refine(cx<double> *work, const double *J, const XYSys &sys, double tol_sol,
                                        double refine_eps, int refine_iters, const EPView &ep, int64_t e) {
    using L = FarLayout<M>;
    const int lane = threadIdx.x & 31;
    const FarPath<M> G{work, J, lane};
    const int64_t cnt = ep.count;
    if (lane < 2 * M) G.at(L::Z, lane) = cx<double>{ep.z_re[lane * cnt + e], ep.z_im[lane * cnt + e]};
    __syncwarp();
    bool finite = true, certified = false, cert_ok = false;
    double beta = INFINITY, inv = INFINITY, res = INFINITY;
#pragma unroll 1
    for (int it = 0; it < refine_iters; it++) {
        const double r = G.minus_p();
        if (!G.factor()) break;
        const double dn = sqrt(G.solve()), z2 = G.z_norm2();
        if (!isfinite(dn) || !isfinite(z2)) {
            finite = false;
            break;
        }
        certified = dn <= refine_eps * (1.0 + sqrt(z2));
        if (certified) {
            cert_ok = G.certify(sys, dn, inv);
            beta = dn;
            res = r;
        }
        if (lane < 2 * M) G.at(L::Z, lane) = cadd(G.at(L::Z, lane), G.at(L::D, lane));
        __syncwarp();
        if (!isfinite(G.z_norm2())) {
            finite = false;
            break;
        }
        if (certified) break;
    }
    if (finite && !certified) cert_ok = G.evaluate_and_certify(sys, beta, inv, res);
    double alpha = INFINITY, gam = INFINITY, im2 = 0.0;
    int cls = NPHC_END_SINGULAR;
    bool real_test = false;
    const double zi = G.z_max();
#pragma unroll 1
    for (int k = 0; k < 2 * M; k++) {
        const cx<double> z = G.at(L::Z, k);
        im2 += z.im * z.im;
    }
    const double im = sqrt(im2);
    if (finite && cert_ok) {
        gam = inv * sys.d2norm;
        alpha = beta * gam;
        if (res <= tol_sol * fmax(1.0, zi * zi) && alpha < NPHC_ALPHA_CERT) {
            if (alpha < 0.03 && im < 1.0 / (20.0 * gam)) real_test = true;
            else cls = im > 2.0 * beta ? NPHC_END_NONREAL : NPHC_END_UNDECIDED;
        }
    } else {
        beta = INFINITY;
    }
    if (lane < 2 * M) {
        const cx<double> z = G.at(L::Z, lane);
        ep.z_re[lane * cnt + e] = z.re;
        ep.z_im[lane * cnt + e] = z.im;
    }
    if (real_test) {   // z and Re z share their zero: the test at Re z decides
        __syncwarp();
        if (lane < 2 * M) G.at(L::Z, lane).im = 0.0;
        __syncwarp();
        double br, ir, rr;
        const bool ok = G.evaluate_and_certify(sys, br, ir, rr);
        cls = ok && br * ir * sys.d2norm < NPHC_ALPHA_CERT ? NPHC_END_REAL
              : im > 2.0 * beta                            ? NPHC_END_NONREAL
                                                           : NPHC_END_UNDECIDED;
    }
    if (lane == 0) {
        ep.alpha[e] = alpha;
        ep.beta[e] = beta;
        ep.gamma[e] = gam;
        ep.resid[e] = finite ? res : INFINITY;
        ep.cls[e] = cls;
    }
    __syncwarp();
}
