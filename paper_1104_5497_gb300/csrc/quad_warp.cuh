// quad_warp.cuh -- tracking, refinement and certification of a generic quadratic system
// (QSys: P_i(z) = sum_t c_t w(a_t) w(b_t), w(-1) = 1) in FP64 with one path or endpoint per
// warp.
//
// A system has at most 2^12 paths: with one per thread its 32 to 128 warps leave most of the
// chip idle, and a warp's time is the FP64 instruction count of one lane (67 cycles each,
// whatever the number of lanes; a dense residual and QR of n = 10 take 40 k).  So the lanes
// share a path:
//   * sums over an equation's terms: 32 / n lanes per equation, each a share of the terms,
//     their (compensated: gsum in nphc_internal.cuh) sums combined by shuffles;
//   * the Jacobian: one (variable, equation) cell per lane at a time, from the list of the
//     terms that contribute to it;
//   * the linear solve: warp_lu_solve (xy_track_warp.cuh).
// The 1,024 paths of a random n = 10 system (30 terms per equation): tracking 336 -> 21.8 ms,
// refinement 1.60 -> 0.14 ms against one path and endpoint per thread.  What remains is the
// FP64 chain of the longest paths (about 1.7 paths per scheduler).
#pragma once

#include "xy_endgame.cuh"
#include "xy_track_warp.cuh"

template <int N>
struct QuadLayout {   // shared memory per warp, complex doubles
    static constexpr int A = 0;                 // [H_z | r | -H_t], column-major
    static constexpr int Z0 = A + N * (N + 2);
    static constexpr int K1 = Z0 + N;
    static constexpr int AC = K1 + N;
    static constexpr int ZC = AC + N;
    static constexpr int W1 = ZC + N;
    static constexpr int PV = W1 + N;           // P at ZC (from the residual)
    static constexpr int TOTAL = PV + N;
};

struct QuadPath {
    cx<double> *s;
    int lane;
    __device__ __forceinline__ cx<double> &at(int off, int i) const { return s[off + i]; }
};

__device__ __forceinline__ cx<double> quad_w(const cx<double> *z, int a) {
    return a < 0 ? cx<double>{1.0, 0.0} : z[a];
}

// P_i(z) for the equation i = lane / (32 / N) of this lane, complete on the lane's first lane
// (lane % (32 / N) == 0): plain, or with exact products and compensated sums.
template <int N>
struct QuadSum {
    static constexpr int LE = 32 / N;   // lanes per equation
    static __device__ __forceinline__ int eq(int lane) { return lane / LE; }
    static __device__ __forceinline__ bool first(int lane) { return lane < N * LE && lane % LE == 0; }

    static __device__ __forceinline__ cx<double> plain(const QSys &S, const cx<double> *z, int lane) {
        cx<double> p = {0.0, 0.0};
        const int i = lane / LE;
        if (i < N) {
#pragma unroll 1
            for (int t = S.row[i] + lane % LE; t < S.row[i + 1]; t += LE) {
                const QTerm T = S.terms[t];
                p = cfma64(cx<double>{T.cre, T.cim}, cmul(quad_w(z, T.a), quad_w(z, T.b)), p);
            }
        }
#pragma unroll
        for (int o = 1; o < LE; o <<= 1) {
            const cx<double> q = {__shfl_down_sync(0xffffffffu, p.re, o), __shfl_down_sync(0xffffffffu, p.im, o)};
            if (lane % LE % (2 * o) == 0 && lane % LE + o < LE) p = cadd(p, q);
        }
        return p;
    }
    static __device__ __forceinline__ int wexp(const cx<double> *z, int a) {
        return a < 0 ? 0 : max(gexp(z[a].re), gexp(z[a].im));
    }
    // With exact products and compensated sums, on grids (gsum) of each equation's own size: the
    // variables and equations of a system may differ by many orders.  |P_i's parts| < 2^(kp - 1).
    static __device__ __forceinline__ void compensated(const QSys &S, const cx<double> *z, int lane,
                                                       ext<double> &pr, ext<double> &pi, int &kp) {
        const int i = lane / LE;
        int kt = -4000;   // exponent of the equation's largest |c| |w(a)| |w(b)|, in integers
        if (i < N) {
#pragma unroll 1
            for (int t = S.row[i] + lane % LE; t < S.row[i + 1]; t += LE) {
                const QTerm T = S.terms[t];
                kt = max(kt, max(gexp(T.cre), gexp(T.cim)) + wexp(z, T.a) + wexp(z, T.b));
            }
        }
#pragma unroll
        for (int o = 1; o < LE; o++) {   // over the equation's lanes
            const int ko = __shfl_down_sync(0xffffffffu, kt, o);
            if (lane % LE == 0) kt = max(kt, ko);
        }
        kt = __shfl_sync(0xffffffffu, kt, i * LE < 32 ? i * LE : 0);
        // a term's parts are below 2^(kt + 5), the sum of all below their number times that
        kp = kt + 6 + (i < N ? 32 - __clz(S.row[i + 1] - S.row[i]) : 0);
        const double ap = gsum_anchor(kp);
        gsum sr = {ap, 0.0}, si = sr;
        if (i < N) {
#pragma unroll 1
            for (int t = S.row[i] + lane % LE; t < S.row[i + 1]; t += LE) {
                const QTerm T = S.terms[t];
                const cx<double> wa = quad_w(z, T.a), wb = quad_w(z, T.b);
                const double am = gsum_anchor(wexp(z, T.a) + wexp(z, T.b) + 4);
                gsum smr = {am, 0.0}, smi = smr;   // wa wb
                gsum_acc(smr, wa.re, wb.re);
                gsum_acc(smr, -wa.im, wb.im);
                gsum_acc(smi, wa.re, wb.im);
                gsum_acc(smi, wa.im, wb.re);
                const ext<double> mr = gsum_ext(smr, am), mi = gsum_ext(smi, am);
                gsum_acc_ext(sr, T.cre, mr);
                gsum_acc_ext(sr, -T.cim, mi);
                gsum_acc_ext(si, T.cre, mi);
                gsum_acc_ext(si, T.cim, mr);
            }
        }
        pr = gsum_ext(sr, ap);
        pi = gsum_ext(si, ap);
#pragma unroll
        for (int o = 1; o < LE; o <<= 1) {
            const ext<double> qr = {__shfl_down_sync(0xffffffffu, pr.hi, o), __shfl_down_sync(0xffffffffu, pr.lo, o)};
            const ext<double> qi = {__shfl_down_sync(0xffffffffu, pi.hi, o), __shfl_down_sync(0xffffffffu, pi.lo, o)};
            if (lane % LE % (2 * o) == 0 && lane % LE + o < LE) {
                pr = grid_add(pr, qr);
                pi = grid_add(pi, qi);
            }
        }
    }
};

// dP_i/dz_v at z for cell = v N + i
template <int N>
__device__ __forceinline__ cx<double> quad_jac(const QSys &S, const cx<double> *z, int cell) {
    cx<double> d = {0.0, 0.0};
#pragma unroll 1
    for (int t = S.jrow[cell]; t < S.jrow[cell + 1]; t++) {
        const QTerm T = S.jac[t];
        d = cfma64(cx<double>{T.cre, T.cim}, quad_w(z, T.a), d);
    }
    return d;
}

// Tracker policy (see warp_track_body): the state is z itself.
template <int N>
struct WarpQuad {
    using Sys = QSys;
    using L = QuadLayout<N>;
    using Path = QuadPath;
    static constexpr int NV = N;
    static constexpr double NORM2 = 1.0;
    static __device__ __forceinline__ void load(const Path &P, const EPView &ep, int64_t e) {
        const int k = P.lane;
        if (k < N) P.at(L::Z0, k) = cx<double>{ep.z_re[k * ep.count + e], ep.z_im[k * ep.count + e]};
    }
    static __device__ __forceinline__ void store(const Path &P, const EPView &ep, int64_t e) {
        const int k = P.lane;
        if (k < N) {
            ep.z_re[k * ep.count + e] = P.at(L::Z0, k).re;
            ep.z_im[k * ep.count + e] = P.at(L::Z0, k).im;
        }
    }
    static __device__ __forceinline__ double norminf(const Path &P) {
        return P.lane < N ? sqrt(cabs2(P.at(L::ZC, P.lane))) : 0.0;
    }
    // z_i = -1 if bit i of the path is set, else +1; dz_i/dt at t = 0 is -P_i(z) / (2 gamma z_i)
    static __device__ __forceinline__ void start(const Path &P, const Sys &S, int64_t p) {
        const int lane = P.lane, i = QuadSum<N>::eq(lane);
        if (lane < N) P.at(L::Z0, lane) = cx<double>{((p >> lane) & 1) ? -1.0 : 1.0, 0.0};
        __syncwarp();
        const cx<double> v = QuadSum<N>::plain(S, P.s + L::Z0, lane);
        if (QuadSum<N>::first(lane))
            P.at(L::K1, i) = cscale(-0.5 * P.at(L::Z0, i).re, cmul(crecip(cx<double>{S.gre, S.gim}), v));
    }
    // -H(ZC, t) into W1 with exact products and compensated sums, rounded once
    static __device__ __forceinline__ void residual(const Path &P, const Sys &S, double s, double omt) {
        using E = EFT<double>;
        const int lane = P.lane, i = QuadSum<N>::eq(lane);
        ext<double> pr, pi;
        int kp;
        QuadSum<N>::compensated(S, P.s + L::ZC, lane, pr, pi, kp);
        if (QuadSum<N>::first(lane)) {
            const double g1r = E::mul(omt, S.gre), g1i = E::mul(omt, S.gim);
            const cx<double> zi = P.at(L::ZC, i);
            const int kq = max(0, 2 * max(gexp(zi.re), gexp(zi.im)) + 2) + 2;
            const double aq = gsum_anchor(kq);
            gsum sqr = gsum_start(aq, -1.0), sqi = {aq, 0.0};   // z_i^2 - 1
            gsum_acc(sqr, zi.re, zi.re);
            gsum_acc(sqr, -zi.im, zi.im);
            gsum_acc(sqi, 2.0 * zi.re, zi.im);
            const ext<double> qr = gsum_ext(sqr, aq), qi = gsum_ext(sqi, aq);
            const double ah = gsum_anchor(max(max(gexp(g1r), gexp(g1i)) + kq + 1, gexp(s) + kp) + 2);
            gsum hr = {ah, 0.0}, hi = hr;
            gsum_acc_ext(hr, g1r, qr);
            gsum_acc_ext(hr, -g1i, qi);
            gsum_acc_ext(hr, s, pr);
            gsum_acc_ext(hi, g1r, qi);
            gsum_acc_ext(hi, g1i, qr);
            gsum_acc_ext(hi, s, pi);
            P.at(L::W1, i) = cx<double>{-ext_val(gsum_ext(hr, ah)), -ext_val(gsum_ext(hi, ah))};
            P.at(L::PV, i) = cx<double>{ext_val(pr), ext_val(pi)};
        }
        __syncwarp();
    }
    // H_z(ZC, t) d = r: r = -H_t, d into W1 (two_rhs false), or r1 = W1 (the residual), d1 into
    // W1, and r2 = -H_t (P from that residual), d2 into out2
    static __device__ __forceinline__ bool solve(const Path &P, const Sys &S, double s, double omt,
                                                 bool two_rhs, int out2) {
        const int lane = P.lane, i = QuadSum<N>::eq(lane);
        const cx<double> *z = P.s + L::ZC;
        const cx<double> gam = {S.gre, S.gim}, g2 = cscale(2.0 * omt, gam);
        const cx<double> p = two_rhs ? P.at(L::PV, i < N ? i : 0) : QuadSum<N>::plain(S, z, lane);
        if (QuadSum<N>::first(lane)) {
            const cx<double> zi = z[i], z2 = cmul(zi, zi);
            const cx<double> mht = csub(cmul(gam, cx<double>{z2.re - 1.0, z2.im}), p);   // gamma Q - P
            P.s[L::A + N * N + i] = two_rhs ? P.at(L::W1, i) : mht;
            if (two_rhs) P.s[L::A + N * (N + 1) + i] = mht;
        }
#pragma unroll 1
        for (int c = lane; c < N * N; c += 32) {
            cx<double> d = cscale(s, quad_jac<N>(S, z, c));
            if (c / N == c % N) d = cadd(d, cmul(g2, z[c % N]));
            P.s[L::A + c] = d;
        }
        __syncwarp();
        cx<double> cur;
        const bool ok = warp_lu_solve<N>(P.s + L::A, lane, two_rhs, cur);
        const int row = lane & 15, r = lane >> 4;
        double chk = 0.0;
        if (row < N && (r == 0 || two_rhs)) {
            P.at(r ? out2 : L::W1, row) = cur;
            chk = cabs2(cur);
        }
        __syncwarp();
        return ok && isfinite(warp_sum(chk));
    }
};

// ------------------------------------------------- refinement, certification --
template <int N>
struct QuadRefineLayout {   // shared memory per warp, complex doubles
    static constexpr int Z = 0;
    static constexpr int A = Z + N;              // [DP | -P | I], column-major, 2 N + 1 columns
    static constexpr int TOTAL = A + N * (2 * N + 1);
};

struct QuadEval {
    double res, dn, z2, zi, fro, inv;   // ||P||_inf, ||DP^-1 P||, ||z||_2^2, ||z||_inf, ||DP||_F, ||DP^-1||_F
    cx<double> d;                       // Newton correction, component `lane`
    bool ok;                            // false: DP is singular
};

// P, its Newton correction and the norms of DP and DP^-1 at Z: LU with partial pivoting of
// [DP | -P | I], then a back substitution per right-hand side, one on each lane.
template <int N>
__device__ QuadEval quad_evaluate(const QuadPath &W, const QSys &S) {
    using L = QuadRefineLayout<N>;
    constexpr int NC = 2 * N + 1;
    const int lane = W.lane, i = QuadSum<N>::eq(lane);
    cx<double> *const A = W.s + L::A;
    const cx<double> *z = W.s + L::Z;
    QuadEval v;
    ext<double> pr, pi;
    int kp;
    QuadSum<N>::compensated(S, z, lane, pr, pi, kp);
    double pm = 0.0;
    if (QuadSum<N>::first(lane)) {
        const cx<double> p = {ext_val(pr), ext_val(pi)};
        pm = cabs2(p);
        A[N * N + i] = cx<double>{-p.re, -p.im};
    }
    v.res = sqrt(warp_max(pm));
    double f = 0.0;
#pragma unroll 1
    for (int c = lane; c < N * N; c += 32) {
        const cx<double> d = quad_jac<N>(S, z, c);
        A[c] = d;
        A[N * (N + 1) + c] = cx<double>{c / N == c % N ? 1.0 : 0.0, 0.0};
        f += cabs2(d);
    }
    v.fro = sqrt(warp_sum(f));
    const cx<double> zl = lane < N ? z[lane] : cx<double>{0.0, 0.0};
    v.z2 = warp_sum(cabs2(zl));
    v.zi = sqrt(warp_max(cabs2(zl)));
    __syncwarp();
    v.ok = true;
#pragma unroll 1
    for (int k = 0; k < N; k++) {
        unsigned long long key = 0ull;
        if (lane >= k && lane < N) {
            const cx<double> a = A[k * N + lane];
            key = ((unsigned long long)__double_as_longlong(fabs(a.re) + fabs(a.im)) & ~31ull) |
                  (unsigned long long)(31 - lane);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
        key = __shfl_sync(0xffffffffu, key, 0);
        int p = 31 - (int)(key & 31ull);
        if ((key >> 5) == 0) {
            v.ok = false;
            p = k;
        }
        if (p != k) {
#pragma unroll 1
            for (int c = k + lane; c < NC; c += 32) {
                const cx<double> t = A[c * N + k];
                A[c * N + k] = A[c * N + p];
                A[c * N + p] = t;
            }
            __syncwarp();
        }
        const cx<double> a = A[k * N + k];
        const double rd = 1.0 / fma(a.re, a.re, a.im * a.im);
        const cx<double> ip = cx<double>{a.re * rd, -a.im * rd};
        if (lane > k && lane < N) A[k * N + lane] = cmul(A[k * N + lane], ip);
        __syncwarp();
        const int nr = N - 1 - k, nc = NC - 1 - k;
#pragma unroll 1
        for (int q = lane; q < nr * nc; q += 32) {
            const int c = k + 1 + q / nr, r = k + 1 + q % nr;
            A[c * N + r] = cfnms(A[c * N + r], A[k * N + r], A[c * N + k]);
        }
        if (lane == 31) A[k * N + k] = ip;   // nothing reads the pivot in this step's update
        __syncwarp();
    }
    // right-hand side `lane`: 0 the Newton correction, 1 .. N the columns of DP^-1
    double n2 = 0.0;
    if (lane <= N) {
        cx<double> *const b = A + (N + lane) * N;
#pragma unroll 1
        for (int k = N - 1; k >= 0; k--) {
            cx<double> x = b[k];
#pragma unroll 1
            for (int c = k + 1; c < N; c++) x = cfnms(x, A[c * N + k], b[c]);
            x = cmul(x, A[k * N + k]);
            b[k] = x;
            n2 += cabs2(x);
        }
    }
    v.dn = sqrt(__shfl_sync(0xffffffffu, n2, 0));
    v.inv = sqrt(warp_sum(lane >= 1 ? n2 : 0.0));
    __syncwarp();
    v.d = lane < N ? A[N * N + lane] : cx<double>{0.0, 0.0};
    __syncwarp();
    return v;
}

// Refinement, certification and the real test of every selected entry that reached t = 1 (the
// rules of xy_refine_group.cuh).  One endpoint per warp, the control flow uniform over it.
template <int N, int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
    quad_refine_warp_kernel(const __grid_constant__ QSys S, double tol_sol, double refine_eps,
                            int refine_iters, const EPView ep, const WorkList wl) {
    using L = QuadRefineLayout<N>;
    extern __shared__ __align__(16) unsigned char wraw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const QuadPath W{reinterpret_cast<cx<double> *>(wraw) + (size_t)wid * L::TOTAL, lane};
    const double alpha0 = NPHC_ALPHA_CERT;
    const int64_t cnt = ep.count, total = worklist_size(wl, cnt);
    for (int64_t q = (int64_t)wid * gridDim.x + blockIdx.x; q < total; q += (int64_t)WARPS * gridDim.x) {
        const int64_t e = worklist_entry(wl, q, cnt);
        if (e < 0) continue;   // rejected by the debug build's check
        const int st = ep.status[e];
        if (st != NPHC_PATH_REACHED) {
            if (lane == 0) {
                ep.alpha[e] = ep.beta[e] = ep.gamma[e] = ep.resid[e] = INFINITY;
                ep.cls[e] = st == NPHC_PATH_DIVERGED ? NPHC_END_NONE : NPHC_END_FAILED;
            }
            continue;
        }
        cx<double> z = {0.0, 0.0};   // component `lane`
        if (lane < N) z = cx<double>{ep.z_re[lane * cnt + e], ep.z_im[lane * cnt + e]};
        auto put = [&](cx<double> v) {
            __syncwarp();
            if (lane < N) W.at(L::Z, lane) = v;
            __syncwarp();
        };
        put(z);
        // Newton refinement; the iteration whose correction meets refine_eps certifies its own
        // point, and the output is that point's Newton iterate
        QuadEval v;
        bool finite = true, certified = false;
#pragma unroll 1
        for (int it = 0; it < refine_iters; it++) {
            v = quad_evaluate<N>(W, S);
            if (!v.ok) break;
            if (!isfinite(v.dn) || !isfinite(v.z2)) {
                finite = false;
                break;
            }
            z = cadd(z, v.d);
            put(z);
            if (!isfinite(warp_sum(cabs2(z)))) {
                finite = false;
                break;
            }
            if (v.dn <= refine_eps * (1.0 + sqrt(v.z2))) {
                certified = true;
                break;
            }
        }
        if (finite && !certified) v = quad_evaluate<N>(W, S);
        auto cond_ok = [&](const QuadEval &x) {
            return x.ok && isfinite(x.dn) && isfinite(x.inv) &&
                   x.fro * x.inv <= S.kappa_sing * fmax(1.0, x.zi * x.zi);
        };
        double alpha = INFINITY, beta = INFINITY, gam = INFINITY;
        int cls = NPHC_END_SINGULAR;
        if (finite && cond_ok(v)) {
            beta = v.dn;
            gam = v.inv * S.d2norm;
            alpha = beta * gam;
            const double zi2 = warp_max(cabs2(z)), im = sqrt(warp_sum(z.im * z.im));
            if (v.res <= tol_sol * fmax(1.0, zi2) && alpha < alpha0) {
                cls = im > 2.0 * beta ? NPHC_END_NONREAL : NPHC_END_UNDECIDED;
                if (alpha < 0.03 && im < 1.0 / (20.0 * gam)) {   // z and Re z share their zero
                    put(cx<double>{z.re, 0.0});
                    const QuadEval r = quad_evaluate<N>(W, S);
                    if (cond_ok(r) && r.dn * r.inv * S.d2norm < alpha0) cls = NPHC_END_REAL;
                }
            }
        }
        if (lane < N) {
            ep.z_re[lane * cnt + e] = z.re;
            ep.z_im[lane * cnt + e] = z.im;
        }
        if (lane == 0) {
            ep.alpha[e] = alpha;
            ep.beta[e] = beta;
            ep.gamma[e] = gam;
            ep.resid[e] = finite ? v.res : INFINITY;
            ep.cls[e] = cls;
        }
    }
}

template <int N, int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
    quad_track_warp_kernel(const __grid_constant__ QSys S, const __grid_constant__ XYCtl C,
                           const EPView ep, const WorkList wl) {
    warp_track_body<WarpQuad<N>>(S, C, ep, wl);
}
