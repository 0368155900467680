// xy_refine_group.cuh -- refinement and certification of the XY ring's endpoints (the method
// and its formulas: xy_endgame.cuh), four lanes per endpoint, eight endpoints per warp.
//
// The kernel is bound by the FP64 pipe, which takes a warp instruction every 67 cycles per
// scheduler (measured, dependent or not, whatever the number of active lanes): its time is
// the FP64 instruction count of the longest lane times the warps per scheduler.  So the work
// of an endpoint is laid over lanes until the rows fill them (lane g owns the sites and
// matrix rows j = g + 4 q), and the instruction count is what it is written for:
//   * P by sums on grids (gsum in nphc_internal.cuh, as in the trackers' residuals): four
//     instructions per term where an exact product and a two-sum took ten (15,013 points of
//     N = 10 2.72 -> 2.06 ms);
//   * the Schur right-hand side as J times per-site vectors;
//   * LU with partial pivoting instead of Householder QR (half the operations, no square
//     roots; the pivot search compares |re| + |im| as integers);
//   * ||DP^-1||_F from 2 M triangular solves, dealt out over the four lanes.
// A few hundred endpoints fill the chip.  Against one endpoint per thread with double-double sums
// and a QR (solve's launches, ms): N = 5 0.7 -> 0.15, N = 8 (3,432 endpoints) 2.96 -> 0.45, N = 10
// (47,100) 14.4 -> 6.1; called step by step, 15,013 points of N = 10 6.0 -> 2.06 and N = 13 (2,900)
// 26.4 -> 2.0.
//
// An endpoint is in one of two states: it waits for an evaluation (P, the factorisation of DP
// and the Newton correction at its point) or for a certificate from the factorisation just
// made.  A warp runs evaluations while any of its endpoints waits for one, then the
// certificates together; a finished slot takes the next entry.  Far endpoints are the whole warp's
// (xy_refine_far.cuh), one at a time, as the slots come upon them.
#pragma once

#include "xy_refine_far.cuh"

constexpr int RG_PATHS = 8;   // endpoints per warp (one warp per block)

// Shared memory per endpoint, in complex doubles ([index * 8 + endpoint]).
template <int M>
struct RGLayout {
    static constexpr int Z = 0;              // x_1..x_M, y_1..y_M
    static constexpr int A = Z + 2 * M;      // [S | rhs], row-major, M + 1 columns; then its LU
    static constexpr int AH = A + M * (M + 1);   // frame a^
    static constexpr int BH = AH + M;        // frame b^
    static constexpr int QA = BH + M;        // conj(a^_j) q_j, then the Newton correction dx_j
    static constexpr int QB = QA + M;        // conj(b^_j) q_j, then dy_j
    static constexpr int U = QB + M;         // u_j
    static constexpr int W = U + M;          // w_j
    static constexpr int IV = W + M;         // (1 / |(a_j, b_j)|, -)
    static constexpr int V = IV + M;         // a column per lane, 4 M; of all endpoints together,
    static constexpr int TOTAL = V + 4 * M;  // between certificates, the working set of a far one,
    static constexpr int FAR = FarLayout<M>::TOTAL > RG_PATHS * 4 * M   // which takes so many more at M = 12
                                   ? FarLayout<M>::TOTAL - RG_PATHS * 4 * M : 0;
};

template <int M>
constexpr size_t rg_smem_per_block() {
    return sizeof(cx<double>) * (size_t)(RG_PATHS * RGLayout<M>::TOTAL + RGLayout<M>::FAR) +
           sizeof(double) * (size_t)(M * (M + 2));   // J rows (the pinned column too), sums of squares
}

__device__ __forceinline__ cx<double> rg_cfma(cx<double> a, cx<double> b, cx<double> c) {   // c + a b
    return cx<double>{fma(-a.im, b.im, fma(a.re, b.re, c.re)), fma(a.im, b.re, fma(a.re, b.im, c.im))};
}
__device__ __forceinline__ cx<double> rg_cfms(cx<double> a, cx<double> b, cx<double> c) {   // c - a b
    return cx<double>{fma(a.im, b.im, fma(-a.re, b.re, c.re)), fma(-a.im, b.re, fma(-a.re, b.im, c.im))};
}
__device__ __forceinline__ double rg_sum(unsigned m, double v) {
    v += __shfl_xor_sync(m, v, 8);
    return v + __shfl_xor_sync(m, v, 16);
}
__device__ __forceinline__ double rg_max(unsigned m, double v) {
    v = fmax(v, __shfl_xor_sync(m, v, 8));
    return fmax(v, __shfl_xor_sync(m, v, 16));
}
__device__ __forceinline__ int gexp_max(cx<double> x, cx<double> y) {
    return max(max(gexp(x.re), gexp(x.im)), max(gexp(y.re), gexp(y.im)));
}

// One endpoint's lanes: slot memory, own rows.
template <int M>
struct RGPath {
    using L = RGLayout<M>;
    static constexpr int SL = (M + 3) / 4;
    cx<double> *sm;      // this endpoint's column of the shared memory
    const double *J;     // J[k * (M + 1) + l], l = M the pinned site
    const double *jj;    // sum over free l of J_kl^2
    int g;               // lane of the endpoint
    unsigned m;          // the lanes that run this code together (whole endpoints)
    __device__ __forceinline__ cx<double> &at(int off, int i) const { return sm[(off + i) * RG_PATHS]; }
    __device__ __forceinline__ cx<double> &A(int i, int c) const { return sm[(L::A + i * (M + 1) + c) * RG_PATHS]; }
    __device__ __forceinline__ void sync() const { __syncwarp(m); }
};

// Warps (one-warp blocks) of a launch with up to two per scheduler that share `total` items,
// `slots` side by side in each: half of them while that is enough, so that no scheduler runs
// two FP64 chains where one would do.
__device__ __forceinline__ int fill_warps(int64_t total, int slots) {
    const int half = ((int)gridDim.x + 1) / 2;
    return total <= (int64_t)half * slots ? half : (int)gridDim.x;
}

// P's rows of site j, as sums on grids: f = y u - x w and g = x^2 + y^2 - 1, and u, w.
template <int M>
__device__ __forceinline__ void rg_row(const RGPath<M> &G, int j, cx<double> &f, cx<double> &gg, cx<double> &u,
                                       cx<double> &w) {
    using L = RGLayout<M>;
    const double *Jj = G.J + j * (M + 1);
    int er = gexp(Jj[M]);
#pragma unroll 1
    for (int l = 0; l < M; l++) er = max(er, gexp(Jj[l]) + gexp_max(G.at(L::Z, l), G.at(L::Z, M + l)));
    const int ku = gsum_row(er);   // |u|, |w| < 2^(ku - 1)
    const double au = gsum_anchor(ku);
    gsum sur = gsum_start(au, Jj[M]), sui = {au, 0.0}, swr = sui, swi = sui;
#pragma unroll 1
    for (int l = 0; l < M; l++) {   // J_jj = 0 adds exact zeros
        const cx<double> xl = G.at(L::Z, l), yl = G.at(L::Z, M + l);
        const double c = Jj[l];
        gsum_acc(sur, c, xl.re);
        gsum_acc(sui, c, xl.im);
        gsum_acc(swr, c, yl.re);
        gsum_acc(swi, c, yl.im);
    }
    const ext<double> ur = gsum_ext(sur, au), ui = gsum_ext(sui, au), wr = gsum_ext(swr, au), wi = gsum_ext(swi, au);
    const cx<double> x = G.at(L::Z, j), y = G.at(L::Z, M + j);
    const int ek = gexp_max(x, y);
    const double af = gsum_anchor(ek + ku + 3), ag = gsum_anchor(max(0, 2 * ek + 4) + 2);
    gsum fr = {af, 0.0}, fi = fr, gr = gsum_start(ag, -1.0), gi = {ag, 0.0};
    gsum_acc_ext(fr, y.re, ur);
    gsum_acc_ext(fr, -y.im, ui);
    gsum_acc_ext(fr, -x.re, wr);
    gsum_acc_ext(fr, x.im, wi);
    gsum_acc_ext(fi, y.re, ui);
    gsum_acc_ext(fi, y.im, ur);
    gsum_acc_ext(fi, -x.re, wi);
    gsum_acc_ext(fi, -x.im, wr);
    gsum_acc(gr, x.re, x.re);
    gsum_acc(gr, -x.im, x.im);
    gsum_acc(gr, y.re, y.re);
    gsum_acc(gr, -y.im, y.im);
    gsum_acc(gi, 2.0 * x.re, x.im);
    gsum_acc(gi, 2.0 * y.re, y.im);
    f = cx<double>{ext_val(gsum_ext(fr, af)), ext_val(gsum_ext(fi, af))};
    gg = cx<double>{ext_val(gsum_ext(gr, ag)), ext_val(gsum_ext(gi, ag))};
    u = cx<double>{ext_val(ur), ext_val(ui)};
    w = cx<double>{ext_val(wr), ext_val(wi)};
}

// P, the factorisation of DP and the Newton correction D = -DP^-1 P (into QA, QB) at Z.  res = ||P||_inf,
// dn2 = ||D||_2^2, z2 = ||z||_2^2; perm: the row of S behind each row of the factor, four bits
// each.  False when the Schur matrix is singular.
template <int M>
__device__ bool rg_evaluate(const RGPath<M> &G, double &res, double &dn2, double &z2, unsigned long long &perm) {
    using L = RGLayout<M>;
    const int g = G.g;
    double pmax = 0.0;
#pragma unroll 1
    for (int j = g; j < M; j += 4) {
        const cx<double> x = G.at(L::Z, j), y = G.at(L::Z, M + j);
        cx<double> f, gg, u, w;
        rg_row<M>(G, j, f, gg, u, w);
        pmax = fmax(pmax, fmax(cabs2(f), cabs2(gg)));
        const cx<double> a = cscale(2.0, x), b = cscale(2.0, y);
        const double iv = rsqrt(cabs2(a) + cabs2(b));
        const cx<double> ah = cscale(iv, a), bh = cscale(iv, b);
        const cx<double> q = cscale(-iv, gg);
        G.at(L::AH, j) = ah;
        G.at(L::BH, j) = bh;
        G.at(L::IV, j) = cx<double>{iv, 0.0};
        G.at(L::U, j) = u;
        G.at(L::W, j) = w;
        G.at(L::QA, j) = cmulc(ah, q);
        G.at(L::QB, j) = cmulc(bh, q);
        G.A(j, M) = cx<double>{-f.re, -f.im};
    }
    G.sync();
    // own rows: S_kj = J_kj (y_k b^_j + x_k a^_j), S_kk = -w_k b^_k - u_k a^_k; right-hand side
    // -f_k - y_k sum_j J_kj QA_j + x_k sum_j J_kj QB_j + w_k QA_k - u_k QB_k
#pragma unroll 1
    for (int k = g; k < M; k += 4) {
        const double *Jk = G.J + k * (M + 1);
        const cx<double> x = G.at(L::Z, k), y = G.at(L::Z, M + k);
        cx<double> sa = {0.0, 0.0}, sb = sa;
#pragma unroll 1
        for (int j = 0; j < M; j++) {
            const double c = Jk[j];
            const cx<double> qa = G.at(L::QA, j), qb = G.at(L::QB, j);
            sa = cx<double>{fma(c, qa.re, sa.re), fma(c, qa.im, sa.im)};
            sb = cx<double>{fma(c, qb.re, sb.re), fma(c, qb.im, sb.im)};
            G.A(k, j) = cscale(c, rg_cfma(x, G.at(L::AH, j), cmul(y, G.at(L::BH, j))));
        }
        const cx<double> u = G.at(L::U, k), w = G.at(L::W, k);
        const cx<double> d = rg_cfma(w, G.at(L::BH, k), cmul(u, G.at(L::AH, k)));
        G.A(k, k) = cx<double>{-d.re, -d.im};
        cx<double> r = G.A(k, M);
        r = rg_cfms(y, sa, r);
        r = rg_cfma(x, sb, r);
        r = rg_cfma(w, G.at(L::QA, k), r);
        r = rg_cfms(u, G.at(L::QB, k), r);
        G.A(k, M) = r;
    }
    G.sync();
    // LU with partial pivoting of [S | rhs]; multipliers below the diagonal, the pivots'
    // reciprocals on it
    bool ok = true;
    perm = 0xba9876543210ull;
#pragma unroll 1
    for (int k = 0; k < M; k++) {
        unsigned long long key = 0;
#pragma unroll 1
        for (int i = g; i < M; i += 4)
            if (i >= k) {
                const cx<double> a = G.A(i, k);
                const unsigned long long v = (unsigned long long)__double_as_longlong(fabs(a.re) + fabs(a.im));
                key = max(key, (v & ~15ull) | (unsigned long long)(15 - i));
            }
        key = max(key, __shfl_xor_sync(G.m, key, 8));
        key = max(key, __shfl_xor_sync(G.m, key, 16));
        int p = 15 - (int)(key & 15ull);
        if ((key >> 4) == 0) {   // zero from row k down
            ok = false;
            p = k;
        }
        if (p != k) {   // the same for the endpoint's four lanes
#pragma unroll 1
            for (int c = g; c <= M; c += 4) {
                const cx<double> t = G.A(k, c);
                G.A(k, c) = G.A(p, c);
                G.A(p, c) = t;
            }
            const unsigned long long x = ((perm >> (4 * k)) ^ (perm >> (4 * p))) & 15ull;
            perm ^= (x << (4 * k)) | (x << (4 * p));
        }
        G.sync();
        const cx<double> a = G.A(k, k);
        const double rd = 1.0 / fma(a.re, a.re, a.im * a.im);
        const cx<double> ip = cx<double>{a.re * rd, -a.im * rd};
#pragma unroll 1
        for (int i = g; i < M; i += 4)
            if (i > k) {
                const cx<double> l = cmul(G.A(i, k), ip);
                G.A(i, k) = l;
#pragma unroll 2
                for (int c = k + 1; c <= M; c++) G.A(i, c) = rg_cfms(l, G.A(k, c), G.A(i, c));
            }
        G.sync();
        if (g == (k & 3)) G.A(k, k) = ip;
    }
    G.sync();
#pragma unroll 1
    for (int k = M - 1; k >= 0; k--) {
        const cx<double> s = cmul(G.A(k, M), G.A(k, k));
        G.sync();
#pragma unroll 1
        for (int i = g; i <= k; i += 4) G.A(i, M) = i == k ? s : rg_cfms(G.A(i, k), s, G.A(i, M));
        G.sync();
    }
    // (dx, dy) = conj(a^, b^) q + (b^, -a^) s
    double d2 = 0.0, n2 = 0.0;
#pragma unroll 1
    for (int j = g; j < M; j += 4) {
        const cx<double> s = G.A(j, M);
        const cx<double> dx = rg_cfma(G.at(L::BH, j), s, G.at(L::QA, j));
        const cx<double> dy = rg_cfms(G.at(L::AH, j), s, G.at(L::QB, j));
        G.at(L::QA, j) = dx;
        G.at(L::QB, j) = dy;
        d2 += cabs2(dx) + cabs2(dy);
        n2 += cabs2(G.at(L::Z, j)) + cabs2(G.at(L::Z, M + j));
    }
    dn2 = rg_sum(G.m, d2);
    z2 = rg_sum(G.m, n2);
    res = sqrt(rg_max(G.m, pmax));
    return ok;
}

// ||DP^-1||_F and ||DP||_F at the point of the last evaluation, and ||z||_inf^2 there.
template <int M>
__device__ void rg_norms(const RGPath<M> &G, unsigned long long perm, double &inv_fro, double &fro, double &zi2) {
    using L = RGLayout<M>;
    const int g = G.g;
    double s = 0.0, f = 0.0, zi = 0.0;
#pragma unroll 1
    for (int j = g; j < M; j += 4) {
        const double iv = G.at(L::IV, j).re;
        s = fma(iv, iv, s);
        const double x2 = cabs2(G.at(L::Z, j)), y2 = cabs2(G.at(L::Z, M + j)), xy = x2 + y2;
        // gradient row j: J_jl y_j, -J_jl x_j (free l != j), -w_j, u_j; constraint row j: 2 x_j, 2 y_j
        f += (G.jj[j] + 4.0) * xy + cabs2(G.at(L::U, j)) + cabs2(G.at(L::W, j));
        zi = fmax(zi, fmax(x2, y2));
    }
    // columns of S^-1 (col < M) and of S^-1 C D^-1, one at a time per lane
    const int v = L::V + g * M;
#pragma unroll 1
    for (int col = g; col < 2 * M; col += 4) {
        const int j = col < M ? col : col - M;
        const cx<double> ah = G.at(L::AH, j), bh = G.at(L::BH, j);
        const double iv = G.at(L::IV, j).re;
#pragma unroll 1
        for (int i = 0; i < M; i++) {
            const int k = (int)(perm >> (4 * i)) & 15;   // row k of S is row i of the factor
            cx<double> b;
            if (col < M) {
                b = cx<double>{k == j ? 1.0 : 0.0, 0.0};
            } else if (k == j) {   // C_jj = -conj(a^) w + conj(b^) u
                b = cscale(iv, csub(cmulc(bh, G.at(L::U, j)), cmulc(ah, G.at(L::W, j))));
            } else {               // C_kj = J_kj (conj(a^) y_k - conj(b^) x_k)
                b = cscale(iv * G.J[k * (M + 1) + j],
                           csub(cmulc(ah, G.at(L::Z, M + k)), cmulc(bh, G.at(L::Z, k))));
            }
#pragma unroll 1
            for (int c = 0; c < i; c++) b = rg_cfms(G.A(i, c), G.at(v, c), b);
            G.at(v, i) = b;
        }
#pragma unroll 1
        for (int i = M - 1; i >= 0; i--) {
            cx<double> b = G.at(v, i);
#pragma unroll 1
            for (int c = i + 1; c < M; c++) b = rg_cfms(G.A(i, c), G.at(v, c), b);
            b = cmul(b, G.A(i, i));
            G.at(v, i) = b;
            s += cabs2(b);
        }
    }
    inv_fro = sqrt(rg_sum(G.m, s));
    fro = sqrt(rg_sum(G.m, f));
    zi2 = rg_max(G.m, zi);
}

// Refinement, certification and the real test of every selected entry that reached t = 1.
template <int M>
__global__ void __launch_bounds__(32)
    xy_refine_group_kernel(const __grid_constant__ XYSys S, double tol_sol, double refine_eps,
                           int refine_iters, const __grid_constant__ EPView ep, const WorkList wl,
                           int shortcut, int far_exp) {
    using L = RGLayout<M>;
    extern __shared__ __align__(16) unsigned char rgraw[];
    cx<double> *const base = reinterpret_cast<cx<double> *>(rgraw);
    double *const J = reinterpret_cast<double *>(base + RG_PATHS * L::TOTAL + L::FAR);
    double *const jj = J + M * (M + 1);
    const int lane = threadIdx.x, g = lane >> 3, pth = lane & 7;
    for (int i = lane; i < M * (M + 1); i += 32) J[i] = S.Jd[(i / (M + 1)) * NPHC_JSTRIDE + i % (M + 1)];
    __syncwarp();
    if (lane < M) {
        double s = 0.0;
        for (int l = 0; l < M; l++) s = fma(J[lane * (M + 1) + l], J[lane * (M + 1) + l], s);
        jj[lane] = s;
    }
    __syncwarp();
    RGPath<M> G{base + pth, J, jj, g, 0xffffffffu};
    const unsigned mine = 0x01010101u << pth;   // this endpoint's four lanes
    const double alpha0 = NPHC_ALPHA_CERT;
    const int64_t cnt = ep.count, total = worklist_size(wl, cnt);

    // entries one per warp before more per warp: i = endpoint slot * warps + warp
    const int warps = fill_warps(total, RG_PATHS);
    if ((int)blockIdx.x >= warps) return;
    int64_t next = (int64_t)pth * warps + blockIdx.x;
    const int64_t stride = (int64_t)RG_PATHS * warps;
    enum { IDLE, EVALUATE, CERTIFY, FAR, DONE };
    enum { NEWTON, LAST, FINAL, REAL };   // what the evaluation is for: a Newton step, the one
                                          // whose correction met the tolerance, a certificate
                                          // without a step, the real test at Re z
    int state = IDLE, mode = NEWTON, it = 0;
    int64_t e = -1;
    bool sc = false;
    double dn = INFINITY, beta = INFINITY, res = INFINITY, im = 0.0;
    unsigned long long perm = 0;

    for (;;) {
        // ---- idle slots take the next entry that needs work
#pragma unroll 1
        while (state == IDLE) {
            if (next >= total) {
                state = DONE;
                break;
            }
            e = worklist_entry(wl, next, cnt);   // -1: rejected (debug)
            next += stride;
            if (e < 0) continue;
            const int st = ep.status[e];
            sc = shortcut && (st == NPHC_PATH_HANDOFF || st == NPHC_PATH_HANDOFF_COND);
            if (sc || st == NPHC_PATH_REACHED) {
#pragma unroll 1
                for (int k = g; k < 2 * M; k += 4)
                    G.at(L::Z, k) = cx<double>{ep.z_re[k * cnt + e], ep.z_im[k * cnt + e]};
                state = EVALUATE;
                if (!sc) {
                    int ez = -2000;
#pragma unroll 1
                    for (int k = g; k < 2 * M; k += 4) {
                        const cx<double> z = G.at(L::Z, k);
                        ez = max(ez, max(gexp(z.re), gexp(z.im)));
                    }
                    ez = max(ez, __shfl_xor_sync(mine, ez, 8));
                    ez = max(ez, __shfl_xor_sync(mine, ez, 16));
                    if (ez >= far_exp) state = FAR;
                }
                it = 0;
                mode = refine_iters > 0 ? NEWTON : FINAL;
            } else if (g == 0) {
                ep.alpha[e] = ep.beta[e] = ep.gamma[e] = ep.resid[e] = INFINITY;
                ep.cls[e] = st == NPHC_PATH_DIVERGED ? NPHC_END_NONE : NPHC_END_FAILED;
            }
        }
        __syncwarp();
        unsigned fa = __ballot_sync(0xffffffffu, state == FAR) & 0xffu;   // slots with a far endpoint
        if (fa) {
            for (; fa; fa &= fa - 1)
                far_refine<M>(base + RG_PATHS * L::V, J, S, tol_sol, refine_eps, refine_iters, ep,
                              __shfl_sync(0xffffffffu, e, __ffs(fa) - 1));
            if (state == FAR) state = IDLE;
            continue;
        }
        const unsigned ev = __ballot_sync(0xffffffffu, state == EVALUATE);
        const unsigned ce = __ballot_sync(0xffffffffu, state == CERTIFY);
        if (!ev && !ce) break;   // every slot is done
        bool settle = false;                  // the endpoint's outcome is known
        bool finite = true, cert_ok = false;
        double inv = INFINITY;
        auto step = [&]() -> double {         // z += the Newton correction; the new ||z||_2^2
            double zn = 0.0;
#pragma unroll 1
            for (int j = g; j < M; j += 4) {
                const cx<double> x = cadd(G.at(L::Z, j), G.at(L::QA, j));
                const cx<double> y = cadd(G.at(L::Z, M + j), G.at(L::QB, j));
                G.at(L::Z, j) = x;
                G.at(L::Z, M + j) = y;
                zn += cabs2(x) + cabs2(y);
            }
            return rg_sum(mine, zn);   // only some of the endpoints may be here
        };
        if (ev) {
            if (state == EVALUATE) {
                G.m = ev;
                double r, dn2, z2;
                const bool ok = rg_evaluate<M>(G, r, dn2, z2, perm);
                dn = sqrt(dn2);
                if (mode != REAL) res = r;
                if (!ok) {                    // singular: never certified
                    state = CERTIFY;
                    settle = mode != REAL;
                    dn = INFINITY;
                } else if (mode != NEWTON) {
                    state = CERTIFY;
                } else if (sc && it == 0 && !(dn <= SHORTCUT_TRUST * (1.0 + sqrt(z2)))) {
                    state = IDLE;             // not in a basin: left for FP64 tracking
                } else if (!isfinite(dn) || !isfinite(z2)) {
                    finite = false;
                    settle = true;
                } else if (dn <= refine_eps * (1.0 + sqrt(z2))) {
                    mode = LAST;
                    state = CERTIFY;
                } else if (!isfinite(step())) {
                    finite = false;
                    settle = true;
                } else if (++it >= refine_iters) {
                    mode = FINAL;
                }
                if (mode != REAL) beta = dn;
            }
        } else if (state == CERTIFY) {
            G.m = ce;
            double fro, zi2;
            rg_norms<M>(G, perm, inv, fro, zi2);
            cert_ok = isfinite(dn) && isfinite(inv) && fro * inv <= S.kappa_sing * fmax(1.0, zi2);
            if (mode == REAL) {
                if (g == 0)
                    ep.cls[e] = cert_ok && dn * inv * S.d2norm < alpha0 ? NPHC_END_REAL
                                : im > 2.0 * beta                       ? NPHC_END_NONREAL
                                                                        : NPHC_END_UNDECIDED;
                state = IDLE;
            } else {
                if (mode == LAST) finite = isfinite(step());
                settle = true;
            }
        }
        const unsigned se = __ballot_sync(0xffffffffu, settle);
        if (settle) {
            double alpha = INFINITY, gam = INFINITY, zi2 = 0.0, im2 = 0.0;
            int cls = NPHC_END_SINGULAR;
            bool real_test = false;
#pragma unroll 1
            for (int j = g; j < M; j += 4) {
                const cx<double> x = G.at(L::Z, j), y = G.at(L::Z, M + j);
                zi2 = fmax(zi2, fmax(cabs2(x), cabs2(y)));
                im2 = fma(x.im, x.im, fma(y.im, y.im, im2));
            }
            zi2 = rg_max(se, zi2);
            im = sqrt(rg_sum(se, im2));
            if (finite && cert_ok) {
                gam = inv * S.d2norm;
                alpha = beta * gam;
                // Delta_sol relative to the size of the (quadratic) terms: max(1, ||z||_inf^2)
                if (res <= tol_sol * fmax(1.0, zi2) && alpha < alpha0) {
                    // z and Re z share their zero when alpha < 0.03 and ||Im z|| < 1 / (20 gamma):
                    // then the test at Re z decides
                    if (alpha < 0.03 && im < 1.0 / (20.0 * gam)) real_test = true;
                    else cls = im > 2.0 * beta ? NPHC_END_NONREAL : NPHC_END_UNDECIDED;
                }
            } else {
                beta = INFINITY;
            }
            state = IDLE;
            // a hand-off point that does not certify is left for FP64 tracking
            if (!sc || real_test || cls != NPHC_END_SINGULAR) {
                if (g == 0) {
                    ep.alpha[e] = alpha;
                    ep.beta[e] = beta;
                    ep.gamma[e] = gam;
                    ep.resid[e] = finite ? res : INFINITY;
                    if (sc) {
                        ep.status[e] = NPHC_PATH_REACHED;
                        ep.t[e] = 1.0;
                    }
                    if (!real_test) ep.cls[e] = cls;
                }
#pragma unroll 1
                for (int k = g; k < M; k += 4)
#pragma unroll 1
                    for (int i = k; i < 2 * M; i += M) {
                        const cx<double> z = G.at(L::Z, i);
                        ep.z_re[i * cnt + e] = z.re;
                        ep.z_im[i * cnt + e] = z.im;
                        G.at(L::Z, i) = cx<double>{z.re, 0.0};
                    }
                if (real_test) {
                    mode = REAL;
                    state = EVALUATE;
                }
            }
        }
        // an entry's unknowns are loaded by other lanes than those that have just written out the
        // slot's last one
        __syncwarp();
    }
}
