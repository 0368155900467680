// xy_track_group64.cuh -- the FP64 tracker of the XY ring: four lanes per path, eight paths per
// warp (the method: xy_track.cuh; the linear algebra: xy_solve.cuh).
//
// Bound by the FP64 pipe: a warp instruction every 67 cycles per scheduler, whatever the number
// of active lanes and dependent or not (measured), so the time is the FP64 instruction count of
// the longest lane of every warp.  Against one path per thread the count per solve falls with
// the lanes (rows of the last lanes idle), a ring's paths make four times as many warps, and no
// warp waits in lockstep:
//   * lane g owns the sites and rows g + 4 q; the matrix and the vectors are in shared memory,
//     every loop is rolled (the pipe hides the loads, and the code stays small);
//   * the light-cone scales are powers of two taken from the exponents (any scale solves the
//     same system; a power of two adds no rounding and no FP64 instruction);
//   * the corrector's residual is sums on grids (gsum in nphc_internal.cuh): four instructions per
//     term where compensated sums with two-sums took ten (N = 8, 16,384 paths: 121 -> 97 ms);
//   * each path is in its own phase (RK4 stage or corrector iteration); a warp runs whichever
//     kind of solve more of its paths wait for, as the FP32 pass does (xy_track_group.cuh).
// Against one path per warp (xy_track_warp.cuh) a solve's chain is three times as long but eight
// paths share it: the better choice once there are ten paths for every scheduler.  16,384 paths
// of N = 8: 248 ms with one path per thread, 170 with one per warp, 97 here.
#pragma once

#include "xy_track_warp.cuh"

constexpr int G64_PATHS = 8;   // paths per warp (one warp per block)

template <int M>
struct G64Layout {   // complex doubles per path ([index * 8 + path])
    static constexpr int PQ = 0;              // evaluation point: p_j, then q_j
    static constexpr int Z0 = PQ + 2 * M;     // accepted point
    static constexpr int K1 = Z0 + 2 * M;     // dz/dt there
    static constexpr int AC = K1 + 2 * M;     // RK4 sum; in a corrector solve X1, Y1, then dz/dt
    static constexpr int W = AC + 2 * M;      // X0, Y0 of the first right-hand side, then its d
    static constexpr int FR = W + 2 * M;      // sp b^_j, sq a^_j
    static constexpr int A = FR + 2 * M;      // [S | b0 | b1], row-major, M + 2 columns
    static constexpr int TOTAL = A + M * (M + 2);
};

template <int M>
constexpr size_t g64_smem_per_block() {
    return sizeof(cx<double>) * (size_t)(G64_PATHS * G64Layout<M>::TOTAL) + sizeof(double) * (size_t)(M * (M + 1));
}

template <int M>
struct G64Path {
    using L = G64Layout<M>;
    cx<double> *sm;
    const double *J;     // J[k * (M + 1) + l], l = M the pinned site
    int g;
    unsigned m;          // the lanes that run this code together (whole paths)
    __device__ __forceinline__ cx<double> &at(int off, int i) const { return sm[(off + i) * G64_PATHS]; }
    __device__ __forceinline__ cx<double> &A(int i, int c) const { return sm[(L::A + i * (M + 2) + c) * G64_PATHS]; }
    __device__ __forceinline__ void sync() const { __syncwarp(m); }
    __device__ __forceinline__ double sum(double v) const {
        v += __shfl_xor_sync(m, v, 8);
        return v + __shfl_xor_sync(m, v, 16);
    }
    __device__ __forceinline__ double most(double v) const {
        v = fmax(v, __shfl_xor_sync(m, v, 8));
        return fmax(v, __shfl_xor_sync(m, v, 16));
    }
};

// -H rows of one site (f32_residual_rows in f32_step.cuh, in FP64), as sums on grids (gsum).
// |U_p|, |U_q| < 2^(ku - 1).
__device__ __forceinline__ void f64_residual_rows(cx<double> p, cx<double> q, const ext<double> &upr,
                                                  const ext<double> &upi, const ext<double> &uqr,
                                                  const ext<double> &uqi, int ku, double s, double hs,
                                                  double gr, double gi, cx<double> &rf, cx<double> &rg) {
    const int ep = max(gexp(p.re), gexp(p.im)), eq = max(gexp(q.re), gexp(q.im)), ek = max(ep, eq);
    const int eg = max(gexp(gr), gexp(gi)), kd = ek + ku + 3;
    // h has a grid of its own: near infinity p q stays near 1 where p^2 or q^2 is huge
    const int kh = max(0, ep + eq + 2) + 2, kx = max(2 * ek + 3, kh) + 1;
    const double ad = gsum_anchor(kd), ah = gsum_anchor(kh), ax = gsum_anchor(kx);
    gsum sdr = {ad, 0.0}, sdi = sdr;   // D = q U_p - p U_q, f = i D / 2
    gsum_acc_ext(sdr, q.re, upr);
    gsum_acc_ext(sdr, -q.im, upi);
    gsum_acc_ext(sdr, -p.re, uqr);
    gsum_acc_ext(sdr, p.im, uqi);
    gsum_acc_ext(sdi, q.re, upi);
    gsum_acc_ext(sdi, q.im, upr);
    gsum_acc_ext(sdi, -p.re, uqi);
    gsum_acc_ext(sdi, -p.im, uqr);
    const ext<double> dr = gsum_ext(sdr, ad), di = gsum_ext(sdi, ad);
    // h = (p q - 2) / 2, B = (p^2 + q^2) / 4: x^2 - 1 = h + B, y^2 - 1 = h - B, p q - 1 = 2 h + 1
    const cx<double> ph = cscale(0.5, p), qh = cscale(0.5, q);
    gsum shr = gsum_start(ah, -1.0), shi = {ah, 0.0}, sbr = {ax, 0.0}, sbi = sbr;
    gsum_acc(shr, ph.re, q.re);
    gsum_acc(shr, -ph.im, q.im);
    gsum_acc(shi, ph.re, q.im);
    gsum_acc(shi, ph.im, q.re);
    gsum_acc(sbr, ph.re, ph.re);
    gsum_acc(sbr, -ph.im, ph.im);
    gsum_acc(sbr, qh.re, qh.re);
    gsum_acc(sbr, -qh.im, qh.im);
    gsum_acc(sbi, ph.re, p.im);
    gsum_acc(sbi, qh.re, q.im);
    const ext<double> hr = gsum_ext(shr, ah), hi = gsum_ext(shi, ah), br = gsum_ext(sbr, ax), bi = gsum_ext(sbi, ax);
    gsum tr = {__dsub_rn(ax, br.hi), -br.lo}, ti = {__dsub_rn(ax, bi.hi), -bi.lo};   // -B
    gsum_add(sbr, hr);
    gsum_add(sbi, hi);
    gsum_add(tr, hr);
    gsum_add(ti, hi);
    const ext<double> xr = gsum_ext(sbr, ax), xi = gsum_ext(sbi, ax), yr = gsum_ext(tr, ax), yi = gsum_ext(ti, ax);
    // H_f = gomt X + t f ;  H_g = gomt Y + t (2 h + 1)
    const double s2 = 2.0 * s;
    const double af = gsum_anchor(max(eg + kx + 2, gexp(hs) + kd) + 2);
    const double ag = gsum_anchor(max(eg + kx + 2, gexp(s2) + kh + 1) + 2);
    gsum fr = {af, 0.0}, fi = fr, kr = gsum_start(ag, s), ki = {ag, 0.0};
    gsum_acc_ext(fr, gr, xr);
    gsum_acc_ext(fr, -gi, xi);
    gsum_acc_ext(fr, -hs, di);
    gsum_acc_ext(fi, gr, xi);
    gsum_acc_ext(fi, gi, xr);
    gsum_acc_ext(fi, hs, dr);
    gsum_acc_ext(kr, gr, yr);
    gsum_acc_ext(kr, -gi, yi);
    gsum_acc_ext(kr, s2, hr);
    gsum_acc_ext(ki, gr, yi);
    gsum_acc_ext(ki, gi, yr);
    gsum_acc_ext(ki, s2, hi);
    rf = cx<double>{-ext_val(gsum_ext(fr, af)), -ext_val(gsum_ext(fi, af))};
    rg = cx<double>{-ext_val(gsum_ext(kr, ag)), -ext_val(gsum_ext(ki, ag))};
}

// -H's rows of site j at PQ, and U_p, U_q.
template <int M>
__device__ __forceinline__ void g64_residual(const G64Path<M> &G, int j, double s, double gr, double gi, cx<double> &Up,
                                             cx<double> &Uq, cx<double> &rf, cx<double> &rg) {
    using L = G64Layout<M>;
    const double *Jj = G.J + j * (M + 1);
    int er = gexp(Jj[M]);
#pragma unroll 1
    for (int l = 0; l < M; l++) {
        const cx<double> pl = G.at(L::PQ, l), ql = G.at(L::PQ, M + l);
        er = max(er, gexp(Jj[l]) + max(max(gexp(pl.re), gexp(pl.im)), max(gexp(ql.re), gexp(ql.im))));
    }
    const int ku = gsum_row(er);
    const double au = gsum_anchor(ku);
    gsum spr = gsum_start(au, Jj[M]), spi = {au, 0.0}, sqr = spr, sqi = spi;
#pragma unroll 1
    for (int l = 0; l < M; l++) {   // J_jj = 0 adds exact zeros
        const cx<double> pl = G.at(L::PQ, l), ql = G.at(L::PQ, M + l);
        const double c = Jj[l];
        gsum_acc(spr, c, pl.re);
        gsum_acc(spi, c, pl.im);
        gsum_acc(sqr, c, ql.re);
        gsum_acc(sqi, c, ql.im);
    }
    const ext<double> upr = gsum_ext(spr, au), upi = gsum_ext(spi, au), uqr = gsum_ext(sqr, au), uqi = gsum_ext(sqi, au);
    f64_residual_rows(G.at(L::PQ, j), G.at(L::PQ, M + j), upr, upi, uqr, uqi, ku, s, 0.5 * s, gr, gi, rf, rg);
    Up = cx<double>{ext_val(upr), ext_val(upi)};
    Uq = cx<double>{ext_val(uqr), ext_val(uqi)};
}

// One solve of H_z(z, t) d = r at PQ: r = -H_t, d into W (corr false); r = -H (compensated), d into
// W, and r = -H_t, d into AC (corr true; uniform over G.m).  False when the system is singular or
// the result is not finite.
template <int M>
__device__ bool g64_solve(const G64Path<M> &G, double s, double omt, cx<double> gam, bool corr) {
    using L = G64Layout<M>;
    const int g = G.g;
    const cx<double> gomt = cscale(omt, gam);
    const double hs = 0.5 * s;
    // ---- site by site: U sums, residual rows, frames, the diagonal's terms
#pragma unroll 1
    for (int j = g; j < M; j += 4) {
        const double *Jj = G.J + j * (M + 1);
        const cx<double> p = G.at(L::PQ, j), q = G.at(L::PQ, M + j);
        cx<double> Up = {Jj[M], 0.0}, Uq = Up, rf, rg;
        if (corr) {
            g64_residual<M>(G, j, s, EFT<double>::mul(omt, gam.re), EFT<double>::mul(omt, gam.im), Up, Uq, rf, rg);
        } else {
#pragma unroll 1
            for (int l = 0; l < M; l++) {
                const cx<double> pl = G.at(L::PQ, l), ql = G.at(L::PQ, M + l);
                const double c = Jj[l];
                Up = cx<double>{fma(c, pl.re, Up.re), fma(c, pl.im, Up.im)};
                Uq = cx<double>{fma(c, ql.re, Uq.re), fma(c, ql.im, Uq.im)};
            }
        }
        cx<double> htf, htg;
        lc_minus_ht_rows<double>(p, q, Up, Uq, gam, htf, htg);
        if (!corr) {
            rf = htf;
            rg = htg;
        }
        // frame of the constraint row (g_frame_lc), the scales powers of two
        const double sp = pow2_scale(p), sq = pow2_scale(q);
        const cx<double> hd = cscale(0.5, cmul(gomt, csub(p, q)));
        const cx<double> a = cscale(sp, csub(cscale(s, q), hd)), b = cscale(sq, cadd(cscale(s, p), hd));
        const double iv = rsqrt(cabs2(a) + cabs2(b));
        const cx<double> ah = cscale(iv, a), bh = cscale(iv, b);
        const cx<double> gpq = cmul(gomt, cadd(p, q));
        const cx<double> Ajj = cscale(0.5 * sp, csub(gpq, cmul_i(cscale(s, Uq))));
        const cx<double> Bjj = cscale(0.5 * sq, cadd(gpq, cmul_i(cscale(s, Up))));
        const cx<double> q0 = cscale(iv, rg);
        const cx<double> px = cmulc(ah, q0), py = cmulc(bh, q0);
        G.at(L::W, j) = cscale(sp, px);
        G.at(L::W, M + j) = cscale(sq, py);
        G.at(L::FR, j) = cscale(sp, bh);
        G.at(L::FR, M + j) = cscale(sq, ah);
        G.A(j, j) = cfnms(cmul(Ajj, bh), Bjj, ah);
        G.A(j, M) = cfnms(cfnms(rf, Ajj, px), Bjj, py);
        if (corr) {
            const cx<double> q1 = cscale(iv, htg);
            const cx<double> px1 = cmulc(ah, q1), py1 = cmulc(bh, q1);
            G.at(L::AC, j) = cscale(sp, px1);
            G.at(L::AC, M + j) = cscale(sq, py1);
            G.A(j, M + 1) = cfnms(cfnms(htf, Ajj, px1), Bjj, py1);
        }
    }
    G.sync();
    // ---- the own rows: S_kj = (i t / 2) J_kj (q_k sp b^_j + p_k sq a^_j), right-hand sides
    // b_k -= (i t / 2) (q_k sum_j J_kj X_j - p_k sum_j J_kj Y_j)
#pragma unroll 1
    for (int k = g; k < M; k += 4) {
        const double *Jk = G.J + k * (M + 1);
        const cx<double> p = G.at(L::PQ, k), q = G.at(L::PQ, M + k);
        const cx<double> ip = cmul_i(cscale(hs, p)), iq = cmul_i(cscale(hs, q));
        cx<double> sx = {0.0, 0.0}, sy = sx, tx = sx, ty = sx;
#pragma unroll 1
        for (int j = 0; j < M; j++) {
            const double c = Jk[j];
            const cx<double> x = G.at(L::W, j), y = G.at(L::W, M + j);
            sx = cx<double>{fma(c, x.re, sx.re), fma(c, x.im, sx.im)};
            sy = cx<double>{fma(c, y.re, sy.re), fma(c, y.im, sy.im)};
            if (corr) {
                const cx<double> u = G.at(L::AC, j), v = G.at(L::AC, M + j);
                tx = cx<double>{fma(c, u.re, tx.re), fma(c, u.im, tx.im)};
                ty = cx<double>{fma(c, v.re, ty.re), fma(c, v.im, ty.im)};
            }
            if (j != k)
                G.A(k, j) = cscale(c, cfma64(ip, G.at(L::FR, M + j), cmul(iq, G.at(L::FR, j))));
        }
        G.A(k, M) = cfma64(ip, sy, cfnms(G.A(k, M), iq, sx));
        if (corr) G.A(k, M + 1) = cfma64(ip, ty, cfnms(G.A(k, M + 1), iq, tx));
    }
    G.sync();
    // ---- LU with partial pivoting (the pivot search compares |re| + |im| as integers); the
    // pivots' reciprocals on the diagonal
    const int nc = corr ? M + 2 : M + 1;
    bool ok = true;
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
        int piv = 15 - (int)(key & 15ull);
        if ((key >> 4) == 0) {
            ok = false;
            piv = k;
        }
        if (piv != k)
#pragma unroll 1
            for (int c = k + g; c < nc; c += 4) {
                const cx<double> t = G.A(k, c);
                G.A(k, c) = G.A(piv, c);
                G.A(piv, c) = t;
            }
        G.sync();
        const cx<double> a = G.A(k, k);
        const double rd = 1.0 / fma(a.re, a.re, a.im * a.im);
        const cx<double> ip = cx<double>{a.re * rd, -a.im * rd};
#pragma unroll 1
        for (int i = g; i < M; i += 4)
            if (i > k) {
                const cx<double> l = cmul(G.A(i, k), ip);
#pragma unroll 2
                for (int c = k + 1; c < nc; c++) G.A(i, c) = cfnms(G.A(i, c), l, G.A(k, c));
            }
        G.sync();
        if (g == (k & 3)) G.A(k, k) = ip;
    }
    G.sync();
#pragma unroll 1
    for (int k = M - 1; k >= 0; k--) {
        const cx<double> ip = G.A(k, k);
        const cx<double> s0 = cmul(G.A(k, M), ip);
        cx<double> s1 = {0.0, 0.0};
        if (corr) s1 = cmul(G.A(k, M + 1), ip);
        G.sync();
#pragma unroll 1
        for (int i = g; i <= k; i += 4) {
            if (i == k) {
                G.A(k, M) = s0;
                if (corr) G.A(k, M + 1) = s1;
            } else {
                const cx<double> u = G.A(i, k);
                G.A(i, M) = cfnms(G.A(i, M), u, s0);
                if (corr) G.A(i, M + 1) = cfnms(G.A(i, M + 1), u, s1);
            }
        }
        G.sync();
    }
    // ---- back to (dp, dq) = (X + sp b^ s, Y - sq a^ s)
    double chk = 0.0;
#pragma unroll 1
    for (int j = g; j < M; j += 4) {
        const cx<double> sb = G.at(L::FR, j), sa = G.at(L::FR, M + j), s0 = G.A(j, M);
        const cx<double> dp = cfma64(sb, s0, G.at(L::W, j)), dq = cfnms(G.at(L::W, M + j), sa, s0);
        G.at(L::W, j) = dp;
        G.at(L::W, M + j) = dq;
        chk += cabs2(dp) + cabs2(dq);
        if (corr) {
            const cx<double> s1 = G.A(j, M + 1);
            const cx<double> ep = cfma64(sb, s1, G.at(L::AC, j)), eq = cfnms(G.at(L::AC, M + j), sa, s1);
            G.at(L::AC, j) = ep;
            G.at(L::AC, M + j) = eq;
            chk += cabs2(ep) + cabs2(eq);
        }
    }
    return ok && isfinite(G.sum(chk));
}

// min_paths: the launch leaves lists shorter than that to the one-path-per-warp kernel (which
// leaves the others to this one); the length of a list is on the device.
template <int M>
__global__ void __launch_bounds__(32)
    xy_track_group64_kernel(const __grid_constant__ XYSys S, const __grid_constant__ XYCtl C,
                            const EPView ep, const WorkList wl, int64_t min_paths) {
    using L = G64Layout<M>;
    extern __shared__ __align__(16) unsigned char g64raw[];
    const int64_t total = worklist_size(wl, ep.count), cnt = ep.count;
    if (total < min_paths) return;
    cx<double> *const base = reinterpret_cast<cx<double> *>(g64raw);
    double *const J = reinterpret_cast<double *>(base + G64_PATHS * L::TOTAL);
    const int lane = threadIdx.x, g = lane >> 3, pth = lane & 7;
    for (int i = lane; i < M * (M + 1); i += 32) J[i] = S.Jd[(i / (M + 1)) * NPHC_JSTRIDE + i % (M + 1)];
    G64Path<M> G{base + pth, J, g, 0xffffffffu};
    const cx<double> gam = {S.gre, S.gim};
    // few paths: fewer per warp, so that every scheduler has some
    const int64_t want = (total + gridDim.x - 1) / gridDim.x;
    const int per = want < G64_PATHS ? (want < 1 ? 1 : (int)want) : G64_PATHS;

    int64_t e = pth < per ? -1 : -2;   // -1 idle, -2 drained
    int ph = 0, run = 0, attempts = 0, steps = 0, solves = 0, newton = 0;
    bool far = false, bad = false, start = false;
    double t = 0.0, h = 0.0, zlast = 0.0, zpn = 0.0;
    __syncwarp();
#pragma unroll 1
    for (;;) {
        // ---- hand new entries to idle paths
        const unsigned need = __ballot_sync(0xffffffffu, e == -1) & 0xffu;
        if (need) {
            unsigned long long first = 0;
            if (lane == 0) first = atomicAdd(wl.queue, (unsigned long long)__popc(need));
            first = __shfl_sync(0xffffffffu, first, 0);
            if (e == -1) {
                const int64_t i = (int64_t)first + __popc(need & ((1u << pth) - 1u));
                bool fresh = false;
                if (i >= total) {
                    e = -2;
                } else {
                    e = worklist_entry(wl, i, cnt);   // -1 (skipped) if the debug build rejects it
                    fresh = e >= 0;
                }
                if (fresh) {
                    run = attempts = steps = solves = newton = 0;
                    far = bad = false;
                    zlast = 0.0;
                    if (C.resume || C.accumulate) {
                        steps = ep.steps[e];
                        solves = ep.solves[e];
                        newton = ep.newton[e];
                    }
                    if (C.resume) {
#pragma unroll 1
                        for (int k = g; k < M; k += 4) {   // (x, y) to (p, q)
                            const double xr = ep.z_re[k * cnt + e], xi = ep.z_im[k * cnt + e];
                            const double yr = ep.z_re[(M + k) * cnt + e], yi = ep.z_im[(M + k) * cnt + e];
                            const cx<double> p = {xr - yi, xi + yr}, q = {xr + yi, xi - yr};
                            G.at(L::Z0, k) = G.at(L::PQ, k) = p;
                            G.at(L::Z0, M + k) = G.at(L::PQ, M + k) = q;
                        }
                        t = ep.t[e];
                        h = fmin(fmax(ep.h[e], 0.125 * (1.0 - t)), C.hmax);
                        h = fmax(h, C.hmin * 4.0);
                        ph = 0;
                    } else {
                        const int64_t path = ep.path[e];
                        const cx<double> ig = crecip(gam);
#pragma unroll 1
                        for (int k = g; k < M; k += 4) {   // dz/dt at t = 0: -P_i(z) / (2 gamma z_i)
                            double u = J[k * (M + 1) + M], v = 0.0;
#pragma unroll 1
                            for (int l = 0; l < M; l++) {
                                const double c = J[k * (M + 1) + l];
                                u += ((path >> l) & 1) ? -c : c;
                                v += ((path >> (M + l)) & 1) ? -c : c;
                            }
                            const double x = ((path >> k) & 1) ? -1.0 : 1.0;
                            const double y = ((path >> (M + k)) & 1) ? -1.0 : 1.0;
                            cx<double> rf, rg;
                            minus_ht_rows<double>(cx<double>{x, 0.0}, cx<double>{y, 0.0}, cx<double>{u, 0.0},
                                                  cx<double>{v, 0.0}, gam, rf, rg);
                            const cx<double> dx = cscale(0.5 * x, cmul(ig, rf)), dy = cscale(0.5 * y, cmul(ig, rg));
                            G.at(L::Z0, k) = cx<double>{x, y};   // p = x + i y, q = x - i y
                            G.at(L::Z0, M + k) = cx<double>{x, -y};
                            G.at(L::K1, k) = cadd(dx, cmul_i(dy));
                            G.at(L::K1, M + k) = csub(dx, cmul_i(dy));
                        }
                        t = 0.0;
                        h = C.h0;
                        start = true;
                    }
                }
            }
        }
        if (__all_sync(0xffffffffu, e < 0)) break;

        // ---- a new attempt: its first stage's point z0 + h/2 k1
        const bool act = e >= 0;
        if (start && far && h > KAPPA_FAR * (1.0 - t)) h = KAPPA_FAR * (1.0 - t);
        double hh = h, t1 = t + h;
        if (t1 >= C.t_end) {
            t1 = C.t_end;
            hh = C.t_end - t;
        }
        if (start) {
#pragma unroll 1
            for (int k = g; k < M; k += 4) {
                G.at(L::PQ, k) = cadd(G.at(L::Z0, k), cscale(0.5 * hh, G.at(L::K1, k)));
                G.at(L::PQ, M + k) = cadd(G.at(L::Z0, M + k), cscale(0.5 * hh, G.at(L::K1, M + k)));
            }
            ph = 1;
            bad = start = false;
        }

        // ---- which solve runs now, and for whom
        const bool wants_c = act && (ph == 0 || ph >= 4);
        const unsigned mc = __ballot_sync(0xffffffffu, wants_c);
        const unsigned mp = __ballot_sync(0xffffffffu, act && !wants_c);
        const bool corr = mc != 0 && 2 * __popc(mc) >= __popc(mp);
        if (!(act && wants_c == corr)) continue;
        G.m = corr ? mc : mp;
        int verdict = STEP_GO_ON, status = NPHC_PATH_RUNNING;
        double zi = 0.0;
        G.sync();
        const double te = ph == 0 ? t : ph < 3 ? t + 0.5 * hh : t1;
        const bool oks = g64_solve<M>(G, te, 1.0 - te, gam, corr);
        solves++;
        if (!corr) {
            // ---- RK4: the next stage's point, or the predicted one
            bad = bad || !oks;
            const double c = ph == 1 ? 0.5 * hh : ph == 2 ? hh : hh / 6.0;
            double zz = 0.0;
#pragma unroll 1
            for (int j = g; j < M; j += 4)
#pragma unroll 1
                for (int k = j; k < 2 * M; k += M) {   // p_j, q_j
                    const cx<double> w = G.at(L::W, k);
                    const cx<double> sum = cadd(G.at(ph == 1 ? L::K1 : L::AC, k), cscale(ph == 3 ? 1.0 : 2.0, w));
                    G.at(L::AC, k) = sum;
                    const cx<double> z = cadd(G.at(L::Z0, k), cscale(c, ph == 3 ? sum : w));
                    G.at(L::PQ, k) = z;
                    zz += cabs2(z);
                }
            zpn = sqrt(0.5 * G.sum(zz));   // ||(x, y)||_2 of the predicted point
            if (++ph == 4 && bad) verdict = STEP_REJECT;
        } else {
            // ---- corrector iteration (phase 0: a resumed point pulled onto the FP64 path)
            newton++;
            double dd = 0.0, zz = 0.0;
#pragma unroll 1
            for (int k = g; k < M; k += 4) {
                const cx<double> dp = G.at(L::W, k), dq = G.at(L::W, M + k);
                const cx<double> p = cadd(G.at(L::PQ, k), dp), q = cadd(G.at(L::PQ, M + k), dq);
                dd += cabs2(dp) + cabs2(dq);
                zz += cabs2(p) + cabs2(q);
                zi = fmax(zi, fmax(cabs2(cadd(p, q)), cabs2(csub(p, q))));
                G.at(L::PQ, k) = p;
                G.at(L::PQ, M + k) = q;
            }
            const double dn = sqrt(0.5 * G.sum(dd));
            zz = G.sum(zz);
            zi = 0.5 * sqrt(G.most(zi));   // ||(x, y)||_inf
            if (ph == 0) {
                verdict = STEP_ANCHORED;
                if (!oks) status = NPHC_PATH_NONFINITE;
            } else if (!oks || !isfinite(dn) || (ph == 4 && dn > C.trust * (1.0 + zpn))) {
                verdict = STEP_REJECT;
            } else if (dn <= C.eps * (1.0 + sqrt(0.5 * zz))) {
                verdict = STEP_ACCEPT;
            } else if (++ph >= 4 + C.max_newton) {
                verdict = STEP_REJECT;
            }
            if (verdict == STEP_ACCEPT || verdict == STEP_ANCHORED) {
#pragma unroll 1
                for (int k = g; k < M; k += 4) {
                    G.at(L::Z0, k) = G.at(L::PQ, k);
                    G.at(L::Z0, M + k) = G.at(L::PQ, M + k);
                    G.at(L::K1, k) = G.at(L::AC, k);
                    G.at(L::K1, M + k) = G.at(L::AC, M + k);
                }
            }
        }
        // ---- the step attempt is over
        if (verdict != STEP_GO_ON) {
            if (verdict == STEP_ACCEPT) {
                attempts++;
                t = t1;
                far = 1.0 - t < CRAWL_ZONE && zi > FAR_NORM && zi > FAR_GROWTH * zlast;
                zlast = zi;
                steps++;
                if (++run >= C.grow_after) {
                    run = 0;
                    h = fmin(2.0 * h, C.hmax);
                }
                if (zi > C.rdiv) status = NPHC_PATH_DIVERGED;
                else if (t >= C.t_end) status = NPHC_PATH_REACHED;
            } else if (verdict == STEP_REJECT) {
                attempts++;
                run = 0;
                h *= 0.5;
                if (h < C.hmin) status = NPHC_PATH_MIN_STEP;
            }
            if (status == NPHC_PATH_RUNNING && attempts >= C.max_steps) status = NPHC_PATH_STEP_BUDGET;
            start = status == NPHC_PATH_RUNNING;
            if (!start) {
#pragma unroll 1
                for (int k = g; k < M; k += 4) {   // x = (p + q) / 2, y = -i (p - q) / 2
                    const cx<double> p = G.at(L::Z0, k), q = G.at(L::Z0, M + k);
                    ep.z_re[k * cnt + e] = 0.5 * (p.re + q.re);
                    ep.z_im[k * cnt + e] = 0.5 * (p.im + q.im);
                    ep.z_re[(M + k) * cnt + e] = 0.5 * (p.im - q.im);
                    ep.z_im[(M + k) * cnt + e] = -0.5 * (p.re - q.re);
                }
                if (g == 0) {
                    ep.t[e] = t;
                    ep.h[e] = h;
                    ep.status[e] = status;
                    ep.steps[e] = steps;
                    ep.solves[e] = solves;
                    ep.newton[e] = newton;
                }
                e = -1;
            }
        }
    }
}
