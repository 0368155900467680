// xy_track_warp32.cuh -- the FP32 tracker of the XY ring with one path per warp, for the far endpoints
// of a pass (xy_track.cuh says which and why): tens or hundreds of paths out of 10^4 to 10^6.
//
// Every path's arithmetic is that of the per-thread tracker (xy_track.cuh, xy_solve.cuh), operation by
// operation and in its order, so that its endpoint is the same bit for bit; only what is
// independent is shared out over the lanes: sites, matrix entries, rows, the two right-hand
// sides and the p and q sides of a site (half-warps).  Sums and norms keep their order, and the
// expressions are written as they are there, so that the compiler fuses the same products and
// sums (the tests compare the two kernels' endpoints bit for bit).
//
// A pass is followed by one path's chain of dependent solves, so the time is that chain's latency:
// per thread a solve is ten thousand instructions on one lane (193 paths of N = 10 14.1 ms, 144 of N = 13
// 16.9), here some two thousand (2.9 and 3.5 ms).  Very long lists are left to the per-thread kernel, which needs
// fewer instructions per path (kFarPerScheduler in nphc_api.cu).
#pragma once

#include "xy_track.cuh"

template <int M>
struct Warp32Layout {   // shared memory per warp, complex floats
    static constexpr int NV = 2 * M;
    static constexpr int A = 0;                 // [S | b0 | b1], column-major
    static constexpr int ZC = A + M * (M + 2);  // evaluation point (p, q)
    static constexpr int W1 = ZC + NV;          // residual, solution of the first right-hand side
    static constexpr int Z0 = W1 + NV;          // accepted point
    static constexpr int K1 = Z0 + NV;          // dz/dt there
    static constexpr int AC = K1 + NV;          // RK4 sum; in a corrector solve dz/dt
    static constexpr int CK = AC + NV;          // hand-off checkpoint
    static constexpr int CB = CK + NV;          // of column j of S: J_kj (q_k i cb_j + p_k i ca_j)
    static constexpr int CA = CB + M;
    static constexpr int X0 = CA + M;           // sums of the right-hand sides
    static constexpr int Y0 = X0 + M;
    static constexpr int X1 = Y0 + M;
    static constexpr int Y1 = X1 + M;
    static constexpr int TOTAL = Y1 + M;
};

template <int M>
struct Warp32 {
    using C = cx<float>;
    using E = ext<float>;
    using L = Warp32Layout<M>;
    C *s;
    const float *J;   // J[k * NPHC_JSTRIDE + l], in shared memory
    int lane;
    __device__ __forceinline__ C &at(int off, int i) const { return s[off + i]; }
    __device__ __forceinline__ C &A(int i, int c) const { return s[L::A + c * M + i]; }
    static __device__ __forceinline__ C other(C v) {   // the other half's
        return C{__shfl_xor_sync(0xffffffffu, v.re, 16), __shfl_xor_sync(0xffffffffu, v.im, 16)};
    }
    static __device__ __forceinline__ E other(E v) {
        return E{__shfl_xor_sync(0xffffffffu, v.hi, 16), __shfl_xor_sync(0xffffffffu, v.lo, 16)};
    }

    // -H(z, t) at ZC into W1 (xy_residual_comp): lane k the f row of site k, lane 16 + k its g row
    __device__ void residual(float t, float omt, C gam) const {
        using F = EFT<float>;
        const int k = (lane & 15) < M ? lane & 15 : 0;
        const bool hi = lane >= 16;
        const C gomt = {F::mul(omt, gam.re), F::mul(omt, gam.im)};
        const float hs = 0.5f * t;
        const C p = at(L::ZC, k), q = at(L::ZC, M + k);
        const float *Jk = J + k * NPHC_JSTRIDE;
        const E zero = {0.0f, 0.0f};
        E ur = {Jk[M], 0.0f}, ui = zero;   // U_p on the lower half, U_q on the upper
        const int off = hi ? L::ZC + M : L::ZC;
#pragma unroll 4
        for (int l = 0; l < M; l++) {   // J_kk = 0 adds exact zeros
            const C v = at(off, l);
            ext_acc(ur, Jk[l], v.re);
            ext_acc(ui, Jk[l], v.im);
        }
        const E vr = other(ur), vi = other(ui);
        const E upr = hi ? vr : ur, upi = hi ? vi : ui, uqr = hi ? ur : vr, uqi = hi ? ui : vi;
        E dr = zero, di = zero;   // D = q U_p - p U_q, f = i D / 2
        ext_acc_ext(dr, q.re, upr);
        ext_acc_ext(dr, -q.im, upi);
        ext_acc_ext(dr, -p.re, uqr);
        ext_acc_ext(dr, p.im, uqi);
        ext_acc_ext(di, q.re, upi);
        ext_acc_ext(di, q.im, upr);
        ext_acc_ext(di, -p.re, uqi);
        ext_acc_ext(di, -p.im, uqr);
        // X = x^2 - 1 (lower half) or Y = y^2 - 1 (upper), and G = p q - 1
        const float c4 = hi ? -0.25f : 0.25f, c2 = hi ? -0.5f : 0.5f;
        E xr = {-1.0f, 0.0f}, xi = zero, gr = {-1.0f, 0.0f}, gi = zero;
        ext_acc(xr, c4 * p.re, p.re);
        ext_acc(xr, -c4 * p.im, p.im);
        ext_acc(xr, 0.5f * p.re, q.re);
        ext_acc(xr, -0.5f * p.im, q.im);
        ext_acc(xr, c4 * q.re, q.re);
        ext_acc(xr, -c4 * q.im, q.im);
        ext_acc(xi, c2 * p.re, p.im);
        ext_acc(xi, 0.5f * p.re, q.im);
        ext_acc(xi, 0.5f * p.im, q.re);
        ext_acc(xi, c2 * q.re, q.im);
        ext_acc(gr, p.re, q.re);
        ext_acc(gr, -p.im, q.im);
        ext_acc(gi, p.re, q.im);
        ext_acc(gi, p.im, q.re);
        // H_f = gomt X + t f, H_g = gomt Y + t G
        E hr = zero, hm = zero;
        ext_acc_ext(hr, gomt.re, xr);
        ext_acc_ext(hr, -gomt.im, xi);
        ext_acc_ext(hr, hi ? t : -hs, hi ? gr : di);
        ext_acc_ext(hm, gomt.re, xi);
        ext_acc_ext(hm, gomt.im, xr);
        ext_acc_ext(hm, hi ? t : hs, hi ? gi : dr);
        if ((lane & 15) < M) at(L::W1, hi ? M + k : k) = C{-ext_val(hr), -ext_val(hm)};
        __syncwarp();
    }

    // H_z(ZC, t) d = r (xy_solve): r = -H_t into W1, or with two the residual in W1 into W1 and
    // -H_t into AC.  False when the system is singular or the result is not finite.
    __device__ bool solve(float t, float omt, C gam, bool two, float &kest) const {
        const int row = lane & 15, r = lane >> 4, j = row < M ? row : 0;
        const bool on = row < M && (r == 0 || two);
        const C gomt = cscale(omt, gam);
        const float hs = 0.5f * t;
        // ---- the sites, on both halves
        const C p = at(L::ZC, j), q = at(L::ZC, M + j);
        C U = {J[j * NPHC_JSTRIDE + M], 0.0f};
        const int off = r ? L::ZC + M : L::ZC;
#pragma unroll 4
        for (int l = 0; l < M; l++) {
            const float Jl = J[j * NPHC_JSTRIDE + l];
            const C v = at(off, l);
            U.re += Jl * v.re;
            U.im += Jl * v.im;
        }
        const C V = other(U), Up = r ? V : U, Uq = r ? U : V;
        C htf, htg, ah, bh;
        lc_minus_ht_rows<float>(p, q, Up, Uq, gam, htf, htg);
        const C rf0 = two ? at(L::W1, j) : htf, rg0 = two ? at(L::W1, M + j) : htg;
        float iv, sp, sq;
        g_frame_lc<float>(p, q, t, gomt, ah, bh, iv, sp, sq);
        const C gpq = cmul(gomt, cadd(p, q));
        const C Ajj = cscale(0.5f * sp, csub(gpq, cmul_i(cscale(t, Uq))));
        const C Bjj = cscale(0.5f * sq, cadd(gpq, cmul_i(cscale(t, Up))));
        const C rf = r ? htf : rf0, rg = r ? htg : rg0;   // this half's right-hand side
        const C qr = cscale(iv, rg), px = cmulc(ah, qr), py = cmulc(bh, qr);
        __syncwarp();   // W1 has been read
        if (on) {
            A(j, M + r) = csub(rf, cadd(cmul(Ajj, px), cmul(Bjj, py)));
            at(r ? L::X1 : L::X0, j) = cscale(sp, px);
            at(r ? L::Y1 : L::Y0, j) = cscale(sq, py);
            if (r == 0) {
                at(L::CB, j) = cscale(hs * sp, bh);
                at(L::CA, j) = cscale(hs * sq, ah);
                A(j, j) = csub(cmul(Ajj, bh), cmul(Bjj, ah));
            }
        }
        __syncwarp();
        // ---- off-diagonal entries (the factor i is applied here: the compiler then fuses the products as
        // it does in xy_solve); right-hand sides
#pragma unroll 1
        for (int e = lane; e < M * M; e += 32) {
            const int c = e / M, k = e - c * M;
            if (k != c)
                A(k, c) = cscale(J[k * NPHC_JSTRIDE + c],
                                 cadd(cmul(at(L::ZC, M + k), cmul_i(at(L::CB, c))), cmul(at(L::ZC, k), cmul_i(at(L::CA, c)))));
        }
        if (on) {
            C sx = {0.0f, 0.0f}, sy = sx;
#pragma unroll 4
            for (int c = 0; c < M; c++) {
                const float Jkc = J[j * NPHC_JSTRIDE + c];
                const C x = at(r ? L::X1 : L::X0, c), y = at(r ? L::Y1 : L::Y0, c);
                sx = C{fma(Jkc, x.re, sx.re), fma(Jkc, x.im, sx.im)};
                sy = C{fma(Jkc, y.re, sy.re), fma(Jkc, y.im, sy.im)};
            }
            A(j, M + r) = csub(A(j, M + r), cmul_i(cscale(hs, csub(cmul(q, sx), cmul(p, sy)))));
        }
        __syncwarp();
        // ---- LU with partial pivoting (aug_lu_solve): the first row of the largest |a|^2
        const int ncol = two ? M + 2 : M + 1;
        bool ok = true;
        float umax = 0.0f, umin = 0.0f;
#pragma unroll 1
        for (int k = 0; k < M; k++) {
            const bool in = lane >= k && lane < M;
            const unsigned key = in ? __float_as_uint(cabs2(A(in ? lane : 0, k))) : 0u;
            const unsigned best = __reduce_max_sync(0xffffffffu, key);
            const int pr = __ffs(__ballot_sync(0xffffffffu, in && key == best)) - 1;
            const float b = __uint_as_float(best);
            ok = ok && b > 0.0f;
            const float um = sqrt_r(b);
            umax = fmax(umax, um);
            umin = k == 0 ? um : fmin(umin, um);
            const C ip = crecip(A(pr, k));
            C l = {0.0f, 0.0f};
            if (lane > k && lane < M) l = cmul(lane == pr ? A(k, k) : A(lane, k), ip);
            if (pr != k && lane > k && lane < ncol) {
                const C a = A(k, lane);
                A(k, lane) = A(pr, lane);
                A(pr, lane) = a;
            }
            __syncwarp();
            if (lane > k && lane < M) A(lane, k) = l;
            if (lane == k) A(k, k) = ip;
            __syncwarp();
            const int nr = M - 1 - k, n = nr * (ncol - 1 - k);
#pragma unroll 1
            for (int e = lane; e < n; e += 32) {
                const int c = k + 1 + e / nr, i = k + 1 + (e - (e / nr) * nr);
                const C x = A(i, c), m = A(i, k), ap = A(k, c);
                A(i, c) = C{fma(m.im, ap.im, fma(-m.re, ap.re, x.re)), fma(-m.im, ap.re, fma(-m.re, ap.im, x.im))};
            }
            __syncwarp();
        }
        kest = umin > 0.0f ? umax / umin : INFINITY;
        // ---- back substitution: right-hand side r, row `row`
        C cur = {0.0f, 0.0f};
        if (on) cur = A(row, M + r);
#pragma unroll 1
        for (int k = M - 1; k >= 0; k--) {
            const int src = (lane & 16) | k;
            const C bk = {__shfl_sync(0xffffffffu, cur.re, src), __shfl_sync(0xffffffffu, cur.im, src)};
            const C sk = cmul(bk, A(k, k));
            if (row == k) cur = sk;
            else if (row < k) cur = csub(cur, cmul(A(row, k), sk));
        }
        // ---- back to (dp, dq)
        float chk = 0.0f;
        if (on) {
            const C dp = cscale(sp, cadd(cmulc(ah, qr), cmul(bh, cur)));
            const C dq = cscale(sq, csub(cmulc(bh, qr), cmul(ah, cur)));
            const int o = r ? L::AC : L::W1;
            at(o, j) = dp;
            at(o, M + j) = dq;
            chk = cabs2(dp) + cabs2(dq);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) chk += __shfl_xor_sync(0xffffffffu, chk, o);
        __syncwarp();
        return ok && isfinite(chk);
    }

    __device__ __forceinline__ float norm2(int off) const {   // of the state: sum of |v_i|^2 in order
        float v = 0.0f;
#pragma unroll 4
        for (int i = 0; i < 2 * M; i++) v += cabs2(at(off, i));
        return v;
    }
    __device__ __forceinline__ float norminf() const {   // ||(x, y)||_inf at ZC
        float v = 0.0f;
        if (lane < M) {
            const C p = at(L::ZC, lane), q = at(L::ZC, M + lane);
            v = fmax(cabs2(cadd(p, q)), cabs2(csub(p, q)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
        return 0.5f * sqrt_r(v);
    }

    // the start point of path n and dz/dt there
    __device__ void start(int64_t n, C gam) const {
        if (lane < M) {
            const int k = lane;
            const float *Jk = J + k * NPHC_JSTRIDE;
            C u = {Jk[M], 0.0f}, w = {0.0f, 0.0f}, rf, rg;
#pragma unroll 4
            for (int l = 0; l < M; l++) {
                const float Jl = Jk[l];
                u.re += Jl * (((n >> l) & 1) ? -1.0f : 1.0f);
                w.re += Jl * (((n >> (M + l)) & 1) ? -1.0f : 1.0f);
            }
            const C x = {((n >> k) & 1) ? -1.0f : 1.0f, 0.0f}, y = {((n >> (M + k)) & 1) ? -1.0f : 1.0f, 0.0f};
            minus_ht_rows<float>(x, y, u, w, gam, rf, rg);
            const C ig = crecip(gam);
            const C dx = cscale(0.5f * x.re, cmul(ig, rf)), dy = cscale(0.5f * y.re, cmul(ig, rg));
            at(L::Z0, k) = C{x.re, y.re};
            at(L::Z0, M + k) = C{x.re, -y.re};
            at(L::K1, k) = cadd(dx, cmul_i(dy));
            at(L::K1, M + k) = csub(dx, cmul_i(dy));
        }
        __syncwarp();
    }
    __device__ void store(int off, const EPView &ep, int64_t e) const {
        const int64_t cnt = ep.count;
        if (lane < M) {
            const int k = lane;
            const C p = at(off, k), q = at(off, M + k);
            const double pr = p.re, pi = p.im, qr = q.re, qi = q.im;
            ep.z_re[k * cnt + e] = 0.5 * (pr + qr);
            ep.z_im[k * cnt + e] = 0.5 * (pi + qi);
            ep.z_re[(M + k) * cnt + e] = 0.5 * (pi - qi);
            ep.z_im[(M + k) * cnt + e] = -0.5 * (pr - qr);
        }
        __syncwarp();
    }
};

// Tracks the listed paths from t = 0 (the control flow is track_body's in FP32, uniform over the
// warp).  total: the list's length; src.take(q, inst, e) gives its entry q.
template <int M, int WARPS, class Src>
__device__ __forceinline__ void warp32_track_body(const Src &src, const XYCtl &C, int64_t total,
                                                  unsigned long long *queue) {
    using L = Warp32Layout<M>;
    constexpr int NV = 2 * M;
    __shared__ cx<float> work[WARPS * L::TOTAL];
    __shared__ float Js[WARPS * M * NPHC_JSTRIDE];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, i = lane;   // i: vector component
    float *const J = Js + wid * (M * NPHC_JSTRIDE);
    const Warp32<M> P{work + wid * L::TOTAL, J, lane};
    const float eps = (float)C.eps, trust = (float)C.trust, scale = 0.70710678118654752440f;
    int inst = 0, have = -1;   // the instance whose couplings are in J
    cx<float> gam = {1.0f, 0.0f};
    for (;;) {
        unsigned long long take = 0;
        if (lane == 0) take = atomicAdd(queue, 1ull);
        take = __shfl_sync(0xffffffffu, take, 0);
        if ((int64_t)take >= total) break;
        int64_t e;
        src.take((int64_t)take, inst, e);
        if (e < 0) continue;   // rejected by the debug build's check
        if (inst != have) {
            const XYSys &S = src.sys(inst);
            for (int k = lane; k < M * NPHC_JSTRIDE; k += 32) J[k] = S.Jf[k];
            gam = cx<float>{(float)S.gre, (float)S.gim};
            have = inst;
            __syncwarp();
        }
        const EPView &ep = src.eps(inst);
        P.start(ep.path[e], gam);
        double t = 0.0, h = C.h0, hacc = h, tck = 0.0, hck = 0.0, tmark = 1.0, zlast = 0.0;
        bool have_ck = false, far = false;
        int status = NPHC_PATH_RUNNING, run = 0, rejects = 0, attempts = 0, clean = 0, since = 0;
        int steps = C.accumulate ? ep.steps[e] : 0, solves = C.accumulate ? ep.solves[e] : 0;
        int newton = C.accumulate ? ep.newton[e] : 0;
        while (status == NPHC_PATH_RUNNING) {
            if (far && h > KAPPA_FAR * (1.0 - t)) h = KAPPA_FAR * (1.0 - t);
            double hh = h, t1 = t + h;
            if (t1 >= C.t_end) {
                t1 = C.t_end;
                hh = C.t_end - t;
            }
            const float hr = (float)hh;
            bool conv = false, bad = false;
            float zpn = 0.0f, kstep = 0.0f;
#pragma unroll 1
            for (int ph = 1; ph < 4 + C.max_newton; ph++) {
                const bool corr = ph >= 4;
                if (corr && (conv || bad)) break;
                const double te = ph >= 3 ? t1 : t + 0.5 * hh;
                if (!corr) {   // z0 + h/2 k1, z0 + h/2 k2, z0 + h k3
                    const float c = ph == 3 ? hr : 0.5f * hr;
                    if (i < NV)
                        P.at(L::ZC, i) = cadd(P.at(L::Z0, i), cscale(c, ph == 1 ? P.at(L::K1, i) : P.at(L::W1, i)));
                    __syncwarp();
                }
                const float tr = (float)te, omt = (float)(1.0 - te);
                if (corr) P.residual(tr, omt, gam);
                float kest;
                const bool oks = P.solve(tr, omt, gam, corr, kest);
                solves++;
                kstep = fmax(kstep, kest);
                if (!corr) {
                    bad = bad || !oks;
                    if (i < NV) {
                        const cx<float> w = P.at(L::W1, i);
                        if (ph == 1) P.at(L::AC, i) = cadd(P.at(L::K1, i), cscale(2.0f, w));
                        else if (ph == 2) P.at(L::AC, i) = cadd(P.at(L::AC, i), cscale(2.0f, w));
                        else P.at(L::ZC, i) = cadd(P.at(L::Z0, i), cscale(hr / 6.0f, cadd(P.at(L::AC, i), w)));
                    }
                    __syncwarp();
                    if (ph == 3) zpn = sqrt_r(P.norm2(L::ZC)) * scale;
                } else {
                    newton++;
                    const float dn = sqrt_r(P.norm2(L::W1)) * scale;
                    if (!oks || !isfinite(dn) || (ph == 4 && dn > trust * (1.0f + zpn))) {
                        bad = true;
                    } else {
                        if (i < NV) P.at(L::ZC, i) = cadd(P.at(L::ZC, i), P.at(L::W1, i));
                        __syncwarp();
                        if (dn <= eps * (1.0f + sqrt_r(P.norm2(L::ZC)) * scale)) conv = true;
                    }
                    __syncwarp();
                }
            }
            if (conv && C.kappa > 0.0 && !((double)kstep <= C.kappa)) {
                status = NPHC_PATH_HANDOFF_COND;
                break;
            }
            attempts++;
            if (conv) {
                if (i < NV) {
                    P.at(L::Z0, i) = P.at(L::ZC, i);
                    P.at(L::K1, i) = P.at(L::AC, i);
                }
                const double zi = (double)P.norminf();
                __syncwarp();
                clean = rejects == 0 ? clean + 1 : 1;
                t = t1;
                const double left = 1.0 - t;
                far = left < CRAWL_ZONE && zi > FAR_NORM && zi > FAR_GROWTH * zlast;
                zlast = zi;
                steps++;
                rejects = 0;
                hacc = h;
                if (++run >= C.grow_after) {
                    run = 0;
                    h = fmin(2.0 * h, C.hmax);
                }
                if (zi > C.rdiv)
                    status = left < NEAR_END && zi <= C.rdiv * (1.0 + RDIV_BAND) ? NPHC_PATH_HANDOFF : NPHC_PATH_DIVERGED;
                else if (t >= C.t_end)
                    status = NPHC_PATH_REACHED;
                if ((clean >= 2 || !have_ck) && status == NPHC_PATH_RUNNING && left < CRAWL_ZONE) {
                    if (i < NV) P.at(L::CK, i) = P.at(L::Z0, i);
                    tck = t;
                    hck = hacc;
                    have_ck = true;
                }
                if (status == NPHC_PATH_RUNNING && C.crawl_steps > 0 && left < CRAWL_ZONE) {
                    if (++since >= C.crawl_steps) {
                        if (left > 0.5 * tmark) status = NPHC_PATH_HANDOFF;
                        tmark = left;
                        since = 0;
                    }
                } else {
                    tmark = left;
                    since = 0;
                }
            } else {
                run = 0;
                rejects++;
                h *= 0.5;
                if (h < C.hmin || rejects >= 10) status = NPHC_PATH_HANDOFF;
            }
            if (status == NPHC_PATH_RUNNING && attempts >= C.max_steps) status = NPHC_PATH_HANDOFF;
        }
        __syncwarp();
        const bool handed = status == NPHC_PATH_HANDOFF || status == NPHC_PATH_HANDOFF_COND;
        const bool from_ck = handed && have_ck;
        P.store(from_ck ? L::CK : L::Z0, ep, e);
        if (lane == 0) {
            ep.t[e] = from_ck ? tck : t;
            ep.h[e] = from_ck ? hck : (handed ? hacc : h);
            ep.status[e] = status;
            ep.steps[e] = steps;
            ep.solves[e] = solves;
            ep.newton[e] = newton;
        }
        __syncwarp();
    }
}

// One ring's list, when it is shorter than max_paths (longer ones are the per-thread kernel's).
template <int M, int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
    xy_track_warp32_kernel(const __grid_constant__ XYSys S, const __grid_constant__ XYCtl C,
                           const __grid_constant__ EPView ep, const WorkList wl, int64_t max_paths) {
    const int64_t total = worklist_size(wl, ep.count);
    if (total < max_paths) warp32_track_body<M, WARPS>(SingleSrc<XYSys>{S, ep, wl}, C, total, wl.queue);
}

// A batch group's: list[q] is an item of the group (BatchSrc).
template <int M, int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
    xy_track_warp32_batch_kernel(const XYSys *__restrict__ sys, const EPView *__restrict__ eps,
                                 const int64_t *__restrict__ off, int n, const __grid_constant__ XYCtl C,
                                 const int32_t *list, const int32_t *count, unsigned long long *queue) {
    struct Src : BatchSrc<XYSys> {
        const int32_t *list;
        __device__ __forceinline__ void take(int64_t q, int &g, int64_t &e) const {
            BatchSrc<XYSys>::take(list[q], g, e);
        }
    };
    Src src;
    src.S = sys;
    src.ep = eps;
    src.off = off;
    src.n = n;
    src.list = list;
    warp32_track_body<M, WARPS>(src, C, *count, queue);
}

// The items of a batch group that reached a far endpoint (launch_far_list for a batch).
template <int M>
__global__ void far_list_batch_kernel(const XYSys *__restrict__ sys, const EPView *__restrict__ eps,
                                      const int64_t *__restrict__ off, int n, int32_t *list, int32_t *count) {
    const BatchSrc<XYSys> src = {sys, eps, off, n};
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= src.total()) return;
    int g;
    int64_t e;
    src.take(i, g, e);
    if (e < 0 || eps[g].status[e] != NPHC_PATH_REACHED) return;
    const EPView &ep = eps[g];
    int ez = -2000;
    for (int k = 0; k < 2 * M; k++) ez = max(ez, max(gexp(ep.z_re[k * ep.count + e]), gexp(ep.z_im[k * ep.count + e])));
    if (ez >= sys[g].far_exp) list[atomicAdd(count, 1)] = (int32_t)i;   // every item once: at most total
}
