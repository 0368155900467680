// xy_track_warp.cuh -- FP64 path tracking of the XY ring with one path per warp, for
// short lists (paths handed off by the FP32 pass, re-tracks).
//
// GB300 runs FP64 at 1/64 of the FP32 rate, and its FP64 pipe takes a warp instruction
// at the same cost whatever the number of active lanes: a solve costs 67 cycles of an SM
// sub-partition per FP64 instruction on the longest chain that any lane runs.  So
// the 32 lanes share one path, and every stage is laid out to keep each lane's own FP64
// chain short rather than to save lanes:
//   * per-site quantities (couplings sums, frames, the diagonal's terms): the p side of
//     site j on lane j, the q side on lane 16 + j, both halves on the same instructions;
//     the frames' scales are powers of two from the exponents (no square root);
//   * the off-diagonal Schur entries: one entry per lane, strided over the M x M matrix;
//   * the right-hand sides: sums of J times per-site vectors, right-hand side r on the
//     lanes 16 r + k (row k);
//   * the factorisation: LU with partial pivoting (one reciprocal per column and no
//     square root; the pivot search compares the bit patterns of |re| + |im| as integers
//     and costs one FP64 add), the rank-one update strided over the trailing block;
//   * the back substitution in registers (right-hand side r on lanes 16 r + row);
//   * the compensated residual of row pair k on lanes k and 16 + k, as sums on grids (gsum in
//     nphc_internal.cuh: four instructions per term where two-sums took ten).
// The 9,493 hand-offs of an N = 10 ring: 20.0 ms with two-sums, one lane per site and square
// roots, 13.5 now; 1,400 of N = 13 6.4 -> 5.0.
// The step logic (RK4 predictor, Newton corrector, step control, divergence radius,
// budget) is the per-thread FP64 tracker's, as are the state in light-cone coordinates,
// the equations and the scaled light-cone frames of the Schur reduction (xy_solve.cuh):
// the same algorithm with a different linear solver, so the endpoints agree to the
// tracking tolerance.  The Cauchy endgame (cauchy_warp.cuh) calls the same solve and
// residual on points in (x, y).
//
// Storage: everything of a path in per-warp shared memory (complex doubles): the
// augmented Schur matrix [S | b0 | b1] (column-major, M x (M + 2)), the five step
// vectors Z0, K1, AC, ZC, W1 (2M each) and eight per-site arrays.
#pragma once

#include "xy_track.cuh"

template <int M>
struct WarpLayout {
    static constexpr int NV = 2 * M;
    static constexpr int A = 0;
    static constexpr int Z0 = A + M * (M + 2);
    static constexpr int K1 = Z0 + NV;
    static constexpr int AC = K1 + NV;
    static constexpr int ZC = AC + NV;
    static constexpr int W1 = ZC + NV;
    static constexpr int SB = W1 + NV;    // sp b^_j of the scaled frame: Schur column j is J_kj (IQ_k SB_j + IP_k SA_j)
    static constexpr int SA = SB + M;     // sq a^_j
    static constexpr int X0 = SA + M;     // sp_j conj(a^_j) q0_j, sq_j conj(b^_j) q0_j (right-hand side 0),
    static constexpr int Y0 = X0 + M;
    static constexpr int X1 = Y0 + M;     // the same with q1_j (right-hand side 1)
    static constexpr int Y1 = X1 + M;
    static constexpr int IP = Y1 + M;     // (i t / 2) p_j, (i t / 2) q_j
    static constexpr int IQ = IP + M;
    static constexpr int TOTAL = IQ + M;
};

template <int M>
constexpr size_t warp_track_smem_per_warp() {
    return sizeof(cx<double>) * (size_t)WarpLayout<M>::TOTAL;
}

// Warp reductions whose result is lane 0's, broadcast: the butterfly leaves each lane a
// sum in its own association order, and the step logic branches on these values, so
// every lane must see the same bits.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return __shfl_sync(0xffffffffu, v, 0);
}

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return __shfl_sync(0xffffffffu, v, 0);
}

// c - a b with four fused multiply-adds
__device__ __forceinline__ cx<double> cfnms(cx<double> c, cx<double> a, cx<double> b) {
    return cx<double>{fma(a.im, b.im, fma(-a.re, b.re, c.re)), fma(-a.im, b.re, fma(-a.re, b.im, c.im))};
}

// c + a b
__device__ __forceinline__ cx<double> cfma64(cx<double> a, cx<double> b, cx<double> c) {
    return cx<double>{fma(-a.im, b.im, fma(a.re, b.re, c.re)), fma(a.im, b.re, fma(a.re, b.im, c.im))};
}

// The largest power of two <= max(1, |re|, |im|), from the exponents alone.
__device__ __forceinline__ double pow2_scale(cx<double> a) {
    const int hi = max(__double2hiint(a.re) & 0x7fffffff, __double2hiint(a.im) & 0x7fffffff) & 0x7ff00000;
    return __hiloint2double(min(max(hi, 0x3ff00000), 0x7fd00000), 0);
}

__device__ __forceinline__ cx<double> shfl_xor16(cx<double> v) {
    return cx<double>{__shfl_xor_sync(0xffffffffu, v.re, 16), __shfl_xor_sync(0xffffffffu, v.im, 16)};
}

__device__ __forceinline__ ext<double> shfl_down16(ext<double> v) {
    return ext<double>{__shfl_down_sync(0xffffffffu, v.hi, 16), __shfl_down_sync(0xffffffffu, v.lo, 16)};
}

__device__ __forceinline__ ext<double> shfl_up16(ext<double> v) {
    return ext<double>{__shfl_up_sync(0xffffffffu, v.hi, 16), __shfl_up_sync(0xffffffffu, v.lo, 16)};
}

template <int M>
struct WarpPath {
    cx<double> *s;   // this warp's shared memory
    int lane;
    __device__ __forceinline__ cx<double> &at(int off, int i) const { return s[off + i]; }
    __device__ __forceinline__ cx<double> &A(int i, int c) const { return s[WarpLayout<M>::A + c * M + i]; }
};

// -H(z, t) at ZC into W1 with compensated sums (on grids: gsum).  LC == false: ZC holds (x, y) (the
// Cauchy endgame), f = y u - x w; LC == true: the light-cone coordinates (p, q), f = i D / 2 with
// D = q U_p - p U_q (xy_residual_comp in xy_solve.cuh).  Row pair k: lane k sums u_k (U_p,k) and forms
// the f row, lane 16 + k sums w_k (U_q,k), hands its share of f (D) to lane k and forms the g row;
// both halves run the same instructions.
template <int M, bool LC = false>
__device__ void warp_residual(const WarpPath<M> &P, const double *__restrict__ J, double s,
                              double omt, cx<double> gam) {
    static_assert(M <= 16, "one row pair per lane pair");
    using L = WarpLayout<M>;
    using E = EFT<double>;
    const int k = P.lane & 15;
    const bool hi = P.lane >= 16, on = k < M;
    cx<double> zk = {1.0, 0.0}, wk = zk;   // (x_k, y_k) or (p_k, q_k)
    if (on) {
        zk = P.at(L::ZC, k);
        wk = P.at(L::ZC, M + k);
    }
    const int ez = max(gexp(zk.re), gexp(zk.im)), ew = max(gexp(wk.re), gexp(wk.im)), ek = max(ez, ew);
    const double *Jk = J + (on ? k : 0) * NPHC_JSTRIDE;
    int er = gexp(Jk[M]);
#pragma unroll 1
    for (int l = 0; l < M; l++) er = max(er, gexp(Jk[l]) + __shfl_sync(0xffffffffu, ek, l));
    const int ku = gsum_row(er), kd = ek + ku + 3;   // the same on both halves
    const double au = gsum_anchor(ku), ad = gsum_anchor(kd);
    const int off = hi ? L::ZC + M : L::ZC;
    gsum sr = gsum_start(au, (hi && !LC) ? 0.0 : Jk[M]), si = {au, 0.0};
#pragma unroll 1
    for (int l = 0; l < M; l++) {   // J_kk = 0 adds exact zeros
        const cx<double> v = P.at(off, l);
        gsum_acc(sr, Jk[l], v.re);
        gsum_acc(si, Jk[l], v.im);
    }
    const ext<double> ur = gsum_ext(sr, au), ui = gsum_ext(si, au);
    // (x, y): lane k y_k u_k, lane 16 + k -x_k w_k;  (p, q): lane k q_k U_p, lane 16 + k -p_k U_q
    const cx<double> c = hi ? cx<double>{-zk.re, -zk.im} : wk;
    gsum sfr = {ad, 0.0}, sfi = sfr;
    gsum_acc_ext(sfr, c.re, ur);
    gsum_acc_ext(sfr, -c.im, ui);
    gsum_acc_ext(sfi, c.re, ui);
    gsum_acc_ext(sfi, c.im, ur);
    ext<double> fr = gsum_ext(sfr, ad), fi = gsum_ext(sfi, ad);
    fr = grid_add(fr, shfl_down16(fr));
    fi = grid_add(fi, shfl_down16(fi));
    // lane k: X = x^2 - 1, lane 16 + k: Y = y^2 - 1 and G = x^2 + y^2 - 1
    // (h has a grid of its own: near infinity p q stays near 1 where p^2 or q^2 is huge)
    const int kh = max(0, (LC ? ez + ew : 2 * ek) + 2) + 2, kx = LC ? max(2 * ek + 3, kh) + 1 : kh;
    const double ah = gsum_anchor(kh);
    ext<double> ar, ai, tr, ti;   // X or Y; what t multiplies: f (or D), or G - 1
    double cr, ci;
    if (LC) {   // h = (p q - 2) / 2, B = (p^2 + q^2) / 4: X = h + B, Y = h - B, G = p q - 1 = 2 h + 1
        const cx<double> ph = cscale(0.5, zk), qh = cscale(0.5, wk);
        const double ax = gsum_anchor(kx);
        gsum shr = gsum_start(ah, -1.0), shi = {ah, 0.0}, sbr = {ax, 0.0}, sbi = sbr;
        gsum_acc(shr, ph.re, wk.re);
        gsum_acc(shr, -ph.im, wk.im);
        gsum_acc(shi, ph.re, wk.im);
        gsum_acc(shi, ph.im, wk.re);
        gsum_acc(sbr, ph.re, ph.re);
        gsum_acc(sbr, -ph.im, ph.im);
        gsum_acc(sbr, qh.re, qh.re);
        gsum_acc(sbr, -qh.im, qh.im);
        gsum_acc(sbi, ph.re, zk.im);
        gsum_acc(sbi, qh.re, wk.im);
        const ext<double> br = gsum_ext(sbr, ax), bi = gsum_ext(sbi, ax);
        if (hi) {   // -B
            sbr = gsum{__dsub_rn(ax, br.hi), -br.lo};
            sbi = gsum{__dsub_rn(ax, bi.hi), -bi.lo};
        }
        const ext<double> hr = gsum_ext(shr, ah), hm = gsum_ext(shi, ah);
        gsum_add(sbr, hr);
        gsum_add(sbi, hm);
        ar = gsum_ext(sbr, ax);
        ai = gsum_ext(sbi, ax);
        tr = hi ? hr : fi;
        ti = hi ? hm : fr;
        cr = hi ? 2.0 * s : -0.5 * s;
        ci = hi ? 2.0 * s : 0.5 * s;
    } else {
        const cx<double> v = hi ? wk : zk;
        gsum svr = gsum_start(ah, -1.0), svi = {ah, 0.0};
        gsum_acc(svr, v.re, v.re);
        gsum_acc(svr, -v.im, v.im);
        gsum_acc(svi, 2.0 * v.re, v.im);
        ar = gsum_ext(svr, ah);
        ai = gsum_ext(svi, ah);
        const ext<double> xr = shfl_up16(ar), xi = shfl_up16(ai);
        tr = hi ? grid_add(ar, xr) : fr;   // X + Y = G - 1
        ti = hi ? grid_add(ai, xi) : fi;
        cr = ci = s;
    }
    // H_f = gomt X + t f, H_g = gomt Y + t G
    const double gr = E::mul(omt, gam.re), gi = E::mul(omt, gam.im);
    const int kt = hi ? kh + 1 : kd;
    const double av = gsum_anchor(max(max(gexp(gr), gexp(gi)) + kx + 2, gexp(cr) + kt + 1) + 2);
    gsum vr = gsum_start(av, hi ? s : 0.0), vi = {av, 0.0};
    gsum_acc_ext(vr, gr, ar);
    gsum_acc_ext(vr, -gi, ai);
    gsum_acc_ext(vr, cr, tr);
    gsum_acc_ext(vi, gr, ai);
    gsum_acc_ext(vi, gi, ar);
    gsum_acc_ext(vi, ci, ti);
    if (on)
        P.at(L::W1, hi ? M + k : k) = cx<double>{-ext_val(gsum_ext(vr, av)), -ext_val(gsum_ext(vi, av))};
    __syncwarp();
}

// Solves the M x M system [A | b0 | b1] (column-major, M rows; b1 only when two_rhs) by LU with
// partial pivoting over the warp; cur: entry lane % 16 of the solution for right-hand side
// lane / 16.  False when the matrix is singular.
template <int M>
__device__ __forceinline__ bool warp_lu_solve(cx<double> *A, int lane, bool two_rhs, cx<double> &cur) {
    static_assert(M <= 16, "one row per lane of each half-warp");
    auto at = [&](int i, int c) -> cx<double> & { return A[c * M + i]; };
    const int hrow = lane & 15, r = lane >> 4;
    // ---- LU with partial pivoting of [S | b0 | b1]; the pivot's reciprocal replaces it
    const int ncol = two_rhs ? M + 2 : M + 1;
    bool ok = true;
#pragma unroll 1
    for (int k = 0; k < M; k++) {
        // the row of the largest |re| + |im| at or below k (ties: the lowest row); the
        // bit patterns of non-negative doubles order as the values do
        unsigned long long key = 0ull;
        int idx = lane;
        if (lane >= k && lane < M) {
            const cx<double> a = at(lane, k);
            key = (unsigned long long)__double_as_longlong(fabs(a.re) + fabs(a.im));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ko = __shfl_xor_sync(0xffffffffu, key, o);
            const int io = __shfl_xor_sync(0xffffffffu, idx, o);
            if (ko > key || (ko == key && io < idx)) {
                key = ko;
                idx = io;
            }
        }
        int p = idx;
        if (key == 0ull) {   // the column is zero from row k down: S is singular
            ok = false;
            p = k;
        }
        if (p != k) {   // uniform
            if (lane >= k && lane < ncol) {
                const cx<double> a = at(k, lane);
                at(k, lane) = at(p, lane);
                at(p, lane) = a;
            }
            __syncwarp();
        }
        const cx<double> a = at(k, k);
        const double rd = 1.0 / fma(a.re, a.re, a.im * a.im);
        const cx<double> ip = cx<double>{a.re * rd, -a.im * rd};
        if (lane > k && lane < M) at(lane, k) = cmul(at(lane, k), ip);
        __syncwarp();
        const int nr = M - 1 - k, nc = ncol - 1 - k;
#pragma unroll 1
        for (int e = lane; e < nr * nc; e += 32) {
            const int c = k + 1 + e / nr, i = k + 1 + (e - (e / nr) * nr);
            at(i, c) = cfnms(at(i, c), at(i, k), at(k, c));
        }
        if (lane == 31) at(k, k) = ip;   // nothing reads the pivot in this step's update
        __syncwarp();
    }

    // ---- back substitution U x = b in registers: right-hand side r, row hrow
    const bool act = r == 0 || two_rhs;
    cur = cx<double>{0.0, 0.0};
    if (act && hrow < M) cur = at(hrow, M + r);
#pragma unroll 1
    for (int k = M - 1; k >= 0; k--) {
        const int src = (lane & 16) | k;
        const cx<double> bk = cx<double>{__shfl_sync(0xffffffffu, cur.re, src),
                                         __shfl_sync(0xffffffffu, cur.im, src)};
        if (hrow <= k) {
            const cx<double> xk = cmul(bk, at(k, k));   // the pivot's reciprocal
            cur = hrow == k ? xk : cfnms(cur, at(hrow, k), xk);
        }
    }

    return ok;
}

// H_z(ZC, t) d = r, the Schur reduction of xy_solve.cuh shared out over the warp; ZC and d in
// (x, y) (LC == false) or in the light-cone coordinates (p, q).
//   two_rhs false: r = -H_t, d into W1.
//   two_rhs true:  r1 = W1 (the residual), d1 into W1; r2 = -H_t, d2 into `out2`.
// Returns false (in every lane) when S is singular or the result is not finite.
template <int M, bool LC = false>
__device__ bool warp_solve(const WarpPath<M> &P, const double *__restrict__ J, double s,
                           double omt, cx<double> gam, bool two_rhs, int out2) {
    static_assert(M <= 16, "one site per lane of each half-warp");
    using L = WarpLayout<M>;
    const int lane = P.lane;
    const int hrow = lane & 15, r = lane >> 4;   // row and right-hand side of the half-warp layout
    const bool hi = lane >= 16, on = hrow < M;
    const cx<double> hg = cscale(0.5 * omt, gam);
    const double hs = 0.5 * s;

    // ---- per-site quantities of site j: its p side (U_p, a^, sp, A, -H_t's f row) on lane j, its q
    // side (U_q, b^, sq, B, the g row) on lane 16 + j.  o: the own one of p_j and q_j, x the other.
    {
        const int j = on ? hrow : 0;
        const double *Jj = J + j * NPHC_JSTRIDE;
        const cx<double> z = P.at(L::ZC, j), w = P.at(L::ZC, M + j);
        cx<double> U = {(hi && !LC) ? 0.0 : Jj[M], 0.0};
        const int off = hi ? L::ZC + M : L::ZC;
#pragma unroll 1
        for (int l = 0; l < M; l++) {
            const cx<double> v = P.at(off, l);
            U.re = fma(Jj[l], v.re, U.re);
            U.im = fma(Jj[l], v.im, U.im);
        }
        cx<double> V = shfl_xor16(U), p = z, q = w;   // V: the other side's sum
        if (!LC) {   // U_p = u + i w, U_q = u - i w
            const cx<double> su = hi ? V : U, sw = hi ? U : V;
            const cx<double> up = {su.re - sw.im, su.im + sw.re}, uq = {su.re + sw.im, su.im - sw.re};
            U = hi ? uq : up;
            V = hi ? up : uq;
            p = cx<double>{z.re - w.im, z.im + w.re};
            q = cx<double>{z.re + w.im, z.im - w.re};
        }
        const cx<double> o = hi ? q : p, x = hi ? p : q;
        // -H_t's rows: gamma X - f, f = i D / 2, D = q U_p - p U_q; gamma Y - G, G = p q - 1
        const cx<double> m = cmul(x, U), mo = shfl_xor16(m), pq = cmul(p, q);
        const cx<double> D = csub(hi ? mo : m, hi ? m : mo);
        const cx<double> sum = cadd(p, q), dif = csub(o, x);
        const cx<double> e = hi ? dif : sum, e2 = cmul(e, e);
        const double quarter = hi ? -0.25 : 0.25;
        const cx<double> t = {fma(quarter, e2.re, -1.0), quarter * e2.im};
        const cx<double> sub = hi ? cx<double>{pq.re - 1.0, pq.im} : cx<double>{-0.5 * D.im, 0.5 * D.re};
        const cx<double> ht = csub(cmul(gam, t), sub), ho = shfl_xor16(ht);
        const cx<double> htg = hi ? ht : ho;
        // the scaled frame (g_frame_lc in xy_solve.cuh) with powers of two for scales
        const double so = pow2_scale(o);
        const cx<double> hd = cmul(hg, dif);
        const cx<double> v = {so * fma(s, x.re, -hd.re), so * fma(s, x.im, -hd.im)};
        const double n2 = cabs2(v), iv = rsqrt(n2 + __shfl_xor_sync(0xffffffffu, n2, 16));
        const cx<double> vh = cscale(iv, v), xh = shfl_xor16(vh);
        const cx<double> g2 = cmul(hg, sum);
        const double hsu = hi ? hs : -hs;
        const cx<double> A = {so * fma(-hsu, V.im, g2.re), so * fma(hsu, V.re, g2.im)};
        const cx<double> dg = cmul(A, xh), dgo = shfl_xor16(dg);
        const cx<double> px0 = cmulc(vh, cscale(iv, two_rhs ? P.at(L::W1, M + j) : htg));
        const cx<double> b0 = cmul(A, px0), b0o = shfl_xor16(b0);
        cx<double> px1 = px0, b1 = b0, b1o = b0o;
        if (two_rhs) {
            px1 = cmulc(vh, cscale(iv, htg));
            b1 = cmul(A, px1);
            b1o = shfl_xor16(b1);
        }
        if (on) {
            P.at(hi ? L::SA : L::SB, j) = cscale(so, xh);
            P.at(hi ? L::IQ : L::IP, j) = cx<double>{-hs * o.im, hs * o.re};
            P.at(hi ? L::Y0 : L::X0, j) = cscale(so, px0);
            if (two_rhs) P.at(hi ? L::Y1 : L::X1, j) = cscale(so, px1);
            if (!hi) {   // the diagonal entry, and the diagonal's own terms of the right-hand sides
                P.A(j, j) = csub(dg, dgo);
                P.A(j, M) = csub(csub(two_rhs ? P.at(L::W1, j) : ht, b0), b0o);
                if (two_rhs) P.A(j, M + 1) = csub(csub(ht, b1), b1o);
            }
        }
    }
    __syncwarp();

    // ---- off-diagonal entries of S, one per lane (consecutive lanes: consecutive rows);
    // right-hand side r of row k on lane 16 r + k:
    //   b_k -= (i t / 2) (q_k sum_j J_kj X_j - p_k sum_j J_kj Y_j)   (J_kk = 0)
#pragma unroll 1
    for (int e = lane; e < M * M; e += 32) {
        const int j = e / M, k = e - j * M;
        if (k != j)
            P.A(k, j) = cscale(J[k * NPHC_JSTRIDE + j],
                               cfma64(P.at(L::IP, k), P.at(L::SA, j), cmul(P.at(L::IQ, k), P.at(L::SB, j))));
    }
    const bool act = r == 0 || two_rhs;
    if (on && act) {
        const int k = hrow;
        const double *Jk = J + k * NPHC_JSTRIDE;
        const int ox = r ? L::X1 : L::X0, oy = r ? L::Y1 : L::Y0;
        cx<double> sx = cx<double>{0.0, 0.0}, sy = sx;
#pragma unroll 1
        for (int j = 0; j < M; j++) {
            const double Jkj = Jk[j];
            const cx<double> xv = P.at(ox, j), yv = P.at(oy, j);
            sx.re = fma(Jkj, xv.re, sx.re);
            sx.im = fma(Jkj, xv.im, sx.im);
            sy.re = fma(Jkj, yv.re, sy.re);
            sy.im = fma(Jkj, yv.im, sy.im);
        }
        P.A(k, M + r) = cfma64(P.at(L::IP, k), sy, cfnms(P.A(k, M + r), P.at(L::IQ, k), sx));
    }
    __syncwarp();

    cx<double> cur;   // the solution: right-hand side r, row hrow
    const bool ok = warp_lu_solve<M>(P.s + L::A, lane, two_rhs, cur);

    // ---- back to (dp, dq) = (X + sp b^ s, Y - sq a^ s): site j of right-hand side r on lane 16 r + j
    bool finite = true;   // a square that overflows counts as not finite
    if (act && on) {
        const int j = hrow;
        cx<double> dp = cfma64(P.at(L::SB, j), cur, P.at(r ? L::X1 : L::X0, j));
        cx<double> dq = cfnms(P.at(r ? L::Y1 : L::Y0, j), P.at(L::SA, j), cur);
        finite = max(max(gexp(dp.re), gexp(dp.im)), max(gexp(dq.re), gexp(dq.im))) < 511;
        if (!LC) {
            const cx<double> x = {0.5 * (dp.re + dq.re), 0.5 * (dp.im + dq.im)};
            dq = cx<double>{0.5 * (dp.im - dq.im), -0.5 * (dp.re - dq.re)};
            dp = x;
        }
        const int o = r ? out2 : L::W1;   // W1's entries j and M + j were read above only
        P.at(o, j) = dp;
        P.at(o, M + j) = dq;
    }
    __syncwarp();
    return ok && __all_sync(0xffffffffu, finite);
}

// The problem a warp tracker runs on, as a policy for warp_track_body: the unknowns (NV), the
// shared layout with the step vectors Z0, K1, AC, ZC, W1, the start point with its dz/dt, the
// residual -H at ZC into W1, the linear solve, and the state's relation to the endpoint
// arrays' z (load, store, NORM2: the factor from the state's squared 2-norm to z's, and this
// lane's share of ||z||_inf at ZC).  WarpXY: the XY ring, its state in light-cone coordinates
// (p_k, q_k) = (x_k + i y_k, x_k - i y_k), like the per-thread trackers' (xy_track.cuh): near
// infinity one of them is far below x_k and y_k, and in (x, y) FP64 would lose it to
// cancellation.  ||(x, y)||_2 = sqrt(1/2) ||(p, q)||_2, ||(x, y)||_inf = max_k max(|p + q|, |p - q|) / 2.
template <int M>
struct WarpXY {
    using Sys = XYSys;
    using L = WarpLayout<M>;
    using Path = WarpPath<M>;
    static constexpr int NV = 2 * M;
    static constexpr double NORM2 = 0.5;
    static __device__ __forceinline__ void load(const Path &P, const EPView &ep, int64_t e) {
        const int64_t cnt = ep.count;
        const int lane = P.lane;
        if (lane < M) {   // (x, y) to (p, q)
            const int k = lane;
            const double xr = ep.z_re[k * cnt + e], xi = ep.z_im[k * cnt + e];
            const double yr = ep.z_re[(M + k) * cnt + e], yi = ep.z_im[(M + k) * cnt + e];
            P.at(L::Z0, k) = cx<double>{xr - yi, xi + yr};
            P.at(L::Z0, M + k) = cx<double>{xr + yi, xi - yr};
        }
    }
    static __device__ __forceinline__ void start(const Path &P, const Sys &S, int64_t p) {
        const int lane = P.lane, i = lane;
        const double *J = S.Jd;
        const cx<double> gam = cx<double>{S.gre, S.gim};
        if (i < NV) P.at(L::Z0, i) = cx<double>{((p >> i) & 1) ? -1.0 : 1.0, 0.0};
        __syncwarp();
        if (lane < M) {   // dz/dt at t = 0: -P_i(z) / (2 gamma z_i)
            const int k = lane;
            const cx<double> xk = P.at(L::Z0, k), yk = P.at(L::Z0, M + k);
            const double *Jk = J + k * NPHC_JSTRIDE;
            cx<double> u = cx<double>{Jk[M], 0.0}, w = cx<double>{0.0, 0.0};
#pragma unroll 1
            for (int l = 0; l < M; l++) {
                u.re += Jk[l] * P.at(L::Z0, l).re;
                w.re += Jk[l] * P.at(L::Z0, M + l).re;
            }
            cx<double> rf, rg;
            minus_ht_rows<double>(xk, yk, u, w, gam, rf, rg);
            const cx<double> ig = crecip(gam);
            const cx<double> dx = cscale(0.5 * xk.re, cmul(ig, rf));
            const cx<double> dy = cscale(0.5 * yk.re, cmul(ig, rg));
            P.at(L::K1, k) = cadd(dx, cmul_i(dy));       // dp = dx + i dy
            P.at(L::K1, M + k) = csub(dx, cmul_i(dy));   // dq = dx - i dy
        }
        __syncwarp();
        if (lane < M) {   // p = x + i y, q = x - i y (x, y real at the start)
            const int k = lane;
            const double xk = P.at(L::Z0, k).re, yk = P.at(L::Z0, M + k).re;
            P.at(L::Z0, k) = cx<double>{xk, yk};
            P.at(L::Z0, M + k) = cx<double>{xk, -yk};
        }
    }
    static __device__ __forceinline__ void residual(const Path &P, const Sys &S, double s, double omt) {
        warp_residual<M, true>(P, S.Jd, s, omt, cx<double>{S.gre, S.gim});
    }
    static __device__ __forceinline__ bool solve(const Path &P, const Sys &S, double s, double omt,
                                                 bool two_rhs, int out2) {
        return warp_solve<M, true>(P, S.Jd, s, omt, cx<double>{S.gre, S.gim}, two_rhs, out2);
    }
    static __device__ __forceinline__ double norminf(const Path &P) {
        if (P.lane >= M) return 0.0;
        const cx<double> pk = P.at(L::ZC, P.lane), qk = P.at(L::ZC, M + P.lane);
        return 0.5 * sqrt(fmax(cabs2(cadd(pk, qk)), cabs2(csub(pk, qk))));
    }
    static __device__ __forceinline__ void store(const Path &P, const EPView &ep, int64_t e) {
        const int64_t cnt = ep.count;
        const int lane = P.lane;
        if (lane < M) {   // x = (p + q) / 2, y = -i (p - q) / 2
            const int k = lane;
            const cx<double> pk = P.at(L::Z0, k), qk = P.at(L::Z0, M + k);
            ep.z_re[k * cnt + e] = 0.5 * (pk.re + qk.re);
            ep.z_im[k * cnt + e] = 0.5 * (pk.im + qk.im);
            ep.z_re[(M + k) * cnt + e] = 0.5 * (pk.im - qk.im);
            ep.z_im[(M + k) * cnt + e] = -0.5 * (pk.re - qk.re);
        }
    }
};

// One path per warp; the control flow of track_body in FP64, uniform over the warp.
// A list of max_paths entries or more is left to the group kernel (xy_track_group64.cuh).
template <class Q>
__device__ __forceinline__ void warp_track_body(const typename Q::Sys &S, const XYCtl &C,
                                                const EPView &ep, const WorkList &wl,
                                                int64_t max_paths = INT64_MAX) {
    using L = typename Q::L;
    constexpr int NV = Q::NV;
    extern __shared__ __align__(16) unsigned char wraw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const typename Q::Path P{reinterpret_cast<cx<double> *>(wraw) + (size_t)wid * L::TOTAL, lane};
    const int64_t total = worklist_size(wl, ep.count);
    if (total >= max_paths) return;
    const int i = lane;   // vector component of this lane (i < NV)
    for (;;) {
        unsigned long long q = 0;
        if (lane == 0) q = atomicAdd(wl.queue, 1ull);
        q = __shfl_sync(0xffffffffu, q, 0);
        if ((int64_t)q >= total) break;
        const int64_t e = worklist_entry(wl, (int64_t)q, ep.count);
        if (e < 0) continue;   // rejected by the debug build's check
        int status = NPHC_PATH_RUNNING, run = 0, attempts = 0, steps, solves, newton;
        double t, h;
        bool need_k1;
        if (C.resume) {
            Q::load(P, ep, e);
            t = ep.t[e];
            h = fmin(fmax(ep.h[e], 0.125 * (1.0 - t)), C.hmax);
            h = fmax(h, C.hmin * 4.0);
            steps = ep.steps[e];
            solves = ep.solves[e];
            newton = ep.newton[e];
            need_k1 = true;
        } else {
            Q::start(P, S, ep.path[e]);
            t = 0.0;
            h = C.h0;
            steps = C.accumulate ? ep.steps[e] : 0;
            solves = C.accumulate ? ep.solves[e] : 0;
            newton = C.accumulate ? ep.newton[e] : 0;
            need_k1 = false;
        }
        bool far = false;      // heading out: steps capped at KAPPA_FAR (1 - t) (xy_track.cuh)
        double zlast = 0.0;
        __syncwarp();
        while (status == NPHC_PATH_RUNNING) {
            if (far && h > KAPPA_FAR * (1.0 - t)) h = KAPPA_FAR * (1.0 - t);
            double hh = h, t1 = t + h;
            if (t1 >= C.t_end) {
                t1 = C.t_end;
                hh = C.t_end - t;
            }
            bool conv = false, bad = false;
            double zpn = 0.0;
            const int ph0 = need_k1 ? 0 : 1;
            const int nph = 4 + C.max_newton;
#pragma unroll 1
            for (int ph = ph0; ph < nph; ph++) {
                const bool corr = ph >= 4 || ph == 0;
                if (ph >= 4 && (conv || bad)) break;
                const double te = ph == 0 ? t : (ph >= 4 || ph == 3) ? t1 : t + 0.5 * hh;
                if (ph < 4) {   // evaluation point: z0, z0 + h/2 k1, z0 + h/2 k2, z0 + h k3
                    const double c = ph == 3 ? hh : 0.5 * hh;
                    if (i < NV) {
                        const cx<double> z0 = P.at(L::Z0, i);
                        P.at(L::ZC, i) = ph == 0 ? z0
                                                 : cadd(z0, cscale(c, ph == 1 ? P.at(L::K1, i) : P.at(L::W1, i)));
                    }
                    __syncwarp();
                }
                if (corr) Q::residual(P, S, te, 1.0 - te);
                const bool oks = Q::solve(P, S, te, 1.0 - te, corr, L::AC);
                solves++;
                if (ph == 0) {   // pull the resumed point onto the FP64 path; dz/dt there
                    if (i < NV) {
                        P.at(L::Z0, i) = cadd(P.at(L::ZC, i), P.at(L::W1, i));
                        P.at(L::K1, i) = P.at(L::AC, i);
                    }
                    __syncwarp();
                    newton++;
                    need_k1 = false;
                    if (!oks) status = NPHC_PATH_NONFINITE;
                    if (status != NPHC_PATH_RUNNING) break;
                } else if (!corr) {
                    bad = bad || !oks;
                    if (i < NV) {
                        const cx<double> w1 = P.at(L::W1, i);
                        if (ph == 1) P.at(L::AC, i) = cadd(P.at(L::K1, i), cscale(2.0, w1));
                        else if (ph == 2) P.at(L::AC, i) = cadd(P.at(L::AC, i), cscale(2.0, w1));
                    }
                    if (ph == 3) {   // predicted point z0 + h/6 (k1 + 2 k2 + 2 k3 + k4)
                        double zz = 0.0;
                        if (i < NV) {
                            const cx<double> zp = cadd(P.at(L::Z0, i),
                                                       cscale(hh / 6.0, cadd(P.at(L::AC, i), P.at(L::W1, i))));
                            P.at(L::ZC, i) = zp;
                            zz = cabs2(zp);
                        }
                        zpn = sqrt(Q::NORM2 * warp_sum(zz));
                    }
                    __syncwarp();
                } else {
                    newton++;
                    const double dn = sqrt(Q::NORM2 * warp_sum(i < NV ? cabs2(P.at(L::W1, i)) : 0.0));
                    if (!oks || !isfinite(dn)) {
                        bad = true;
                    } else if (ph == 4 && dn > C.trust * (1.0 + zpn)) {
                        bad = true;
                    } else {
                        double zz = 0.0;
                        if (i < NV) {
                            const cx<double> zn = cadd(P.at(L::ZC, i), P.at(L::W1, i));
                            P.at(L::ZC, i) = zn;
                            zz = cabs2(zn);
                        }
                        zz = Q::NORM2 * warp_sum(zz);
                        if (dn <= C.eps * (1.0 + sqrt(zz))) conv = true;
                    }
                    __syncwarp();
                }
            }
            if (status != NPHC_PATH_RUNNING) break;
            attempts++;
            if (conv) {
                if (i < NV) {
                    P.at(L::Z0, i) = P.at(L::ZC, i);
                    P.at(L::K1, i) = P.at(L::AC, i);
                }
                const double zi = warp_max(Q::norminf(P));   // of the endpoint arrays' z
                __syncwarp();
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
            } else {
                run = 0;
                h *= 0.5;
                if (h < C.hmin) status = NPHC_PATH_MIN_STEP;
            }
            if (status == NPHC_PATH_RUNNING && attempts >= C.max_steps) status = NPHC_PATH_STEP_BUDGET;
        }
        Q::store(P, ep, e);
        if (lane == 0) {
            ep.t[e] = t;
            ep.h[e] = h;
            ep.status[e] = status;
            ep.steps[e] = steps;
            ep.solves[e] = solves;
            ep.newton[e] = newton;
        }
        __syncwarp();
    }
}

template <int M, int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
    xy_track_warp64_kernel(const __grid_constant__ XYSys S, const __grid_constant__ XYCtl C,
                           const EPView ep, const WorkList wl, int64_t max_paths) {
    warp_track_body<WarpXY<M>>(S, C, ep, wl, max_paths);
}
