// xy_track_group.cuh -- the FP32 tracker of the XY ring: four lanes per path, eight paths
// per warp.
//
// The method is that of xy_track.cuh (RK4 predictor, Newton corrector with a compensated
// residual, light-cone state, end-zone rules, hand-offs to FP64) with the linear algebra of
// xy_solve.cuh (scaled light-cone frames, M x M complex Schur system, LU with partial
// pivoting).  The layout is for latency and issue slots: the tracker is bound by neither
// memory (under 1 GB/s) nor the FMA pipe, but by how many instructions the few resident
// warps can issue.
//   * Lane g of a path owns the sites j = g + 4 s and with them row j of the Schur system:
//     U sums, frames, right-hand sides and residual rows of its own sites, and the row's
//     M + 2 complex entries, in registers (72 of them at M = 9).  Nothing of the matrix but
//     the pivot rows passes through shared memory.
//   * LU step k: every lane's largest |a|^2 among its rows not yet pivoted, the path's by two
//     shuffles (the row index rides in the low four bits of the value, ties go to the lowest
//     row); the owner writes the pivot row to shared memory, the four lanes read it back and
//     update their rows.  The written rows are U, from which the back substitution runs
//     (T on even lanes, R on odd ones).  No rows are swapped.
//   * Arithmetic in pairs (fma.rn.f32x2): (re, im) where the coefficient is real or a
//     compensated sum runs, two neighbouring columns where both factors are complex.
//   * Each path is in its own phase (an RK4 stage or a corrector iteration); a warp, or with
//     full warps the block, runs, for all paths that wait for one, whichever of a predictor and a
//     corrector solve has more takers (a corrector solve costs about twice as much, so it needs
//     half as many).  In
//     lockstep a warp runs the correctors its slowest path needs (1.7 per step on average,
//     three at worst).  A path's own sequence of operations does not depend on its company.
//   * Time is an integer number of 2^-53, the grid of the doubles in [1/2, 1): 1 - t is exact
//     and the step logic costs no FP64 instruction (an FP64 instruction takes 67 cycles of
//     a scheduler here, whatever the number of lanes).
#pragma once

#include "f32_step.cuh"

// --------------------------------------------------------------- the layout --
constexpr int GRP_LANES = 4;    // lanes per path
constexpr int GRP_PATHS = 8;    // paths per warp
constexpr int GRP_WARPS = 4;    // warps per block (they share the coupling table)

// Shared memory, in float4 per path ([index * 8 + path in warp]).
template <int M>
struct GrpLayout {
    static constexpr int SL = (M + 3) / 4;        // sites per lane
    static constexpr int ROWS = 4 * SL;           // rows of the coupling table (zero rows from M on)
    static constexpr int NPM = (M + 1) / 2;       // column pairs holding S
    static constexpr int NP = (M + 3) / 2;        // column pairs of [S | T | R]
    static constexpr int NPT = (M + 2) / 2;       // column pairs of [S | T]
    __host__ __device__ static constexpr int uoff(int k) {   // first pair of U's row k
        int o = 0;
        for (int i = 0; i < k; i++) o += NP - i / 2;
        return o;
    }
    static constexpr int USIZE = uoff(M);
    static constexpr int BSIZE = 2 * NPM;         // build: the columns' (cb, ca)
    static constexpr int PQ = 0;                  // evaluation point (p_j, q_j)
    static constexpr int XY = PQ + M;             // X_j, Y_j of right-hand side T
    static constexpr int FR = XY + M;             // (sp b^_j, sq a^_j), read by their owner only
    static constexpr int W0 = FR + M;             // of a site, for its owner: diagonal entry and
    static constexpr int W1 = W0 + M;             // right-hand side T; right-hand side R
    static constexpr int U = W1 + M;              // pivot rows; before them (cb, ca), after them
    static constexpr int Z0 = U + (USIZE > BSIZE ? USIZE : BSIZE);   // the solution (T, R)
    static constexpr int K1 = Z0 + M;             // accepted point, dz/dt there
    static constexpr int AC = K1 + M;             // RK4 sum; in corrector solves X_j, Y_j of R
    static constexpr int TOTAL = AC + M;
    static constexpr int JB = ROWS * (M + 1);     // coupling table entries
    static constexpr int BLOCKS = M <= 10 ? 4 : 3;   // resident blocks per SM aimed at
};

// the coupling table: one per block, or (batch) one per path
template <int M>
constexpr size_t grp_smem_per_block(bool batch) {
    using L = GrpLayout<M>;
    return sizeof(float4) * (size_t)(GRP_WARPS * GRP_PATHS * L::TOTAL) +
           sizeof(float) * (size_t)L::JB * (batch ? GRP_WARPS * GRP_PATHS : 1);
}

template <int M, bool BATCH>
struct GrpJ {
    const float *base;   // this lane's row g of the table
    static constexpr int STEP = BATCH ? GRP_PATHS : 1;
    __device__ __forceinline__ float val(int s, int l) const { return base[(4 * s * (M + 1) + l) * STEP]; }
    __device__ __forceinline__ float2 dup(int s, int l) const { return f2dup(val(s, l)); }
};

__device__ __forceinline__ float grp_sum(float v) {   // over a path's four lanes
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    return v + __shfl_xor_sync(0xffffffffu, v, 16);
}
__device__ __forceinline__ float grp_max(float v) {
    v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
    return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
}

template <int SL>
struct GrpStep {       // (dp, dq) of a lane's own sites
    float2 p[SL], q[SL];
};

// One solve of H_z(z, t) d = r at the points in PQ (see xy_solve and xy_residual_comp in
// xy_solve.cuh): d of r = -H_t into dt and, when corr (uniform over the warp), d of r = -H
// (compensated) into dr.  sm: the path's column of the warp's shared memory.  The R scratch
// is written only when w (it aliases the RK4 sum, which paths outside this solve still need).
// Returns false when the system is singular or the result is not finite.
template <int M, bool BATCH>
__device__ __forceinline__ bool grp_solve(float4 *__restrict__ sm, const GrpJ<M, BATCH> &J, int g,
                                          float s, float omt, cx<float> gam, bool corr, bool w,
                                          GrpStep<GrpLayout<M>::SL> &dt,
                                          GrpStep<GrpLayout<M>::SL> &dr, float &kest) {
    using L = GrpLayout<M>;
    constexpr int SL = L::SL, NP = L::NP, NPT = L::NPT;
    // the sums over l unrolled where the kernel stays under 4,000 instructions (M <= 8: 256 paths of
    // N = 5 0.84 -> 0.77 ms, 16,384 of N = 8 4.15 -> 4.0); at M = 9 (5,100) even three at a time cost 4%
    constexpr int UL = M <= 8 ? M : 1, UP = M <= 8 ? M : 3;
    const float2 gm = f2(gam.re, gam.im), hgomt = f2scale(0.5f * omt, gm);
    const float hs = 0.5f * s;
    auto at = [&](int off, int i) -> float4 & { return sm[(off + i) * GRP_PATHS]; };
    auto own = [&](int q) { return q < SL - 1 || M % 4 == 0 || g + 4 * q < M; };   // site g + 4 q exists
    auto site = [&](int q) { return own(q) ? g + 4 * q : M - 1; };

    // ---- site by site (one copy of the code: straight-line code for every site outgrows the
    // instruction cache): U_p, U_q (compensated for the corrector), residual rows, frames,
    // diagonal entries, the diagonal's share of the right-hand sides
#pragma unroll 1
    for (int q = 0; q < SL; q++) {
        const int j = site(q);
        const float4 z = at(L::PQ, j);
        ext2 up = {f2(J.val(q, M), 0.0f), f2dup(0.0f)}, uq = up;
        float2 rf = f2dup(0.0f), rg = rf;   // -H rows
        if (corr) {
#pragma unroll UL
            for (int l = 0; l < M; l++) {
                const float4 v = at(L::PQ, l);
                const float2 c = J.dup(q, l);
                acc2(up, c, f2(v.x, v.y));
                acc2(uq, c, f2(v.z, v.w));
            }
            f32_residual_rows(f2(z.x, z.y), f2(z.z, z.w), up, uq, s, hs, __fmul_rn(omt, gam.re),
                              __fmul_rn(omt, gam.im), rf, rg);
        } else {
#pragma unroll UP
            for (int l = 0; l < M; l++) {
                const float4 v = at(L::PQ, l);
                const float2 c = J.dup(q, l);
                up.hi = f2fma(c, f2(v.x, v.y), up.hi);
                uq.hi = f2fma(c, f2(v.z, v.w), uq.hi);
            }
        }
        float2 htf, htg, x, y, d;
        const F32Site v = f32_site(f2(z.x, z.y), f2(z.z, z.w), up.hi, uq.hi, s, hs, hgomt, gm, htf, htg);
        v.rhs(htf, htg, x, y, d);
        if (own(q)) {
            at(L::XY, j) = make_float4(x.x, x.y, y.x, y.y);
            at(L::FR, j) = make_float4(v.sb.x, v.sb.y, v.sa.x, v.sa.y);
            at(L::W0, j) = make_float4(v.sjj.x, v.sjj.y, d.x, d.y);
            // column pair j / 2: (re, re', im, im') of cb = i t/2 sp b^ and ca = i t/2 sq a^
            float *cb = reinterpret_cast<float *>(&at(L::U, j >> 1)) + (j & 1);
            float *ca = reinterpret_cast<float *>(&at(L::U, L::NPM + (j >> 1))) + (j & 1);
            cb[0] = -hs * v.sb.y;
            cb[2] = hs * v.sb.x;
            ca[0] = -hs * v.sa.y;
            ca[2] = hs * v.sa.x;
        }
        if (corr) {
            v.rhs(rf, rg, x, y, d);
            if (own(q)) {
                if (w) at(L::AC, j) = make_float4(x.x, x.y, y.x, y.y);
                at(L::W1, j) = make_float4(d.x, d.y, 0.0f, 0.0f);
            }
        }
    }
    __syncwarp();

    // ---- the own rows: S_kj = J_kj (q_k cb_j + p_k ca_j), two columns at a time, ...
    float2 re[SL][NP], im[SL][NP];
#pragma unroll
    for (int q = 0; q < SL; q++) {
        const float4 z = at(L::PQ, site(q));
        const float2 pr = f2dup(z.x), pi = f2dup(z.y), npi = f2dup(-z.y);
        const float2 qr = f2dup(z.z), qi = f2dup(z.w), nqi = f2dup(-z.w);
#pragma unroll
        for (int jp = 0; jp < L::NPM; jp++) {
            const float4 cb = at(L::U, jp), ca = at(L::U, L::NPM + jp);
            const float2 cbr = f2(cb.x, cb.y), cbi = f2(cb.z, cb.w);
            const float2 car = f2(ca.x, ca.y), cai = f2(ca.z, ca.w);
            const float2 jj = f2(J.val(q, 2 * jp), 2 * jp + 1 < M ? J.val(q, 2 * jp + 1) : 0.0f);
            const float2 a = f2fma(npi, cai, f2fma(pr, car, f2fma(nqi, cbi, f2mul(qr, cbr))));
            const float2 b = f2fma(pi, car, f2fma(pr, cai, f2fma(qi, cbr, f2mul(qr, cbi))));
            re[q][jp] = f2mul(jj, a);
            im[q][jp] = f2mul(jj, b);
        }
        // the diagonal entry: column g + 4 q, in pair 2 q + g / 2
        const float4 dg = at(L::W0, site(q));
#pragma unroll
        for (int h = 0; h < 2; h++) {
            if (2 * q + h < L::NPM) {
                if (g == 2 * h && own(q)) {
                    re[q][2 * q + h].x = dg.x;
                    im[q][2 * q + h].x = dg.y;
                }
                if (g == 2 * h + 1 && own(q)) {
                    re[q][2 * q + h].y = dg.x;
                    im[q][2 * q + h].y = dg.y;
                }
            }
        }
    }
    // ---- ... and right-hand sides b_k = d_k - (i t / 2) (q_k sum_j J_kj X_j - p_k sum_j J_kj Y_j)
    {
        float2 sx[SL], sy[SL], rx[SL], ry[SL];
#pragma unroll
        for (int q = 0; q < SL; q++) sx[q] = sy[q] = rx[q] = ry[q] = f2dup(0.0f);
        if (corr) {
#pragma unroll UL
            for (int j = 0; j < M; j++) {
                const float4 v = at(L::XY, j), r = at(L::AC, j);
#pragma unroll
                for (int q = 0; q < SL; q++) {
                    const float2 c = J.dup(q, j);
                    sx[q] = f2fma(c, f2(v.x, v.y), sx[q]);
                    sy[q] = f2fma(c, f2(v.z, v.w), sy[q]);
                    rx[q] = f2fma(c, f2(r.x, r.y), rx[q]);
                    ry[q] = f2fma(c, f2(r.z, r.w), ry[q]);
                }
            }
        } else {
#pragma unroll UL
            for (int j = 0; j < M; j++) {
                const float4 v = at(L::XY, j);
#pragma unroll
                for (int q = 0; q < SL; q++) {
                    const float2 c = J.dup(q, j);
                    sx[q] = f2fma(c, f2(v.x, v.y), sx[q]);
                    sy[q] = f2fma(c, f2(v.z, v.w), sy[q]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < SL; q++) {
            const float4 z = at(L::PQ, site(q));
            const float2 ip = f2scale(hs, f2i(f2(z.x, z.y))), iq = f2scale(-hs, f2i(f2(z.z, z.w)));
            const float4 dg = at(L::W0, site(q)), dr1 = at(L::W1, site(q));
            const float mine = own(q) ? 1.0f : 0.0f;   // rows that do not exist are zero
            const float2 t = f2scale(mine, f2cfma(ip, sy[q], f2cfma(iq, sx[q], f2(dg.z, dg.w))));
            float2 r = f2dup(0.0f);
            if (corr) r = f2scale(mine, f2cfma(ip, ry[q], f2cfma(iq, rx[q], f2(dr1.x, dr1.y))));
            const float tr = t.x, ti = t.y, rr = r.x, ri = r.y;
            if (M % 2) {
                re[q][M / 2].y = tr;
                im[q][M / 2].y = ti;
                re[q][NP - 1] = f2(rr, 0.0f);
                im[q][NP - 1] = f2(ri, 0.0f);
            } else {
                re[q][M / 2] = f2(tr, rr);
                im[q][M / 2] = f2(ti, ri);
            }
        }
    }
    __syncwarp();

    // ---- LU with partial pivoting; U's rows go to shared memory
    unsigned live[SL];   // all but the low four bits while own row g + 4 q waits to be a pivot row, else 0
#pragma unroll
    for (int q = 0; q < SL; q++) live[q] = own(q) ? ~15u : 0u;
    bool ok = true;
    float umax = 0.0f, umin = INFINITY;   // of |U_kk|^2
    float2 ip[M];
#pragma unroll
    for (int k = 0; k < M; k++) {
        const int kp = k / 2;
        float2 a[SL];
        unsigned key = 0;   // rows done or absent count as zeros
#pragma unroll
        for (int q = 0; q < SL; q++) {
            a[q] = k % 2 ? f2(re[q][kp].y, im[q][kp].y) : f2(re[q][kp].x, im[q][kp].x);
            key = max(key, (__float_as_uint(f2abs2(a[q])) & live[q]) | (unsigned)(15 - 4 * q - g));
        }
        key = max(key, __shfl_xor_sync(0xffffffffu, key, 8));
        key = max(key, __shfl_xor_sync(0xffffffffu, key, 16));
        ok = ok && key > 15u;
        const int prow = 15 - (int)(key & 15u);
        const int uo = L::U + L::uoff(k) - kp;
#pragma unroll
        for (int q = 0; q < SL; q++) {
            if (g + 4 * q == prow) {
#pragma unroll
                for (int c = kp; c < NP; c++) at(uo, c) = make_float4(re[q][c].x, re[q][c].y, im[q][c].x, im[q][c].y);
                live[q] = 0;
            }
        }
        __syncwarp();
        const float4 u0 = at(uo, kp);
        const float2 piv = k % 2 ? f2(u0.y, u0.w) : f2(u0.x, u0.z);
        const float best = f2abs2(piv);
        umax = fmaxf(umax, best);
        umin = fminf(umin, best);
        ip[k] = f2scale(f32_recip(best), f2(piv.x, -piv.y));
        if (k < M - 1) {
            float2 lr[SL], li[SL], nli[SL];   // -Re, Im, -Im of the multipliers
#pragma unroll
            for (int q = 0; q < SL; q++) {
                const float2 l = f2cmul(a[q], ip[k]);
                lr[q] = f2dup(-l.x);
                li[q] = f2dup(l.y);
                nli[q] = f2dup(-l.y);
            }
            auto update = [&](int c) {
                const float4 u = c == kp ? u0 : at(uo, c);
                const float2 ur = f2(u.x, u.y), ui = f2(u.z, u.w);
#pragma unroll
                for (int q = 0; q < SL; q++) {
                    re[q][c] = f2fma(li[q], ui, f2fma(lr[q], ur, re[q][c]));
                    im[q][c] = f2fma(nli[q], ur, f2fma(lr[q], ui, im[q][c]));
                }
            };
#pragma unroll
            for (int c = (k + 1) / 2; c < NPT; c++) update(c);
            if (M % 2 && corr) update(NP - 1);
        }
    }
    kest = sqrtf(umax / umin);
    __syncwarp();

    // ---- back substitution: T on even lanes, R on odd ones (T again without corr)
    const bool mine_r = corr && (g & 1);
    float2 xr[L::NPM], xi[L::NPM];
#pragma unroll
    for (int c = 0; c < L::NPM; c++) xr[c] = xi[c] = f2dup(0.0f);
#pragma unroll
    for (int k = M - 1; k >= 0; k--) {
        const int uo = L::U + L::uoff(k) - k / 2;
        float2 sr = f2dup(0.0f), si = f2dup(0.0f);
#pragma unroll
        for (int c = L::NPM - 1; c >= (k + 1) / 2; c--) {
            const float4 u = at(uo, c);
            const float2 ur = f2(u.x, u.y), ui = f2(u.z, u.w);
            sr = f2fma(f2neg(ui), xi[c], f2fma(ur, xr[c], sr));
            si = f2fma(ui, xr[c], f2fma(ur, xi[c], si));
        }
        const float4 ut = at(uo, M / 2);
        float2 b = M % 2 ? f2(ut.y, ut.w) : f2(ut.x, ut.z);
        if (mine_r) {
            const float4 ub = at(uo, NP - 1);
            b = M % 2 ? f2(ub.x, ub.z) : f2(ub.y, ub.w);
        }
        const float2 x = f2cmul(f2(b.x - (sr.x + sr.y), b.y - (si.x + si.y)), ip[k]);
        if (k % 2) {
            xr[k / 2].y = x.x;
            xi[k / 2].y = x.y;
        } else {
            xr[k / 2].x = x.x;
            xi[k / 2].x = x.y;
        }
    }
    __syncwarp();
    if (g < 2) {
#pragma unroll
        for (int k = 0; k < M; k++) {
            float2 *o = reinterpret_cast<float2 *>(&at(L::U, k)) + g;
            *o = k % 2 ? f2(xr[k / 2].y, xi[k / 2].y) : f2(xr[k / 2].x, xi[k / 2].x);
        }
    }
    __syncwarp();

    // ---- back to (dp, dq) = (X + sp b^ s, Y - sq a^ s)
    float chk = 0.0f;
#pragma unroll
    for (int q = 0; q < SL; q++) {
        const int j = site(q);
        const float4 x = at(L::U, j), f = at(L::FR, j), v = at(L::XY, j);
        const float2 sb = f2(f.x, f.y), sa = f2(f.z, f.w), sT = f2(x.x, x.y);
        dt.p[q] = f2cfma(sb, sT, f2(v.x, v.y));
        dt.q[q] = f2cfms(sa, sT, f2(v.z, v.w));
        chk += f2abs2(dt.p[q]) + f2abs2(dt.q[q]);
        if (corr) {
            const float4 r = at(L::AC, j);
            const float2 sR = f2(x.z, x.w);
            dr.p[q] = f2cfma(sb, sR, f2(r.x, r.y));
            dr.q[q] = f2cfms(sa, sR, f2(r.z, r.w));
            chk += f2abs2(dr.p[q]) + f2abs2(dr.q[q]);
        }
    }
    chk = grp_sum(chk);
    return ok && isfinite(chk);
}

template <int M, bool BATCH, class Src>
__device__ __forceinline__ void grp_track_body(const Src &src, const XYCtl &C, const WorkList &wl) {
    using L = GrpLayout<M>;
    constexpr int SL = L::SL;
    extern __shared__ __align__(16) float4 grp_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int g = lane >> 3, pth = lane & 7;
    float4 *const sm = grp_raw + wid * (GRP_PATHS * L::TOTAL) + pth;
    float *const jtab = reinterpret_cast<float *>(grp_raw + GRP_WARPS * (GRP_PATHS * L::TOTAL));
    auto at = [&](int off, int i) -> float4 & { return sm[(off + i) * GRP_PATHS]; };
    auto own = [&](int q) { return q < SL - 1 || M % 4 == 0 || g + 4 * q < M; };
    auto site = [&](int q) { return own(q) ? g + 4 * q : M - 1; };
    float *const jpath = jtab + wid * (GRP_PATHS * L::JB) + pth;   // batch
    const GrpJ<M, BATCH> J{BATCH ? jpath + g * (M + 1) * GRP_PATHS : jtab + g * (M + 1)};
    if (!BATCH) {
        const float *Jf = src.sys(0).Jf;
        for (int i = threadIdx.x; i < L::JB; i += blockDim.x) {
            const int r = i / (M + 1), l = i - r * (M + 1);
            jtab[i] = r < M ? Jf[r * NPHC_JSTRIDE + l] : 0.0f;
        }
        __syncthreads();
    }
    // every slot starts at a finite point (paths that never come still run the arithmetic)
#pragma unroll
    for (int q = 0; q < SL; q++)
        if (own(q)) at(L::PQ, g + 4 * q) = at(L::AC, g + 4 * q) = make_float4(1.0f, 0.0f, 1.0f, 0.0f);
    if (BATCH)
        for (int i = g; i < L::JB; i += GRP_LANES) jpath[i * GRP_PATHS] = 0.0f;

    // hand-off checkpoints: in the launch's global scratch (written now and then, read once)
    const int64_t slots = (int64_t)gridDim.x * (GRP_WARPS * GRP_PATHS);
    float4 *const ck = reinterpret_cast<float4 *>(wl.state) +
                       ((int64_t)blockIdx.x * GRP_WARPS + wid) * GRP_PATHS + pth;

    const int64_t total = src.total();
    // few paths: one warp per scheduler before more paths per warp (fewer to wait for, and
    // the warp's time is its slowest path's either way)
    int per = GRP_PATHS;
    {
        const int64_t warps = (int64_t)gridDim.x * GRP_WARPS;
        const int64_t want = (total + warps - 1) / warps;
        if (want < per) per = want < 1 ? 1 : (int)want;
    }
    // With full warps the block decides which solve runs, so that its four warps go through the same
    // code at the same time: an SM's warps (eight at M = 12 to fourteen at M <= 9) in as many places of a
    // kernel of 60 to 90 KB waited for instructions two cycles per issue.  The pool of 32 paths fills the phases as well as
    // eight do (85% in a simulation of the mix).  N = 13 80,000 paths 58 -> 41 ms, N = 12 32,768
    // 24.4 -> 18.6, N = 11 19.1 -> 15.8, N = 9 65,536 13.7 -> 12.7.  With fewer paths no path waits for
    // the others of its block.
    const bool together = per == GRP_PATHS;
    const F32Ctl K(C);
    int64_t e = pth < per ? -1 : -2;   // entry of this path slot; -1 idle, -2 drained
    int inst = 0;                      // instance of the entry (batches)
    int ph = 1;                        // phase: 1 .. 3 RK4 stages, 4 .. corrector
    F32Step P;
    P.start(0, 0);
    bool bad = false, start = false;   // start: a new step attempt begins
    float zpn = 0.0f, kstep = 0.0f;
    cx<float> gam = {1.0f, 0.0f};
    if (!BATCH) gam = cx<float>{(float)src.sys(0).gre, (float)src.sys(0).gim};

#pragma unroll 1
    for (;;) {
        // ---- hand new entries to idle paths
        const unsigned need = __ballot_sync(0xffffffffu, e == -1) & 0xffu;
        if (need) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(wl.queue, (unsigned long long)__popc(need));
            base = __shfl_sync(0xffffffffu, base, 0);
            bool fresh = false;
            if (e == -1) {
                const int64_t i = (int64_t)base + __popc(need & ((1u << pth) - 1u));
                if (i >= total) e = -2;
                else src.take(i, inst, e);   // -1 (skipped) if the debug build rejects it
                fresh = e >= 0;
            }
            if (BATCH) {
                if (fresh) {
                    const XYSys &S = src.sys(inst);
                    for (int i = g; i < L::JB; i += GRP_LANES) {
                        const int r = i / (M + 1), l = i - r * (M + 1);
                        jpath[i * GRP_PATHS] = r < M ? S.Jf[r * NPHC_JSTRIDE + l] : 0.0f;
                    }
                    gam = cx<float>{(float)S.gre, (float)S.gim};
                }
                __syncwarp();
            }
            if (fresh) {
                P.steps = P.solves = P.newton = 0;
                kstep = 0.0f;
                bad = false;
                const int64_t path = src.eps(inst).path[e];
                const cx<float> ig = crecip(gam);
#pragma unroll 1
                for (int q = 0; q < SL; q++) {
                    const int k = site(q);
                    float u = J.val(q, M), v = 0.0f;
#pragma unroll 1
                    for (int l = 0; l < M; l++) {
                        const float jl = J.val(q, l);
                        u += ((path >> l) & 1) ? -jl : jl;
                        v += ((path >> (M + l)) & 1) ? -jl : jl;
                    }
                    const float x = ((path >> k) & 1) ? -1.0f : 1.0f;
                    const float y = ((path >> (M + k)) & 1) ? -1.0f : 1.0f;
                    cx<float> rf, rg;
                    minus_ht_rows<float>(cx<float>{x, 0.0f}, cx<float>{y, 0.0f}, cx<float>{u, 0.0f},
                                         cx<float>{v, 0.0f}, gam, rf, rg);
                    const cx<float> dx = cscale(0.5f * x, cmul(ig, rf)), dy = cscale(0.5f * y, cmul(ig, rg));
                    if (own(q)) {
                        at(L::Z0, k) = make_float4(x, y, x, -y);   // p = x + i y, q = x - i y
                        at(L::K1, k) = make_float4(dx.re - dy.im, dx.im + dy.re, dx.re + dy.im, dx.im - dy.re);
                    }
                }
                P.start(0, K.h0);
                start = true;
            }
        }
        const bool any = __any_sync(0xffffffffu, e >= 0);
        if (!together && !any) break;

        // ---- a new attempt: its first stage's point z0 + h/2 k1
        const bool act = e >= 0;
        f32_time hh, t1;
        if (start) P.cap();
        P.len(K, hh, t1);
        if (start) {
            const float2 c = f2dup(0.5f * time_float(hh));
#pragma unroll
            for (int q = 0; q < SL; q++)
                if (own(q)) {
                    const int j = g + 4 * q;
                    const float4 z = at(L::Z0, j), k = at(L::K1, j);
                    const float2 a = f2fma(c, f2(k.x, k.y), f2(z.x, z.y)), b = f2fma(c, f2(k.z, k.w), f2(z.z, z.w));
                    at(L::PQ, j) = make_float4(a.x, a.y, b.x, b.y);
                }
            ph = 1;
            bad = start = false;
        }

        // ---- which solve runs now, and for whom
        const bool wants_c = act && ph >= 4;
        int nc, np;
        if (together) {
            nc = __syncthreads_count(wants_c);
            np = __syncthreads_count(act && !wants_c);
            if (nc + np == 0) break;
        } else {
            nc = __popc(__ballot_sync(0xffffffffu, wants_c));
            np = __popc(__ballot_sync(0xffffffffu, act && !wants_c));
        }
        const bool corr = nc > 0 && 2 * nc >= np;
        const bool w = act && wants_c == corr;
        if (together && !__any_sync(0xffffffffu, w)) continue;
        const f32_time te = ph < 3 ? P.t + hh / 2 : t1;
        int verdict = STEP_GO_ON, status = NPHC_PATH_RUNNING;
        float zi = 0.0f;
        GrpStep<SL> dt, dr;
        float kest;
        __syncwarp();
        const bool oks = grp_solve<M, BATCH>(sm, J, g, time_float(te), time_float(F32_ONE - te), gam, corr, w,
                                             dt, dr, kest);

        if (!corr) {
            // ---- RK4: the next stage's point, or the predicted one
            float zz = 0.0f;
            if (w) {
                const float hr = time_float(hh);
                const float2 c = f2dup(ph == 1 ? 0.5f * hr : ph == 2 ? hr : hr * (1.0f / 6.0f));
                bad = bad || !oks;
                P.solves++;
                kstep = fmaxf(kstep, kest);
#pragma unroll
                for (int q = 0; q < SL; q++) {
                    const int j = site(q);
                    const float4 z = at(L::Z0, j), o = at(ph == 1 ? L::K1 : L::AC, j);
                    const float2 m = f2dup(ph == 3 ? 1.0f : 2.0f);
                    const float2 sp = f2fma(m, dt.p[q], f2(o.x, o.y)), sq = f2fma(m, dt.q[q], f2(o.z, o.w));
                    const float2 a = f2fma(c, ph == 3 ? sp : dt.p[q], f2(z.x, z.y));
                    const float2 b = f2fma(c, ph == 3 ? sq : dt.q[q], f2(z.z, z.w));
                    if (own(q)) {
                        at(L::AC, j) = make_float4(sp.x, sp.y, sq.x, sq.y);
                        at(L::PQ, j) = make_float4(a.x, a.y, b.x, b.y);
                        zz += a.x * a.x + a.y * a.y + b.x * b.x + b.y * b.y;
                    }
                }
            }
            zz = grp_sum(zz);
            if (w) {
                zpn = sqrtf(0.5f * zz);   // ||(x, y)||_2 of the predicted point
                ph++;
                if (ph == 4 && bad) verdict = STEP_REJECT;
            }
        } else {
            // ---- corrector iteration
            float dd = 0.0f;
#pragma unroll
            for (int q = 0; q < SL; q++)
                if (own(q)) dd += dr.p[q].x * dr.p[q].x + dr.p[q].y * dr.p[q].y + dr.q[q].x * dr.q[q].x + dr.q[q].y * dr.q[q].y;
            const float dn = sqrtf(0.5f * grp_sum(dd));
            const bool fail = !oks || !isfinite(dn) || (ph == 4 && dn > K.trust * (1.0f + zpn));
            const bool move = w && !fail;
            float zz = 0.0f;
            zi = 0.0f;
            if (move) {
#pragma unroll
                for (int q = 0; q < SL; q++) {
                    const int j = site(q);
                    const float4 z = at(L::PQ, j);
                    const float2 a = f2add(f2(z.x, z.y), dr.p[q]), b = f2add(f2(z.z, z.w), dr.q[q]);
                    if (own(q)) {
                        at(L::PQ, j) = make_float4(a.x, a.y, b.x, b.y);
                        zz += a.x * a.x + a.y * a.y + b.x * b.x + b.y * b.y;
                        const float2 u = f2add(a, b), v = f2sub(a, b);
                        zi = fmaxf(zi, fmaxf(u.x * u.x + u.y * u.y, v.x * v.x + v.y * v.y));
                    }
                }
            }
            zz = grp_sum(zz);
            zi = 0.5f * sqrtf(grp_max(zi));   // ||(x, y)||_inf
            if (w) {
                P.solves++;
                P.newton++;
                kstep = fmaxf(kstep, kest);
                if (move && dn <= K.eps * (1.0f + sqrtf(0.5f * zz))) {
                    // a converged step whose systems' condition estimate exceeds kappa (0: no
                    // test) is not taken: FP64 continues the path from its last accepted
                    // point (or the end zone's clean checkpoint)
                    verdict = STEP_ACCEPT;
                    if (K.kappa > 0.0f && !(kstep <= K.kappa)) status = NPHC_PATH_HANDOFF_COND;
                } else if (fail || ph + 1 >= 4 + C.max_newton) {
                    verdict = STEP_REJECT;
                } else {
                    ph++;
                }
                if (verdict == STEP_ACCEPT && status == NPHC_PATH_RUNNING) {
#pragma unroll
                    for (int q = 0; q < SL; q++)
                        if (own(q)) {
                            const int j = g + 4 * q;
                            at(L::Z0, j) = at(L::PQ, j);
                            at(L::K1, j) = make_float4(dt.p[q].x, dt.p[q].y, dt.q[q].x, dt.q[q].y);
                        }
                }
            }
        }
        // ---- the step attempt is over
        if (verdict != STEP_GO_ON) {
            bool save = false;
            if (verdict == STEP_ACCEPT && status == NPHC_PATH_RUNNING) status = P.accept(K, C, t1, zi, save);
            else if (verdict == STEP_REJECT) status = P.reject(K, C);
            status = P.budget(C, status);
            if (save) {
#pragma unroll
                for (int q = 0; q < SL; q++)
                    if (own(q)) ck[(g + 4 * q) * slots] = at(L::PQ, g + 4 * q);
            }
            kstep = 0.0f;
            start = status == NPHC_PATH_RUNNING;
            if (!start) {
                const EPView &ep = src.eps(inst);
                const int64_t cnt = ep.count;
                const bool from_ck = P.from_checkpoint(status);
                // (p, q) to x = (p + q) / 2, y = -i (p - q) / 2, in FP64 (halving is exact)
#pragma unroll 1
                for (int q = 0; q < SL; q++)
                    if (own(q)) {
                        const int k = g + 4 * q;
                        const float4 z = from_ck ? ck[k * slots] : at(L::Z0, k);
                        const double pr = 0.5f * z.x, pi = 0.5f * z.y, qr = 0.5f * z.z, qi = 0.5f * z.w;
                        ep.z_re[k * cnt + e] = pr + qr;
                        ep.z_im[k * cnt + e] = pi + qi;
                        ep.z_re[(M + k) * cnt + e] = pi - qi;
                        ep.z_im[(M + k) * cnt + e] = qr - pr;
                    }
                if (g == 0) P.store(ep, e, status);
                e = -1;
            }
        }
    }
}

template <int M>
__global__ void __launch_bounds__(32 * GRP_WARPS, GrpLayout<M>::BLOCKS)
    xy_track_group_kernel(const __grid_constant__ XYSys S, const __grid_constant__ XYCtl C,
                          const EPView ep, const WorkList wl) {
    grp_track_body<M, false>(SingleSrc<XYSys>{S, ep, wl}, C, wl);
}

// The FP32 pass of a batch: every path of every instance of one ring size in one
// persistent launch, pulled from one queue (BatchSrc).
template <int M>
__global__ void __launch_bounds__(32 * GRP_WARPS, GrpLayout<M>::BLOCKS)
    xy_track_group_batch_kernel(const XYSys *__restrict__ sys, const EPView *__restrict__ eps,
                                const int64_t *__restrict__ off, int n,
                                const __grid_constant__ XYCtl C, const WorkList wl) {
    grp_track_body<M, true>(BatchSrc<XYSys>{sys, eps, off, n}, C, wl);
}
