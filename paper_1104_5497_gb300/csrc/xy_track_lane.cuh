// xy_track_lane.cuh -- the FP32 tracker of the XY ring with one path per thread, for launches with
// paths for every lane of the chip (the method: xy_track.cuh; the linear algebra: xy_solve.cuh).
//
// Bound by latency at the residency that a matrix per thread leaves (28 KB of shared memory per
// warp at M = 9: seven warps per SM), so it is written for few instructions and short waits:
//   * arithmetic in pairs (fma.rn.f32x2, f32_step.cuh): complex times real, the two halves of a
//     complex product, and the compensated sums;
//   * the augmented matrix [S | T | R] in shared memory, two neighbouring columns to a 128-bit
//     word, interleaved across the threads (entry (i, pair c) at [(i NPC + c) 32 + lane]): the
//     rank-one update of LU is a load, the paired FMAs and a store for two entries;
//   * every thread is in its own phase (an RK4 stage or a corrector iteration); the warp runs
//     whichever kind of solve more of its paths wait for (a corrector solve costs about twice
//     a predictor's).  In lockstep every step took the slowest path's three corrector solves
//     where a path needs 1.7;
//   * what a step keeps in global scratch (L2, 600 cycles away) is read LANE_CHUNK sites ahead of
//     its use, the first of them before the back substitution; an accepted step's copies and
//     the next step's first point are one pass;
//   * step control on integer time (f32_step.cuh).
// The elimination and build loops are rolled: the kernel is 4,000 instructions, and with
// another 1,000 (everything unrolled) it waited a quarter of the time for instructions, 73 -> 90 ms.
// Measured (GB300, 262,144 paths of N = 10): 109 ms for a lockstep kernel with a path per thread
// and scalar arithmetic, 73 ms here (issue slots 32% used, the rest waits on shared memory and on
// results); N = 11 154 -> 93.  Up to M = 10 (xy_inst.cu).
#pragma once

#include "f32_step.cuh"

constexpr int LANE_CHUNK = 3;   // sites whose scratch words are in flight together (registers: 15 each)

template <int M>
struct LaneLayout {   // shared memory per thread, in float4 (16 bytes) but R
    static constexpr int NPC = (M + 2) / 2;              // column pairs of [S | T] (M even: with R)
    static constexpr int PQ = M * NPC;                   // evaluation point (p_k, q_k)
    static constexpr int TOTAL4 = PQ + M;
    static constexpr bool RSEP = M % 2 == 1;             // R in a column of its own (float2)
    static constexpr size_t BYTES = sizeof(float4) * TOTAL4 + (RSEP ? sizeof(float2) * M : 0);
    static constexpr int JROW = (M + 4) / 4 * 4;         // a row of the coupling table (J_k1 .. J_kM, J_kN)
};

template <int M>
constexpr size_t lane_smem_per_block(bool batch) {
    return 32 * LaneLayout<M>::BYTES + (batch ? 0 : sizeof(float) * M * LaneLayout<M>::JROW);
}

// Row k of the couplings: the block's table in shared memory, or (batch) the instance's.
template <int M, bool BATCH>
struct LaneJ {
    const float *base;
    static constexpr int ROW = BATCH ? NPHC_JSTRIDE : LaneLayout<M>::JROW;
    __device__ __forceinline__ void row(int k, float (&c)[LaneLayout<M>::JROW]) const {
        const float4 *r = reinterpret_cast<const float4 *>(base + k * ROW);
#pragma unroll
        for (int i = 0; i < LaneLayout<M>::JROW / 4; i++) {
            const float4 v = r[i];
            c[4 * i] = v.x;
            c[4 * i + 1] = v.y;
            c[4 * i + 2] = v.z;
            c[4 * i + 3] = v.w;
        }
    }
};

// One thread's shared memory.
template <int M>
struct LaneMem {
    using L = LaneLayout<M>;
    float4 *a;    // this thread's word 0
    float2 *r;    // its R column (M odd)
    __device__ __forceinline__ float4 &A(int i, int c) const { return a[(i * L::NPC + c) * 32]; }   // column pair c
    __device__ __forceinline__ float2 &col(int i, int c) const {   // one column
        return reinterpret_cast<float2 *>(&A(i, c >> 1))[c & 1];
    }
    __device__ __forceinline__ float2 &R(int i) const { return L::RSEP ? r[i * 32] : col(i, M + 1); }
    __device__ __forceinline__ float4 &pq(int k) const { return a[(L::PQ + k) * 32]; }
};

// Per-thread vectors in global scratch: a word of site k at [k stride].
struct LaneVec {
    float4 *p;
    int64_t stride;
    __device__ __forceinline__ float4 &at(int k) const { return p[k * stride]; }
};

// One solve of H_z(z, t) d = r at PQ (see xy_solve and xy_residual_comp in xy_solve.cuh): r = -H_t
// (T), and with corr (uniform over the warp) r = -H (R, compensated) too.  Hands site k's (dp, dq)
// to post(i, k, T's dp, dq, R's dp, dq), k = 0 .. M - 1 (R is meaningless without corr), i its place
// in the chunk that post.fetch(i, k) has loaded and post.next() handed over.  XT, XR, FR: scratch for the sites' X, Y of either side and frames, from the build to the recovery.
// Returns false when the system is singular or the result is not finite.
template <int M, bool BATCH, class Post>
__device__ __forceinline__ bool lane_solve(const LaneMem<M> &m, const LaneJ<M, BATCH> &J, const LaneVec &XT,
                                           const LaneVec &XR, const LaneVec &FR, float s, float omt,
                                           float2 gam, bool corr, float &kest, Post &post) {
    using L = LaneLayout<M>;
    const float2 hgomt = f2scale(0.5f * omt, gam);
    const float hs = 0.5f * s;
    float2 p[M], q[M];
#pragma unroll
    for (int k = 0; k < M; k++) {
        const float4 z = m.pq(k);
        p[k] = f2(z.x, z.y);
        q[k] = f2(z.z, z.w);
    }
    if (corr) {
        // -H rows: the f row waits in R(k), the g row in T's place (both are read back when
        // column k is built, before anything is written there)
        const float gr = __fmul_rn(omt, gam.x), gi = __fmul_rn(omt, gam.y);
#pragma unroll 1
        for (int k = 0; k < M; k++) {
            const float4 z = m.pq(k);
            float c[L::JROW];
            J.row(k, c);
            ext2 up = {f2(c[M], 0.0f), f2dup(0.0f)}, uq = up;
#pragma unroll
            for (int l = 0; l < M; l++) {   // J_kk = 0 adds exact zeros
                acc2(up, f2dup(c[l]), p[l]);
                acc2(uq, f2dup(c[l]), q[l]);
            }
            float2 rf, rg;
            f32_residual_rows(f2(z.x, z.y), f2(z.z, z.w), up, uq, s, hs, gr, gi, rf, rg);
            m.R(k) = rf;
            m.col(k, M) = rg;
        }
    }

    // ---- build S column by column; right-hand sides as sums over the columns:
    // b_k = d_k - (i t / 2) (q_k sum_j J_kj X_j - p_k sum_j J_kj Y_j)
    float2 sxT[M], syT[M], sxR[M], syR[M];
#pragma unroll
    for (int k = 0; k < M; k++) sxT[k] = syT[k] = sxR[k] = syR[k] = f2dup(0.0f);
#pragma unroll 1
    for (int j = 0; j < M; j++) {
        const float4 z = m.pq(j);
        float c[L::JROW];   // J is symmetric: row j is column j
        J.row(j, c);
        float2 up = f2(c[M], 0.0f), uq = up;
#pragma unroll
        for (int l = 0; l < M; l++) {
            up = f2fma(f2dup(c[l]), p[l], up);
            uq = f2fma(f2dup(c[l]), q[l], uq);
        }
        float2 htf, htg, xT, yT, d, xR, yR;
        const F32Site v = f32_site(f2(z.x, z.y), f2(z.z, z.w), up, uq, s, hs, hgomt, gam, htf, htg);
        v.rhs(htf, htg, xT, yT, d);
        if (corr) {
            const float2 rf = m.R(j), rg = m.col(j, M);
            float2 dR;
            v.rhs(rf, rg, xR, yR, dR);
            m.R(j) = dR;   // the diagonal's own terms wait in the right-hand sides' columns
            XR.at(j) = make_float4(xR.x, xR.y, yR.x, yR.y);
        }
        m.col(j, M) = d;
        XT.at(j) = make_float4(xT.x, xT.y, yT.x, yT.y);
        FR.at(j) = make_float4(v.sb.x, v.sb.y, v.sa.x, v.sa.y);
        const float2 cb = f2scale(hs, f2i(v.sb)), ca = f2scale(hs, f2i(v.sa));
#pragma unroll
        for (int k = 0; k < M; k++) {   // S_kj = J_kj (q_k cb + p_k ca)
            const float2 ck = f2dup(c[k]);
            m.col(k, j) = f2mul(ck, f2cfma(ca, p[k], f2cmul(cb, q[k])));
            sxT[k] = f2fma(ck, xT, sxT[k]);
            syT[k] = f2fma(ck, yT, syT[k]);
            if (corr) {
                sxR[k] = f2fma(ck, xR, sxR[k]);
                syR[k] = f2fma(ck, yR, syR[k]);
            }
        }
        m.col(j, j) = v.sjj;
    }
#pragma unroll
    for (int k = 0; k < M; k++) {
        const float2 ip = f2scale(hs, f2i(p[k])), iq = f2scale(-hs, f2i(q[k]));
        m.col(k, M) = f2cfma(ip, syT[k], f2cfma(iq, sxT[k], m.col(k, M)));
        if (corr) m.R(k) = f2cfma(ip, syR[k], f2cfma(iq, sxR[k], m.R(k)));
    }

    // ---- LU with partial pivoting; the pivots' reciprocals on the diagonal
    bool ok = true;
    float umax = 0.0f, umin = INFINITY;   // of |U_kk|^2
#pragma unroll 1
    for (int k = 0; k < M; k++) {
        const int n = M - k;   // active rows k .. M - 1, relative index i = 0 .. n - 1
        const LaneMem<M> mk{m.a + k * L::NPC * 32, m.r + k * 32};   // mk.A(i, c) = row k + i
        float2 v[M];
        unsigned key = 0;   // the largest |a|^2, its row in the low four bits (ties: the lowest row)
#pragma unroll
        for (int i = 0; i < M; i++) {
            if (i >= n) break;
            v[i] = mk.col(i, k);
            key = max(key, (__float_as_uint(f2abs2(v[i])) & ~15u) | (unsigned)(15 - i));
        }
        const int pr = 15 - (int)(key & 15u);
        const float2 piv = mk.col(pr, k);
        const float best = f2abs2(piv);
        ok = ok && best > 0.0f;
        umax = fmaxf(umax, best);
        umin = fminf(umin, best);
        const float2 ip = f2scale(f32_recip(best), f2(piv.x, -piv.y));
#pragma unroll
        for (int i = 1; i < M; i++) {   // multipliers of rows 1 .. n - 1 after the swap
            if (i >= n) break;
            v[i] = f2cmul(i == pr ? v[0] : v[i], ip);
        }
#pragma unroll 1
        for (int c = (k + 1) >> 1; c < L::NPC; c++) {
            const float4 a0 = mk.A(0, c), ap = mk.A(pr, c);
            mk.A(pr, c) = a0;
            mk.A(0, c) = ap;
            const float2 u = f2(ap.x, ap.y), w = f2(ap.z, ap.w);
#pragma unroll
            for (int i = 1; i < M; i++) {
                if (i >= n) break;
                const float4 x = mk.A(i, c);
                const float2 y0 = f2cfms(v[i], u, f2(x.x, x.y)), y1 = f2cfms(v[i], w, f2(x.z, x.w));
                mk.A(i, c) = make_float4(y0.x, y0.y, y1.x, y1.y);
            }
        }
        if (L::RSEP && corr) {
            const float2 a0 = mk.R(0), ap = mk.R(pr);
            mk.R(pr) = a0;
            mk.R(0) = ap;
#pragma unroll
            for (int i = 1; i < M; i++) {
                if (i >= n) break;
                mk.R(i) = f2cfms(v[i], ap, mk.R(i));
            }
        }
        mk.col(0, k) = ip;   // after the swap of the pair that holds column k too
    }
    kest = sqrtf(umax / umin);

    // what the recovery reads from global scratch, one chunk of sites ahead
    float4 gf[LANE_CHUNK], gx[LANE_CHUNK], gr[LANE_CHUNK];
    auto fetch = [&](int j0) {
#pragma unroll
        for (int i = 0; i < LANE_CHUNK; i++) {
            const int j = j0 + i;
            if (j >= M) break;
            gf[i] = FR.at(j);
            gx[i] = XT.at(j);
            if (corr) gr[i] = XR.at(j);
            else post.fetch(i, j);
        }
    };
    fetch(0);

    // ---- back substitution U x = b, in place in T's column, then in R's
#pragma unroll 1
    for (int h = 0; h < (corr ? 2 : 1); h++) {
        float2 x[M];
#pragma unroll
        for (int k = M - 1; k >= 0; k--) {
            float2 b = h ? m.R(k) : m.col(k, M);
#pragma unroll
            for (int c = M - 1; c > k; c--) b = f2cfms(m.col(k, c), x[c], b);
            x[k] = f2cmul(b, m.col(k, k));
            if (h) m.R(k) = x[k];
            else m.col(k, M) = x[k];
        }
    }

    // ---- back to (dp, dq) = (X + sp b^ s, Y - sq a^ s)
    float chk = 0.0f;
#pragma unroll 1
    for (int j0 = 0; j0 < M; j0 += LANE_CHUNK) {
        float4 cf[LANE_CHUNK], cx[LANE_CHUNK], cr[LANE_CHUNK];
#pragma unroll
        for (int i = 0; i < LANE_CHUNK; i++) {
            cf[i] = gf[i];
            cx[i] = gx[i];
            cr[i] = gr[i];
        }
        post.next();
        fetch(j0 + LANE_CHUNK);
#pragma unroll
        for (int i = 0; i < LANE_CHUNK; i++) {
            const int j = j0 + i;
            if (j >= M) break;
            const float4 f = cf[i], x = cx[i];
            const float2 sb = f2(f.x, f.y), sa = f2(f.z, f.w), sT = m.col(j, M);
            const float2 pT = f2cfma(sb, sT, f2(x.x, x.y)), qT = f2cfms(sa, sT, f2(x.z, x.w));
            chk += f2abs2(pT) + f2abs2(qT);
            float2 pR = f2dup(0.0f), qR = pR;
            if (corr) {
                const float4 r = cr[i];
                const float2 sR = m.R(j);
                pR = f2cfma(sb, sR, f2(r.x, r.y));
                qR = f2cfms(sa, sR, f2(r.z, r.w));
                chk += f2abs2(pR) + f2abs2(qR);
            }
            post(i, j, pT, qT, pR, qR);
        }
    }
    return ok && isfinite(chk);
}

// What a solve's recovery does with site j's step, in the phase the path is in (w: it takes part):
// an RK4 stage adds to the RK4 sum and moves on to the next stage's point, a corrector
// iteration moves the point and keeps dz/dt.
template <int M>
struct LanePost {
    const LaneMem<M> &m;
    const LaneVec &Z0, &K1, &AC;
    bool w, corr;
    int ph;
    float c;                    // the next point is z0 + c k (phase 3: z0 + c (sum + k))
    float dd, zz, zi;           // ||d||^2, ||z||^2, max |p +- q|^2
    float4 gz[LANE_CHUNK], go[LANE_CHUNK], cz[LANE_CHUNK], co[LANE_CHUNK];
    __device__ __forceinline__ void fetch(int i, int j) {
        gz[i] = Z0.at(j);
        go[i] = (ph == 1 ? K1 : AC).at(j);
    }
    __device__ __forceinline__ void next() {
#pragma unroll
        for (int i = 0; i < LANE_CHUNK; i++) {
            cz[i] = gz[i];
            co[i] = go[i];
        }
    }
    __device__ __forceinline__ void operator()(int i, int j, float2 pT, float2 qT, float2 pR, float2 qR) {
        if (!w) return;
        float2 a, b;
        if (corr) {
            const float4 z = m.pq(j);
            a = f2add(f2(z.x, z.y), pR);
            b = f2add(f2(z.z, z.w), qR);
            AC.at(j) = make_float4(pT.x, pT.y, qT.x, qT.y);
            dd += f2abs2(pR) + f2abs2(qR);
            zi = fmaxf(zi, fmaxf(f2abs2(f2add(a, b)), f2abs2(f2sub(a, b))));
        } else {
            const float4 z = cz[i], o = co[i];
            const float f = ph == 3 ? 1.0f : 2.0f;
            const float2 sp = f2fma(f2dup(f), pT, f2(o.x, o.y)), sq = f2fma(f2dup(f), qT, f2(o.z, o.w));
            a = f2fma(f2dup(c), ph == 3 ? sp : pT, f2(z.x, z.y));
            b = f2fma(f2dup(c), ph == 3 ? sq : qT, f2(z.z, z.w));
            AC.at(j) = make_float4(sp.x, sp.y, sq.x, sq.y);
        }
        m.pq(j) = make_float4(a.x, a.y, b.x, b.y);
        zz += f2abs2(a) + f2abs2(b);
    }
};

template <int M, bool BATCH, class Src>
__device__ __forceinline__ void lane_track_body(const Src &src, const XYCtl &C, const WorkList &wl) {
    using L = LaneLayout<M>;
    extern __shared__ __align__(16) unsigned char lane_raw[];
    const int lane = threadIdx.x;   // one warp per block
    float4 *const words = reinterpret_cast<float4 *>(lane_raw);
    const LaneMem<M> mem{words + lane, reinterpret_cast<float2 *>(words + 32 * L::TOTAL4) + lane};
    float *const jtab = reinterpret_cast<float *>(lane_raw + 32 * L::BYTES);
    LaneJ<M, BATCH> J{BATCH ? src.sys(0).Jf : jtab};
    if (!BATCH) {
        const float *Jf = src.sys(0).Jf;
        for (int i = lane; i < M * L::JROW; i += 32) jtab[i] = Jf[i / L::JROW * NPHC_JSTRIDE + i % L::JROW];
    }
    // a finite point for lanes that get no path (they still run the arithmetic)
#pragma unroll 1
    for (int k = 0; k < M; k++) mem.pq(k) = make_float4(1.0f, 0.0f, 1.0f, 0.0f);
    __syncwarp();
    const int64_t nth = wl.state_threads, gtid = (int64_t)blockIdx.x * 32 + lane;
    float4 *const st = reinterpret_cast<float4 *>(wl.state) + gtid;
    // accepted point, dz/dt there, RK4 sum (in corrector solves dz/dt), hand-off checkpoint; the
    // solve's scratch (the trackers' scratch holds eight such vectors per thread)
    const LaneVec Z0{st, nth}, K1{st + M * nth, nth}, AC{st + 2 * M * nth, nth}, CK{st + 3 * M * nth, nth};
    const LaneVec XT{st + 4 * M * nth, nth}, XR{st + 5 * M * nth, nth}, FR{st + 6 * M * nth, nth};
    const int64_t total = src.total();
    const F32Ctl K(C);
    int64_t e = -1;   // entry; -1 idle, -2 drained
    int inst = 0;     // its instance (batches)
    int ph = 1;       // phase: 1 .. 3 RK4 stages, 4 .. corrector
    F32Step P;
    P.start(0, 0);
    bool bad = false, start = false, take = false, save = false;
    float zpn = 0.0f, kstep = 0.0f;
    float2 gam = f2((float)src.sys(0).gre, (float)src.sys(0).gim);

#pragma unroll 1
    for (;;) {
        // ---- hand new entries to idle lanes
        const unsigned need = __ballot_sync(0xffffffffu, e == -1);
        if (need) {
            unsigned long long base = 0;
            const int leader = __ffs(need) - 1;
            if (lane == leader) base = atomicAdd(wl.queue, (unsigned long long)__popc(need));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (e == -1) {
                const int64_t i = (int64_t)base + __popc(need & ((1u << lane) - 1u));
                if (i >= total) e = -2;
                else src.take(i, inst, e);   // -1 (skipped) if the debug build rejects it
                if (e >= 0) {
                    if (BATCH) {
                        J.base = src.sys(inst).Jf;
                        gam = f2((float)src.sys(inst).gre, (float)src.sys(inst).gim);
                    }
                    P.steps = P.solves = P.newton = 0;
                    kstep = 0.0f;
                    bad = false;
                    const int64_t path = src.eps(inst).path[e];
                    const cx<float> cg = {gam.x, gam.y}, ig = crecip(cg);
#pragma unroll 1
                    for (int k = 0; k < M; k++) {
                        const float *Jk = J.base + k * J.ROW;
                        float u = Jk[M], v = 0.0f;
#pragma unroll 1
                        for (int l = 0; l < M; l++) {
                            const float jl = Jk[l];
                            u += ((path >> l) & 1) ? -jl : jl;
                            v += ((path >> (M + l)) & 1) ? -jl : jl;
                        }
                        const float x = ((path >> k) & 1) ? -1.0f : 1.0f;
                        const float y = ((path >> (M + k)) & 1) ? -1.0f : 1.0f;
                        cx<float> rf, rg;
                        minus_ht_rows<float>(cx<float>{x, 0.0f}, cx<float>{y, 0.0f}, cx<float>{u, 0.0f},
                                             cx<float>{v, 0.0f}, cg, rf, rg);
                        const cx<float> dx = cscale(0.5f * x, cmul(ig, rf)), dy = cscale(0.5f * y, cmul(ig, rg));
                        Z0.at(k) = make_float4(x, y, x, -y);   // p = x + i y, q = x - i y
                        K1.at(k) = make_float4(dx.re - dy.im, dx.im + dy.re, dx.re + dy.im, dx.im - dy.re);
                    }
                    P.start(0, K.h0);
                    start = true;
                }
            }
        }
        if (__all_sync(0xffffffffu, e < 0)) break;

        // ---- a new attempt: its first stage's point z0 + h/2 k1.  An accepted step's copies ride along.
        const bool act = e >= 0;
        f32_time hh, t1;
        if (start) P.cap();
        P.len(K, hh, t1);
        const float hr = time_float(hh);
        if (start) {
            const float2 c = f2dup(0.5f * hr);
#pragma unroll 3
            for (int k = 0; k < M; k++) {
                const float4 d = (take ? AC : K1).at(k);
                float4 z;
                if (take) {
                    z = mem.pq(k);
                    Z0.at(k) = z;
                    K1.at(k) = d;
                    if (save) CK.at(k) = z;
                } else {
                    z = Z0.at(k);
                }
                const float2 a = f2fma(c, f2(d.x, d.y), f2(z.x, z.y)), b = f2fma(c, f2(d.z, d.w), f2(z.z, z.w));
                mem.pq(k) = make_float4(a.x, a.y, b.x, b.y);
            }
            ph = 1;
            bad = start = take = save = false;
        }

        // ---- which solve runs now, and for whom
        const bool wants_c = act && ph >= 4;
        const int nc = __popc(__ballot_sync(0xffffffffu, wants_c));
        const int np = __popc(__ballot_sync(0xffffffffu, act && !wants_c));
        const bool corr = nc > 0 && 2 * nc >= np;
        const bool w = act && wants_c == corr;
        const f32_time te = ph < 3 ? P.t + hh / 2 : t1;
        LanePost<M> post{mem, Z0, K1, AC, w, corr, ph, ph == 1 ? 0.5f * hr : ph == 2 ? hr : hr * (1.0f / 6.0f),
                         0.0f, 0.0f, 0.0f};
        float kest;
        const bool oks = lane_solve<M, BATCH>(mem, J, XT, XR, FR, time_float(te), time_float(F32_ONE - te), gam,
                                              corr, kest, post);
        if (!w) continue;
        int verdict = STEP_GO_ON, status = NPHC_PATH_RUNNING;
        float zi = 0.0f;
        P.solves++;
        kstep = fmaxf(kstep, kest);
        if (!corr) {
            bad = bad || !oks;
            zpn = sqrtf(0.5f * post.zz);   // ||(x, y)||_2 of the predicted point
            if (++ph == 4 && bad) verdict = STEP_REJECT;
        } else {
            P.newton++;
            const float dn = sqrtf(0.5f * post.dd);
            zi = 0.5f * sqrtf(post.zi);    // ||(x, y)||_inf
            const bool fail = !oks || !isfinite(dn) || (ph == 4 && dn > K.trust * (1.0f + zpn));
            if (!fail && dn <= K.eps * (1.0f + sqrtf(0.5f * post.zz))) {
                // a converged step whose systems' condition estimate exceeds kappa (0: no test) is
                // not taken: FP64 continues the path from its last accepted point (or the
                // end zone's clean checkpoint)
                verdict = STEP_ACCEPT;
                if (K.kappa > 0.0f && !(kstep <= K.kappa)) status = NPHC_PATH_HANDOFF_COND;
            } else if (fail || ph + 1 >= 4 + C.max_newton) {
                verdict = STEP_REJECT;
            } else {
                ph++;
            }
        }
        if (verdict == STEP_GO_ON) continue;

        // ---- the step attempt is over
        take = verdict != STEP_REJECT && status == NPHC_PATH_RUNNING;
        if (verdict == STEP_ACCEPT && take) status = P.accept(K, C, t1, zi, save);
        else if (verdict == STEP_REJECT) status = P.reject(K, C);
        status = P.budget(C, status);
        kstep = 0.0f;
        start = status == NPHC_PATH_RUNNING;
        if (!start) {
            const EPView &ep = src.eps(inst);
            const int64_t cnt = ep.count;
            const bool from_ck = P.from_checkpoint(status) && !save;   // save: the checkpoint is PQ itself
            const bool from_pq = take || (P.from_checkpoint(status) && save);
            // (p, q) to x = (p + q) / 2, y = -i (p - q) / 2, in FP64 (halving is exact)
#pragma unroll 1
            for (int k = 0; k < M; k++) {
                const float4 z = from_ck ? CK.at(k) : from_pq ? mem.pq(k) : Z0.at(k);
                const double pr = 0.5f * z.x, pi = 0.5f * z.y, qr = 0.5f * z.z, qi = 0.5f * z.w;
                ep.z_re[k * cnt + e] = pr + qr;
                ep.z_im[k * cnt + e] = pi + qi;
                ep.z_re[(M + k) * cnt + e] = pi - qi;
                ep.z_im[(M + k) * cnt + e] = qr - pr;
            }
            P.store(ep, e, status);
            e = -1;
            take = save = false;
        }
    }
}

template <int M>
__global__ void __launch_bounds__(32)
    xy_track_lane_kernel(const __grid_constant__ XYSys S, const __grid_constant__ XYCtl C,
                         const EPView ep, const WorkList wl) {
    lane_track_body<M, false>(SingleSrc<XYSys>{S, ep, wl}, C, wl);
}

// The FP32 pass of a batch: every path of every instance of one ring size in one
// persistent launch, pulled from one queue (BatchSrc).
template <int M>
__global__ void __launch_bounds__(32)
    xy_track_lane_batch_kernel(const XYSys *__restrict__ sys, const EPView *__restrict__ eps,
                               const int64_t *__restrict__ off, int n,
                               const __grid_constant__ XYCtl C, const WorkList wl) {
    lane_track_body<M, true>(BatchSrc<XYSys>{sys, eps, off, n}, C, wl);
}
