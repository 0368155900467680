// f32_step.cuh -- what the FP32 trackers (xy_track_group.cuh, xy_track_lane.cuh) share: arithmetic
// in pairs (f32x2), compensated sums of pairs, the terms of one site, one path's step control.
#pragma once

#include "xy_track.cuh"

// ------------------------------------------------------------- f32x2 pairs --
// A pair is a complex number (re, im) or two neighbours.  The paired instructions take their
// operands negated, swapped or one half twice at no cost (static instruction counts), so
// f2dup, f2neg and f2i below are free as operands, and a complex product is two instructions.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 f2dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 f2neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __fadd2_rn(a, f2neg(b)); }
__device__ __forceinline__ float2 f2i(float2 a) { return make_float2(-a.y, a.x); }   // i a
__device__ __forceinline__ float2 f2scale(float s, float2 a) { return f2mul(f2dup(s), a); }
__device__ __forceinline__ float f2abs2(float2 a) { return fmaf(a.x, a.x, a.y * a.y); }
// complex a b, conj(a) b, c + a b, c - a b
__device__ __forceinline__ float2 f2cmul(float2 a, float2 b) { return f2fma(f2dup(a.y), f2i(b), f2mul(f2dup(a.x), b)); }
__device__ __forceinline__ float2 f2cmulc(float2 a, float2 b) {
    return f2fma(f2dup(-a.y), f2i(b), f2mul(f2dup(a.x), b));
}
__device__ __forceinline__ float2 f2cfma(float2 a, float2 b, float2 c) {
    return f2fma(f2dup(a.y), f2i(b), f2fma(f2dup(a.x), b, c));
}
__device__ __forceinline__ float2 f2cfms(float2 a, float2 b, float2 c) {
    return f2fma(f2dup(-a.y), f2i(b), f2fma(f2dup(-a.x), b, c));
}

// Square root and reciprocal square root for the light-cone scales and frames (any scale solves
// the same system, and the frame's error of two ulp is the row's own rounding), and a pivot's
// reciprocal with one Newton step: a few instructions where the IEEE forms take thirteen to
// fifteen.  Without flushing: |pivot|^2 beyond 2^126 has a subnormal reciprocal, and a reciprocal
// flushed to 0 stays 0 in the Newton step, sets its unknown to 0 and passes every test of the
// solve.  (A square root flushed to 0 is below the scales' bound of 1.)
__device__ __forceinline__ float f32_sqrt(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float f32_rsqrt(float x) {
    float r;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float f32_recip(float x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(fmaf(-x, r, 1.0f), r, r);
}

// A pair of two-word numbers (EFT, nphc_internal.cuh): the same error-free transformations
// on both halves.
struct ext2 {
    float2 hi, lo;
};

// acc += c v; as ext_acc
__device__ __forceinline__ void acc2(ext2 &acc, float2 c, float2 v) {
    const float2 p = f2mul(c, v);
    const float2 e = f2fma(c, v, f2neg(p));   // the product's rounding error
    const float2 s = f2add(acc.hi, p);
    const float2 bb = f2sub(s, acc.hi);
    const float2 e2 = f2add(f2sub(acc.hi, f2sub(s, bb)), f2sub(p, bb));
    acc.hi = s;
    acc.lo = f2add(acc.lo, f2add(e, e2));
}
// acc += c (v.hi + v.lo); as ext_acc_ext
__device__ __forceinline__ void acc2_ext(ext2 &acc, float c, const ext2 &v) {
    acc2(acc, f2dup(c), v.hi);
    acc.lo = f2fma(f2dup(c), v.lo, acc.lo);
}
// (a.hi + a.lo) + (b.hi + b.lo)
__device__ __forceinline__ ext2 ext2_add(const ext2 &a, const ext2 &b) {
    const float2 s = f2add(a.hi, b.hi);
    const float2 bb = f2sub(s, a.hi);
    const float2 e = f2add(f2sub(a.hi, f2sub(s, bb)), f2sub(b.hi, bb));
    return ext2{s, f2add(e, f2add(a.lo, b.lo))};
}
__device__ __forceinline__ ext2 ext2_scale(float c, const ext2 &a) {   // c a power of two
    return ext2{f2mul(f2dup(c), a.hi), f2mul(f2dup(c), a.lo)};
}
__device__ __forceinline__ ext2 ext2_i(const ext2 &v) { return ext2{f2i(v.hi), f2i(v.lo)}; }
// acc += a b for complex a, b: exact products
__device__ __forceinline__ void acc2_cmul(ext2 &acc, float2 a, float2 b) {
    acc2(acc, f2dup(a.x), b);
    acc2(acc, f2dup(a.y), f2i(b));
}

// The rows (-H_f, -H_g) of one site at (p, q), compensated, from the compensated sums
// U_p, U_q (xy_residual_comp in xy_solve.cuh, with the squares shared:
// x^2 - 1 = B + h, y^2 - 1 = -B + h, B = (p^2 + q^2) / 4, h = G / 2 - 1 / 2, G = p q - 1).
__device__ __forceinline__ void f32_residual_rows(float2 pk, float2 qk, const ext2 &up, const ext2 &uq,
                                                  float s, float hs, float gr, float gi, float2 &rf,
                                                  float2 &rg) {
    const ext2 zero = {f2dup(0.0f), f2dup(0.0f)};
    ext2 d = zero;   // D = q U_p - p U_q, f = i D / 2
    acc2_ext(d, qk.x, up);
    acc2_ext(d, qk.y, ext2_i(up));
    acc2_ext(d, -pk.x, uq);
    acc2_ext(d, -pk.y, ext2_i(uq));
    ext2 G = {f2(-1.0f, 0.0f), f2dup(0.0f)}, B = zero;
    acc2_cmul(G, pk, qk);
    acc2_cmul(B, pk, pk);
    acc2_cmul(B, qk, qk);
    B = ext2_scale(0.25f, B);
    const ext2 nB = {f2neg(B.hi), f2neg(B.lo)};
    const ext2 half = {f2(-0.5f, 0.0f), f2dup(0.0f)};
    const ext2 h = ext2_add(ext2_scale(0.5f, G), half);
    const ext2 X = ext2_add(h, B), Y = ext2_add(h, nB);
    ext2 hf = zero, hg = zero;   // H_f = gomt X + t f ;  H_g = gomt Y + t G
    acc2_ext(hf, gr, X);
    acc2_ext(hf, gi, ext2_i(X));
    acc2_ext(hf, hs, ext2_i(d));
    acc2_ext(hg, gr, Y);
    acc2_ext(hg, gi, ext2_i(Y));
    acc2_ext(hg, s, G);
    rf = f2neg(f2add(hf.hi, hf.lo));
    rg = f2neg(f2add(hg.hi, hg.lo));
}

// The terms of site j at (p, q) = (p_j, q_j) with U_p, U_q (xy_solve.cuh): the scaled light-cone
// frame (g_frame_lc) sb = sp b^, sa = sq a^, the Schur matrix's diagonal entry sjj, and for a
// right-hand side (rf, rg) X, Y (xy_solve.cuh) and the site's own share d = rf - A px - B py.
struct F32Site {
    float2 ah, bh, sb, sa, sjj, Ajj, Bjj;
    float iv, sp, sq;
    __device__ __forceinline__ void rhs(float2 rf, float2 rg, float2 &x, float2 &y, float2 &d) const {
        const float2 c = f2scale(iv, rg);
        const float2 px = f2cmulc(ah, c), py = f2cmulc(bh, c);
        x = f2scale(sp, px);
        y = f2scale(sq, py);
        d = f2cfms(Bjj, py, f2cfms(Ajj, px, rf));
    }
};

// Also -H_t's rows (lc_minus_ht_rows) into htf, htg.  hs = t / 2, hgomt = gamma (1 - t) / 2.
__device__ __forceinline__ F32Site f32_site(float2 p, float2 q, float2 Up, float2 Uq, float s, float hs,
                                            float2 hgomt, float2 gam, float2 &htf, float2 &htg) {
    F32Site v;
    const float2 one = f2(1.0f, 0.0f), a = f2add(p, q), d = f2sub(p, q);
    const float2 D = f2cfms(p, Uq, f2cmul(q, Up));   // f = i D / 2
    htf = f2cfma(gam, f2fma(f2dup(0.25f), f2cmul(a, a), f2neg(one)), f2scale(-0.5f, f2i(D)));
    htg = f2cfma(gam, f2fma(f2dup(-0.25f), f2cmul(d, d), f2neg(one)), f2cfms(p, q, one));
    v.sp = fmaxf(1.0f, f32_sqrt(f2abs2(p)));
    v.sq = fmaxf(1.0f, f32_sqrt(f2abs2(q)));
    const float2 hd = f2cmul(hgomt, d);
    const float2 ra = f2scale(v.sp, f2fma(f2dup(s), q, f2neg(hd))), rb = f2scale(v.sq, f2fma(f2dup(s), p, hd));
    v.iv = f32_rsqrt(f2abs2(ra) + f2abs2(rb));
    v.ah = f2scale(v.iv, ra);
    v.bh = f2scale(v.iv, rb);
    v.sb = f2scale(v.sp, v.bh);
    v.sa = f2scale(v.sq, v.ah);
    const float2 g = f2cmul(hgomt, a);
    v.Ajj = f2scale(v.sp, f2fma(f2dup(-hs), f2i(Uq), g));
    v.Bjj = f2scale(v.sq, f2fma(f2dup(hs), f2i(Up), g));
    v.sjj = f2cfms(v.Bjj, v.ah, f2cmul(v.Ajj, v.bh));
    return v;
}

// ------------------------------------------------------------ step control --
// Time in units of 2^-53, the grid of the doubles in [1/2, 1): 1 - t is exact, and the step
// logic costs no FP64 instruction (67 cycles of a scheduler each, measured, whatever the
// number of lanes).  Steps below one unit (an initial or largest step under 1.1e-16) are one unit: a
// step rounded to 0 would never grow.
typedef long long f32_time;
#define F32_ONE (1ll << 53)
__device__ __forceinline__ f32_time to_f32_time(double t) {   // clamped: beyond 256 no step differs
    return __double2ll_rn(fmin(fmax(t, -256.0), 256.0) * 9007199254740992.0);
}
__device__ __forceinline__ float time_float(f32_time t) { return __ll2float_rn(t) * 1.1102230246251565e-16f; }
__device__ __forceinline__ double time_double(f32_time t) { return __ll2double_rn(t) * 1.1102230246251565e-16; }

struct F32Ctl {   // XYCtl in the trackers' own units
    f32_time h0, hmax, hmin, tend, zone, near_end;
    float rdiv, rband, eps, trust, kappa;
    __device__ __forceinline__ explicit F32Ctl(const XYCtl &C)
        : h0(max(to_f32_time(C.h0), (f32_time)1)), hmax(max(to_f32_time(C.hmax), (f32_time)1)),
          hmin(max(to_f32_time(C.hmin), (f32_time)1)),
          tend(to_f32_time(C.t_end)), zone(to_f32_time(CRAWL_ZONE)), near_end(to_f32_time(NEAR_END)),
          rdiv((float)C.rdiv), rband((float)(C.rdiv * (1.0 + RDIV_BAND))), eps((float)C.eps),
          trust((float)C.trust), kappa((float)C.kappa) {}
};

// One path's step control: the rules of xy_track.cuh (track_body) for the FP32 pass.
struct F32Step {
    f32_time t, h, hacc, tck, hck, tmark;
    float zlast;
    int clean, since, run, rejects, attempts, steps, solves, newton;
    bool have_ck, far;

    __device__ __forceinline__ void start(f32_time t0, f32_time h0) {
        t = t0;
        h = hacc = h0;
        tmark = F32_ONE - t0;
        tck = hck = 0;
        zlast = 0.0f;
        clean = since = run = rejects = attempts = 0;
        have_ck = far = false;
    }
    // a path heading out takes steps of at most KAPPA_FAR (1 - t)
    __device__ __forceinline__ void cap() {
        if (far) h = min(h, (f32_time)__umul64hi((unsigned long long)(F32_ONE - t),
                                                 (unsigned long long)(KAPPA_FAR * 18446744073709551616.0)));
    }
    // length and end of the step
    __device__ __forceinline__ void len(const F32Ctl &K, f32_time &hh, f32_time &t1) const {
        const bool last = t + h >= K.tend;
        t1 = last ? K.tend : t + h;
        hh = last ? K.tend - t : h;
    }
    // The step to t1 is accepted at ||z||_inf = zi; returns the path's status.  save: the
    // point becomes the hand-off checkpoint (the last clean point of the end zone: accepted,
    // with the step before it accepted too).
    __device__ __forceinline__ int accept(const F32Ctl &K, const XYCtl &C, f32_time t1, float zi, bool &save) {
        int status = NPHC_PATH_RUNNING;
        attempts++;
        clean = rejects == 0 ? clean + 1 : 1;
        t = t1;
        const f32_time left = F32_ONE - t;
        const bool zone = left < K.zone;
        far = zone && zi > (float)FAR_NORM && zi > (float)FAR_GROWTH * zlast;
        zlast = zi;
        steps++;
        rejects = 0;
        hacc = h;
        if (++run >= C.grow_after) {
            run = 0;
            h = min(2 * h, K.hmax);
        }
        if (zi > K.rdiv)   // marginal crossings close to t = 1 are FP64's to judge
            status = (C.handoff && left < K.near_end && zi <= K.rband) ? NPHC_PATH_HANDOFF : NPHC_PATH_DIVERGED;
        else if (t >= K.tend)
            status = NPHC_PATH_REACHED;
        save = C.handoff && (clean >= 2 || !have_ck) && status == NPHC_PATH_RUNNING && zone;
        if (save) {
            tck = t;
            hck = hacc;
            have_ck = true;
        }
        // crawl test near t = 1: 1 - t must at least halve every crawl_steps accepted steps
        if (status == NPHC_PATH_RUNNING && C.crawl_steps > 0 && zone) {
            if (++since >= C.crawl_steps) {
                if (2 * left > tmark) status = C.handoff ? NPHC_PATH_HANDOFF : NPHC_PATH_MIN_STEP;
                tmark = left;
                since = 0;
            }
        } else {
            tmark = left;
            since = 0;
        }
        return status;
    }
    __device__ __forceinline__ int reject(const F32Ctl &K, const XYCtl &C) {
        attempts++;
        run = 0;
        rejects++;
        h >>= 1;
        if (h < K.hmin) return C.handoff ? NPHC_PATH_HANDOFF : NPHC_PATH_MIN_STEP;
        return C.handoff && rejects >= 10 ? NPHC_PATH_HANDOFF : NPHC_PATH_RUNNING;
    }
    // the step budget, after an attempt that left the path running
    __device__ __forceinline__ int budget(const XYCtl &C, int status) const {
        if (status != NPHC_PATH_RUNNING || attempts < C.max_steps) return status;
        return C.handoff ? NPHC_PATH_HANDOFF : NPHC_PATH_STEP_BUDGET;
    }
    // what the endpoint arrays get besides the point (the checkpoint's, for a path handed off
    // after one)
    __device__ __forceinline__ bool from_checkpoint(int status) const {
        return have_ck && (status == NPHC_PATH_HANDOFF || status == NPHC_PATH_HANDOFF_COND);
    }
    __device__ __forceinline__ void store(const EPView &ep, int64_t e, int status) const {
        const bool handed = status == NPHC_PATH_HANDOFF || status == NPHC_PATH_HANDOFF_COND;
        const bool ck = handed && have_ck;
        ep.t[e] = time_double(ck ? tck : t);
        ep.h[e] = time_double(ck ? hck : (handed ? hacc : h));
        ep.status[e] = status;
        ep.steps[e] = steps;
        ep.solves[e] = solves;
        ep.newton[e] = newton;
    }
};
