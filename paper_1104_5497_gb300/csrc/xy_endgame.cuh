// xy_endgame.cuh -- FP64 work at t = 1 on the endpoints of the XY ring:
//   refinement: Newton's method on P to full double precision (section "Numerical
//     Polynomial Homotopy Continuation Method" refines every endpoint to machine
//     precision before certifying it), with P evaluated by exact products and
//     compensated sums (at ||z|| >> 1 the terms of P are ~||z||^2, and a plain sum's
//     rounding would limit the refinement and inflate beta);
//   the solution tolerance Delta_sol on ||P(z)||_inf;
//   alpha-theory certification (the alphaCertified step of the same section):
//     beta = ||DP^-1 P||_2, gamma <= ||DP^-1||_F ||D^2 P / 2|| (P is quadratic, so
//     D^k P = 0 for k >= 3 and Smale's gamma is ||DP^-1 D^2P/2|| exactly), certified when
//     alpha = beta gamma < (13 - 3 sqrt 17) / 4; real when z and Re z share their zero
//     (alpha < 0.03 and ||Im z|| < 1 / (20 gamma)) and the test passes at Re z (a real
//     point of a real system: Newton's iterates stay real), otherwise non-real when
//     ||z - conj z|| > 2 (beta(z) + beta(conj z)), i.e. ||Im z|| > 2 beta, else undecided;
//   classification of real stationary points (introduction and section "A First
//     Application"): theta_k = atan2(s_k, c_k) in (-pi, pi], the Hessian of
//     V = sum_{i<j} J_ij (1 - cos(theta_i - theta_j)) in theta_1..theta_M, its number of
//     negative eigenvalues (cyclic Jacobi), and V.
//
// Linear algebra at t = 1 (the structure of xy_solve.cuh): in the unitary per-site frame
// W, (dx_j, dy_j) = conj(a^_j, b^_j) q_j + (b^_j, -a^_j) s_j, the Jacobian becomes
//   DP W = [[C, S], [D, 0]],   D = diag(nu_j), nu_j = |(a_j, b_j)| = 1 / iv_j,
//   C_kj = A_kj conj(a^_j) + B_kj conj(b^_j),  S_kj = A_kj b^_j - B_kj a^_j,
// (A, B: derivatives of the gradient rows in c and s) with inverse
//   [[0, D^-1], [S^-1, -S^-1 C D^-1]],
// so a solve costs one M x M system, and, W being unitary,
//   ||DP^-1||_F^2 = sum_j iv_j^2 + ||S^-1||_F^2 + ||S^-1 C D^-1||_F^2
// needs only 2M triangular solves after one factorisation of S.  The XY ring's kernel is
// xy_refine_group.cuh (four lanes per endpoint), a quadratic system's quad_warp.cuh (one
// endpoint per warp); this file holds what they share, the classification and the adjoint.
//
// The refinement certifies the iterate whose Newton correction met the tolerance, from
// the factorisation of that iteration, and outputs its Newton iterate.
#pragma once

#include "nphc_internal.cuh"

// The certification threshold: half of Smale's (13 - 3 sqrt 17) / 4.  alphaCertified
// decides in exact arithmetic; an FP64 test keeps a factor of two so that rounding cannot
// carry a point near a singular solution set across the constant (on the N = 4 ring a
// point of the positive-dimensional family reached alpha = 0.115 < 0.158).
#define NPHC_ALPHA_CERT (0.5 * (13.0 - 3.0 * sqrt(17.0)) / 4.0)

// shortcut = 1: entries handed off by the FP32 pass close to t = 1 are refined at t = 1
// directly (Newton on P from the hand-off point: for a path to a nonsingular solution xi,
// z(t) = xi + (1 - t) z'(1) + ..., so the point is already in xi's Newton basin).  The
// first Newton correction must stay below SHORTCUT_TRUST (1 + ||z||); an entry that
// certifies becomes NPHC_PATH_REACHED, any other entry is left untouched.
#define SHORTCUT_TRUST 1e-2

// Classification: theta, V, the Hessian's eigenvalues (cyclic Jacobi) for every entry of class
// NPHC_END_REAL, or the listed ones; the other entries' outputs are the caller's defaults.
// Four lanes per point, eight points per warp, bound by the FP64 pipe (67 cycles of a scheduler
// per instruction, whatever the number of lanes): a sweep visits the pairs (p, q) in rounds of
// disjoint ones (the circle method), so that the lanes compute the rotations of a round side
// by side and share the rows and columns they touch.  One point per thread ran every rotation's
// square roots and divisions and 8 M updates on one lane: 1.20 ms for the 1,170 points of a ring
// of N = 10, now 0.32 (the FP64 chain of one point).
#define CLS_PATHS 8
template <int M>
struct ClsLayout {   // doubles per point ([index * 8 + point])
    static constexpr int N = M + 1;
    static constexpr int ME = M + M % 2;       // players of the circle method (one idles if M is odd)
    static constexpr int C = 0;                // cos theta_k, sin theta_k (theta_N = 0)
    static constexpr int S = C + N;
    static constexpr int H = S + N;            // M x M, row-major
    static constexpr int RC = H + M * M;       // the round's rotations, by pair
    static constexpr int RS = RC + ME / 2;
    static constexpr int TOTAL = RS + ME / 2;
    // pair k of round r
    static __device__ __forceinline__ void pair(int r, int k, int &p, int &q) {
        const int m = ME - 1;
        p = k == 0 ? m : r + k < m ? r + k : r + k - m;
        q = k == 0 ? r : r >= k ? r - k : r - k + m;
        if (p > q) {
            const int t = p;
            p = q;
            q = t;
        }
    }
};

template <int M>
constexpr size_t cls_smem_per_block() {
    return sizeof(double) * (size_t)(CLS_PATHS * ClsLayout<M>::TOTAL + M * (M + 1));
}

__device__ __forceinline__ double cls_sum(double v) {   // over a point's four lanes
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    return v + __shfl_xor_sync(0xffffffffu, v, 16);
}

template <int M>
__global__ void __launch_bounds__(32)
    xy_classify_kernel(const __grid_constant__ XYSys S, const EPView ep, double *theta,
                       int32_t *index, double *energy, double *min_eig, double *log_abs_det,
                       const int32_t *list, const int32_t *list_count) {
    using L = ClsLayout<M>;
    constexpr int N = M + 1;
    extern __shared__ __align__(16) double cls_raw[];
    const int lane = threadIdx.x, g = lane >> 3, pth = lane & 7;
    double *const sm = cls_raw + pth;
    double *const J = cls_raw + CLS_PATHS * L::TOTAL;   // M x N
    for (int i = lane; i < M * N; i += 32) J[i] = S.Jd[(i / N) * NPHC_JSTRIDE + i % N];
    auto at = [&](int off, int i) -> double & { return sm[(off + i) * CLS_PATHS]; };
    auto H = [&](int i, int c) -> double & { return sm[(L::H + i * M + c) * CLS_PATHS]; };
    const int64_t cnt = ep.count, total = list ? (int64_t)*list_count : cnt;
    int64_t next = (int64_t)pth * gridDim.x + blockIdx.x;   // points one per warp first
    const int64_t stride = (int64_t)CLS_PATHS * gridDim.x;
    for (;;) {
        int64_t e = -1;
#pragma unroll 1
        while (e < 0 && next < total) {   // the next real point
            const int64_t i = list ? (int64_t)list[next] : next;
            next += stride;
            if (!NPHC_VALID(i >= 0 && i < cnt, 5)) continue;
            if (ep.cls[i] == NPHC_END_REAL) e = i;
        }
        __syncwarp();
        if (!__any_sync(0xffffffffu, e >= 0)) break;
#pragma unroll 1
        for (int k = g; k < N; k += 4) {
            double c = 1.0, s = 0.0;   // theta_N = 0
            if (e >= 0 && k < M) {
                const double x = ep.z_re[k * cnt + e], y = ep.z_re[(M + k) * cnt + e];
                double a = atan2(y, x);
                if (a <= -M_PI) a = M_PI;
                theta[k * cnt + e] = a;
                const double r2 = fma(x, x, y * y);
                if (r2 > 1e-280 && isfinite(r2)) {   // a subnormal r2 has lost its digits
                    const double ir = rsqrt(r2);
                    c = x * ir;
                    s = y * ir;
                } else {
                    sincos(a, &s, &c);
                }
            }
            at(L::C, k) = c;
            at(L::S, k) = s;
        }
        __syncwarp();
        // V = sum_{i<j} J_ij (1 - cos(theta_i - theta_j)), cos(a - b) = c_a c_b + s_a s_b, and the
        // Hessian in theta_1..theta_M; off, tot: its squares off the diagonal, and all of them
        double V = 0.0, off = 0.0, tot = 0.0;
#pragma unroll 1
        for (int k = g; k < M; k += 4) {
            const double ck = at(L::C, k), sk = at(L::S, k);
            double d = 0.0;
#pragma unroll 1
            for (int j = 0; j < N; j++) {
                const double Jkj = J[k * N + j], cd = ck * at(L::C, j) + sk * at(L::S, j);
                const double v = j == k ? 0.0 : Jkj * cd;
                if (j > k) V = fma(Jkj, 1.0 - cd, V);
                d += v;
                if (j < M) {
                    H(k, j) = -v;
                    off = fma(v, v, off);
                }
            }
            H(k, k) = d;
            tot = fma(d, d, tot);
        }
        V = cls_sum(V);
        off = cls_sum(off);
        tot = cls_sum(tot) + off;
        __syncwarp();
        // cyclic Jacobi rotations until the off-diagonal part is negligible
        bool busy = e >= 0;
#pragma unroll 1
        for (int sweep = 0; sweep < 64; sweep++) {
            busy = busy && !(off <= 1e-30 * tot);
            if (!__any_sync(0xffffffffu, busy)) break;
#pragma unroll 1
            for (int r = 0; r < L::ME - 1; r++) {
#pragma unroll 1
                for (int k = g; k < L::ME / 2; k += 4) {
                    int p, q;
                    L::pair(r, k, p, q);
                    double cs = 1.0, sn = 0.0;
                    const double apq = q < M ? H(p, q) : 0.0;
                    if (busy && apq != 0.0) {   // tan of the smaller angle: 2 apq / (d +- sqrt(d^2 + 4 apq^2))
                        double d = H(q, q) - H(p, p), h = 2.0 * apq;
                        const int ex = max(gexp(d), gexp(h));
                        if (ex < -400 || ex > 400) {   // the squares below must neither vanish nor overflow
                            const double by = __hiloint2double((1023 - min(max(ex, -1000), 1000)) << 20, 0);
                            d *= by;
                            h *= by;
                        }
                        const double w = sqrt(fma(d, d, h * h));
                        const double tn = h / (d >= 0.0 ? d + w : d - w);
                        cs = rsqrt(fma(tn, tn, 1.0));
                        sn = tn * cs;
                    }
                    at(L::RC, k) = cs;
                    at(L::RS, k) = sn;
                }
                __syncwarp();
#pragma unroll 1
                for (int i = g; i < M; i += 4)   // columns p and q of the own rows
#pragma unroll 1
                    for (int k = 0; k < L::ME / 2; k++) {
                        int p, q;
                        L::pair(r, k, p, q);
                        if (q < M) {
                            const double cs = at(L::RC, k), sn = at(L::RS, k), x = H(i, p), y = H(i, q);
                            H(i, p) = cs * x - sn * y;
                            H(i, q) = sn * x + cs * y;
                        }
                    }
                __syncwarp();
#pragma unroll 1
                for (int i = g; i < M; i += 4)   // rows p and q of the own columns
#pragma unroll 1
                    for (int k = 0; k < L::ME / 2; k++) {
                        int p, q;
                        L::pair(r, k, p, q);
                        if (q < M) {
                            const double cs = at(L::RC, k), sn = at(L::RS, k), x = H(p, i), y = H(q, i);
                            H(p, i) = cs * x - sn * y;
                            H(q, i) = sn * x + cs * y;
                        }
                    }
                __syncwarp();
            }
            off = tot = 0.0;
#pragma unroll 1
            for (int i = g; i < M; i += 4)
#pragma unroll 1
                for (int j = 0; j < M; j++) {
                    const double v = H(i, j);
                    if (i == j) tot = fma(v, v, tot);
                    else off = fma(v, v, off);
                }
            off = cls_sum(off);
            tot = cls_sum(tot) + off;
        }
        double mn = INFINITY, ld = 0.0;
        int neg = 0;
#pragma unroll 1
        for (int k = g; k < M; k += 4) {
            const double w = H(k, k);
            neg += w < 0.0;
            mn = fmin(mn, fabs(w));
            ld += log(fabs(w));   // log |det H| = sum of log |eigenvalue|
        }
        ld = cls_sum(ld);
        mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, 8));
        mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, 16));
        neg += __shfl_xor_sync(0xffffffffu, neg, 8);
        neg += __shfl_xor_sync(0xffffffffu, neg, 16);
        if (e >= 0 && g == 0) {
            index[e] = neg;
            energy[e] = V;
            if (min_eig) min_eig[e] = mn;
            if (log_abs_det) log_abs_det[e] = ld;
        }
        __syncwarp();
    }
}

// Gradient with respect to the couplings of a loss L(V*, theta*) summed over real
// stationary points (not part of the paper's method: derivatives of its outputs).  At
// theta* the gradient G = grad_theta V vanishes, so dV*/dJ_ij = 1 - cos(theta_i - theta_j)
// (envelope), and d theta*/dJ_ij = -H^-1 dG/dJ_ij (implicit function theorem); with
// H lambda = dL/dtheta (lambda_N = 0) and dG_i/dJ_ij = sin(theta_i - theta_j) = -dG_j/dJ_ij:
//   dL/dJ_ij = gV (1 - cos(theta_i - theta_j)) - (lambda_i - lambda_j) sin(theta_i - theta_j).
// Four lanes per point, eight points per warp (FP64: an instruction costs 67 cycles of a
// scheduler whatever the number of lanes, so the rows of H fill them): lane g owns the sites
// and rows g + 4 q and the couplings g + 4 u of the pair list, whose sums it keeps in registers
// over the points of its slot.  1,670 points of N = 10: 277 -> 33 us against one point per thread
// (14 blocks, and shared-memory FP64 atomics contended by 128 threads).  theta: [count * M], one row per point; g_energy [count] and
// g_theta [count * M] may be NULL.  One atomic add per coupling and block into dJ (N x N,
// symmetric: both J_ij and J_ji get the value of the one parameter).
#define ADJ_WARPS 4
#define ADJ_PATHS 8
template <int M>
struct AdjLayout {   // doubles per point ([index * 8 + point])
    static constexpr int N = M + 1;
    static constexpr int C = 0;                 // cos theta_k (theta_N = 0)
    static constexpr int S = C + N;
    static constexpr int LAM = S + N;
    static constexpr int H = LAM + N;           // [H | g], row-major, M + 1 columns
    static constexpr int TOTAL = H + M * (M + 1);
    static constexpr int PAIRS = N * (N - 1) / 2;
};

template <int M>
constexpr size_t adj_smem_per_block() {
    return sizeof(double) * (size_t)(ADJ_WARPS * (ADJ_PATHS * AdjLayout<M>::TOTAL + AdjLayout<M>::PAIRS) +
                                     (M + 1) * (M + 1));
}

template <int M>
__global__ void __launch_bounds__(32 * ADJ_WARPS)
    xy_adjoint_kernel(const __grid_constant__ XYSys S, int64_t count, const double *theta,
                      const double *g_energy, const double *g_theta, double *dJ) {
    using L = AdjLayout<M>;
    constexpr int N = M + 1, U = (L::PAIRS + 3) / 4;
    extern __shared__ __align__(16) double adj_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, g = lane >> 3, pth = lane & 7;
    double *const sm = adj_raw + wid * (ADJ_PATHS * L::TOTAL) + pth;
    double *const sums = adj_raw + ADJ_WARPS * (ADJ_PATHS * L::TOTAL);   // [warp][pair]
    double *const J = sums + ADJ_WARPS * L::PAIRS;                       // N x N
    for (int i = threadIdx.x; i < N * N; i += blockDim.x) J[i] = S.Jd[(i / N) * NPHC_JSTRIDE + i % N];
    __syncthreads();
    auto at = [&](int off, int i) -> double & { return sm[(off + i) * ADJ_PATHS]; };
    auto H = [&](int i, int c) -> double & { return sm[(L::H + i * (M + 1) + c) * ADJ_PATHS]; };
    double acc[U];
#pragma unroll
    for (int u = 0; u < U; u++) acc[u] = 0.0;
    // points one per warp before more per warp
    const int64_t warps = (int64_t)gridDim.x * ADJ_WARPS;
    const int64_t first = (int64_t)pth * warps + (int64_t)wid * gridDim.x + blockIdx.x;
    for (int64_t base = 0; base < count; base += warps * ADJ_PATHS) {   // uniform over the block
        const int64_t e = base + first;
        const bool on = e < count;
        if (!__any_sync(0xffffffffu, on)) break;
#pragma unroll 1
        for (int k = g; k < N; k += 4) {
            double s = 0.0, c = 1.0;   // theta_N = 0, and points that do not exist
            if (on && k < M) sincos(theta[e * M + k], &s, &c);
            at(L::C, k) = c;
            at(L::S, k) = s;
            at(L::LAM, k) = 0.0;
        }
        __syncwarp();
        bool ok = true;
        if (g_theta) {
            // H lambda = g by LU with partial pivoting; cos(a - b) = c_a c_b + s_a s_b
#pragma unroll 1
            for (int k = g; k < M; k += 4) {
                const double ck = at(L::C, k), sk = at(L::S, k);
                double d = 0.0;
#pragma unroll 1
                for (int j = 0; j < N; j++) {
                    const double v = J[k * N + j] * (ck * at(L::C, j) + sk * at(L::S, j));   // J_kk = 0
                    d += v;
                    if (j < M) H(k, j) = -v;
                }
                H(k, k) = d;
                H(k, M) = on ? g_theta[e * M + k] : 0.0;
            }
            __syncwarp();
#pragma unroll 1
            for (int k = 0; k < M; k++) {
                unsigned long long key = 0;
#pragma unroll 1
                for (int i = g; i < M; i += 4)
                    if (i >= k) {
                        const unsigned long long v = (unsigned long long)__double_as_longlong(fabs(H(i, k)));
                        key = max(key, (v & ~15ull) | (unsigned long long)(15 - i));
                    }
                key = max(key, __shfl_xor_sync(0xffffffffu, key, 8));
                key = max(key, __shfl_xor_sync(0xffffffffu, key, 16));
                int p = 15 - (int)(key & 15ull);
                if ((key >> 4) == 0) {   // singular: the point adds nothing
                    ok = false;
                    p = k;
                }
                if (p != k)
#pragma unroll 1
                    for (int c = k + g; c <= M; c += 4) {
                        const double t = H(k, c);
                        H(k, c) = H(p, c);
                        H(p, c) = t;
                    }
                __syncwarp();
                const double ip = 1.0 / H(k, k);
#pragma unroll 1
                for (int i = g; i < M; i += 4)
                    if (i > k) {
                        const double f = H(i, k) * ip;
#pragma unroll 2
                        for (int c = k + 1; c <= M; c++) H(i, c) = fma(-f, H(k, c), H(i, c));
                    }
                __syncwarp();
                if (g == (k & 3)) H(k, k) = ip;
            }
            __syncwarp();
#pragma unroll 1
            for (int k = M - 1; k >= 0; k--) {
                const double x = H(k, M) * H(k, k);
                __syncwarp();
#pragma unroll 1
                for (int i = g; i <= k; i += 4) {
                    if (i == k) at(L::LAM, k) = x;
                    else H(i, M) = fma(-H(i, k), x, H(i, M));
                }
                __syncwarp();
            }
        }
        const double gv = on && g_energy ? g_energy[e] : 0.0;
        int i = 0, j = 1 + g;   // pair g + 4 u of (0,1), (0,2), .., (1,2), ..
#pragma unroll
        for (int u = 0; u < U; u++) {
            while (j >= N && i < N - 1) {
                i++;
                j += i + 1 - N;
            }
            if (on && ok && g + 4 * u < L::PAIRS) {
                const double ci = at(L::C, i), si = at(L::S, i), cj = at(L::C, j), sj = at(L::S, j);
                const double cd = ci * cj + si * sj;   // cos(theta_i - theta_j)
                const double sd = si * cj - ci * sj;   // sin(theta_i - theta_j)
                acc[u] += gv * (1.0 - cd) - (at(L::LAM, i) - at(L::LAM, j)) * sd;
            }
            j += 4;
        }
        __syncwarp();
    }
    // sums over the warp's points, then over the block's warps
#pragma unroll
    for (int u = 0; u < U; u++) {
        double v = acc[u];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        if (pth == 0 && g + 4 * u < L::PAIRS) sums[wid * L::PAIRS + g + 4 * u] = v;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < L::PAIRS; t += blockDim.x) {
        double v = 0.0;
        for (int w = 0; w < ADJ_WARPS; w++) v += sums[w * L::PAIRS + t];
        int i = 0, j = t + 1;
        while (j >= N) {
            i++;
            j += i + 1 - N;
        }
        if (v != 0.0) {
            atomicAdd(&dJ[i * N + j], v);
            atomicAdd(&dJ[j * N + i], v);
        }
    }
}
