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

template <int M>
__global__ void __launch_bounds__(128)
    xy_classify_kernel(const __grid_constant__ XYSys S, const EPView ep, double *theta,
                       int32_t *index, double *energy, double *min_eig, double *log_abs_det,
                       const int32_t *list, const int32_t *list_count) {
    // every entry, or the listed ones: the real stationary points packed 32 to a warp, so
    // that the FP64 Jacobi runs on full warps (GB300's FP64 pipe charges a warp instruction
    // whatever the number of active lanes, and scattered real points cost a warp each)
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t cnt = ep.count;
    int64_t e = i;
    if (list) {
        if (i >= *list_count) return;
        e = list[i];
        if (!NPHC_VALID(e >= 0 && e < cnt, 5)) return;
    }
    if (e >= cnt) return;
    if (ep.cls[e] != NPHC_END_REAL) {
        index[e] = -1;
        energy[e] = 0.0;
        if (min_eig) min_eig[e] = 0.0;
        if (log_abs_det) log_abs_det[e] = 0.0;
        for (int k = 0; k < M; k++) theta[k * cnt + e] = 0.0;
        return;
    }
    const double *J = S.Jd;
    constexpr int N = M + 1;
    double c[N], s[N];
#pragma unroll 1
    for (int k = 0; k < M; k++) {
        const double x = ep.z_re[k * cnt + e], y = ep.z_re[(M + k) * cnt + e];
        double a = atan2(y, x);
        if (a <= -M_PI) a = M_PI;
        sincos(a, &s[k], &c[k]);
        theta[k * cnt + e] = a;
    }
    c[M] = 1.0;   // theta_N = 0
    s[M] = 0.0;
    // V = sum_{i<j} J_ij (1 - cos(theta_i - theta_j)), cos(a - b) = c_a c_b + s_a s_b
    double V = 0.0;
#pragma unroll 1
    for (int i = 0; i < N; i++)
        for (int j = i + 1; j < N; j++) V += J[i * NPHC_JSTRIDE + j] * (1.0 - (c[i] * c[j] + s[i] * s[j]));
    // Hessian in theta_1..theta_M (row-major, flat)
    double H[M * M];
#pragma unroll 1
    for (int k = 0; k < M; k++) {
        double d = 0.0;
        for (int j = 0; j < N; j++)
            if (j != k) d += J[k * NPHC_JSTRIDE + j] * (c[k] * c[j] + s[k] * s[j]);
        for (int l = 0; l < M; l++)
            H[k * M + l] = (k == l) ? d : -J[k * NPHC_JSTRIDE + l] * (c[k] * c[l] + s[k] * s[l]);
    }
    // cyclic Jacobi rotations until the off-diagonal part is negligible
#pragma unroll 1
    for (int sweep = 0; sweep < 64; sweep++) {
        double off = 0.0, tot = 0.0;
        for (int i = 0; i < M * M; i++) {
            tot += H[i] * H[i];
            if (i / M != i % M) off += H[i] * H[i];
        }
        if (off <= 1e-30 * tot) break;
#pragma unroll 1
        for (int p = 0; p < M - 1; p++)
#pragma unroll 1
            for (int q = p + 1; q < M; q++) {
                const double apq = H[p * M + q];
                if (apq == 0.0) continue;
                const double tq = (H[q * M + q] - H[p * M + p]) / (2.0 * apq);
                const double tn = (tq >= 0.0 ? 1.0 : -1.0) / (fabs(tq) + sqrt(tq * tq + 1.0));
                const double cs = 1.0 / sqrt(tn * tn + 1.0), sn = tn * cs;
#pragma unroll 1
                for (int k = 0; k < M; k++) {   // columns p and q
                    const double akp = H[k * M + p], akq = H[k * M + q];
                    H[k * M + p] = cs * akp - sn * akq;
                    H[k * M + q] = sn * akp + cs * akq;
                }
#pragma unroll 1
                for (int k = 0; k < M; k++) {   // rows p and q
                    const double apk = H[p * M + k], aqk = H[q * M + k];
                    H[p * M + k] = cs * apk - sn * aqk;
                    H[q * M + k] = sn * apk + cs * aqk;
                }
            }
    }
    int neg = 0;
    double mn = INFINITY, ld = 0.0;
    for (int k = 0; k < M; k++) {
        const double w = H[k * M + k];
        if (w < 0.0) neg++;
        mn = fmin(mn, fabs(w));
        ld += log(fabs(w));   // log |det H| = sum of log |eigenvalue|
    }
    index[e] = neg;
    energy[e] = V;
    if (min_eig) min_eig[e] = mn;
    if (log_abs_det) log_abs_det[e] = ld;
}

// Gradient with respect to the couplings of a loss L(V*, theta*) summed over real
// stationary points (not part of the paper's method: derivatives of its outputs).  At
// theta* the gradient G = grad_theta V vanishes, so dV*/dJ_ij = 1 - cos(theta_i - theta_j)
// (envelope), and d theta*/dJ_ij = -H^-1 dG/dJ_ij (implicit function theorem); with
// H lambda = dL/dtheta (lambda_N = 0) and dG_i/dJ_ij = sin(theta_i - theta_j) = -dG_j/dJ_ij:
//   dL/dJ_ij = gV (1 - cos(theta_i - theta_j)) - (lambda_i - lambda_j) sin(theta_i - theta_j).
// One stationary point per thread (theta: [count * M] row per point; g_energy [count] and
// g_theta [count * M] may be NULL), the block's sum in shared memory, then one atomic add
// per coupling and block into dJ (N x N, symmetric: both J_ij and J_ji get the value of
// the one parameter).
template <int M>
__global__ void __launch_bounds__(128)
    xy_adjoint_kernel(const __grid_constant__ XYSys S, int64_t count, const double *theta,
                      const double *g_energy, const double *g_theta, double *dJ) {
    constexpr int N = M + 1;
    __shared__ double acc[N * N];
    for (int i = threadIdx.x; i < N * N; i += blockDim.x) acc[i] = 0.0;
    __syncthreads();
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < count) {
        const double *J = S.Jd;
        double c[N], s[N], lam[N];
#pragma unroll 1
        for (int k = 0; k < M; k++) sincos(theta[e * M + k], &s[k], &c[k]);
        c[M] = 1.0;
        s[M] = 0.0;
#pragma unroll 1
        for (int k = 0; k < N; k++) lam[k] = 0.0;
        bool ok = true;
        if (g_theta) {
            // H lambda = g by Gaussian elimination with partial pivoting; cos(a - b) =
            // c_a c_b + s_a s_b
            double H[M * M], b[M];
#pragma unroll 1
            for (int k = 0; k < M; k++) {
                double d = 0.0;
#pragma unroll 1
                for (int j = 0; j < N; j++)
                    if (j != k) d += J[k * NPHC_JSTRIDE + j] * (c[k] * c[j] + s[k] * s[j]);
#pragma unroll 1
                for (int l = 0; l < M; l++)
                    H[k * M + l] = (k == l) ? d : -J[k * NPHC_JSTRIDE + l] * (c[k] * c[l] + s[k] * s[l]);
                b[k] = g_theta[e * M + k];
            }
#pragma unroll 1
            for (int k = 0; k < M; k++) {
                int p = k;
#pragma unroll 1
                for (int i = k + 1; i < M; i++)
                    if (fabs(H[i * M + k]) > fabs(H[p * M + k])) p = i;
                if (H[p * M + k] == 0.0) {
                    ok = false;
                    break;
                }
                if (p != k) {
#pragma unroll 1
                    for (int l = 0; l < M; l++) {
                        const double tmp = H[k * M + l];
                        H[k * M + l] = H[p * M + l];
                        H[p * M + l] = tmp;
                    }
                    const double tb = b[k];
                    b[k] = b[p];
                    b[p] = tb;
                }
                const double ip = 1.0 / H[k * M + k];
#pragma unroll 1
                for (int i = k + 1; i < M; i++) {
                    const double f = H[i * M + k] * ip;
#pragma unroll 1
                    for (int l = k + 1; l < M; l++) H[i * M + l] -= f * H[k * M + l];
                    b[i] -= f * b[k];
                }
            }
            if (ok) {
#pragma unroll 1
                for (int k = M - 1; k >= 0; k--) {
                    double v = b[k];
#pragma unroll 1
                    for (int l = k + 1; l < M; l++) v -= H[k * M + l] * lam[l];
                    lam[k] = v / H[k * M + k];
                }
            }
        }
        if (ok) {
            const double gv = g_energy ? g_energy[e] : 0.0;
#pragma unroll 1
            for (int i = 0; i < N; i++)
#pragma unroll 1
                for (int j = i + 1; j < N; j++) {
                    const double cd = c[i] * c[j] + s[i] * s[j];   // cos(theta_i - theta_j)
                    const double sd = s[i] * c[j] - c[i] * s[j];   // sin(theta_i - theta_j)
                    const double v = gv * (1.0 - cd) - (lam[i] - lam[j]) * sd;
                    atomicAdd(&acc[i * N + j], v);
                    atomicAdd(&acc[j * N + i], v);
                }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < N * N; i += blockDim.x)
        if (acc[i] != 0.0) atomicAdd(&dJ[i], acc[i]);
}

