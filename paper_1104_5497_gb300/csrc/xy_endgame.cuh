// xy_endgame.cuh -- FP64 work at t = 1 on the endpoints of the XY ring:
//   refinement: Newton's method on P to full double precision (section "Numerical
//     Polynomial Homotopy Continuation Method" refines every endpoint to machine
//     precision before certifying it), with P evaluated by exact products and
//     double-double sums (eg_minus_p);
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
// xy_refine_group.cuh (four lanes per endpoint); this file holds the classification and the
// adjoint, and the rules of refinement and certification as a generic body, one endpoint per
// thread with a Householder QR of DP, for quadratic systems (quad.cuh).
//
// The refinement certifies the iterate whose Newton correction met the tolerance, from
// the factorisation of that iteration, and outputs its Newton iterate.
//
// Storage of the generic body: interleaved across the 32 threads of a block in shared memory
// (element i of a thread's array at [i * 32 + lane]), so that the rolled loops index it at run
// time without local memory.
#pragma once

#include "nphc_internal.cuh"

#define EG_BLOCK 32

// The certification threshold: half of Smale's (13 - 3 sqrt 17) / 4.  alphaCertified
// decides in exact arithmetic; an FP64 test keeps a factor of two so that rounding cannot
// carry a point near a singular solution set across the constant (on the N = 4 ring a
// point of the positive-dimensional family reached alpha = 0.115 < 0.158).
#define NPHC_ALPHA_CERT (0.5 * (13.0 - 3.0 * sqrt(17.0)) / 4.0)


// One thread's array of complex doubles in shared memory.
struct EGVec {
    cx<double> *p;
    __device__ __forceinline__ cx<double> get(int i) const { return p[i * EG_BLOCK]; }
    __device__ __forceinline__ void set(int i, cx<double> v) const { p[i * EG_BLOCK] = v; }
};

// Per-thread working set of the refinement (complex doubles, in this order).
template <int M>
struct EGLayout {
    static constexpr int TQ = 0;                // conj(tau) of the reflectors
    static constexpr int X = TQ + M;            // z
    static constexpr int R = X + M;             // right-hand side / residual (and one scalar)
    static constexpr int D = R + M + 1;         // solution
    static constexpr int S = D + M;             // M x M, column-major: entry (i, c) at c M + i
    static constexpr int TOTAL = S + M * M;
};

template <int M>
constexpr size_t eg_smem_per_thread() {
    return sizeof(cx<double>) * (size_t)EGLayout<M>::TOTAL;
}

template <int M>
struct EG {
    cx<double> *base;   // this thread's first entry in shared memory (stride EG_BLOCK)
    cx<double> *sp;     // this thread's entry (0, 0) of S
    __device__ __forceinline__ EGVec v(int off) const { return EGVec{base + off * EG_BLOCK}; }
    __device__ __forceinline__ cx<double> S(int i, int c) const { return sp[(c * M + i) * EG_BLOCK]; }
    __device__ __forceinline__ void setS(int i, int c, cx<double> a) const { sp[(c * M + i) * EG_BLOCK] = a; }
};

// Householder QR of the M x M matrix G.S in place: R above the diagonal with a real
// diagonal (stored as (beta, 0)), the reflectors (1, v) below it, conj(tau) in TQ.
// Returns false when the matrix is singular.
template <int M>
__device__ bool eg_qr(const EG<M> &G) {
    const EGVec TQ = G.v(EGLayout<M>::TQ);
    bool ok = true;
#pragma unroll 1
    for (int k = 0; k < M; k++) {
        const cx<double> al = G.S(k, k);
        double xn2 = 0.0;
#pragma unroll 1
        for (int i = k + 1; i < M; i++) xn2 += cabs2(G.S(i, k));
        const double an = sqrt(cabs2(al) + xn2);
        ok = ok && an > 0.0;
        const double beta = al.re >= 0.0 ? -an : an;
        const cx<double> tauc = cx<double>{(beta - al.re) / beta, al.im / beta};
        const cx<double> sc = crecip(cx<double>{al.re - beta, al.im});
#pragma unroll 1
        for (int i = k + 1; i < M; i++) G.setS(i, k, cmul(G.S(i, k), sc));
        G.setS(k, k, cx<double>{beta, 0.0});
        TQ.set(k, tauc);
#pragma unroll 1
        for (int c = k + 1; c < M; c++) {
            cx<double> wv = G.S(k, c);
#pragma unroll 1
            for (int i = k + 1; i < M; i++) wv = cadd(wv, cmulc(G.S(i, k), G.S(i, c)));
            wv = cmul(tauc, wv);
            G.setS(k, c, csub(G.S(k, c), wv));
#pragma unroll 1
            for (int i = k + 1; i < M; i++) G.setS(i, c, csub(G.S(i, c), cmul(G.S(i, k), wv)));
        }
    }
    return ok;
}

// b <- R^-1 Q^H b (b: M entries of a per-thread array); returns ||b||^2 afterwards.
template <int M>
__device__ double eg_schur_solve(const EG<M> &G, const EGVec &b) {
    const EGVec TQ = G.v(EGLayout<M>::TQ);
#pragma unroll 1
    for (int k = 0; k < M; k++) {
        cx<double> wv = b.get(k);
#pragma unroll 1
        for (int i = k + 1; i < M; i++) wv = cadd(wv, cmulc(G.S(i, k), b.get(i)));
        wv = cmul(TQ.get(k), wv);
        b.set(k, csub(b.get(k), wv));
#pragma unroll 1
        for (int i = k + 1; i < M; i++) b.set(i, csub(b.get(i), cmul(G.S(i, k), wv)));
    }
    double n2 = 0.0;
#pragma unroll 1
    for (int k = M - 1; k >= 0; k--) {
        cx<double> acc = b.get(k);
#pragma unroll 1
        for (int c = k + 1; c < M; c++) acc = csub(acc, cmul(G.S(k, c), b.get(c)));
        acc = cscale(1.0 / G.S(k, k).re, acc);
        b.set(k, acc);
        n2 += cabs2(acc);
    }
    return n2;
}

// shortcut = 1: entries handed off by the FP32 pass close to t = 1 are refined at t = 1
// directly (Newton on P from the hand-off point: for a path to a nonsingular solution xi,
// z(t) = xi + (1 - t) z'(1) + ..., so the point is already in xi's Newton basin).  The
// first Newton correction must stay below SHORTCUT_TRUST (1 + ||z||); an entry that
// certifies becomes NPHC_PATH_REACHED, any other entry is left untouched.
#define SHORTCUT_TRUST 1e-2

// The system a refinement kernel works on is a policy Q for refine_body (EGQuad in quad.cuh):
// the unknowns (NZ of them, stored in G's X), -P into R, the factorisation of DP, the Newton
// step D = DP^-1 R, ||DP||_F, ||DP^-1||_F and ||D^2 P / 2||.  The XY ring has a kernel of its own
// (xy_refine_group.cuh) that follows the same rules.

// beta = ||DP^-1 P||, ||DP^-1||_F and ||P||_inf at the point in G.  False if singular:
// at a point of a positive-dimensional solution set P vanishes to double-double precision
// (beta is tiny) while rounding leaves the computed DP^-1 merely huge, and the soft alpha
// test alone can pass there, so a Frobenius condition number ||DP||_F ||DP^-1||_F above
// kappa_sing max(1, ||z||_inf^2) counts as singular.  The bound grows with ||z||_inf^2 like
// the solution tolerance: the equations are quadratic, the Jacobian's entries grow like
// ||z|| and an isolated solution near the solution set at infinity has a smallest singular
// value shrinking like 1 / ||z|| (a solution of norm 1e6 has a condition number ~1e12).
// The same from a factorisation already made at the point in G: fro = ||DP||_F, dn =
// ||DP^-1 P|| from its solve (inv_fro takes D as scratch).
template <class Q>
__device__ bool eg_certify_factored(const EG<Q::DIM> &G, const typename Q::Sys &S, double fro,
                                    double dn, double &beta, double &invF) {
    beta = dn;
    invF = Q::inv_fro(G, S);
    double zi = 0.0;
#pragma unroll 1
    for (int k = 0; k < Q::NZ; k++) zi = fmax(zi, sqrt(cabs2(Q::zget(G, k))));
    return isfinite(beta) && isfinite(invF) && fro * invF <= S.kappa_sing * fmax(1.0, zi * zi);
}

template <class Q>
__device__ bool eg_beta_invnorm_p(const EG<Q::DIM> &G, const typename Q::Sys &S, double &beta,
                                  double &invF, double &res) {
    res = Q::minus_p(G, S);
    if (!Q::factor(G, S)) return false;
    const double fro = Q::jac_fro(G, S);
    const double dn = sqrt(Q::solve(G, S));
    return eg_certify_factored<Q>(G, S, fro, dn, beta, invF);
}

// Refinement and certification of entry e.  Returns true when e still needs the
// alpha-test at Re z (its refined z is already written out; the caller runs the test).
template <class Q>
__device__ bool eg_refine_certify_one(const EG<Q::DIM> &G, const typename Q::Sys &S,
                                      double tol_sol, double refine_eps, int refine_iters,
                                      const EPView &ep, int64_t e) {
    constexpr int NZ = Q::NZ;
    const EGVec Dv = G.v(EGLayout<Q::DIM>::D);
    const int64_t cnt = ep.count;
    const double alpha0 = NPHC_ALPHA_CERT;
    const int st = ep.status[e];
    ep.alpha[e] = INFINITY;
    ep.beta[e] = INFINITY;
    ep.gamma[e] = INFINITY;
    ep.resid[e] = INFINITY;
    if (st == NPHC_PATH_DIVERGED) {
        ep.cls[e] = NPHC_END_NONE;
        return false;
    }
    if (st != NPHC_PATH_REACHED) {
        ep.cls[e] = NPHC_END_FAILED;
        return false;
    }
#pragma unroll 1
    for (int k = 0; k < NZ; k++) Q::zset(G, k, cx<double>{ep.z_re[k * cnt + e], ep.z_im[k * cnt + e]});
    int cls = NPHC_END_SINGULAR;
    bool finite = true;
    double beta = INFINITY, invF = INFINITY, res = INFINITY;
    bool certified = false, cert_ok = false;
    // Newton refinement on P.  The iteration whose correction meets refine_eps certifies its
    // own point z_k from the factorisation it has just made (beta = ||dz_k||, exactly what a
    // separate certification at z_k computes), and the output is z_k's Newton iterate
    // z_k + dz_k, closer still to the same zero: one evaluation, factorisation and solve
    // less than certifying the output point afresh
#pragma unroll 1
    for (int it = 0; it < refine_iters; it++) {
        const double rk = Q::minus_p(G, S);
        if (!Q::factor(G, S)) break;
        const double dn = sqrt(Q::solve(G, S));
        double z2 = 0.0;
#pragma unroll 1
        for (int k = 0; k < NZ; k++) z2 += cabs2(Q::zget(G, k));
        if (!isfinite(dn) || !isfinite(z2)) {
            finite = false;
            break;
        }
        const bool last = dn <= refine_eps * (1.0 + sqrt(z2));
        const EGVec Step = last ? G.v(EGLayout<Q::DIM>::R) : Dv;
        if (last) {
#pragma unroll 1
            for (int k = 0; k < NZ; k++) Step.set(k, Dv.get(k));   // inv_fro takes D as scratch
            const double fro = Q::jac_fro(G, S);
            cert_ok = eg_certify_factored<Q>(G, S, fro, dn, beta, invF);
            res = rk;
            certified = true;
        }
        double zn = 0.0;
#pragma unroll 1
        for (int k = 0; k < NZ; k++) {
            const cx<double> zk = cadd(Q::zget(G, k), Step.get(k));
            Q::zset(G, k, zk);
            zn += cabs2(zk);
        }
        if (!isfinite(zn)) {
            finite = false;
            break;
        }
        if (last) break;
    }
    if (finite && !certified) cert_ok = eg_beta_invnorm_p<Q>(G, S, beta, invF, res);
    double alpha = INFINITY, gam = INFINITY;
    bool real_test = false;
    if (finite && cert_ok) {
        gam = invF * Q::d2norm(S);
        alpha = beta * gam;
        // Delta_sol relative to the size of the (quadratic) terms: max(1, ||z||_inf^2)
        double zi = 0.0, im2 = 0.0;
#pragma unroll 1
        for (int k = 0; k < NZ; k++) {
            const cx<double> zk = Q::zget(G, k);
            zi = fmax(zi, sqrt(cabs2(zk)));
            im2 += zk.im * zk.im;
        }
        if (res <= tol_sol * fmax(1.0, zi * zi) && alpha < alpha0) {
            // z and Re z share their associated zero when alpha < 0.03 and
            // ||Im z|| < 1 / (20 gamma): then the real test at Re z decides (queued)
            const double im = sqrt(im2);
            if (alpha < 0.03 && im < 1.0 / (20.0 * gam))
                real_test = true;
            else
                cls = im > 2.0 * beta ? NPHC_END_NONREAL : NPHC_END_UNDECIDED;
        }
    } else {
        beta = INFINITY;
    }
    ep.alpha[e] = alpha;
    ep.beta[e] = beta;
    ep.gamma[e] = gam;
    ep.resid[e] = finite ? res : INFINITY;
#pragma unroll 1
    for (int k = 0; k < NZ; k++) {
        const cx<double> zk = Q::zget(G, k);
        ep.z_re[k * cnt + e] = zk.re;
        ep.z_im[k * cnt + e] = zk.im;
    }
    if (!real_test) ep.cls[e] = cls;
    return real_test;
}

// The alpha-test at Re z of a certified entry e that shares its zero with Re z: real
// when it passes there; otherwise non-real when ||Im z|| > 2 beta (z and conj z then
// have distinct zeros), else undecided.
template <class Q>
__device__ void eg_real_test(const EG<Q::DIM> &G, const typename Q::Sys &S, const EPView &ep,
                             int64_t e) {
    const int64_t cnt = ep.count;
    const double alpha0 = NPHC_ALPHA_CERT;
    double im2 = 0.0;
#pragma unroll 1
    for (int k = 0; k < Q::NZ; k++) {
        const double yi = ep.z_im[k * cnt + e];
        im2 += yi * yi;
        Q::zset(G, k, cx<double>{ep.z_re[k * cnt + e], 0.0});
    }
    double br, ir, rr;
    if (eg_beta_invnorm_p<Q>(G, S, br, ir, rr) && br * ir * Q::d2norm(S) < alpha0)
        ep.cls[e] = NPHC_END_REAL;
    else
        ep.cls[e] = sqrt(im2) > 2.0 * ep.beta[e] ? NPHC_END_NONREAL : NPHC_END_UNDECIDED;
}

// One warp per block.  Entries are taken 32 at a time; the few that need the real test go to
// a per-warp queue that is drained 32 at a time, so that the test runs on full warps.
template <class Q>
__device__ __forceinline__ void refine_body(const typename Q::Sys &S, double tol_sol,
                                            double refine_eps, int refine_iters, const EPView &ep,
                                            const WorkList &wl) {
    using L = EGLayout<Q::DIM>;
    extern __shared__ __align__(16) unsigned char egraw[];
    __shared__ int64_t rq[2 * EG_BLOCK];
    const int lane = threadIdx.x;
    cx<double> *const sb = reinterpret_cast<cx<double> *>(egraw) + lane;
    const EG<Q::DIM> G{sb, sb + L::S * EG_BLOCK};
    const int64_t total = worklist_size(wl, ep.count);
    int qn = 0;   // queued real tests (the same in every lane)
    for (int64_t base = (int64_t)blockIdx.x * EG_BLOCK; base < total;
         base += (int64_t)gridDim.x * EG_BLOCK) {
        const int64_t i = base + lane;
        int64_t e = -1;
        bool rt = false;
        if (i < total) e = worklist_entry(wl, i, ep.count);   // -1: rejected (debug)
        if (e >= 0)
            rt = eg_refine_certify_one<Q>(G, S, tol_sol, refine_eps, refine_iters, ep, e);
        const unsigned m = __ballot_sync(0xffffffffu, rt);
        if (rt) rq[qn + __popc(m & ((1u << lane) - 1u))] = e;
        qn += __popc(m);
        __syncwarp();
        if (qn >= EG_BLOCK) {
            eg_real_test<Q>(G, S, ep, rq[qn - EG_BLOCK + lane]);
            qn -= EG_BLOCK;
            __syncwarp();
        }
    }
    if (lane < qn) eg_real_test<Q>(G, S, ep, rq[lane]);
}

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

