// k_vn.cu -- von Neumann analysis of the D2Q9 scheme on the GPU (Sec. V.A of the paper):
// batched eigenvalues of the amplification matrix M = E (delta + J) (Eq. eq:VN_eigen) and
// the linear-stability limit of Sec. V.A.2, in FP64.
//
// J is the Jacobian of the collision operator Omega_i = 2 beta (f_i^eq - f_i) at the
// equilibrium state f = f^eq(rho, u).  The derivative of a locally corrected 2 beta
// multiplies f^eq - f = 0 there, so J = 2 beta (d f^eq / d f - I) with
//   d f_i^eq / d f_j = d f_i^eq / d rho + sum_a d f_i^eq / d u_a (c_ja - u_a) / rho
// (rho = sum f, rho u = sum c f).  The partial derivatives of f^eq(rho, u) come from
// forward-mode dual numbers evaluated through the same equilibrium formulas as the step
// kernels, so they are exact to rounding.  E_ij = exp(-i c_i . k) delta_ij.
//
// Eigenvalues: reduction to upper Hessenberg form by complex Givens rotations, then
// single-shift QR with Wilkinson shifts and deflation (the standard complex Schur
// iteration), on a 9 x 9 matrix held by G lanes of a warp.
#include <algorithm>
#include <cmath>

#include "lbm.h"
#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbmd {

// ------------------------------------------------------------------------- dual numbers

struct Dual {  // value and derivatives with respect to (rho, u_x, u_y)
    double v, d[3];
};
__device__ __forceinline__ Dual dconst(double c) { return {c, {0, 0, 0}}; }
__device__ __forceinline__ Dual operator+(Dual a, Dual b) {
    return {a.v + b.v, {a.d[0] + b.d[0], a.d[1] + b.d[1], a.d[2] + b.d[2]}};
}
__device__ __forceinline__ Dual operator-(Dual a, Dual b) {
    return {a.v - b.v, {a.d[0] - b.d[0], a.d[1] - b.d[1], a.d[2] - b.d[2]}};
}
__device__ __forceinline__ Dual operator*(Dual a, Dual b) {
    return {a.v * b.v, {a.d[0] * b.v + a.v * b.d[0], a.d[1] * b.v + a.v * b.d[1], a.d[2] * b.v + a.v * b.d[2]}};
}
__device__ __forceinline__ Dual operator*(double c, Dual a) { return {c * a.v, {c * a.d[0], c * a.d[1], c * a.d[2]}}; }
__device__ __forceinline__ Dual dsqrt(Dual a) {
    const double s = sqrt(a.v), h = 0.5 / s;
    return {s, {h * a.d[0], h * a.d[1], h * a.d[2]}};
}

// f^eq_i(rho, u) of D2Q9 as dual numbers (same formulas as the step kernels' equilibria).
template <int EQ>
__device__ __forceinline__ void feq_dual(Dual rho, Dual ux, Dual uy, Dual (&f)[9]) {
    if (EQ == EQ_POLY2) {
        const Dual uu = ux * ux + uy * uy;
        for (int i = 0; i < 9; ++i) {
            const Dual cu = (double)cxo(i) * ux + (double)cyo(i) * uy;
            const Dual p = dconst(1.0) + 3.0 * cu + 4.5 * (cu * cu) - 1.5 * uu;
            f[i] = wq<2>(i) * (rho * p);
        }
        return;
    }
    Dual tx[3], ty[3];  // per-axis factors t(c) = a(c) / w(c), indexed by c + 1
    const Dual u[2] = {ux, uy};
    for (int a = 0; a < 2; ++a) {
        Dual *t = a == 0 ? tx : ty;
        if (EQ == EQ_ENT) {
            const Dual S = dsqrt(dconst(1.0) + 3.0 * (u[a] * u[a]));
            t[1] = dconst(2.0) - S;
            t[2] = 2.0 * S - dconst(1.0) + 3.0 * u[a];
            t[0] = 2.0 * S - dconst(1.0) - 3.0 * u[a];
        } else {
            const Dual u2 = u[a] * u[a];
            t[1] = dconst(1.0) - 1.5 * u2;
            t[2] = dconst(1.0) + 3.0 * u[a] + 3.0 * u2;
            t[0] = dconst(1.0) - 3.0 * u[a] + 3.0 * u2;
        }
    }
    for (int i = 0; i < 9; ++i) f[i] = wq<2>(i) * (rho * (tx[cxo(i) + 1] * ty[cyo(i) + 1]));
}

// ------------------------------------------------------------------ matrices in shared memory
//
// G lanes of a warp hold one matrix, 32 / G matrices to a block of one warp.  What bounds the
// solver is the FP64 pipe: an SM quarter takes 64 clocks for a warp's instruction, however many
// lanes are active (measured 68 in a full sweep), or with few matrices the latency of one solve
// (about 140 000 instructions, 12 clocks each).  The 9 x 9 complex matrix does not fit one thread's registers (324 of them),
// and the iteration indexes it by run-time bounds; in local memory the warps of an SM overran
// its L1.  In shared memory element (i, j) of the block's matrices lies together (16 bytes each).
// The lanes of a matrix share out the columns of a row rotation and the rows of a column
// rotation; moduli and quotients that a rotation needs in pairs are formed in one instruction
// stream by different lanes.  Which lane computes a value does not change it: the eigenvalues of a
// defective matrix move by the square root of a rounding error, more than a stability tolerance,
// so the operations and their order are kept as they are.
constexpr int kN = 9;
constexpr int kVnThreads = 32;

struct cplx {
    double re, im;
};
__device__ __forceinline__ cplx cadd(cplx a, cplx b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cplx csub(cplx a, cplx b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cplx cmul(cplx a, cplx b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ cplx cconj(cplx a) { return {a.re, -a.im}; }
__device__ __forceinline__ cplx cscale(double s, cplx a) { return {s * a.re, s * a.im}; }
__device__ __forceinline__ double cabs2(cplx a) { return a.re * a.re + a.im * a.im; }
__device__ __forceinline__ double cabsd(cplx a) { return hypot(a.re, a.im); }
__device__ __forceinline__ cplx cdiv(cplx a, cplx b) {
    const double d = cabs2(b);
    return {(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
__device__ __forceinline__ cplx csqrt_(cplx z) {
    const double r = cabsd(z);
    if (r == 0.0) return {0.0, 0.0};
    double x = sqrt(0.5 * (r + fabs(z.re)));
    double y = 0.5 * z.im / x;
    if (z.re >= 0.0) return {x, y};
    return {fabs(y), z.im >= 0.0 ? x : -x};
}


// Order-preserving integer of a modulus within a factor sqrt(2): the larger component's high word.
__device__ __forceinline__ unsigned cmag(cplx a) {
    return max(__double2hiint(a.re) & 0x7fffffffu, __double2hiint(a.im) & 0x7fffffffu);
}

// One matrix, seen by one of its G lanes.
template <int G> struct Mat {
    double2 *p;
    int g;          // lane within the group
    unsigned mask;  // the group's lanes
    __device__ __forceinline__ explicit Mat(double2 *sm) {
        const int lane = threadIdx.x & 31;
        p = sm + lane / G;
        g = lane % G;
        mask = (G == 32 ? 0xffffffffu : ((1u << G) - 1u)) << (lane / G * G);
    }
    __device__ __forceinline__ cplx get(int i, int j) const {
        const double2 v = p[(i * kN + j) * (kVnThreads / G)];
        return {v.x, v.y};
    }
    __device__ __forceinline__ void set(int i, int j, cplx v) const {
        p[(i * kN + j) * (kVnThreads / G)] = make_double2(v.re, v.im);
    }
    __device__ __forceinline__ void sync() const {
        if (G > 1) __syncwarp(mask);
    }
    __device__ __forceinline__ double from(double v, int src) const { return __shfl_sync(mask, v, src, G); }
    // Row i of delta + J times its phase exp(-i c_i . k).
    __device__ __forceinline__ void set_row(int i, const double (&row)[9], double kx, double ky) const {
        const double ph = -(cxo(i) * kx + cyo(i) * ky);
        cplx e;
        sincos(ph, &e.im, &e.re);
#pragma unroll
        for (int j = 0; j < kN; ++j) set(i, j, {e.re * row[j], e.im * row[j]});
    }
};

// Givens rotation G = [[c, s], [-conj(s), c]] (c real) with G [a; b] = [r; 0].
template <int G>
__device__ __forceinline__ void givens(const Mat<G> &M, cplx a, cplx b, double &c, cplx &s) {
    double na, nb;
    if constexpr (G > 1) {
        const double n = cabsd(M.g & 1 ? b : a);
        na = M.from(n, 0);
        nb = M.from(n, 1);
    } else {
        na = cabsd(a);
        nb = cabsd(b);
    }
    if (nb == 0.0) {
        c = 1.0;
        s = {0.0, 0.0};
        return;
    }
    if (na == 0.0) {
        c = 0.0;
        s = {1.0, 0.0};
        return;
    }
    const double r = hypot(na, nb);
    double q;
    if constexpr (G > 1) {
        const double v = (M.g & 1 ? 1.0 : na) / (M.g & 1 ? na * r : r);
        c = M.from(v, 0);
        q = M.from(v, 1);
    } else {
        c = na / r;
        q = 1.0 / (na * r);
    }
    s = cscale(q, cmul(a, cconj(b)));
}

// Rotate rows p, q of H (columns lo..hi) by G.
template <int G>
__device__ __forceinline__ void rot_rows(const Mat<G> &H, int p, int q, double c, cplx s, int lo, int hi) {
    for (int j = lo + H.g; j <= hi; j += G) {
        const cplx x = H.get(p, j), y = H.get(q, j);
        H.set(p, j, cadd(cscale(c, x), cmul(s, y)));
        H.set(q, j, csub(cscale(c, y), cmul(cconj(s), x)));
    }
    H.sync();
}

// Multiply columns p, q of H (rows lo..hi) by G^H on the right.
template <int G>
__device__ __forceinline__ void rot_cols(const Mat<G> &H, int p, int q, double c, cplx s, int lo, int hi) {
    for (int j = lo + H.g; j <= hi; j += G) {
        const cplx x = H.get(j, p), y = H.get(j, q);
        H.set(j, p, cadd(cscale(c, x), cmul(cconj(s), y)));
        H.set(j, q, csub(cscale(c, y), cmul(s, x)));
    }
    H.sync();
}

// Whether |sub| <= eps (|a| + |b|): by the exponents where they decide (the moduli are known
// within a factor sqrt(2)), by the moduli themselves in between.
__device__ __forceinline__ bool negligible(cplx sub, cplx a, cplx b) {
    const double eps = 2.220446049250313e-16;  // 2^-52
    const unsigned m = cmag(sub), d = max(cmag(a), cmag(b));
    if (d < 0x7ff00000u && m < 0x7ff00000u) {
        if (m > d - (49u << 20) && d > (60u << 20)) return false;  // > 2^-50 max > eps (|a| + |b|)
        if (m + (54u << 20) < d) return true;                      // < sqrt(2) 2^-53 max < eps |max|
    }
    return cabsd(sub) <= eps * (cabsd(a) + cabsd(b));
}

// Eigenvalues of H (overwritten; they are left on its diagonal).  Returns false if the
// iteration limit was reached.
template <int G>
__device__ bool eig_hessenberg_qr(const Mat<G> &H) {
    H.sync();
    // Hessenberg reduction (the entries below the subdiagonal are never looked at again)
    for (int k = 0; k < kN - 2; ++k) {
        for (int i = kN - 1; i >= k + 2; --i) {
            double c;
            cplx s;
            givens(H, H.get(i - 1, k), H.get(i, k), c, s);
            rot_rows(H, i - 1, i, c, s, k, kN - 1);
            rot_cols(H, i - 1, i, c, s, 0, kN - 1);
        }
    }
    int hi = kN - 1, iters = 0, since = 0;
    while (hi > 0) {
        // deflation: smallest l with a negligible subdiagonal above the active block
        int l = hi;
        while (l > 0 && !negligible(H.get(l, l - 1), H.get(l - 1, l - 1), H.get(l, l))) --l;
        if (l > 0) {
            H.sync();
            if (H.g == 0) H.set(l, l - 1, {0.0, 0.0});
            H.sync();
        }
        if (l == hi) {
            --hi;
            since = 0;
            continue;
        }
        if (++iters > 60 * kN) return false;
        ++since;
        // Wilkinson shift: eigenvalue of the trailing 2 x 2 block closest to H[hi][hi]
        const cplx a = H.get(hi - 1, hi - 1), b = H.get(hi - 1, hi), cc = H.get(hi, hi - 1), d = H.get(hi, hi);
        const cplx half = cscale(0.5, csub(a, d));
        const cplx disc = csqrt_(cadd(cmul(half, half), cmul(b, cc)));
        cplx mu1 = cadd(d, csub(half, disc)), mu2 = cadd(d, cadd(half, disc));
        cplx mu = cabs2(csub(mu1, d)) <= cabs2(csub(mu2, d)) ? mu1 : mu2;
        if (since % 11 == 10) mu = cadd(d, cscale(0.75, {cabsd(cc), 0.0}));  // exceptional shift
        // one QR step on the active block l..hi: H - mu I = Q R, H <- R Q + mu I
        H.sync();
        for (int k = l + H.g; k <= hi; k += G) H.set(k, k, csub(H.get(k, k), mu));
        H.sync();
        double c0 = 0.0;
        cplx s0 = {0.0, 0.0};
        for (int k = l; k < hi; ++k) {
            double c;
            cplx s;
            givens(H, H.get(k, k), H.get(k + 1, k), c, s);
            H.sync();
            rot_rows(H, k, k + 1, c, s, k, hi);
            if (H.g == 0) H.set(k + 1, k, {0.0, 0.0});
            H.sync();
            // columns k - 1, k are finished with the row rotations: their own now
            if (k > l) rot_cols(H, k - 1, k, c0, s0, l, k);
            c0 = c;
            s0 = s;
        }
        rot_cols(H, hi - 1, hi, c0, s0, l, hi);
        for (int k = l + H.g; k <= hi; k += G) H.set(k, k, cadd(H.get(k, k), mu));
        H.sync();
    }
    return true;
}

// The real matrix delta + J of the D2Q9 scheme at (tau, rho, u), row i into row[].
template <int EQ, bool BULK>
__device__ __forceinline__ void vn_row(double tau, double rho, double ux, double uy, int i, double (&row)[9]) {
    Dual f[9];
    feq_dual<EQ>(Dual{rho, {1, 0, 0}}, Dual{ux, {0, 1, 0}}, Dual{uy, {0, 0, 1}}, f);
    double om = 1.0 / tau;
    if (BULK) {
        const double nu = (tau - 0.5) / 3.0;
        double A;
        if (EQ == EQ_ENT) {
            const double S = fmax(sqrt(1.0 + 3.0 * ux * ux), sqrt(1.0 + 3.0 * uy * uy));
            A = (2.0 - S) / (S * S);
        } else {
            A = 1.0 - 4.5 * fmax(ux * ux, uy * uy);
        }
        om = 2.0 * A / (6.0 * nu + A);
    }
    Dual fi = f[0];
#pragma unroll
    for (int q = 1; q < 9; ++q)
        if (q == i) fi = f[q];
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const double dfdf = fi.d[0] + fi.d[1] * (cxo(j) - ux) / rho + fi.d[2] * (cyo(j) - uy) / rho;
        row[j] = (i == j ? 1.0 : 0.0) + om * (dfdf - (i == j ? 1.0 : 0.0));
    }
}

template <int G, int EQ, bool BULK>
__global__ void __launch_bounds__(kVnThreads) k_vn_eigs(int64_t count, const double *params, double *out,
                                                        int32_t *status) {
    constexpr int per = kVnThreads / G;
    __shared__ double2 sm[kN * kN * per];
    const Mat<G> M(sm);
    for (int64_t p0 = (int64_t)blockIdx.x * per; p0 < count; p0 += (int64_t)gridDim.x * per) {
        const int64_t p = p0 + (threadIdx.x & 31) / G;
        if (p < count) {
            const double *q = params + 6 * p;
            for (int i = M.g; i < kN; i += G) {
                double row[9];
                vn_row<EQ, BULK>(q[0], q[1], q[2], q[3], i, row);
                M.set_row(i, row, q[4], q[5]);
            }
            if (!eig_hessenberg_qr(M) && M.g == 0) atomicExch(status, 1);
            if (M.g == 0) {
                // sort by decreasing modulus (insertion sort on the diagonal)
                for (int a = 1; a < kN; ++a) {
                    const cplx v = M.get(a, a);
                    const double m = cabs2(v);
                    int b = a - 1;
                    while (b >= 0) {
                        const cplx w = M.get(b, b);
                        if (!(cabs2(w) < m)) break;
                        M.set(b + 1, b + 1, w);
                        --b;
                    }
                    M.set(b + 1, b + 1, v);
                }
                for (int a = 0; a < kN; ++a) {
                    const cplx v = M.get(a, a);
                    out[(p * kN + a) * 2] = v.re;
                    out[(p * kN + a) * 2 + 1] = v.im;
                }
            }
            M.sync();
        }
        __syncwarp();
    }
}

// The bisection state of one (nu, theta) pair.  A round sweeps all wave vectors at the pair's
// next trial speed.  Beside it the round looks ahead: it tries the one wave vector that made the last
// unstable trial unstable at the trial speeds that follow as long as trials are unstable, after an
// unstable swept trial and after a stable one (vn_look_node; in the tree of trials below the swept
// one, node 1, node n has children 2 n after an unstable and 2 n + 1 after a stable trial).
// Where that is unstable again the trial is decided, and needs no sweep.
struct VnPair {
    double tau, theta, lo, hi, trial;
    double A[81];              // delta + J at the trial speed
    unsigned long long worst;  // bits of the largest spectral radius seen at the trial speed
    unsigned long long cand;   // the most unstable wave vector of the last unstable trial: growth
                               // (float bits) and, below it, its number + 1; 0: none yet
    int level;                 // trials decided (the first is u_hi itself)
    int done;                  // the limit is known
    unsigned long long look;   // `cand` as the round began
    int unstable[lbmh::kVnLooks];  // what the look-ahead found
};

// The bisection interval of tree node n below [lo, hi] (whose midpoint is node 1).
__device__ __forceinline__ double vn_node(double &lo, double &hi, int n) {
    for (int bit = 30 - __clz(n); bit >= 0; --bit) {
        const double mid = 0.5 * (lo + hi);
        if (n >> bit & 1) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

// One round (54 pairs x 25 x 25 wave vectors, 14 trials: a search took 15 sweeps of 4.1 ms and now
// 42 ms in all, 4.1 ms for the equilibrium that is stable at u_hi).  Blocks of the look-ahead (32 / G
// trial speeds of one pair each), then of the sweep (32 / G wave vectors of one pair each); without the
// look-ahead 32 / G wave vectors of whichever pairs they belong to.  A pair whose limit is known, or that some wave vector has already shown to be unstable,
// is skipped: one is enough.  The largest radius is kept per pair by an integer atomicMax on its bits
// (order-preserving for values >= 0).  A look-ahead that does not converge decides nothing.
template <int G, int EQ>
__global__ void __launch_bounds__(kVnThreads) k_vn_round(int64_t npairs, VnPair *pairs, int nk, double tol,
                                                         bool ahead, int32_t *status) {
    constexpr int per = kVnThreads / G;
    __shared__ double2 sm[kN * kN * per];
    const Mat<G> M(sm);
    const int m = (threadIdx.x & 31) / G;
    const int nkk = nk * nk;
    const int64_t looks = ahead ? npairs * ((lbmh::kVnLooks + per - 1) / per) : 0;
    const int64_t work = ahead ? looks + npairs * ((nkk + per - 1) / per) : (npairs * nkk + per - 1) / per;
    for (int64_t w = blockIdx.x; w < work; w += gridDim.x) {
        const bool look = w < looks;
        // the pair, and the number of the trial looked at or of the wave vector
        int64_t pr;
        int q;
        if (ahead) {
            const int64_t v = look ? w : w - looks, chunk = v / npairs;
            pr = v - chunk * npairs;
            q = (int)chunk * per + m;
        } else {
            const int64_t v = w * per + m;
            pr = v / nkk;
            q = pr < npairs ? (int)(v - pr * nkk) : nkk;
            pr = pr < npairs ? pr : 0;
        }
        VnPair *P = pairs + pr;
        const int kk = look ? (int)(unsigned)P->look - 1 : q;
        // (one lane reads what other blocks write, so that the group takes one branch)
        unsigned long long seen = 0;
        if (M.g == 0 && !look) seen = *(volatile unsigned long long *)&P->worst;
        seen = __shfl_sync(0xffffffffu, seen, threadIdx.x & 31 & ~(G - 1));
        const bool todo = !P->done && kk >= 0 && kk < nkk &&
                          (look ? q < lbmh::kVnLooks && P->level > 0 : !(__longlong_as_double((long long)seen) > 1.0 + tol));
        if (todo) {
            const int ix = kk % nk, iy = kk / nk;
            const double pi = 3.14159265358979323846;
            const double kx = nk > 1 ? pi * ix / (nk - 1) : 0.0, ky = nk > 1 ? pi * iy / (nk - 1) : 0.0;
            double ux = 0.0, uy = 0.0;
            if (look) {
                double lo = P->lo, hi = P->hi, st, ct;
                const double u = vn_node(lo, hi, lbmh::vn_look_node(q));
                sincos(P->theta, &st, &ct);
                ux = u * ct;
                uy = u * st;
            }
            for (int i = M.g; i < kN; i += G) {
                double row[9];
                if (look) {
                    vn_row<EQ, false>(P->tau, 1.0, ux, uy, i, row);
                } else {
#pragma unroll
                    for (int j = 0; j < 9; ++j) row[j] = P->A[9 * i + j];
                }
                M.set_row(i, row, kx, ky);
            }
            const bool converged = eig_hessenberg_qr(M);
            if (!converged && !look && M.g == 0) atomicExch(status, 1);
            if (M.g == 0) {
                double r = 0.0;
                for (int a = 0; a < kN; ++a) r = fmax(r, cabsd(M.get(a, a)));
                if (!(r >= 0.0)) r = 1e300;  // NaN: treat as unstable
                const bool unstable = r > 1.0 + tol;
                if (look) {
                    P->unstable[q] = converged && unstable;
                } else {
                    atomicMax(&P->worst, (unsigned long long)__double_as_longlong(r));
                    if (unstable)
                        atomicMax(&P->cand, (unsigned long long)__float_as_uint((float)fmin(r - 1.0, 1e30)) << 32 |
                                                (unsigned)(kk + 1));
                }
            }
            M.sync();
        }
        __syncwarp();
    }
}

// After a round: narrow each pair's interval by the swept trial and by what the look-ahead decided, set
// its next trial speed and form delta + J there, one pair to a block; before the first (`start`): the
// pair's state from in[2 p] = tau and in[2 p + 1] = theta.  limit[p]: the largest speed known to be stable.
template <int EQ>
__global__ void __launch_bounds__(32) k_vn_bisect(int64_t npairs, VnPair *pairs, const double *in, double *limit, int start,
                                                  int iterations, double u_hi, double tol) {
    for (int64_t p = blockIdx.x; p < npairs; p += gridDim.x) {
        VnPair *P = pairs + p;
        const double tau = in[2 * p], theta = in[2 * p + 1];
        double lo = 0.0, hi = u_hi, trial = u_hi;
        int done = 0, level = 0;
        if (!start) {
            lo = P->lo;
            hi = P->hi;
            trial = P->trial;
            done = P->done;
            level = P->level;
        }
        if (!start && !done) {
            const bool stable = __longlong_as_double((long long)P->worst) <= 1.0 + tol;
            int next = 0, last = 0;  // the look-ahead's trials that follow
            if (level == 0) {  // the trial was u_hi itself: a pair stable there reports u_hi
                if (stable) {
                    lo = hi = u_hi;
                    done = 1;
                }
                next = last = 0;  // nothing was looked up yet
            } else {
                if (lo < hi) {
                    if (stable) lo = trial;
                    else hi = trial;
                }
                next = stable ? lbmh::kVnLooks / 2 : 0;
                last = next + lbmh::kVnLooks / 2;
            }
            ++level;
            trial = 0.5 * (lo + hi);
            while (level <= iterations && next < last && P->unstable[next]) {
                if (lo < hi) hi = trial;
                ++next;
                ++level;
                trial = 0.5 * (lo + hi);
            }
            if (level > iterations) done = 1;
        }
        __syncwarp();
        if (threadIdx.x < lbmh::kVnLooks) P->unstable[threadIdx.x] = 0;
        if (threadIdx.x == 0) {
            P->lo = lo;
            P->hi = hi;
            P->trial = trial;
            P->level = level;
            P->done = done;
            P->worst = 0;
            if (start) {
                P->tau = tau;
                P->theta = theta;
                P->look = 0;
            } else if (P->cand) {
                P->look = P->cand;
            }
            P->cand = 0;
            limit[p] = lo;
        }
        if (threadIdx.x < kN && !done) {
            double st, ct, row[9];
            sincos(theta, &st, &ct);
            vn_row<EQ, false>(tau, 1.0, trial * ct, trial * st, threadIdx.x, row);
            for (int j = 0; j < 9; ++j) P->A[9 * threadIdx.x + j] = row[j];
        }
        __syncwarp();
    }
}

}  // namespace lbmd

namespace lbmh {

using namespace lbmd;

static int grid_n(int64_t blocks) { return (int)(blocks < 1 ? 1 : (blocks > 152 * 64 ? 152 * 64 : blocks)); }

// Lanes a matrix: 4 while that gives every SM quarter (608) one warp at most, where the latency of
// one solve is the time and more lanes shorten it; then 2, and 1 where the FP64 pipe's throughput
// counts, which shared-out rotations waste (4096 spectra 2.69 -> 1.35 ms, 16384 5.1 -> 4.7 ms with
// 2 lanes (5.3 with one), 65536 15.2 -> 13.4 ms with one lane (14.7 with two)).
static int vn_lanes(int64_t matrices) {
    const int64_t slots = (int64_t)608 * kVnThreads;
    return matrices * 4 <= slots ? 4 : (matrices <= slots ? 2 : 1);
}

template <int G>
static cudaError_t vn_eigs_g(int eq, int bulk, int64_t count, const double *params, double *out, int32_t *status,
                             cudaStream_t s) {
    const int g = grid_n((count * G + kVnThreads - 1) / kVnThreads);
#define LBM_VN(EQv)                                                                                  \
    if (eq == EQv) {                                                                                 \
        if (bulk) k_vn_eigs<G, EQv, true><<<g, kVnThreads, 0, s>>>(count, params, out, status);      \
        else k_vn_eigs<G, EQv, false><<<g, kVnThreads, 0, s>>>(count, params, out, status);          \
        return cudaGetLastError();                                                                   \
    }
    LBM_VN(EQ_ENT)
    LBM_VN(EQ_POLY2)
    LBM_VN(EQ_PROD)
#undef LBM_VN
    return cudaErrorInvalidValue;
}

cudaError_t vn_eigs(int eq, int bulk, int64_t count, const double *params, double *out, int32_t *status,
                    cudaStream_t s) {
    switch (vn_lanes(count)) {
    case 4: return vn_eigs_g<4>(eq, bulk, count, params, out, status, s);
    case 2: return vn_eigs_g<2>(eq, bulk, count, params, out, status, s);
    default: return vn_eigs_g<1>(eq, bulk, count, params, out, status, s);
    }
}

size_t vn_limit_bytes(int64_t npairs) { return sizeof(VnPair) * (size_t)npairs; }

template <int EQ, int G>
static cudaError_t vn_limit_g(int64_t npairs, VnPair *P, const double *in, double *limit, int nk, double u_hi, int iterations, double tol,
                               int32_t *status, cudaStream_t s) {
    constexpr int per = kVnThreads / G;
    const int gb = grid_n(npairs);
    // The look-ahead where it costs little: at most an eighth of a sweep, or no more than there are SM
    // quarters to run it beside the sweep.  Otherwise the wave vectors of the pairs lie densely on the lanes
    // (2000 pairs, 3 x 3 wave vectors: look-ahead and a block for each pair 132 ms, no look-ahead 83, densely 28; one
    // matrix a thread and all sweeps took 34).
    const int64_t looks = (kVnLooks + per - 1) / per, sweep = ((int64_t)nk * nk + per - 1) / per;
    const bool ahead = 8 * looks <= sweep || npairs * (looks + sweep) <= 608;
    const int gr = grid_n(ahead ? npairs * (sweep + looks) : (npairs * nk * nk + per - 1) / per);
    k_vn_bisect<EQ><<<gb, 32, 0, s>>>(npairs, P, in, limit, 1, iterations, u_hi, tol);
    for (int it = 0; it <= iterations; ++it) {  // every round decides at least one trial of a pair
        k_vn_round<G, EQ><<<gr, kVnThreads, 0, s>>>(npairs, P, nk, tol, ahead, status);
        k_vn_bisect<EQ><<<gb, 32, 0, s>>>(npairs, P, in, limit, 0, iterations, u_hi, tol);
    }
    return cudaGetLastError();
}

template <int EQ>
static cudaError_t vn_limit_eq(int64_t npairs, VnPair *P, const double *in, double *limit, int nk, double u_hi, int iterations, double tol,
                               int32_t *status, cudaStream_t s) {
    if (vn_lanes(npairs * nk * nk) == 4) return vn_limit_g<EQ, 4>(npairs, P, in, limit, nk, u_hi, iterations, tol, status, s);
    return vn_limit_g<EQ, 1>(npairs, P, in, limit, nk, u_hi, iterations, tol, status, s);
}

cudaError_t vn_limit(int eq, int64_t npairs, void *pairs, const double *in, double *limit, int nk, double u_hi, int iterations, double tol,
                     int32_t *status, cudaStream_t s) {
    VnPair *P = static_cast<VnPair *>(pairs);
    if (eq == EQ_ENT) return vn_limit_eq<EQ_ENT>(npairs, P, in, limit, nk, u_hi, iterations, tol, status, s);
    if (eq == EQ_POLY2) return vn_limit_eq<EQ_POLY2>(npairs, P, in, limit, nk, u_hi, iterations, tol, status, s);
    if (eq == EQ_PROD) return vn_limit_eq<EQ_PROD>(npairs, P, in, limit, nk, u_hi, iterations, tol, status, s);
    return cudaErrorInvalidValue;
}

}  // namespace lbmh
