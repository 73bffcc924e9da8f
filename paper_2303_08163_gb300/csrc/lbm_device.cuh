// lbm_device.cuh -- device-side lattice constants, storage formats and the fused
// equilibrium + BGK collision of one cell (arXiv 2303.08163, Sec. II and Sec. V.B).
//
// Populations are held shifted, ft_i = f_i - w_i rho0.  The collision of one cell:
//   moments     rho = rho0 + sum ft_i, j = sum c_i ft_i (sum w_i c_i = 0), u = j / rho
//   equilibrium f_i^eq - w_i rho0 = w_i (drho + rho h_i), drho = rho - rho0, with
//     entropic (Eq. eq:Entropic_isothermal_EDF): f^eq_i = w_i rho prod_a t_a(c_ia),
//       t(0) = 2 - S, t(+-1) = (2 - S) Z^{+-1} = 2 S - 1 +- 3u, S = sqrt(1 + 3 u^2).
//       (The identity (2 - S)(2u + S) = (2S - 1 + 3u)(1 - u) follows from S^2 = 1 + 3u^2
//       and removes the division by 1 - u.)  With d = t - 1:
//       d(0) = -(S - 1), d(+-1) = 2 (S - 1) +- 3u, S - 1 = 3u^2 / (1 + S) (no cancellation),
//       h_i = prod_a (1 + d_a) - 1 built by nested fused multiply-adds.
//     product form (Eq. eq:Product_isothermal_EDF): same structure with
//       t(0) = 1 - 3/2 u^2, t(+-1) = 1 +- 3u + 3u^2 (i.e. the 1-D factors divided by w).
//     quadratic (Eq. eq:Poly2_isothermal_EDF): h_i = 3 c.u + 9/2 (c.u)^2 - 3/2 u^2.
//   relaxation  2 beta = 1 / tau, or with the local bulk correction (Eq. eq:redefined_
//     relaxation rate) 2 beta = 2 A vs^2 / (2 nu + A vs^2) = 2 A / (6 nu + A), where
//     A = min_a A(u_a).  For the entropic equilibrium Eq. (eq:entropic_bulk) simplifies,
//     with S^2 = 1 + x^2, to A = (2 - S) / S^2, which decreases with |u|, so the minimum
//     is taken at the largest S.  For the polynomial forms A = 1 - 9/2 u^2 (Eq. eq:LBGK_bulk).
//   collide     ft*_i = ft_i + 2 beta (ft^eq_i - ft_i) = (1 - 2beta) ft_i + 2beta w_i (drho + rho h_i).
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

namespace lbmd {

enum { P_F64 = 0, P_F32 = 1, P_F16S = 2 };
enum { EQ_ENT = 0, EQ_POLY2 = 1, EQ_PROD = 2 };

__host__ __device__ constexpr int qof(int D) { return D == 2 ? 9 : 27; }
// population index i = (cx + 1) + 3 (cy + 1) + 9 (cz + 1); opposite = Q - 1 - i
__host__ __device__ constexpr int cxo(int i) { return i % 3 - 1; }
__host__ __device__ constexpr int cyo(int i) { return (i / 3) % 3 - 1; }
__host__ __device__ constexpr int czo(int i) { return i / 9 - 1; }
__host__ __device__ constexpr double w1d(int c) { return c == 0 ? 2.0 / 3.0 : 1.0 / 6.0; }
template <int D>
__host__ __device__ constexpr double wq(int i) {
    return D == 2 ? w1d(cxo(i)) * w1d(cyo(i)) : w1d(cxo(i)) * w1d(cyo(i)) * w1d(czo(i));
}
// weight class: number of nonzero velocity components (0 .. D); for D = 2 only the
// first two digits of the index are velocity components
template <int D>
__host__ __device__ constexpr int wclass(int i) {
    return (cxo(i) != 0) + (cyo(i) != 0) + (D == 3 && czo(i) != 0);
}
// weight of a population with n nonzero components: (1/6)^n (2/3)^(D - n)
template <int D>
__host__ __device__ constexpr double wclass_weight(int n) {
    return (n >= 1 ? 1.0 / 6.0 : 1.0) * (n >= 2 ? 1.0 / 6.0 : 1.0) * (n >= 3 ? 1.0 / 6.0 : 1.0) *
           (D - n >= 1 ? 2.0 / 3.0 : 1.0) * (D - n >= 2 ? 2.0 / 3.0 : 1.0) *
           (D - n >= 3 ? 2.0 / 3.0 : 1.0);
}

template <int P> struct Storage;
template <> struct Storage<P_F64> {
    using T = double;
    using R = double;
    static __host__ __device__ __forceinline__ R load(T v) { return v; }
    static __host__ __device__ __forceinline__ T store(R v) { return v; }
};
template <> struct Storage<P_F32> {
    using T = float;
    using R = float;
    static __host__ __device__ __forceinline__ R load(T v) { return v; }
    static __host__ __device__ __forceinline__ T store(R v) { return v; }
};
template <> struct Storage<P_F16S> {
    using T = __half;
    using R = float;
    static __host__ __device__ __forceinline__ R load(T v) { return __half2float(v); }
    static __host__ __device__ __forceinline__ T store(R v) { return __float2half_rn(v); }
};

// Arithmetic helpers of the field transfers: FP64 takes IEEE square root and division (the
// collisions have rcp_ulp and sqrt_ulp below); FP32 the hardware reciprocal square root and fast
// division (a few ulp, far below the storage rounding of the FP32 and binary16 formats).
__host__ __device__ __forceinline__ double sqrt_r(double x) { return sqrt(x); }
__host__ __device__ __forceinline__ float sqrt_r(float x) {
#ifdef __CUDA_ARCH__
    return x * rsqrtf(x);
#else
    return sqrtf(x);
#endif
}
__host__ __device__ __forceinline__ double div_r(double a, double b) { return a / b; }
__host__ __device__ __forceinline__ float div_r(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fdividef(a, b);
#else
    return a / b;
#endif
}
__host__ __device__ __forceinline__ double fma_r(double a, double b, double c) { return fma(a, b, c); }
__host__ __device__ __forceinline__ float fma_r(float a, float b, float c) { return fmaf(a, b, c); }

// Products of the FP64 collisions that feed a sum.  Whether the compiler fuses such a product into the
// sum depends on the code around it; the collisions of all kernels (a cell on a thread, a cell on
// three lanes, steps with diagnostics) store the same bits because no operation is left to it.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// FP64 reciprocal and square root of the collisions: the hardware approximation of PTX
// rcp / rsqrt.approx.ftz.f64 (better than 2^-20) and one step of a third-order Householder
// iteration, whose error e^3 lies far below the last bit; what is left is the rounding of the last
// operations, about an ulp.  On the FP64 pipe (64 clocks a warp instruction on an SM quarter) they
// take 3 and 5 instructions; the IEEE division measured 5.5, the square root 9.8.
//   1/x     = y (1 + e + e^2),             e = 1 - x y
//   sqrt(x) = t (1 + e (1/2 + 3/8 e)),     t = x y, e = 1 - t y
// The approximations flush what is no normal number to zero (then 0 x infinity: no number), so x
// and 1/x have to be normal.
__device__ __forceinline__ double rcp_ulp(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double sqrt_ulp(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double t = x * y, e = fma(-t, y, 1.0);
    return fma(t * e, fma(e, 0.375, 0.5), t);
}

// Exponents by integer arithmetic, which costs the FP64 pipe nothing: x / 2^n (exact; what falls below
// the normal numbers becomes some number below them, what rises above them becomes infinite or no
// number), and 1/x within an ulp for every x for which both are normal.
__device__ __forceinline__ int exponent_of(double x) { return (__double2hiint(x) >> 20 & 0x7ff) - 1023; }
__device__ __forceinline__ double scale_down(double x, int n) {
    const int hi = __double2hiint(x), e = hi >> 20 & 0x7ff;
    const int t = min(max(e - n, 0), 0x7ff);
    return e == 0 ? x : __hiloint2double((hi & (int)0x800fffff) | t << 20, __double2loint(x));
}
__device__ __forceinline__ double rcp_any(double x) {
    const int n = exponent_of(x);
    return scale_down(rcp_ulp(scale_down(x, n)), n);
}

template <typename R> struct CellMoments {
    R rho;   // density
    R u[3];  // velocity (u[2] = 0 in 2-D)
};

// Per-axis equilibrium factors d(c) = t(c) - 1 for c = -1, 0, +1; also returns the
// quantity the bulk coefficient depends on (S for the entropic form, u^2 otherwise).
template <int EQ, typename R>
__host__ __device__ __forceinline__ void axis_factors(R u, R &dm, R &d0, R &dp, R &key) {
    const R u2 = u * u;
    if constexpr (EQ == EQ_ENT) {
        const R s2 = fma_r(R(3), u2, R(1));
        const R S = sqrt_r(s2);
        const R sm1 = div_r(R(3) * u2, R(1) + S);  // S - 1 without cancellation
        d0 = -sm1;
        dp = fma_r(R(2), sm1, R(3) * u);
        dm = fma_r(R(2), sm1, R(-3) * u);
        key = S;
    } else {  // product form (also used for the per-axis key of the polynomial form)
        const R t3 = R(3) * u2;
        d0 = R(-1.5) * u2;
        dp = fma_r(R(3), u, t3);
        dm = fma_r(R(-3), u, t3);
        key = u2;
    }
}

// The per-axis factors of all D axes.  In FP64 the entropic form's D divisions
// 3u_a^2 / (1 + S_a) share one reciprocal of the product of the (1 + S_a), each axis
// multiplying it by the other axes' factors (a few ulp, one IEEE division instead of D;
// FP64 divisions are long instruction sequences on the FP64 pipe).
template <int D, int EQ, typename R>
__host__ __device__ __forceinline__ void all_axis_factors(const R (&u)[3], R (&dm)[3], R (&d0)[3],
                                                          R (&dp)[3], R (&key)[3]) {
    if constexpr (EQ == EQ_ENT && sizeof(R) == 8) {
        R u2[3], S[3], op[3];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            u2[a] = u[a] * u[a];
            S[a] = sqrt_r(fma_r(R(3), u2[a], R(1)));
            op[a] = R(1) + S[a];
        }
        R inv[3];
        if constexpr (D == 2) {
            const R r = R(1) / (op[0] * op[1]);
            inv[0] = r * op[1];
            inv[1] = r * op[0];
        } else {
            const R yz = op[1] * op[2];
            const R r = R(1) / (op[0] * yz);
            inv[0] = r * yz;
            inv[1] = r * (op[0] * op[2]);
            inv[2] = r * (op[0] * op[1]);
        }
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const R sm1 = R(3) * u2[a] * inv[a];  // S - 1 without cancellation
            d0[a] = -sm1;
            dp[a] = fma_r(R(2), sm1, R(3) * u[a]);
            dm[a] = fma_r(R(2), sm1, R(-3) * u[a]);
            key[a] = S[a];
        }
    } else {
#pragma unroll
        for (int a = 0; a < D; ++a) axis_factors<EQ>(u[a], dm[a], d0[a], dp[a], key[a]);
    }
}

// Local collision frequency 2 beta from the largest per-axis key (FP64; rate32 for FP32).
template <int EQ, bool BULK, typename R>
__device__ __forceinline__ R collision_rate(R key_max, R omega0, R six_nu) {
    if constexpr (!BULK) {
        return omega0;
    } else if constexpr (EQ == EQ_ENT) {
        const R S = key_max;
        const R A2 = R(2) - S;                      // A S^2
        return mul_rn(R(2) * A2, rcp_ulp(fma_r(six_nu, S * S, A2)));
    } else {
        const R A = fma_r(R(-4.5), key_max, R(1));  // 1 - 3/2 u^2 / vs^2
        return mul_rn(R(2) * A, rcp_ulp(six_nu + A));
    }
}

// h_i such that f^eq_i - w_i rho0 = w_i (drho + rho h_i), for all i; returns the
// largest per-axis key (see axis_factors) for the bulk correction.
template <int D, int EQ, typename R>
__host__ __device__ __forceinline__ R equilibrium_h(const R (&u)[3], R (&h)[qof(D)]) {
    constexpr int Q = qof(D);
    if constexpr (EQ == EQ_POLY2) {
        // h = 3 cu + 9/2 cu^2 - 3/2 u^2
        R uu = u[0] * u[0] + u[1] * u[1];
        if constexpr (D == 3) uu = fma_r(u[2], u[2], uu);
        const R m = R(-1.5) * uu;
        R cxy[9];
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const int cx = cxo(p), cy = cyo(p);
            R v = R(0);
            if (cx == 1) v = u[0];
            if (cx == -1) v = -u[0];
            if (cy == 1) v = v + u[1];
            if (cy == -1) v = v - u[1];
            cxy[p] = v;
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int cz = (D == 3) ? czo(i) : 0;
            R cu = cxy[i % 9];
            if (cz == 1) cu = cu + u[2];
            if (cz == -1) cu = cu - u[2];
            h[i] = fma_r(cu, fma_r(R(4.5), cu, R(3)), m);
        }
        R k = u[0] * u[0];
        k = fmax(k, u[1] * u[1]);
        if constexpr (D == 3) k = fmax(k, u[2] * u[2]);
        return k;
    } else {
        R dm[3], d0[3], dp[3], key[3];
        all_axis_factors<D, EQ>(u, dm, d0, dp, key);
        R kmax = fmax(key[0], key[1]);
        if constexpr (D == 3) kmax = fmax(kmax, key[2]);
        // d and t = 1 + d per axis, indexed by c + 1
        R dx[3] = {dm[0], d0[0], dp[0]};
        R dy[3] = {dm[1], d0[1], dp[1]};
        R tx[3] = {R(1) + dm[0], R(1) + d0[0], R(1) + dp[0]};
        if constexpr (D == 2) {
#pragma unroll
            for (int i = 0; i < 9; ++i) h[i] = fma_r(dy[cyo(i) + 1], tx[cxo(i) + 1], dx[cxo(i) + 1]);
        } else {
            R ty[3] = {R(1) + dm[1], R(1) + d0[1], R(1) + dp[1]};
            R dz[3] = {dm[2], d0[2], dp[2]};
            R exy[9], txy[9];
#pragma unroll
            for (int p = 0; p < 9; ++p) {
                exy[p] = fma_r(dy[cyo(p) + 1], tx[cxo(p) + 1], dx[cxo(p) + 1]);
                txy[p] = tx[cxo(p) + 1] * ty[cyo(p) + 1];
            }
#pragma unroll
            for (int i = 0; i < 27; ++i) h[i] = fma_r(dz[czo(i) + 1], txy[i % 9], exy[i % 9]);
        }
        return kmax;
    }
}

// Density (its difference from rho0 is returned) and momentum of one cell from shifted
// populations.  The partial sums follow the tensor structure of the lattice (first over c_z, then
// c_y, then c_x).
template <int D, typename R>
__host__ __device__ __forceinline__ R moment_sums(const R (&f)[qof(D)], R rho0, R &rho, R (&j)[3]) {
    R a[9], bz[9];
    if constexpr (D == 2) {
#pragma unroll
        for (int p = 0; p < 9; ++p) a[p] = f[p];
    } else {
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            a[p] = (f[p] + f[p + 9]) + f[p + 18];
            bz[p] = f[p + 18] - f[p];
        }
    }
    const R c0 = (a[0] + a[3]) + a[6];  // c_x = -1
    const R c1 = (a[1] + a[4]) + a[7];  // c_x = 0
    const R c2 = (a[2] + a[5]) + a[8];  // c_x = +1
    const R rt = (c0 + c1) + c2;
    j[0] = c2 - c0;
    j[1] = ((a[6] + a[7]) + a[8]) - ((a[0] + a[1]) + a[2]);
    j[2] = R(0);
    if constexpr (D == 3) {
        j[2] = ((bz[0] + bz[1]) + (bz[2] + bz[3])) + ((bz[4] + bz[5]) + (bz[6] + bz[7])) + bz[8];
    }
    rho = rho0 + rt;
    return rt;
}

// Moments of one cell from shifted populations: rho and u = j / rho.
template <int D, typename R>
__host__ __device__ __forceinline__ CellMoments<R> moments_shifted(const R (&f)[qof(D)], R rho0) {
    CellMoments<R> m;
    R jv[3];
    moment_sums<D, R>(f, rho0, m.rho, jv);
    const R jx = jv[0], jy = jv[1], jz = jv[2];
    const R inv = div_r(R(1), m.rho);
    m.u[0] = jx * inv;
    m.u[1] = jy * inv;
    m.u[2] = jz * inv;
    return m;
}

// The terms of the FP64 tensor-product equilibria (entropic, product).  With t_a(c) = 1 + d_a(c)
// the factor of axis a, d = prod t_a - 1 and X_a(c) = rho d_a(c), the deviation of a direction's
// equilibrium over its weight is
//   g = drho + rho d = (drho + X_x) + t_x X_y (+ t_x t_y X_z),
// one FMA per direction and axis beyond the first; the relaxation f* = (1 - 2beta) f + 2beta w g is
// two more.  (FP64 collisions are bound by their instruction count.  Forming rho d from d instead
// took the products 2beta w rho and 2beta w drho per weight and d itself: 4 instructions more in
// 2-D, 10 in 3-D, and no X without a product with 1/rho.)
//
// Entropic form: with j3 = 3 j, T_a = rho S_a = sqrt(rho^2 + j3_a j_a) and q_a = rho + T_a, the term
// rho (S_a - 1) is j3_a j_a / q_a (no cancellation: an ulp of T stays an ulp), and one reciprocal of
// the product rho prod q_a gives 1/rho and every 1/q_a.  Errors against 64-bit references are those
// of the direct forms with IEEE division and square root (2-D and 3-D, all options).
// 4096-lattice sweep: 5.20 -> 4.79 ms a step with the own reciprocal and square root, 4.53 with
// these terms; D3Q27 128^3 882 -> 842 -> 820 us.
// Where rho is negative T is the other root, and the product, of the order rho^(D+1), leaves FP64's
// range long before rho does (rho0 = 1e80).  The product itself tells both (terms_ok): it is negative,
// or too small or large.  Such a cell forms its terms with the sign of rho, and without rho's power of
// two, which changes nothing but the exponents.  (All cells in that way: sweep 4.79 -> 4.92 ms a step;
// only those that need it: 4.79, 64^2 2.67 -> 2.74, 48^3 48 -> 49.5 us a step.)
__device__ __forceinline__ bool terms_ok(double product) { return ((unsigned)__double2hiint(product) >> 20) - 64u < 1920u; }

// e_a = rho (S_a - 1), key_a = S_a and 1/rho; returns the product.  SIGNED: for rho of any sign.
template <int D, bool SIGNED>
__device__ __forceinline__ double entropic_terms(double rho, const double (&j)[3], double (&e)[D], double (&key)[D], double &irho) {
    double jj[D], T[D], q[D], others[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        jj[a] = 3.0 * j[a] * j[a];
        T[a] = sqrt_ulp(fma(rho, rho, jj[a]));
        if constexpr (SIGNED) T[a] = copysign(T[a], rho);
        q[a] = rho + T[a];
    }
    if constexpr (D == 2) {
        others[0] = q[1];
        others[1] = q[0];
    } else {
        others[0] = q[1] * q[2];
        others[1] = q[0] * q[2];
        others[2] = q[0] * q[1];
    }
    const double all = q[0] * others[0], product = rho * all, r = rcp_ulp(product), v = r * rho;  // v = 1 / prod q
    irho = r * all;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        e[a] = mul_rn(jj[a], v * others[a]);
        key[a] = mul_rn(T[a], irho);
    }
    return product;
}
template <int D>
__device__ __forceinline__ void entropic_terms_any(double rho, const double (&j)[3], double (&e)[D], double (&key)[D], double &irho) {
    const int n = exponent_of(rho);
    const double j1[3] = {scale_down(j[0], n), scale_down(j[1], n), scale_down(j[2], n)};
    entropic_terms<D, true>(scale_down(rho, n), j1, e, key, irho);
    irho = scale_down(irho, n);
#pragma unroll
    for (int a = 0; a < D; ++a) e[a] = scale_down(e[a], -n);
}

template <typename R> struct TensorTerms {
    R drho, irho, X[3][3], key[3];  // X by axis and c + 1; key: what the bulk coefficient depends on
};

// The moment sums of the FP64 collision: first over the populations of each last velocity component
// (what one of the three lanes of collide_lanes holds), then over those.
template <int D> __device__ __forceinline__ void last_axis_sums(const double *f, double &sum, double (&part)[2]) {
    if constexpr (D == 2) {
        sum = (f[0] + f[1]) + f[2];
        part[0] = f[2] - f[0];
        part[1] = 0.0;
    } else {
        const double c0 = (f[0] + f[3]) + f[6], c1 = (f[1] + f[4]) + f[7], c2 = (f[2] + f[5]) + f[8];
        sum = (c0 + c1) + c2;
        part[0] = c2 - c0;
        part[1] = ((f[6] + f[7]) + f[8]) - ((f[0] + f[1]) + f[2]);
    }
}
template <int D>
__device__ __forceinline__ double collision_sums(const double (&f)[qof(D)], double rho0, double &rho, double (&j)[3]) {
    constexpr int F = D == 2 ? 3 : 9;
    double s[3], p[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) last_axis_sums<D>(f + F * c, s[c], p[c]);
    const double drho = (s[0] + s[1]) + s[2];
    rho = rho0 + drho;
    j[2] = 0.0;
#pragma unroll
    for (int a = 0; a < D - 1; ++a) j[a] = (p[0][a] + p[1][a]) + p[2][a];
    j[D - 1] = s[2] - s[0];
    return drho;
}

template <int D, int EQ, typename R>
__device__ __forceinline__ void tensor_terms(const R (&f)[qof(D)], R rho0, CellMoments<R> &m, TensorTerms<R> &t) {
    R j[3], j3[3];
    t.drho = collision_sums<D>(f, rho0, m.rho, j);
    const R rho = m.rho;
#pragma unroll
    for (int a = 0; a < D; ++a) j3[a] = R(3) * j[a];
    if constexpr (EQ == EQ_ENT) {
        R e[D], key[D];
        if (!terms_ok(entropic_terms<D, false>(rho, j, e, key, t.irho))) entropic_terms_any<D>(rho, j, e, key, t.irho);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            t.X[a][0] = fma_r(R(2), e[a], -j3[a]);
            t.X[a][1] = -e[a];
            t.X[a][2] = fma_r(R(2), e[a], j3[a]);
            t.key[a] = key[a];
        }
    } else {
        t.irho = rcp_any(rho);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const R u = j[a] * t.irho;
            t.X[a][0] = fma_r(j3[a], u, -j3[a]);
            t.X[a][1] = mul_rn(R(-0.5), j3[a] * u);
            t.X[a][2] = fma_r(j3[a], u, j3[a]);
            t.key[a] = u * u;
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) m.u[a] = a < D ? mul_rn(j[a], t.irho) : R(0);
}

// ------------------------------------------------------------------ FP32 collisions
//
// The FP32 collision is written over a value type V: float (one cell) or f32x2 (two cells,
// one in each half of a 64-bit register pair, advanced by the packed fma / mul / add.f32x2
// instructions of sm_100 and later).  Both forms issue the same correctly rounded operations
// in the same order, so the one-cell and the two-cell kernels store the same bits.  (The
// scalar _rn intrinsics are never contracted; a packed product that only feeds packed sums
// was seen to be, so such sums are written as fma.)
struct f32x2 {
    unsigned long long v;
};
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 a, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ f32x2 vadd(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 vmul(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 vfma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ f32x2 vsub(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
template <typename V> __device__ __forceinline__ V vset(float c);
template <> __device__ __forceinline__ float vset<float>(float c) { return c; }
template <> __device__ __forceinline__ f32x2 vset<f32x2>(float c) { return pack2(c, c); }

// A product that keeps its own rounding when it feeds a sum (adding -0 changes nothing, and
// an fma is never contracted further).
template <typename V> __device__ __forceinline__ V vmul_alone(V a, V b) { return vfma(a, b, vset<V>(-0.0f)); }

// Hardware reciprocal and reciprocal square root (a few ulp, far below the storage rounding
// of the FP32 and binary16 formats).
__device__ __forceinline__ float vrcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// The same for a density that may lie below the normal numbers: FP32 storage with a reference density to
// match (for every FP32 cell 509 x 381 quadratic 3.85 -> 3.91 us a step, 4096^2 binary16, whose storage
// holds no such state, 75.7 -> 77.8).
__device__ __forceinline__ float vrcp_any(float x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float vrsqrt(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ f32x2 vrcp(f32x2 a) {
    float x, y;
    unpack2(a, x, y);
    return pack2(vrcp(x), vrcp(y));
}
__device__ __forceinline__ f32x2 vrcp_any(f32x2 a) {
    float x, y;
    unpack2(a, x, y);
    return pack2(vrcp_any(x), vrcp_any(y));
}
__device__ __forceinline__ f32x2 vrsqrt(f32x2 a) {
    float x, y;
    unpack2(a, x, y);
    return pack2(vrsqrt(x), vrsqrt(y));
}
__device__ __forceinline__ f32x2 vmax(f32x2 a, f32x2 b) {
    float x, y, z, w;
    unpack2(a, x, y);
    unpack2(b, z, w);
    return pack2(fmaxf(x, z), fmaxf(y, w));
}

template <typename V> struct Moments32 {
    V rho, u[3];
};

// 2 beta of the FP32 collision from the largest per-axis key (see collision_rate).
template <int EQ, bool BULK, typename V>
__device__ __forceinline__ V rate32(V key_max, V omega0, V six_nu) {
    if constexpr (!BULK) {
        return omega0;
    } else if constexpr (EQ == EQ_ENT) {
        const V A2 = vsub(vset<V>(2.0f), key_max);
        return vmul(vadd(A2, A2), vrcp(vfma(six_nu, vmul(key_max, key_max), A2)));
    } else {
        const V A = vfma(vset<V>(-4.5f), key_max, vset<V>(1.0f));
        return vmul(vadd(A, A), vrcp(vadd(six_nu, A)));
    }
}

// The relaxation f* = (1 - 2beta) f + 2beta w_i (drho + rho h_i) of one direction of weight
// class c, in one of two forms: factored, 2beta w (rho h + drho) + (1 - 2beta) f, or for D2Q9
// binary16 two FMAs with the per-class products 2beta w rho and 2beta w drho formed once.
// (The results of the two differ in the last bit; each storage keeps its own.)
template <int D, int P, typename V> struct Relax32 {
    static constexpr bool kTwoFma = D == 2 && P == P_F16S;
    V keep, rho, drho, omw[4], wr[4], wd[4];
    __device__ __forceinline__ Relax32(V om, V rho_, V drho_) : keep(vsub(vset<V>(1.0f), om)), rho(rho_), drho(drho_) {
#pragma unroll
        for (int c = 0; c <= D; ++c) {
            omw[c] = vmul(om, vset<V>((float)wclass_weight<D>(c)));
            if constexpr (kTwoFma) {
                wr[c] = vmul(omw[c], rho);
                wd[c] = vmul(omw[c], drho);
            }
        }
    }
    __device__ __forceinline__ V operator()(int c, V h, V f) const {
        if constexpr (kTwoFma) return vfma(wr[c], h, vfma(keep, f, wd[c]));
        else return vfma(omw[c], vfma(rho, h, drho), vmul(keep, f));
    }
};

// The fused FP32 collision, in place on shifted populations; returns the pre-collision
// moments.
template <int D, int P, int EQ, bool BULK, typename V>
__device__ __forceinline__ Moments32<V> collide32(V (&f)[qof(D)], float rho0s, float omega0s, float six_nus) {
    constexpr int Q = qof(D);
    const V rho0 = vset<V>(rho0s), one = vset<V>(1.0f);
    Moments32<V> m;
    V j[3];
    {
        V a[9];
        if constexpr (D == 2) {
#pragma unroll
            for (int p = 0; p < 9; ++p) a[p] = f[p];
        } else {
            V bz[9];
#pragma unroll
            for (int p = 0; p < 9; ++p) {
                a[p] = vadd(vadd(f[p], f[p + 9]), f[p + 18]);
                bz[p] = vsub(f[p + 18], f[p]);
            }
            j[2] = vadd(vadd(vadd(vadd(bz[0], bz[1]), vadd(bz[2], bz[3])), vadd(vadd(bz[4], bz[5]), vadd(bz[6], bz[7]))), bz[8]);
        }
        const V c0 = vadd(vadd(a[0], a[3]), a[6]);  // c_x = -1
        const V c1 = vadd(vadd(a[1], a[4]), a[7]);  // c_x = 0
        const V c2 = vadd(vadd(a[2], a[5]), a[8]);  // c_x = +1
        m.rho = vadd(rho0, vadd(vadd(c0, c1), c2));
        j[0] = vsub(c2, c0);
        j[1] = vsub(vadd(vadd(a[6], a[7]), a[8]), vadd(vadd(a[0], a[1]), a[2]));
    }
    V inv = vrcp(m.rho);
    if constexpr (P == P_F32) {
        if (rho0s < 1e-30f) inv = vrcp_any(m.rho);
    }
    m.u[2] = vset<V>(0.0f);
#pragma unroll
    for (int a = 0; a < D; ++a) m.u[a] = vmul(j[a], inv);
    const V drho = vsub(m.rho, rho0);
    if constexpr (EQ == EQ_POLY2) {
        V uu, k;
        if constexpr (BULK) {
            const V xx = vmul_alone(m.u[0], m.u[0]), yy = vmul_alone(m.u[1], m.u[1]);
            uu = vadd(xx, yy);
            k = vmax(xx, yy);
            if constexpr (D == 3) k = vmax(k, vmul(m.u[2], m.u[2]));
        } else {
            uu = k = vfma(m.u[0], m.u[0], vmul(m.u[1], m.u[1]));
        }
        if constexpr (D == 3) uu = vfma(m.u[2], m.u[2], uu);
        const Relax32<D, P, V> relax(rate32<EQ, BULK, V>(k, vset<V>(omega0s), vset<V>(six_nus)), m.rho, drho);
        const V mh = vmul(vset<V>(-1.5f), uu);
        const V upm = vadd(m.u[0], m.u[1]), umm = vsub(m.u[0], m.u[1]);
        const V four5 = vset<V>(4.5f), three = vset<V>(3.0f), m1 = vset<V>(-1.0f);
        f[Q / 2] = relax(0, mh, f[Q / 2]);
#pragma unroll
        for (int i = Q / 2 + 1; i < Q; ++i) {  // direction i and its opposite Q - 1 - i
            const int cx = cxo(i), cy = cyo(i), cz = (D == 3) ? czo(i) : 0;
            // c.u of i: the planar part (with its sign), then u_z
            V cu;
            bool neg = false;
            if (cx == 0 && cy == 0) cu = m.u[2];
            else if (cx == 0) { cu = m.u[1]; neg = cy < 0; }
            else if (cy == 0) { cu = m.u[0]; neg = cx < 0; }
            else if (cx == cy) { cu = upm; neg = cx < 0; }
            else { cu = umm; neg = cx < 0; }
            if (cz != 0 && (cx != 0 || cy != 0)) cu = neg ? vsub(m.u[2], cu) : vadd(cu, m.u[2]);
            else if (neg) cu = vmul(cu, m1);
            const V ncu = vmul(cu, m1);
            const int c = wclass<D>(i);
            f[i] = relax(c, vfma(cu, vfma(four5, cu, three), mh), f[i]);
            f[Q - 1 - i] = relax(c, vfma(ncu, vfma(four5, ncu, three), mh), f[Q - 1 - i]);
        }
    } else {
        V dm[3], d0[3], dp[3], key[3];  // d(-1), d(0), d(+1)
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const V u2 = vmul(m.u[a], m.u[a]), t3 = vmul(vset<V>(3.0f), u2);
            if constexpr (EQ == EQ_ENT) {
                const V s2 = vfma(vset<V>(3.0f), u2, one);
                const V rs = vrsqrt(s2);  // S = s2 rs
                key[a] = vmul(s2, rs);
                const V sm1 = vmul(t3, vrcp(BULK ? vadd(one, key[a]) : vfma(s2, rs, one)));  // S - 1 without cancellation
                d0[a] = vmul(sm1, vset<V>(-1.0f));
                dp[a] = vfma(vset<V>(2.0f), sm1, vmul(vset<V>(3.0f), m.u[a]));
                dm[a] = vfma(vset<V>(2.0f), sm1, vmul(vset<V>(-3.0f), m.u[a]));
            } else {
                d0[a] = vmul_alone(vset<V>(-1.5f), u2);
                dp[a] = vfma(vset<V>(3.0f), m.u[a], t3);
                dm[a] = vfma(vset<V>(-3.0f), m.u[a], t3);
                key[a] = u2;
            }
        }
        V kmax = key[0];
        if constexpr (BULK) {
            kmax = vmax(key[0], key[1]);
            if constexpr (D == 3) kmax = vmax(kmax, key[2]);
        }
        const Relax32<D, P, V> relax(rate32<EQ, BULK, V>(kmax, vset<V>(omega0s), vset<V>(six_nus)), m.rho, drho);
        const V dx[3] = {dm[0], d0[0], dp[0]}, dy[3] = {dm[1], d0[1], dp[1]};
        const V tx[3] = {vadd(one, dm[0]), vadd(one, d0[0]), vadd(one, dp[0])};
        if constexpr (D == 2) {
#pragma unroll
            for (int i = 0; i < 9; ++i)
                f[i] = relax(wclass<D>(i), vfma(dy[cyo(i) + 1], tx[cxo(i) + 1], dx[cxo(i) + 1]), f[i]);
        } else {
            const V ty[3] = {vadd(one, dm[1]), vadd(one, d0[1]), vadd(one, dp[1])};
            const V dz[3] = {dm[2], d0[2], dp[2]};
#pragma unroll
            for (int p = 0; p < 9; ++p) {
                const V exy = vfma(dy[cyo(p) + 1], tx[cxo(p) + 1], dx[cxo(p) + 1]);
                const V txy = vmul(tx[cxo(p) + 1], ty[cyo(p) + 1]);
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int i = p + 9 * q;
                    f[i] = relax(wclass<D>(i), vfma(dz[q], txy, exy), f[i]);
                }
            }
        }
    }
    return m;
}

// The fused FP64 collision of one cell, in place on shifted populations.  Returns the
// pre-collision moments (the macroscopic state at the current time step).  The
// equilibrium term h_i of each direction is formed inside the relaxation loop from the
// per-axis factors, so only the Q populations and O(D^2) factors stay live.
template <int D, int P, int EQ, bool BULK, typename R>
__device__ __forceinline__ CellMoments<R> collide(R (&f)[qof(D)], R rho0, R omega0, R six_nu) {
    constexpr int Q = qof(D);
    // weights per number of nonzero velocity components, folded at compile time
    constexpr double kW0 = wclass_weight<D>(0), kW1 = wclass_weight<D>(1);
    constexpr double kW2 = wclass_weight<D>(2), kW3 = wclass_weight<D>(D >= 3 ? 3 : 0);
    CellMoments<R> m;
    if constexpr (sizeof(R) == 4) {
        const Moments32<float> v = collide32<D, P, EQ, BULK, float>(f, rho0, omega0, six_nu);
        m.rho = v.rho;
        for (int a = 0; a < 3; ++a) m.u[a] = v.u[a];
        return m;
    } else {
    // 2beta w by weight class and 1 - 2beta
    const auto relaxation = [&](R om, R (&omw)[4]) {
        const double w[4] = {kW0, kW1, kW2, kW3};
#pragma unroll
        for (int c = 0; c < 4; ++c) omw[c] = om * R(w[c]);
        return R(1) - om;
    };
    R omw[4];
    if constexpr (EQ == EQ_POLY2) {
        R j[3];
        const R drho = collision_sums<D>(f, rho0, m.rho, j);
        const R inv = rcp_any(m.rho);
        for (int a = 0; a < 3; ++a) m.u[a] = mul_rn(j[a], inv);
        R uu = fma_r(m.u[0], m.u[0], m.u[1] * m.u[1]);
        if constexpr (D == 3) uu = fma_r(m.u[2], m.u[2], uu);
        R k = fmax(m.u[0] * m.u[0], m.u[1] * m.u[1]);
        if constexpr (D == 3) k = fmax(k, m.u[2] * m.u[2]);
        const R om = collision_rate<EQ, BULK, R>(k, omega0, six_nu);
        const R keep = relaxation(om, omw);
        // drho + rho h with h = 3 u.c + 9/2 (u.c)^2 - 3/2 u^2
        const R base = fma_r(R(-1.5) * m.rho, uu, drho), r3 = R(3) * m.rho, r45 = R(4.5) * m.rho;
        const R upm = m.u[0] + m.u[1], umm = m.u[0] - m.u[1];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int cx = cxo(i), cy = cyo(i), cz = (D == 3) ? czo(i) : 0;
            R cu;
            if (cx == 0 && cy == 0) cu = R(0);
            else if (cx == 0) cu = cy > 0 ? m.u[1] : -m.u[1];
            else if (cy == 0) cu = cx > 0 ? m.u[0] : -m.u[0];
            else if (cx == cy) cu = cx > 0 ? upm : -upm;
            else cu = cx > 0 ? umm : -umm;
            if (cz == 1) cu = cu + m.u[2];
            if (cz == -1) cu = cu - m.u[2];
            const R g = i == Q / 2 ? base : fma_r(cu, fma_r(r45, cu, r3), base);
            f[i] = fma_r(omw[wclass<D>(i)], g, keep * f[i]);
        }
    } else {
        TensorTerms<R> t;
        tensor_terms<D, EQ, R>(f, rho0, m, t);
        R kmax = fmax(t.key[0], t.key[1]);
        if constexpr (D == 3) kmax = fmax(kmax, t.key[2]);
        const R om = collision_rate<EQ, BULK, R>(kmax, omega0, six_nu);
        const R keep = relaxation(om, omw);
        R ex[3], tx[3], ty[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            ex[c] = t.drho + t.X[0][c];
            tx[c] = fma_r(t.X[0][c], t.irho, R(1));
            if constexpr (D == 3) ty[c] = fma_r(t.X[1][c], t.irho, R(1));
        }
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const int x = cxo(p) + 1, y = cyo(p) + 1;
            const R exy = fma_r(tx[x], t.X[1][y], ex[x]);
            if constexpr (D == 2) {
                f[p] = fma_r(omw[wclass<D>(p)], exy, keep * f[p]);
            } else {
                const R txy = tx[x] * ty[y];
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    f[p + 9 * q] = fma_r(omw[wclass<D>(p + 9 * q)], fma_r(txy, t.X[2][q], exy), keep * f[p + 9 * q]);
            }
        }
    }
    return m;
    }
}

// ------------------------------------------------------------------ one FP64 cell on three lanes
//
// An FP64 warp instruction takes an SM quarter 64 clocks however many lanes it has: where there
// are fewer cells than lanes, the lanes of a warp that are left over cost nothing.  Here a cell is
// spread over three neighbouring lanes, lane c of the group holding the populations with
// c_last = c - 1 (c_y in 2-D, c_z in 3-D), f[p] = f_{p + F c}, F = 3 or 9.  A lane sums its own
// populations, forms the terms of one axis and relaxes its own populations; partial sums and terms
// go between the lanes by shuffles.  Every lane adds the partial sums in the same order, so the
// three hold the same bits of rho, u and 2beta, and the operations are those of collide, so the
// populations get the same bits from both.  About 45 FP64 instructions in place of 82 in 2-D,
// 100 of 195 in 3-D (entropic).  All 32 lanes call it; `base` is the first lane of the caller's group.
__host__ __device__ constexpr int lane_pops(int D) { return D == 2 ? 3 : 9; }

template <typename R> __device__ __forceinline__ R from_lane(R v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }

template <int D, int EQ, bool BULK>
__device__ __forceinline__ CellMoments<double> collide_lanes(double (&f)[lane_pops(D)], int c, int base, double rho0,
                                                             double omega0, double six_nu) {
    using R = double;
    constexpr int F = lane_pops(D);
    CellMoments<R> m;
    R j[3] = {0, 0, 0}, sum, part[2];  // sums over the lane's populations: all, c_x f, c_y f (3-D)
    last_axis_sums<D>(f, sum, part);
    const R s0 = from_lane(sum, base), s1 = from_lane(sum, base + 1), s2 = from_lane(sum, base + 2);
    const R drho = (s0 + s1) + s2;
    m.rho = rho0 + drho;
    j[D - 1] = s2 - s0;
#pragma unroll
    for (int a = 0; a < D - 1; ++a) j[a] = (from_lane(part[a], base) + from_lane(part[a], base + 1)) + from_lane(part[a], base + 2);
    const R rho = m.rho;
    R om, base_g = 0, irho = 0, ex[3], tx[3], Y[3], Z = 0, r3 = 0, r45 = 0;
    if constexpr (EQ == EQ_POLY2) {
        irho = rcp_any(rho);
        for (int a = 0; a < 3; ++a) m.u[a] = mul_rn(j[a], irho);
        R uu = fma(m.u[0], m.u[0], m.u[1] * m.u[1]), k = fmax(m.u[0] * m.u[0], m.u[1] * m.u[1]);
        if constexpr (D == 3) {
            uu = fma(m.u[2], m.u[2], uu);
            k = fmax(k, m.u[2] * m.u[2]);
        }
        om = collision_rate<EQ, BULK, R>(k, omega0, six_nu);
        base_g = fma(-1.5 * rho, uu, drho);
        r3 = 3.0 * rho;
        r45 = 4.5 * rho;
    } else {
        // the terms of one axis per lane: lane c forms axis min(c, D - 1)
        const R ja = c == 0 ? j[0] : (D == 2 || c == 1 ? j[1] : j[2]);
        const R j3 = 3.0 * ja;
        R X[3], key;
        if constexpr (EQ == EQ_ENT) {
            // entropic_terms with an axis to a lane; all lanes again where some cell of the warp needs it
            R e;
            const auto terms = [&](R r, R v, auto is_signed) {
                R jj = 3.0 * v * v, T = sqrt_ulp(fma(r, r, jj));
                if constexpr (decltype(is_signed)::value) T = copysign(T, r);
                const R q = r + T;
                const R q0 = from_lane(q, base), q1 = from_lane(q, base + 1);
                R others, all;
                if constexpr (D == 2) {
                    others = c == 0 ? q1 : q0;
                    all = q0 * q1;
                } else {
                    const R q2 = from_lane(q, base + 2);
                    others = (c == 0 ? q1 : q0) * (c == 2 ? q1 : q2);
                    all = q0 * (q1 * q2);
                }
                const R product = r * all, w = rcp_ulp(product), z = w * r;
                irho = w * all;
                e = mul_rn(jj, z * others);
                key = mul_rn(T, irho);
                return product;
            };
            const bool ok = terms_ok(terms(rho, ja, std::false_type()));
            if (!__all_sync(0xffffffffu, ok)) {
                const int n = ok ? 0 : exponent_of(rho);
                terms(scale_down(rho, n), scale_down(ja, n), std::true_type());
                irho = scale_down(irho, n);
                e = scale_down(e, -n);
            }
            X[0] = fma(2.0, e, -j3);
            X[1] = -e;
            X[2] = fma(2.0, e, j3);
        } else {
            irho = rcp_any(rho);
            const R u = ja * irho;
            X[0] = fma(j3, u, -j3);
            X[1] = mul_rn(-0.5, j3 * u);
            X[2] = fma(j3, u, j3);
            key = u * u;
        }
        for (int a = 0; a < 3; ++a) m.u[a] = a < D ? mul_rn(j[a], irho) : 0.0;
        R kmax = 0;
        if constexpr (BULK) {
            kmax = fmax(from_lane(key, base), from_lane(key, base + 1));
            if constexpr (D == 3) kmax = fmax(kmax, from_lane(key, base + 2));
        }
        om = collision_rate<EQ, BULK, R>(kmax, omega0, six_nu);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const R Xx = from_lane(X[i], base);
            Y[i] = from_lane(X[i], base + 1);
            ex[i] = drho + Xx;
            tx[i] = fma(Xx, irho, 1.0);
        }
        if constexpr (D == 3) {
            const R z0 = from_lane(X[0], base + 2), z1 = from_lane(X[1], base + 2), z2 = from_lane(X[2], base + 2);
            Z = c == 0 ? z0 : (c == 1 ? z1 : z2);
        }
    }
    // 2beta w by the number of nonzero components but the last
    const R keep = 1.0 - om;
    R omw[D];
#pragma unroll
    for (int n = 0; n < D; ++n) omw[n] = om * (c == 1 ? wclass_weight<D>(n) : wclass_weight<D>(n + 1));
#pragma unroll
    for (int p = 0; p < F; ++p) {
        const int cx = cxo(p), cy = D == 3 ? cyo(p) : 0;  // the direction's components but the last
        R g;
        if constexpr (EQ == EQ_POLY2) {
            R cu = cx == 0 ? 0.0 : (cx > 0 ? m.u[0] : -m.u[0]);
            if (D == 3 && cy != 0) cu = cy > 0 ? cu + m.u[1] : cu - m.u[1];
            cu = c == 1 ? cu : (c == 2 ? cu + m.u[D - 1] : cu - m.u[D - 1]);
            g = fma(cu, fma(r45, cu, r3), base_g);
        } else if constexpr (D == 2) {
            const R Yc = c == 0 ? Y[0] : (c == 1 ? Y[1] : Y[2]);
            g = fma(tx[cx + 1], Yc, ex[cx + 1]);
        } else {
            const R exy = fma(tx[cx + 1], Y[cy + 1], ex[cx + 1]), txy = tx[cx + 1] * fma(Y[cy + 1], irho, 1.0);
            g = fma(txy, Z, exy);
        }
        f[p] = fma(omw[(cx != 0) + (cy != 0)], g, keep * f[p]);
    }
    return m;
}

}  // namespace lbmd
