// Per-node arithmetic of the thermal MRT lattice-Boltzmann model of
// arXiv:1809.08683, written in deviation form for the GPU kernels.
//
// Storage convention: a node holds f'_i = f_i - f^r_i and g'_i = g_i - g^r_i,
// where f^r = M^-1 m^eq(rho0, u = 0, T0) and g^r = M^-1 n^eq(rho0 E0, u = 0, T0)
// are the rest equilibria.  M f^r has only rows 0, 1, 2 nonzero, so
// m' = M f' equals m - m^r and every cancellation-prone difference
// (rho - rho0, T - T0, p - p0, eta - eta0, rho E - rho0 E0) is formed from
// small quantities.  The same code serves FP64 and FP32 storage.
//
// The collision uses the sparse forms of the modified matrices:
//  (I - S/2) d  from the block structure of S (Sec. 2.1; App. B),
//  m_bar - m = F_m - S d - C = 2 (G - (m - m^eq)) - C,
//  ((m + m_bar)/2 - m^eq)_a = G_a - C_a / 2 for a = 1, 7, 8, where
//  G = (I - S/2) d and C = R G + T grad(rho) + X grad(p),
//  L applied as diag(L) plus the two sigma_q omega_j couplings (Sec. 2.2),
//  M^-1 = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4).
//
// Every fused multiply-add is written as mad() and the library is compiled
// without the compiler's own contraction (-fmad=false), so that a node's bits
// do not depend on the kernel.  One set of bits: the one-node kernels of one
// model class (block strips, warp strips, node kernels, the cluster kernel);
// and the paired block strips with their node kernel.  The packed kernels
// agree with the one-node kernels to rounding: they draw one random number per
// two nodes, and the assembler contracts some packed products that meet an
// addition all the same (those with a literal constant always, which is why
// such a product is a mad() throughout).
#pragma once

#include <cmath>

#if defined(__CUDACC__)
#include "lbm_ff.cuh"
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbm {

// Division in the per-node arithmetic.  FP32: the fast hardware division
// (a few ulp), which the FP32 path's 1e-4 tolerance absorbs.  FP64 on the
// device: a * (1/b), with 1/b from the hardware's approximate FP64
// reciprocal (PTX rcp.approx.ftz.f64, about 20 correct bits) refined by one
// third-order step of the geometric series 1/b = y / (1 - e), e = 1 - b y:
// y (1 + e + e^2) leaves e^3, beyond 53 bits.  Within 2 ulp of the quotient.
// The divisors are O(1) lattice quantities (densities, temperatures, 1 plus
// a viscosity), never subnormal.
LBM_HD double recip(double b) {
#if defined(__CUDA_ARCH__)
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double e = fma(-b, y, 1.0);
    return fma(y, fma(e, e, e), y);
#else
    return 1.0 / b;
#endif
}
LBM_HD double fdiv(double a, double b) {
#if defined(__CUDA_ARCH__)
    return a * recip(b);
#else
    return a / b;
#endif
}
LBM_HD float fdiv(float a, float b) {
#if defined(__CUDA_ARCH__)
    return __fdividef(a, b);
#else
    return a / b;
#endif
}
LBM_HD float recip(float b) { return fdiv(1.0f, b); }

// Square root.  FP64 on the device: x y with y the hardware's approximate
// reciprocal square root (PTX rsqrt.approx.ftz.f64, about 20 correct bits)
// and one third-order step of the binomial series
// x^(1/2) = x y (1 - e)^(-1/2), e = 1 - x y^2: five FP64 instructions, which
// is what counts in the FP64 kernels (see collide).  Zero gives zero, a
// negative number NaN.
LBM_HD double root(double x) {
#if defined(__CUDA_ARCH__)
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    if (((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) == 0) y = 0.0;
    const double t = x * y, e = fma(-t, y, 1.0);
    return fma(t, e * fma(0.375, e, 0.5), t);
#else
    return sqrt(x);
#endif
}
LBM_HD float root(float x) { return sqrtf(x); }

// Whether a number is neither infinite nor NaN, by its exponent bits (an
// FP64 comparison would take an FP64 issue slot).
LBM_HD bool finite(double x) {
#if defined(__CUDA_ARCH__)
    return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
#else
    return std::isfinite(x);
#endif
}
LBM_HD bool finite(float x) {
#if defined(__CUDA_ARCH__)
    return (__float_as_int(x) & 0x7f800000) != 0x7f800000;
#else
    return std::isfinite(x);
#endif
}

// a * b + c in one rounding.
LBM_HD double mad(double a, double b, double c) {
#if defined(__CUDA_ARCH__)
    return fma(a, b, c);
#else
    return a * b + c;
#endif
}
LBM_HD float mad(float a, float b, float c) {
#if defined(__CUDA_ARCH__)
    return fmaf(a, b, c);
#else
    return a * b + c;
#endif
}

// Constants of one lattice, in the arithmetic type R.
template <typename R>
struct Params {
    R rho0, T0, E0, Cv, inv_Cv, Rg, eos_a, eos_b, p0, rho0E0_p0;
    R mu0, mu0S, inv_T0, visc_S, lam_fac;
    R nu_e, mu_j;     // 2 * 3 varsigma / (varpi nu), 4 (1/sigma_j - 1/2) / mu (Rates)
    R x2r, x2p;       // beta2 - 1, -3 beta2; alpha1 = -1, beta1 = 1, alpha2 = 1, beta2 = -2 / (1 - varpi)
    R n1T, n2T;       // -(4 + gamma1) rho0 Cp, (4 - gamma2) rho0 Cp
    R kk, hh, bb, bbm2, omk, k2h, gamma1, gamma2;  // bbm2 = -2 bb
    R k11, k17, k18, k71, k77, k81, k88;  // entries of R per 1/(1 + 6 nu) or 1/(1 + nu_e nu) (collide)
    R Fx, Fy, Fxh, Fyh;  // force (or g) and half of it
    R cs_b0;  // 1 - b rho0 (cubic EOS)
    R cs[7], cs_lo[7];  // Carnahan-Starling constants (cs_constants) and, in FP32, what R leaves of them
    R dither; // FP32 storage: 1 rounds the stored deviations stochastically, 0 to nearest
    int eos, visc, force_mode, corrections;
};

enum { EOS_DECOUPLING = 0, EOS_IDEAL = 1, EOS_CS = 2, EOS_CUBIC = 3 };

// Model classes.  MODEL_ANY reads the EOS, the viscosity law, the force
// mode and the corrections flag from the parameters at run time.
// MODEL_CAVITY fixes the heated-cavity model at compile time (Sutherland
// viscosity, F = rho g with vertical g, corrections on) and keeps only the
// ideal-gas and cubic EOS, chosen at run time.  A fixed model drops the
// branches and the code of the others, and the terms of F_x = 0, without
// which some sums are formed in another order: the classes agree to rounding.
enum { MODEL_ANY = 0, MODEL_CAVITY = 1 };
template <int MC, typename R>
LBM_HD int visc_law(const Params<R>& P) { return MC != MODEL_ANY ? 2 : P.visc; }
template <int MC, typename R>
LBM_HD bool force_is_rho_g(const Params<R>& P) { return MC != MODEL_ANY || P.force_mode != 0; }
template <int MC, typename R>
LBM_HD bool corrections_on(const Params<R>& P) { return MC != MODEL_ANY || P.corrections != 0; }

// Macroscopic state of one node in deviation form.
template <typename R>
struct Mac {
    R rho_d, rho, ir, ux, uy, Fx, Fy, qe, rhoE_d, T_d, T, p_d;
};

// The part of Mac that the fused kernels keep in registers from a row's
// macro pass to its collision; expand() rebuilds the rest with the same
// operations as macros() from it and sum g' (which the collision's moments
// form anyway), so an expanded state equals the original bit for bit.
template <typename R>
struct MacC {
    R rho_d, ir, ux, uy, T_d, p_d;
};

// Carnahan-Starling deviation p - p0 with p = Z(e) rho R T, e = b rho / 4
// (Eq. EOSs.3).  rho Z(rho) is differenced in closed form: with d = e - e0,
// q = 1 - e0, N(e) = e + e^2 + e^3 - e^4 and N(e0 + d) = N0 + N1 d + N2 d^2 +
// N3 d^3 - d^4,
//   N(e) q^3 - N0 (q - d)^3
//     = d [(N1 q^3 + 3 N0 q^2) + d ((N2 q^3 - 3 N0 q) + d ((N3 q^3 + N0) - d q^3))],
// so rho Z - rho0 Z0 = rho' poly(d) / (q - d)^3 without cancellation, and
// p - p0 = R [(rho Z - rho0 Z0) T + rho0 Z0 T'].  Constants: b/4, q, the four
// coefficients of poly times R / q^3, and R rho0 Z0.
inline void cs_constants(double b, double rho0, double Rg, double* c) {
    const double e = 0.25 * b * rho0, q = 1.0 - e, q3 = q * q * q;
    const double N0 = e + e * e + e * e * e - e * e * e * e, N1 = 1.0 + 2.0 * e + 3.0 * e * e - 4.0 * e * e * e;
    const double N2 = 1.0 + 3.0 * e - 6.0 * e * e, N3 = 1.0 - 4.0 * e;
    c[0] = 0.25 * b;
    c[1] = q;
    c[2] = Rg * (N1 + 3.0 * N0 / q);
    c[3] = Rg * (N2 - 3.0 * N0 / (q * q));
    c[4] = Rg * (N3 + N0 / q3);
    c[5] = -Rg;
    c[6] = Rg * rho0 * (1.0 + e + e * e - e * e * e) / q3;
}
LBM_HD double cs_dev(const double* c, const double*, double rho_d, double T, double T_d) {
    const double d = c[0] * rho_d, s = c[1] - d;
    const double poly = mad(mad(mad(c[5], d, c[4]), d, c[3]), d, c[2]);
    return mad(rho_d * poly * recip(s * s * s), T, c[6] * T_d);
}
// FP32: the same in pairs of FP32 numbers (48 bits), rounded once.  In FP64,
// whose instructions and conversions issue once per 76 cycles and scheduler,
// this term was most of the step: 1001 x 777 nodes, 20 steps and the fields,
// 1.97 -> 0.97 ms.
LBM_HD float cs_dev(const float* c, const float* lo, float rho_d, float T, float T_d) {
#if defined(__CUDA_ARCH__)
    auto k = [&](int i) { return ff64(c[i], lo[i]); };
    const ff64 d = k(0) * ff64(rho_d, 0.0f), s = k(1) - d, s3 = s * s * s;
    const ff64 poly = ((k(5) * d + k(4)) * d + k(3)) * d + k(2);
    // 1 / s3 = y (1 + t), t = 1 - s3 y, from the hardware's y: t^2 is below 2^-44
    const float y = recip(s3.hi), t = fmaf(-s3.lo, y, fmaf(-s3.hi, y, 1.0f));
    const ff64 p = poly * ff64(rho_d, 0.0f) * fast_two_sum(y, y * t) * ff64(T, 0.0f) + k(6) * ff64(T_d, 0.0f);
    return p.hi;
#else
    double cd[7];
    for (int i = 0; i < 7; ++i) cd[i] = (double)c[i] + (double)lo[i];
    return (float)cs_dev(cd, cd, (double)rho_d, (double)T, (double)T_d);
#endif
}

// p_EOS(rho, T) - p0.
template <int MC = MODEL_ANY, typename R>
LBM_HD R eos_dev(const Params<R>& P, R rho_d, R rho, R T_d, R T) {
    const int kind = MC == MODEL_CAVITY ? (P.eos == EOS_CUBIC ? EOS_CUBIC : EOS_IDEAL) : P.eos;
    if (MC == MODEL_CAVITY && kind == EOS_IDEAL) return P.Rg * mad(rho_d, T, P.rho0 * T_d);
    switch (kind) {
    case EOS_DECOUPLING:
        return P.Rg * P.T0 * rho_d;
    case EOS_IDEAL:
        return P.Rg * mad(rho_d, T, P.rho0 * T_d);
    case EOS_CS:
        return cs_dev(P.cs, P.cs_lo, rho_d, T, T_d);
    default: {
        // rho R T / (1 - b rho) - a rho^2, differenced exactly:
        // [rho T (1 - b rho0) - rho0 T0 (1 - b rho)] = rho_d T + rho0 T_d (1 - b rho)
        const R om = mad(-P.eos_b, rho, R(1));
        const R num = mad(rho_d, T, P.rho0 * T_d * om);
        return mad(-P.eos_a * rho_d, rho + P.rho0, fdiv(P.Rg * num, om * P.cs_b0));
    }
    }
}

// Body force F = rho g (force_mode 1) or F = g, and q = u . F.
template <int MC = MODEL_ANY, typename R>
LBM_HD void mac_force(const Params<R>& P, Mac<R>& m) {
    if (MC == MODEL_CAVITY) { m.Fx = R(0); m.Fy = m.rho * P.Fy; }
    else if (force_is_rho_g<MC>(P)) { m.Fx = m.rho * P.Fx; m.Fy = m.rho * P.Fy; }
    else { m.Fx = P.Fx; m.Fy = P.Fy; }
}
template <int MC = MODEL_ANY, typename R>
LBM_HD void mac_qe(Mac<R>& m) {
    if (MC == MODEL_CAVITY) m.qe = m.uy * m.Fy;
    else m.qe = mad(m.ux, m.Fx, m.uy * m.Fy);
}

// Eq. (rho.u), Eq. (E), T = eps / Cv, p_EOS.
template <int MC = MODEL_ANY, typename R>
LBM_HD void macros(const Params<R>& P, R rho_d, R jx, R jy, R sg, Mac<R>& m) {
    m.rho_d = rho_d;
    m.rho = P.rho0 + rho_d;
    m.ir = recip(m.rho);
    mac_force<MC>(P, m);
    // u = j / rho + a with a = F / (2 rho), and since q / (2 rho) = u . a,
    // Cv T' = (sum g' - rho' E0) / rho + u . (a - u/2), the small second part
    // first so that its additions round little; q itself only enters the
    // collision
    R ax = P.Fxh, ay = P.Fyh;
    if (!force_is_rho_g<MC>(P)) {
        ax = ax * m.ir;
        ay = ay * m.ir;
    }
    m.ux = MC == MODEL_CAVITY ? jx * m.ir : mad(jx, m.ir, ax);
    m.uy = mad(jy, m.ir, ay);
    const R hx = MC == MODEL_CAVITY ? R(-0.5) * m.ux : mad(R(-0.5), m.ux, ax), hy = mad(R(-0.5), m.uy, ay);
    m.T_d = mad(mad(-P.E0, rho_d, sg), m.ir, mad(m.ux, hx, m.uy * hy)) * P.inv_Cv;
    mac_qe<MC>(m);
    m.rhoE_d = mad(R(0.5), m.qe, sg);
    m.T = P.T0 + m.T_d;
    m.p_d = eos_dev<MC>(P, rho_d, m.rho, m.T_d, m.T);
}

template <typename R>
LBM_HD void compress(const Mac<R>& m, MacC<R>& c) {
    c.rho_d = m.rho_d; c.ir = m.ir; c.ux = m.ux; c.uy = m.uy;
    c.T_d = m.T_d; c.p_d = m.p_d;
}

template <int MC = MODEL_ANY, typename R>
LBM_HD void expand(const Params<R>& P, const MacC<R>& c, R sg, Mac<R>& m) {
    m.rho_d = c.rho_d;
    m.rho = P.rho0 + c.rho_d;
    m.ir = c.ir;
    mac_force<MC>(P, m);
    m.ux = c.ux;
    m.uy = c.uy;
    mac_qe<MC>(m);
    m.rhoE_d = mad(R(0.5), m.qe, sg);
    m.T_d = c.T_d;
    m.T = P.T0 + c.T_d;
    m.p_d = c.p_d;
}

// Macros of a wall node whose density, velocity and total energy are fixed
// by the wall data (Sec. 3.1).
template <typename R>
LBM_HD void wall_macros(const Params<R>& P, R rho_d, R ux, R uy, R rhoE_d, Mac<R>& m) {
    m.rho_d = rho_d;
    m.rho = P.rho0 + rho_d;
    m.ir = recip(m.rho);
    mac_force(P, m);
    m.ux = ux;
    m.uy = uy;
    mac_qe(m);
    m.rhoE_d = rhoE_d;
    R E_d = mad(-P.E0, rho_d, rhoE_d) * m.ir;
    m.T_d = mad(R(-0.5), mad(ux, ux, uy * uy), E_d) * P.inv_Cv;
    m.T = P.T0 + m.T_d;
    m.p_d = eos_dev(P, rho_d, m.rho, m.T_d, m.T);
}

// Relaxation rates of Sec. 4: s_p = 1/tau, (1/s_p - 1/2)(1/s_q - 1/2) = 1/12,
// s_eps = s_e from varsigma = varpi c_s^2 (1/s_e - 1/2) = (varsigma/nu) nu,
// lambda = Cp mu / Pr = coef rho0 Cp0 (1/sigma_j - 1/2), sigma_q = sigma_j,
// (1/sigma_j - 1/2)(1/sigma_e - 1/2) = 1/4, sigma_eps = sigma_p = sigma_e.
// All five follow from four reciprocals:
//   s_p = 2 ia, 1 - s_p/2 = 1 - ia               ia = 1/(1 + 6 nu)
//   s_q = 2 sq2 = 36 nu ib, 1 - s_q/2 = ib       ib = 1/(1 + 18 nu)
//   s_e = 2 ic, 1 - s_e/2 = 1 - ic               ic = 1/(1 + nu_e nu)
//   sigma_j = 2 id, sigma_e = sE = mu_j mu id    id = 1/(1 + mu_j mu / 2)
// s_q and sigma_e vanish with the viscosity, and as products they keep their
// relative accuracy (as 2 - 2 id, sigma_e was off by 9e-5 of itself in FP32
// where it is 0.002).
template <typename R>
struct Rates {
    R ia, ib, ic, id, nu, sq2, sE;
};

template <int MC = MODEL_ANY, typename R>
LBM_HD R viscosity(const Params<R>& P, R T) {
    const int law = visc_law<MC>(P);
    if (law == 1) return P.mu0 * T * P.inv_T0;
    if (law == 2) {
        R th = T * P.inv_T0;
        R n = P.mu0S * th * root(th);
        return fdiv(n, th + P.visc_S);
    }
    return P.mu0;
}

template <int MC = MODEL_ANY, typename R>
LBM_HD void rates(const Params<R>& P, R rho_ir, R T, Rates<R>& r) {
    const R mu = viscosity<MC>(P, T);
    r.nu = mu * rho_ir;
    r.ia = recip(mad(R(6), r.nu, R(1)));
    const R x = R(18) * r.nu, y = P.mu_j * mu;
    r.ib = recip(x + R(1));
    r.sq2 = x * r.ib;
    r.ic = recip(mad(P.nu_e, r.nu, R(1)));
    r.id = recip(mad(R(0.5), y, R(1)));
    r.sE = y * r.id;
}

// Rows 1, 2, 4, 6, 7, 8 of x = m - m^eq and of d = m - m^eq + F_m/2 (rows 0,
// 3, 5 of d vanish identically by the definitions of rho and u).
template <typename R>
struct Dev {
    R x1, x2, x4, x6, x7, x8;
    R d1, d2, d4, d6, d7, d8;
};

// m^eq - m^r of Sec. 2.1 with alpha1 = -1, beta1 = 1, alpha2 = 1 and
// eta' = 3 p' - rho' (eta = p / c_s^2 - rho):
//   2 (eta' - rho') + 3 rho u^2, rho' + beta2 eta' - 3 rho u^2 + 9 rho ux^2 uy^2,
//   -jx + 3 rho ux uy^2, -jy + 3 rho uy ux^2, rho (ux^2 - uy^2), rho ux uy
// with j = rho u, and half of F_m by the product rule:
//   3 q, -3 q + 9 ux uy (Fx uy + Fy ux), -Fx/2 + 3/2 (Fx uy^2 + 2 Fy ux uy),
//   -Fy/2 + 3/2 (Fy ux^2 + 2 Fx ux uy), Fx ux - Fy uy, (Fx uy + Fy ux)/2.
// rho' and p' enter rows 1 and 2 as they are: a rounded eta' or eta' - rho'
// would be multiplied by 2 and more.
template <int MC = MODEL_ANY, typename R>
LBM_HD void neq_density(const Params<R>& P, const Mac<R>& m, R m1, R m2, R m4, R m6, R m7, R m8,
                        Dev<R>& d) {
    const R ux = m.ux, uy = m.uy;
    const R jx = m.rho * ux, jy = m.rho * uy;
    const R jxx = jx * ux, jxy = jx * uy, xy = ux * uy;
    const R r2 = mad(jy, uy, jxx), t3 = R(3) * jxy;
    d.x1 = mad(R(-6), m.p_d, mad(R(4), m.rho_d, mad(R(-3), r2, m1)));
    d.x2 = mad(P.x2p, m.p_d, mad(P.x2r, m.rho_d, mad(R(-3), t3 * xy, mad(R(3), r2, m2))));
    d.x4 = mad(-t3, uy, m4 + jx);
    d.x6 = mad(-t3, ux, m6 + jy);
    d.x7 = mad(jy, uy, m7 - jxx);
    d.x8 = m8 - jxy;
    const R Fx = m.Fx, Fy = m.Fy;
    d.d1 = mad(R(3), m.qe, d.x1);
    if (MC == MODEL_CAVITY) {
        // the same terms with F_x = 0
        const R w = mad(R(3), ux * ux, R(-1)), Fh = R(0.5) * Fy;
        d.d2 = mad(R(3) * m.qe, w, d.x2);
        d.d4 = mad(R(3) * Fy, xy, d.x4);
        d.d6 = mad(Fh, w, d.x6);
        d.d7 = d.x7 - m.qe;
        d.d8 = mad(Fh, ux, d.x8);
    } else {
        const R s8 = mad(Fx, uy, Fy * ux), xy3 = R(3) * xy;
        d.d2 = mad(R(3) * xy3, s8, mad(R(-3), m.qe, d.x2));
        d.d4 = mad(xy3, Fy, mad(R(0.5) * Fx, mad(R(3), uy * uy, R(-1)), d.x4));
        d.d6 = mad(xy3, Fx, mad(R(0.5) * Fy, mad(R(3), ux * ux, R(-1)), d.x6));
        d.d7 = mad(-Fy, uy, mad(Fx, ux, d.x7));
        d.d8 = mad(R(0.5), s8, d.x8);
    }
}

// G = (I - S/2) d on rows 1, 7, 8 (Sec. 2.1 S; App. B block structure); rows
// 2, 4, 6 are (1 - s_e/2) d2, (1 - s_q/2) d4, (1 - s_q/2) d6.
template <typename R>
struct Gv {
    R G1, G7, G8;
};

template <typename R>
LBM_HD void apply_IS2(const Params<R>& P, const Rates<R>& r, R ux, R uy, const Dev<R>& d, Gv<R>& G) {
    const R he = R(1) - r.ic, hp = R(1) - r.ia;  // 1 - s/2
    const R bq = P.bb * r.sq2;
    const R a = mad(ux, d.d4, uy * d.d6), b = mad(ux, d.d4, -(uy * d.d6)), c = mad(uy, d.d4, ux * d.d6);
    G.G1 = he * mad(P.hh * r.sq2, a, mad(P.kk * r.ic, d.d2, d.d1));
    G.G7 = hp * mad(R(2) * bq, b, d.d7);
    G.G8 = hp * mad(bq, c, d.d8);
}

// Moments m' = M f' (Eq. M).
template <typename R>
LBM_HD void moments(const R* f, R* m) {
    const R s1 = f[1] + f[3], s2 = f[2] + f[4], s3 = f[5] + f[7], s4 = f[6] + f[8];
    const R d1 = f[5] - f[7], d2 = f[6] - f[8], e1 = f[1] - f[3], e2 = f[2] - f[4];
    const R a = s1 + s2, b = s3 + s4, dx = d1 - d2, dy = d1 + d2;
    m[0] = f[0] + (a + b);
    m[1] = mad(R(-4), f[0], mad(R(2), b, -a));
    m[2] = mad(R(4), f[0], mad(R(-2), a, b));
    m[3] = e1 + dx;
    m[4] = mad(R(-2), e1, dx);
    m[5] = e2 + dy;
    m[6] = mad(R(-2), e2, dy);
    m[7] = s1 - s2;
    m[8] = s3 - s4;
}

// f = M^-1 m with M^-1 = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4).
template <typename R>
LBM_HD void inverse_moments(const R* m, R* f) {
    const R a0 = m[0] * R(1.0 / 9.0);
    const R A = mad(R(-1.0 / 36.0), mad(R(2), m[2], m[1]), a0);
    const R B = mad(R(1.0 / 36.0), mad(R(2), m[1], m[2]), a0);
    const R X = m[3] - m[4], Y = m[5] - m[6];
    const R p = mad(R(2), m[3], m[4]), q = mad(R(2), m[5], m[6]);
    const R S = p + q, D = p - q;
    const R A1 = mad(R(0.25), m[7], A), A2 = mad(R(-0.25), m[7], A);
    const R B1 = mad(R(0.25), m[8], B), B2 = mad(R(-0.25), m[8], B);
    f[0] = mad(R(1.0 / 9.0), m[2] - m[1], a0);
    f[1] = mad(R(1.0 / 6.0), X, A1);
    f[3] = mad(R(-1.0 / 6.0), X, A1);
    f[2] = mad(R(1.0 / 6.0), Y, A2);
    f[4] = mad(R(-1.0 / 6.0), Y, A2);
    f[5] = mad(R(1.0 / 12.0), S, B1);
    f[7] = mad(R(-1.0 / 12.0), S, B1);
    f[6] = mad(R(-1.0 / 12.0), D, B2);
    f[8] = mad(R(1.0 / 12.0), D, B2);
}

// Sec. 2.2: dn = n - n^eq + Q_m/2 of a node, rows 1..8 (rows 7, 8 are n7, n8).
// With ref = rho0 Cp T', H = rho H and q = u . F:
//   n^eq: -4 (rhoE' - ref) + gamma1 ref, 4 (rhoE' - ref) + gamma2 ref, H u, -H u
//   Q_m:  q (1, gamma1, gamma2, ux, -ux, uy, -uy)
// Rows 3 and 4 (5 and 6) of n^eq and Q are opposite, so dn3 is taken as
// s34 - dn4 with s34 = dn3 + dn4 = n3 + n4.  The sums are ordered so that
// only small ones are rounded: rho H - q/2 as rho0 H0 and the rest, rho E'
// and T' with their own factors.  With this and the orders of T' (macros) and
// rows 1, 2 (neq_density), the rms error of FP32 increments at random nodes,
// against FP64, is 1.17e-9 for g and 2.39e-9 for f at tau0 = 0.5005 (1.43e-9
// and 3.11e-9 with rounded rho H - q/2, rho E' - ref and eta'), 1.18e-9 and
// 0.99e-9 at 0.8 (1.41e-9 and 1.11e-9).
template <typename R>
struct EDev {
    R dn1, dn2, s34, dn4, s56, dn6;
};

template <typename R>
LBM_HD void energy_neq(const Params<R>& P, const Mac<R>& m, R n1, R n2, R n3, R n4, R n5, R n6, EDev<R>& e) {
    const R qh = R(0.5) * m.qe, h = (m.rhoE_d + m.p_d) - qh;
    e.dn1 = mad(P.gamma1, qh, mad(P.n1T, m.T_d, mad(R(4), m.rhoE_d, n1)));
    e.dn2 = mad(P.gamma2, qh, mad(P.n2T, m.T_d, mad(R(-4), m.rhoE_d, n2)));
    e.s34 = n3 + n4;
    e.dn4 = mad(h, m.ux, mad(P.rho0E0_p0, m.ux, n4));
    e.s56 = n5 + n6;
    e.dn6 = mad(h, m.uy, mad(P.rho0E0_p0, m.uy, n6));
}

// Rows 3 and 5 of Y v for the rows 1, 7, 8 of v (rows 4, 6 are their opposites).
template <typename R>
LBM_HD void heating(R ux, R uy, R v1, R v7, R v8, R& Y3, R& Y5) {
    const R a = mad(R(1.0 / 3.0), v1, v7), b = mad(R(1.0 / 3.0), v1, -v7), c = R(2) * v8;
    Y3 = mad(ux, a, uy * c);
    Y5 = mad(uy, b, ux * c);
}

// Leaves f and g as they are between the moments and the final update.
struct KeepDFs {
    template <typename R>
    LBM_HD void operator()(R*, R*) const {}
};

// Three times the gradient of one field at an interior node, from its eight
// neighbours (m, z, p: the rows j - 1, j, j + 1; l, c, r: the columns):
// grad = 3 sum_i w_i e_i phi(x + e_i), w = 1/9 (axis), 1/36 (diagonal).
template <typename R>
LBM_HD void gradient3(R ml, R mc, R mr, R zl, R zr, R pl, R pc, R pr, R& gx, R& gy) {
    const R a = pr - ml, b = mr - pl;
    gx = mad(R(0.25), a + b, zr - zl);
    gy = mad(R(0.25), a - b, pc - mc);
}

// Three times a one-sided second-order derivative along the inward normal
// (s = 1 towards increasing coordinates, -1 otherwise) at a wall node, and
// three times a central one along a wall.
template <typename R>
LBM_HD R onesided3(R s, R v0, R v1, R v2) { return s * R(1.5) * mad(R(4), v1, mad(R(-3), v0, -v2)); }
template <typename R>
LBM_HD R central3(R l, R r) { return R(1.5) * (r - l); }

// Full collision of one node (Eqs. LBE.u.c, LBE.T.c) in increment form: the
// moment changes m_bar - m and n_bar - n are formed from small quantities
// only (force and source moments, non-equilibrium parts, corrections), then
// mapped back with M^-1 and added to the stored deviations through `add`,
// which may round stochastically.  f, g hold deviations on entry and the
// post-collision deviations on exit.  f and g are read twice: for the
// moments, and for the final update after `reload(f, g)`; a caller that can
// fetch them again (from shared memory) passes a reload that does so, and
// the values need not stay in registers through the collision.
// (rx, ry), (px, py): three times grad(rho) and grad(p).
//
// Every form below is chosen for its instruction count, which bounds the
// FP64 kernels (GB300 issues one FP64 warp instruction per 76 cycles and
// scheduler, whatever its active lanes): F_m drops out of m_bar - m =
// 2 (G - x) - C on rows 1, 2, 4, 6, 7, 8; the quotients of rates in R reduce to
// s_p (2 - s_e)/(2 - s_p) = (nu_e/3) ic and s_e (2 - s_p)/(2 - s_e) =
// (12/nu_e) ia by the definitions of ia and ic; and the terms T grad(rho),
// X grad(p) share ux d(rho)/dx, ux d(3 p - rho)/dx and their y counterparts.
// Against the term-by-term form: 512^2 FP64 cavity 0.366 -> 0.275 ms per step,
// 64 small FP64 lattices 0.68 -> 0.50 ms, 4096^2 FP32 0.488 -> 0.441 ms.
template <int MC = MODEL_ANY, typename R, typename Add, typename Reload = KeepDFs>
LBM_HD void collide(const Params<R>& P, const Mac<R>& mc, R* f, R* g, R rx, R ry, R px, R py,
                    const Add& add, const Reload& reload = Reload()) {
    Rates<R> r;
    rates<MC>(P, mc.ir, mc.T, r);
    R m[9], n[9];
    moments(f, m);
    moments(g, n);
    Dev<R> d;
    neq_density<MC>(P, mc, m[1], m[2], m[4], m[6], m[7], m[8], d);
    Gv<R> G;
    const R ux = mc.ux, uy = mc.uy;
    apply_IS2(P, r, ux, uy, d, G);

    // (m + m_bar)/2 - m^eq = G - C/2 on rows 1, 7, 8 with the corrections
    // C = R G + T grad(rho) + X grad(p) (Sec. 2.1)
    R Gt1 = G.G1, Gt7 = G.G7, Gt8 = G.G8;
    if (corrections_on<MC>(P)) {
        const R ux2 = ux * ux, uy2 = uy * uy, sum2 = ux2 + uy2, dif2 = ux2 - uy2, xy = ux * uy;
        const R he = R(1) - r.ic, hp3 = R(1.0 / 3.0) * (R(1) - r.ia);
        const R zx = mad(R(3), px, -rx), zy = mad(R(3), py, -ry);
        const R p1 = ux2 * (ux * rx), p2 = uy2 * (uy * ry), p3 = uy2 * (ux * zx), p4 = ux2 * (uy * zy);
        const R C1 = mad(he, mad(P.omk, p1 + p2, P.k2h * (p3 + p4)),
                         r.ic * mad(P.k11, sum2 * G.G1, mad(P.k17, dif2 * G.G7, P.k18 * (xy * G.G8))));
        const R C7 = mad(hp3, mad(P.bbm2, p3 - p4, p1 - p2),
                         r.ia * mad(P.k71, dif2 * G.G1, P.k77 * (sum2 * G.G7)));
        const R v8 = mad(mad(R(2), ux2, uy2), uy * zx, mad(R(2), uy2, ux2) * (ux * zy));
        const R C8 = mad(P.bb * hp3, v8, r.ia * mad(P.k81, xy * G.G1, P.k88 * (sum2 * G.G8)));
        Gt1 = mad(R(-0.5), C1, Gt1);
        Gt7 = mad(R(-0.5), C7, Gt7);
        Gt8 = mad(R(-0.5), C8, Gt8);
    }

    // half of m_bar - m on rows 1, 2, 4, 6, 7, 8; rows 0, 3, 5 of it: 0, Fx/2, Fy/2
    R df[9], dg[9];
    {
        const R e1 = Gt1 - d.x1, e7 = Gt7 - d.x7, e8 = Gt8 - d.x8;
        const R e2 = mad(R(1) - r.ic, d.d2, -d.x2), e4 = mad(r.ib, d.d4, -d.x4), e6 = mad(r.ib, d.d6, -d.x6);
        const R A = R(-1.0 / 18.0) * mad(R(2), e2, e1), B = R(1.0 / 18.0) * mad(R(2), e1, e2);
        const R A1 = mad(R(0.5), e7, A), A2 = mad(R(-0.5), e7, A);
        const R B1 = mad(R(0.5), e8, B), B2 = mad(R(-0.5), e8, B);
        const R X = MC == MODEL_CAVITY ? R(-2) * e4 : mad(R(-2), e4, mc.Fx), Y = mad(R(-2), e6, mc.Fy);
        const R p = MC == MODEL_CAVITY ? e4 : e4 + mc.Fx, q = e6 + mc.Fy;
        const R S = p + q, D = p - q;
        df[0] = R(2.0 / 9.0) * (e2 - e1);
        df[1] = mad(R(1.0 / 6.0), X, A1);
        df[3] = mad(R(-1.0 / 6.0), X, A1);
        df[2] = mad(R(1.0 / 6.0), Y, A2);
        df[4] = mad(R(-1.0 / 6.0), Y, A2);
        df[5] = mad(R(1.0 / 6.0), S, B1);
        df[7] = mad(R(-1.0 / 6.0), S, B1);
        df[6] = mad(R(-1.0 / 6.0), D, B2);
        df[8] = mad(R(1.0 / 6.0), D, B2);
    }

    // total-energy DF: n_bar - n = Q - L (n - n^eq + Q/2) + Y ((m + m_bar)/2 - m^eq),
    // L applied as its diagonal plus the two sigma_j (sigma_j/2 - 1) couplings
    {
        EDev<R> e;
        energy_neq(P, mc, n[1], n[2], n[3], n[4], n[5], n[6], e);
        R Y3, Y5;
        heating(ux, uy, Gt1, Gt7, Gt8, Y3, Y5);
        const R q = mc.qe, z3 = mad(q, ux, Y3), z5 = mad(q, uy, Y5);
        const R sj = R(2) * r.id, wj = r.id - R(2), sE = r.sE;  // wj: (sigma_j/2 - 1) - 1
        const R b1 = mad(-sE, e.dn1, P.gamma1 * q), b2 = mad(-sE, e.dn2, P.gamma2 * q);
        const R b3 = mad(-sj, mad(wj, e.dn4, e.s34), z3), b4 = -mad(sj, e.dn4, z3);
        const R b5 = mad(-sj, mad(wj, e.dn6, e.s56), z5), b6 = -mad(sj, e.dn6, z5);
        const R q9 = R(1.0 / 9.0) * q, s4 = R(-0.25) * sE;
        const R A = mad(R(-1.0 / 36.0), mad(R(2), b2, b1), q9), B = mad(R(1.0 / 36.0), mad(R(2), b1, b2), q9);
        const R A1 = mad(s4, n[7], A), A2 = mad(-s4, n[7], A), B1 = mad(s4, n[8], B), B2 = mad(-s4, n[8], B);
        const R X = b3 - b4, Y = b5 - b6, p = mad(R(2), b3, b4), t = mad(R(2), b5, b6);
        const R S = p + t, D = p - t;
        dg[0] = mad(R(1.0 / 9.0), b2 - b1, q9);
        dg[1] = mad(R(1.0 / 6.0), X, A1);
        dg[3] = mad(R(-1.0 / 6.0), X, A1);
        dg[2] = mad(R(1.0 / 6.0), Y, A2);
        dg[4] = mad(R(-1.0 / 6.0), Y, A2);
        dg[5] = mad(R(1.0 / 12.0), S, B1);
        dg[7] = mad(R(-1.0 / 12.0), S, B1);
        dg[6] = mad(R(-1.0 / 12.0), D, B2);
        dg[8] = mad(R(1.0 / 12.0), D, B2);
    }
    reload(f, g);
#pragma unroll
    for (int i = 0; i < 9; ++i) add(f[i], df[i], g[i], dg[i]);
}

// Redefined non-equilibrium moments of Eq. (neq.redefinition) at a fluid
// node: mt = (I - S/2) m^neq, nt = (I - L/2) n^neq + (Y/2) mt, with
// m^neq = m - m^eq + F_m/2 and n^neq = n - n^eq + Q_m/2 (Eq. decompose).
// Rows 0, 3, 5 of mt and row 0 of nt vanish identically.
template <typename R>
LBM_HD void tilde_neq(const Params<R>& P, const Mac<R>& mc, const R* f, const R* g, R* mt, R* nt) {
    Rates<R> r;
    rates(P, mc.ir, mc.T, r);
    R m[9];
    moments(f, m);
    Dev<R> d;
    neq_density(P, mc, m[1], m[2], m[4], m[6], m[7], m[8], d);
    Gv<R> G;
    apply_IS2(P, r, mc.ux, mc.uy, d, G);
    mt[0] = R(0); mt[3] = R(0); mt[5] = R(0);
    mt[1] = G.G1; mt[2] = (R(1) - r.ic) * d.d2; mt[4] = r.ib * d.d4; mt[6] = r.ib * d.d6; mt[7] = G.G7; mt[8] = G.G8;
    R n[9];
    moments(g, n);
    EDev<R> e;
    energy_neq(P, mc, n[1], n[2], n[3], n[4], n[5], n[6], e);
    // 1 - sigma_e/2 = id; 1 - sigma_j/2 = -(sigma_j/2 - 1) = 1 - id
    const R hj = R(1) - r.id;
    R Y3, Y5;
    heating(mc.ux, mc.uy, mt[1], mt[7], mt[8], Y3, Y5);
    nt[0] = R(0);
    nt[1] = r.id * e.dn1;
    nt[2] = r.id * e.dn2;
    nt[3] = mad(hj, mad(-hj, e.dn4, e.s34), R(0.5) * Y3);
    nt[4] = mad(hj, e.dn4, R(-0.5) * Y3);
    nt[5] = mad(hj, mad(-hj, e.dn6, e.s56), R(0.5) * Y5);
    nt[6] = mad(hj, e.dn6, R(-0.5) * Y5);
    nt[7] = r.id * n[7];
    nt[8] = r.id * n[8];
}

// Rebuild all 18 DFs of a wall node from its macroscopic state mb and the
// extrapolated redefined non-equilibrium moments mt, nt (Sec. 3.2):
// m^neq = (I - S/2)^-1 mt, n^neq = (I - L/2)^-1 (nt - (Y/2) mt) with the
// closed forms of App. B, then m = m^eq - F_m/2 + m^neq, n = n^eq - Q_m/2 + n^neq
// (m^eq - F_m/2 is -d of neq_density at m = 0, n^eq - Q_m/2 likewise).
template <typename R>
LBM_HD void rebuild(const Params<R>& P, const Mac<R>& mb, const R* mt, const R* nt, R* f, R* g) {
    Rates<R> r;
    rates(P, mb.ir, mb.T, r);
    const R ux = mb.ux, uy = mb.uy;
    // 1/(1 - s_e/2), 1/(1 - s_q/2), 1/(1 - s_p/2)
    const R ihe = recip(R(1) - r.ic), ihq = mad(R(18), r.nu, R(1)), ihp = recip(R(1) - r.ia);
    const R v1 = mt[1] * ihe, v2 = mt[2] * ihe, v4 = mt[4] * ihq, v6 = mt[6] * ihq;
    const R v7 = mt[7] * ihp, v8 = mt[8] * ihp;
    const R bq = P.bb * r.sq2;
    const R mn1 = mad(-(P.hh * r.sq2), mad(ux, v4, uy * v6), mad(-(P.kk * r.ic), v2, v1));
    const R mn7 = mad(R(-2) * bq, mad(ux, v4, -(uy * v6)), v7);
    const R mn8 = mad(-bq, mad(uy, v4, ux * v6), v8);

    Dev<R> d;
    neq_density(P, mb, R(0), R(0), R(0), R(0), R(0), R(0), d);
    R m[9];
    m[0] = mb.rho_d;
    m[1] = mn1 - d.d1;
    m[2] = v2 - d.d2;
    m[3] = mad(mb.rho, ux, R(-0.5) * mb.Fx);
    m[4] = v4 - d.d4;
    m[5] = mad(mb.rho, uy, R(-0.5) * mb.Fy);
    m[6] = v6 - d.d6;
    m[7] = mn7 - d.d7;
    m[8] = mn8 - d.d8;

    R Y3, Y5;
    heating(ux, uy, mt[1], mt[7], mt[8], Y3, Y5);
    const R ihE = recip(r.id), ihj = recip(R(1) - r.id);  // 1/(1 - sigma_e/2), 1/(1 - sigma_j/2)
    const R w4 = mad(R(0.5), Y3, nt[4]) * ihj, w6 = mad(R(0.5), Y5, nt[6]) * ihj;
    const R w3 = mad(-r.id, w4, mad(R(-0.5), Y3, nt[3]) * ihj);
    const R w5 = mad(-r.id, w6, mad(R(-0.5), Y5, nt[5]) * ihj);
    EDev<R> e;
    energy_neq(P, mb, R(0), R(0), R(0), R(0), R(0), R(0), e);
    R n[9];
    n[0] = mad(R(-0.5), mb.qe, mb.rhoE_d);
    n[1] = mad(nt[1], ihE, -e.dn1);
    n[2] = mad(nt[2], ihE, -e.dn2);
    n[3] = w3 + e.dn4;
    n[4] = w4 - e.dn4;
    n[5] = w5 + e.dn6;
    n[6] = w6 - e.dn6;
    n[7] = nt[7] * ihE;
    n[8] = nt[8] * ihE;
    inverse_moments(m, f);
    inverse_moments(n, g);
}

// Equilibrium deviations with zero non-equilibrium part (Eq. decompose):
// f' = M^-1 (m^eq - m^r - F_m/2), g' = M^-1 (n^eq - n^r - Q_m/2).
template <typename R>
LBM_HD void equilibrium(const Params<R>& P, const Mac<R>& mb, R* f, R* g) {
    Dev<R> d;
    neq_density(P, mb, R(0), R(0), R(0), R(0), R(0), R(0), d);
    R m[9];
    m[0] = mb.rho_d;
    m[1] = -d.d1;
    m[2] = -d.d2;
    m[3] = mad(mb.rho, mb.ux, R(-0.5) * mb.Fx);
    m[4] = -d.d4;
    m[5] = mad(mb.rho, mb.uy, R(-0.5) * mb.Fy);
    m[6] = -d.d6;
    m[7] = -d.d7;
    m[8] = -d.d8;
    EDev<R> e;
    energy_neq(P, mb, R(0), R(0), R(0), R(0), R(0), R(0), e);
    R n[9];
    n[0] = mad(R(-0.5), mb.qe, mb.rhoE_d);
    n[1] = -e.dn1;
    n[2] = -e.dn2;
    n[3] = e.dn4;
    n[4] = -e.dn4;
    n[5] = e.dn6;
    n[6] = -e.dn6;
    n[7] = R(0);
    n[8] = R(0);
    inverse_moments(m, f);
    inverse_moments(n, g);
}

// Sums over the 9 populations of a node: rho', j, sum g'.  Added in the order
// of moments(), so that a kernel that calls both adds once.
template <typename R>
LBM_HD R sum9(const R* f) {
    return f[0] + (((f[1] + f[3]) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8])));
}
template <typename R>
LBM_HD void node_sums(const R* f, const R* g, R& rd, R& jx, R& jy, R& sg) {
    const R d1 = f[5] - f[7], d2 = f[6] - f[8];
    rd = sum9(f);
    jx = (f[1] - f[3]) + (d1 - d2);
    jy = (f[2] - f[4]) + (d1 + d2);
    sg = sum9(g);
}

}  // namespace lbm
