// FP64 evaluation of the step.  Every rounded operation is the one that the plain left-to-right
// order of the formulas of Sec. 2 has (dense m = M f and f = M^T diag(1/|M_k|^2) m_bar, divisions
// where the paper divides), so the FP64 path is reproducible bit for bit by any plain FP64
// evaluation of the same formulas and FP64 results can be compared exactly over long, dynamically
// unstable runs.  Compiled without multiply-add contraction.
//
// What bounds it: GB300's FP64 pipe takes one warp instruction per SM every 16 cycles, so an FP64
// kernel's time is its FP64 instruction count and everything else hides behind it.  Operations
// whose result needs no rounding are therefore left out or folded, which changes no bit (but one that
// nothing sees: a quotient of -0 by a positive divisor comes out as +0, and no such dividend of a step is
// -0, since a sum that cancels is +0 and the forces are sums):
//   * entries 0 and +-1 of M cost nothing or one add; entries +-2, +-4 scale by a power of two, so
//     their product is exact and one multiply-add rounds as the separate product and sum do;
//   * a product by 1/2, 2 or 6/2 of a term is folded the same way (0.5 F_m, Q_2 = -Q_1/2, F_m7);
//   * the nine moments m_0, m_3, m_5 are rho, j_x, j_y, and m_bar_0 = rho: computed once;
//   * divisions by 3 and 9 times a power of two multiply by the reciprocal and correct once
//     (div_const), divisions that share a divisor share its reciprocal (Divisor);
//   * the coefficients of Q_m are formed once on the host, in the same order.
// The dense evaluation with 17 general divisions issued 465 FP64 instructions a node in the collide
// pass.  Against it, per step: 256 x 256 banded channel (two-pass) 100 -> 61 us, 1024 x 1024
// periodic (one-pass) 1.58 -> 1.12 ms, 4 x 128 column (latency of one warp per SM) 24 -> 20 us; the
// tile and small-lattice kernels and the general division out of line (below) take the rest of the way to
// 47 us, 0.65 ms and 5.4 us.
#pragma once

namespace lbm {
namespace f64 {

__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }

// a / D for D = 3 or 9, correctly rounded (-0 gives +0).  With r = RN(1/D) (relative error 2^-54 for both) the
// product q = RN(a r) is within one ulp of a/D, and one correction by the exact remainder then
// rounds correctly (Markstein, IBM J. Res. Dev. 34(1), 1990, on division by a correctly rounded
// reciprocal).  Magnitudes outside 2^+-450 (0 excepted), infinities and NaN take the general
// division: the remainder could underflow there.
__device__ __forceinline__ bool in_range(double a)
{
    const unsigned hi = (unsigned)__double2hiint(a) & 0x7fffffffu;
    return hi - (573u << 20) < (900u << 20) || (hi | (unsigned)__double2loint(a)) == 0u;
}
// The general division of those, a function of its own: inlined, its first instructions were executed at
// every quotient, whether it was then needed or not (395 FP64 instructions a node instead of 328; 1024^2
// periodic 0.77 -> 0.65 ms a step, 256^2 55.6 -> 47.3 us, 4 x 128 column 6.5 -> 5.4).
static __device__ __noinline__ double div_general(double a, double b) { return a / b; }
template <int D>
__device__ __forceinline__ double div_const(double a)
{
    static_assert(D == 3 || D == 9, "the error bound of the reciprocal is known for 3 and 9");
    constexpr double r = 1.0 / (double)D;
    const double q = a * r;
    const double t = fma_(fma_(-(double)D, q, a), r, q);
    return in_range(a) ? t : div_general(a, (double)D);
}

// Quotients by one divisor b, each correctly rounded: q = RN(a r) with r = RN(1/b) is within two
// ulps of a/b, the first correction brings it within one (faithful), the second rounds correctly
// (Markstein, as above).  The same fallback outside the range where the remainders are exact.
struct Divisor {
    double b, r;
    bool ok;
    __device__ __forceinline__ double operator()(double a) const
    {
        double q = a * r;
        q = fma_(fma_(-b, q, a), r, q);
        q = fma_(fma_(-b, q, a), r, q);
        return ok && in_range(a) ? q : div_general(a, b);
    }
};
__device__ __forceinline__ bool is_nonzero(double b) { return (((unsigned)__double2hiint(b) & 0x7fffffffu) | (unsigned)__double2loint(b)) != 0u; }
__device__ __forceinline__ Divisor divisor(double b) { return Divisor{b, __drcp_rn(b), in_range(b) && is_nonzero(b)}; }

__device__ __forceinline__ double density(const double (&f)[9])
{
    double r = f[0];
#pragma unroll
    for (int i = 1; i < 9; ++i) r += f[i];
    return r;
}

// p_EOS = K (num/den - a rho^2); psi = sqrt(2 (p_EOS - rho/3)/G).  In pieces, which k_small1 spreads over
// four warps.  Products by a gas constant or a K of 1 (the usual ones) change nothing and are left out.
__device__ __forceinline__ double eos_num(const KParams &kp, double rho)
{
    const double rRT = (kp.unit_R ? rho : rho * kp.eos_R) * kp.eos_T;
    if (kp.eos == 0) return rRT;
    const double eta = kp.eos_b4 * rho, e2 = eta * eta;
    return rRT * (1.0 + eta + e2 - e2 * eta);
}
__device__ __forceinline__ double eos_den(const KParams &kp, double rho)
{
    if (kp.eos == 0) return 1.0 - kp.eos_b * rho;
    const double om = 1.0 - kp.eos_b4 * rho;
    return om * om * om;
}
__device__ __forceinline__ double eos_attraction(const KParams &kp, double rho) { return kp.eos_a * rho * rho; }
// a G that is a power of two (the usual -1) divides exactly
__device__ __forceinline__ double psi_of(const KParams &kp, double ratio, double attraction, double third)
{
    const double p = ratio - attraction;
    const double d = (kp.unit_K ? p : kp.eos_K * p) - third;
    return sqrt(kp.G_pow2 ? d * kp.two_inv_G : 2.0 * d / kp.G);
}
__device__ __forceinline__ double psi_of(const KParams &kp, double rho)
{
    return psi_of(kp, eos_num(kp, rho) / eos_den(kp, rho), eos_attraction(kp, rho), div_const<3>(rho));
}

// S of Eq. (fint), the terms in the order i = 1..8
template <class Ps>
__device__ __forceinline__ double stencil_x(const Ps &ps)
{
    const double w1 = 1.0 / 3.0, w5 = 1.0 / 12.0;
    return w1 * ps(1) - w1 * ps(3) + w5 * ps(5) - w5 * ps(6) - w5 * ps(7) + w5 * ps(8);
}
template <class Ps>
__device__ __forceinline__ double stencil_y(const Ps &ps)
{
    const double w1 = 1.0 / 3.0, w5 = 1.0 / 12.0;
    return w1 * ps(2) - w1 * ps(4) + w5 * ps(5) + w5 * ps(6) - w5 * ps(7) - w5 * ps(8);
}
template <class Ps>
__device__ __forceinline__ void stencil_S(const Ps &ps, double &Sx, double &Sy)
{
    Sx = stencil_x(ps);
    Sy = stencil_y(ps);
}

// f = M^T (m_k/|M_k|^2), the terms in the order k = 0..8, from u_k = m_k/|M_k|^2 without its power of
// two (|M_k|^2 = 9, 36, 36, 6, 12, 6, 12, 4, 4), which the multiply-adds carry exactly.  In the pieces that
// k_small1 spreads over four warps: f_0, f_1 and f_3; f_2 and f_4; f_5 and f_8; f_6 and f_7.
__device__ __forceinline__ double axes(const double (&u)[9]) { return fma_(-0.5, u[2], fma_(-0.25, u[1], u[0])); }
__device__ __forceinline__ double diagonals(const double (&u)[9]) { return fma_(0.25, u[2], fma_(0.5, u[1], u[0])); }
__device__ __forceinline__ void populations_013(const double (&u)[9], double (&f)[9])
{
    f[0] = (u[0] - u[1]) + u[2];
    const double a = axes(u);
    f[1] = fma_(0.25, u[7], fma_(-0.5, u[4], fma_(0.5, u[3], a)));
    f[3] = fma_(0.25, u[7], fma_(0.5, u[4], fma_(-0.5, u[3], a)));
}
__device__ __forceinline__ void populations_24(const double (&u)[9], double (&f)[9])
{
    const double a = axes(u);
    f[2] = fma_(-0.25, u[7], fma_(-0.5, u[6], fma_(0.5, u[5], a)));
    f[4] = fma_(-0.25, u[7], fma_(0.5, u[6], fma_(-0.5, u[5], a)));
}
__device__ __forceinline__ void populations_58(const double (&u)[9], double (&f)[9])
{
    const double p = fma_(0.25, u[4], fma_(0.5, u[3], diagonals(u)));
    f[5] = fma_(0.25, u[8], fma_(0.25, u[6], fma_(0.5, u[5], p)));
    f[8] = fma_(-0.25, u[8], fma_(-0.25, u[6], fma_(-0.5, u[5], p)));
}
__device__ __forceinline__ void populations_67(const double (&u)[9], double (&f)[9])
{
    const double q = fma_(-0.25, u[4], fma_(-0.5, u[3], diagonals(u)));
    f[6] = fma_(-0.25, u[8], fma_(0.25, u[6], fma_(0.5, u[5], q)));
    f[7] = fma_(0.25, u[8], fma_(-0.25, u[6], fma_(-0.5, u[5], q)));
}
__device__ __forceinline__ void populations(const double (&u)[9], double (&f)[9])
{
    populations_013(u, f);
    populations_24(u, f);
    populations_58(u, f);
    populations_67(u, f);
}
__device__ __forceinline__ void from_moments(const double (&m)[9], double (&f)[9])
{
    const double u[9] = {div_const<9>(m[0]), div_const<9>(m[1]), div_const<9>(m[2]), div_const<3>(m[3]), div_const<3>(m[4]),
                         div_const<3>(m[5]), div_const<3>(m[6]), m[7], m[8]};
    populations(u, f);
}

__device__ __forceinline__ void equilibrium_moments(double rho, double ux, double uy, double (&meq)[9])
{
    const double u2 = ux * ux + uy * uy;
    const double r3u2 = 3.0 * rho * u2;
    meq[0] = rho;
    meq[1] = fma_(-2.0, rho, r3u2);
    meq[2] = rho - r3u2;
    meq[3] = rho * ux;
    meq[4] = -meq[3];
    meq[5] = rho * uy;
    meq[6] = -meq[5];
    meq[7] = meq[3] * ux - meq[5] * uy;
    meq[8] = meq[3] * uy;
}

__device__ __forceinline__ void equilibrium(double rho, double ux, double uy, double (&fb)[9])
{
    double meq[9];
    equilibrium_moments(rho, ux, uy, meq);
    from_moments(meq, fb);
}

// ---- the collision, in the pieces that k_small1 spreads over four warps.
// m_1 and m_2 of M f, the terms in the order i = 0..8
__device__ __forceinline__ void moments_12(const double (&f)[9], double &m1, double &m2)
{
    m1 = -4.0 * f[0], m2 = 4.0 * f[0];
#pragma unroll
    for (int i = 1; i < 5; ++i) {
        m1 -= f[i];
        m2 = fma_(-2.0, f[i], m2);
    }
#pragma unroll
    for (int i = 5; i < 9; ++i) {
        m1 = fma_(2.0, f[i], m1);
        m2 += f[i];
    }
}
// s_p and s_q of two relaxation times
__device__ __forceinline__ void relaxation(const KParams &kp, double rho, double &sp, double &sq)
{
    double w = (rho - kp.rho_g) / (kp.rho_l - kp.rho_g);
    w = w < 0.0 ? 0.0 : (w > 1.0 ? 1.0 : w);
    const double nu = kp.nu_g + w * (kp.nu_l - kp.nu_g);
    const double tau = 3.0 * nu + 0.5;
    sp = 1.0 / tau;
    sq = 1.0 / (0.5 + kp.Lambda / (tau - 0.5));
}
// m_bar_k = m + F_m - s (m - m_eq + F_m/2) + s Q (Eq. lbe.col), Q_m with |F_int|^2 / (G psi^2) as written
// in the paper (X = F_int,x^2 / (G psi^2), Y likewise)
struct Stress12 {
    double e1, e2, Fm1;  // m_k - m_eq_k, and F_m1 = -F_m2
};
__device__ __forceinline__ Stress12 stress_12(double rho, double m1, double m2, double Fx, double Fy, double ux, double uy)
{
    const double u2 = ux * ux + uy * uy, r3u2 = 3.0 * rho * u2;
    return Stress12{m1 - fma_(-2.0, rho, r3u2), m2 - (rho - r3u2), 6.0 * (Fx * ux + Fy * uy)};
}
__device__ __forceinline__ void relaxed_12(const KParams &kp, const Stress12 &t, double m1, double m2, double X, double Y, double sp,
                                           double &a1, double &a2)
{
    const double sQ1 = sp * (kp.q1c * (X + Y));
    a1 = (m1 + t.Fm1) - sp * fma_(0.5, t.Fm1, t.e1) + sQ1;
    const double c2 = (m2 - t.Fm1) - sp * fma_(-0.5, t.Fm1, t.e2);
    a2 = kp.q2_full ? c2 - sQ1 : fma_(-0.5, sQ1, c2);  // Q_2 = -Q_1 or -Q_1/2
}
// one direction's momentum (s_j = 1) and energy flux, ru = rho u; X along it, Y across
__device__ __forceinline__ double relaxed_j(double j, double F, double ru) { return (j + F) - fma_(0.5, F, j - ru); }
__device__ __forceinline__ double relaxed_q(const KParams &kp, double q, double F, double ru, double u, double X, double Y, double sq)
{
    const double aq = (q - F) - sq * fma_(-0.5, F, q + ru);
    return kp.improved ? aq + sq * ((kp.q4a * X - kp.q4b * Y) * u) : aq;
}
__device__ __forceinline__ double relaxed_7(double rux, double ruy, double m7, double Fx, double Fy, double ux, double uy, double Q7, double sp)
{
    const double meq7 = rux * ux - ruy * uy;
    const double h7 = Fx * ux - Fy * uy;  // F_m7/2
    return fma_(2.0, h7, m7) - sp * ((m7 - meq7) + h7) + sp * Q7;
}
__device__ __forceinline__ double relaxed_8(double rux, double m8, double Fx, double Fy, double ux, double uy, double Q8, double sp)
{
    const double meq8 = rux * uy;
    const double Fm8 = Fx * uy + Fy * ux;
    return (m8 + Fm8) - sp * fma_(0.5, Fm8, m8 - meq8) + sp * Q8;
}

__device__ __forceinline__ void collide(const KParams &kp, const double (&f)[9], double psi, double Sx, double Sy,
                                        double Fex, double Fey, double (&fb)[9], double &ux, double &uy)
{
    const double rho = density(f);
    const Divisor by_rho = divisor(rho);
    // m = M f, the terms in the order i = 0..8 (m_0 = rho, m_3 = j_x, m_5 = j_y)
    const double jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8];
    const double jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8];
    double m1, m2;
    moments_12(f, m1, m2);
    const double m4 = fma_(2.0, f[3], -2.0 * f[1]) + f[5] - f[6] - f[7] + f[8];
    const double m6 = fma_(2.0, f[4], -2.0 * f[2]) + f[5] + f[6] - f[7] - f[8];
    const double m7 = f[1] - f[2] + f[3] - f[4], m8 = f[5] - f[6] + f[7] - f[8];

    const double Gpsi = kp.G * psi;
    const double Fix = -Gpsi * Sx, Fiy = -Gpsi * Sy;
    const double Fx = Fix + Fex, Fy = Fiy + Fey;
    ux = by_rho(fma_(0.5, Fx, jx)), uy = by_rho(fma_(0.5, Fy, jy));
    const Divisor by_Gpsi2 = divisor(Gpsi * psi);
    const double X = by_Gpsi2(Fix * Fix), Y = by_Gpsi2(Fiy * Fiy);
    double sp = kp.sp, sq = kp.sq;
    if (kp.var_tau) relaxation(kp, rho, sp, sq);
    double mb[9];
    mb[0] = rho;
    relaxed_12(kp, stress_12(rho, m1, m2, Fx, Fy, ux, uy), m1, m2, X, Y, sp, mb[1], mb[2]);
    const double rux = rho * ux, ruy = rho * uy;
    mb[3] = relaxed_j(jx, Fx, rux), mb[4] = relaxed_q(kp, m4, Fx, rux, ux, X, Y, sq);
    mb[5] = relaxed_j(jy, Fy, ruy), mb[6] = relaxed_q(kp, m6, Fy, ruy, uy, Y, X, sq);
    mb[7] = relaxed_7(rux, ruy, m7, Fx, Fy, ux, uy, by_Gpsi2(kp.k1 * (Fix * Fix - Fiy * Fiy)), sp);
    mb[8] = relaxed_8(rux, m8, Fx, Fy, ux, uy, by_Gpsi2(kp.k1 * Fix * Fiy), sp);
    from_moments(mb, fb);
}

}  // namespace f64
}  // namespace lbm
