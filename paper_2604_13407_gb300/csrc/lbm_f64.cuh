// FP64 evaluation of the step.  Every rounded operation is the one that the plain left-to-right
// order of the formulas of Sec. 2 has (dense m = M f and f = M^T diag(1/|M_k|^2) m_bar, divisions
// where the paper divides), so the FP64 path is reproducible bit for bit by any plain FP64
// evaluation of the same formulas and FP64 results can be compared exactly over long, dynamically
// unstable runs.  Compiled without multiply-add contraction.
//
// What bounds it: GB300's FP64 pipe takes one warp instruction per SM every 16 cycles, so an FP64
// kernel's time is its FP64 instruction count and everything else hides behind it.  Operations
// whose result needs no rounding are therefore left out or folded, which changes no bit:
//   * entries 0 and +-1 of M cost nothing or one add; entries +-2, +-4 scale by a power of two, so
//     their product is exact and one multiply-add rounds as the separate product and sum do;
//   * a product by 1/2, 2 or 6/2 of a term is folded the same way (0.5 F_m, Q_2 = -Q_1/2, F_m7);
//   * the nine moments m_0, m_3, m_5 are rho, j_x, j_y, and m_bar_0 = rho: computed once;
//   * divisions by 3 and 9 times a power of two multiply by the reciprocal and correct once
//     (div_const), divisions that share a divisor share its reciprocal (Divisor);
//   * the coefficients of Q_m are formed once on the host, in the same order.
// The dense evaluation with 17 general divisions issued 465 FP64 instructions a node in the collide
// pass.  Against it, per step: 256 x 256 banded channel (two-pass) 100 -> 61 us, 1024 x 1024
// periodic (one-pass) 1.58 -> 1.12 ms, 4 x 128 column (latency of one warp per SM) 24 -> 20 us.
#pragma once

namespace lbm {
namespace f64 {

__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }

// a / D for D = 3 or 9, correctly rounded.  With r = RN(1/D) (relative error 2^-54 for both) the
// product q = RN(a r) is within one ulp of a/D, and one correction by the exact remainder then
// rounds correctly (Markstein, IBM J. Res. Dev. 34(1), 1990, on division by a correctly rounded
// reciprocal).  Magnitudes outside 2^+-450 (0 excepted), infinities and NaN take the general
// division: the remainder could underflow there.
__device__ __forceinline__ bool in_range(double a)
{
    const unsigned hi = (unsigned)__double2hiint(a) & 0x7fffffffu;
    return hi - (573u << 20) < (900u << 20) || (hi | (unsigned)__double2loint(a)) == 0u;
}
template <int D>
__device__ __forceinline__ double div_const(double a)
{
    static_assert(D == 3 || D == 9, "the error bound of the reciprocal is known for 3 and 9");
    constexpr double r = 1.0 / (double)D;
    const double q = a * r;
    const double t = fma_(fma_(-(double)D, q, a), r, q);
    return in_range(a) ? t : a / (double)D;
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
        return ok && in_range(a) ? q : a / b;
    }
};
__device__ __forceinline__ Divisor divisor(double b) { return Divisor{b, __drcp_rn(b), in_range(b) && b != 0.0}; }

__device__ __forceinline__ double density(const double (&f)[9])
{
    double r = f[0];
#pragma unroll
    for (int i = 1; i < 9; ++i) r += f[i];
    return r;
}

__device__ __forceinline__ double p_eos(const KParams &kp, double rho)
{
    if (kp.eos == 0) return kp.eos_K * (rho * kp.eos_R * kp.eos_T / (1.0 - kp.eos_b * rho) - kp.eos_a * rho * rho);
    const double eta = kp.eos_b * rho * 0.25;
    const double e2 = eta * eta, om = 1.0 - eta;
    const double num = 1.0 + eta + e2 - e2 * eta;
    const double den = om * om * om;
    return kp.eos_K * (rho * kp.eos_R * kp.eos_T * num / den - kp.eos_a * rho * rho);
}

// sqrt(2 (p_EOS - rho/3)/G); a G that is a power of two (the usual -1) divides exactly
__device__ __forceinline__ double psi_of(const KParams &kp, double rho)
{
    const double d = 2.0 * (p_eos(kp, rho) - div_const<3>(rho));
    return sqrt(kp.G_pow2 ? d * kp.inv_G : d / kp.G);
}

template <class Ps>
__device__ __forceinline__ void stencil_S(const Ps &ps, double &Sx, double &Sy)
{
    double sx = 0.0, sy = 0.0;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const double p = ((i <= 4) ? 1.0 / 3.0 : 1.0 / 12.0) * ps(i);
        if (ex_(i)) sx = i == 1 ? p : (ex_(i) > 0 ? sx + p : sx - p);
        if (ey_(i)) sy = i == 2 ? p : (ey_(i) > 0 ? sy + p : sy - p);
    }
    Sx = sx;
    Sy = sy;
}

// f = M^T (m_k/|M_k|^2), the terms in the order k = 0..8.  u_k is m_k/|M_k|^2 without its power of
// two (|M_k|^2 = 9, 36, 36, 6, 12, 6, 12, 4, 4), which the multiply-adds carry exactly.
__device__ __forceinline__ void from_moments(const double (&m)[9], double (&f)[9])
{
    const double u0 = div_const<9>(m[0]), u1 = div_const<9>(m[1]), u2 = div_const<9>(m[2]);
    const double u3 = div_const<3>(m[3]), u4 = div_const<3>(m[4]), u5 = div_const<3>(m[5]), u6 = div_const<3>(m[6]);
    f[0] = (u0 - u1) + u2;
    const double a = fma_(-0.5, u2, fma_(-0.25, u1, u0));  // axes
    f[1] = fma_(0.25, m[7], fma_(-0.5, u4, fma_(0.5, u3, a)));
    f[2] = fma_(-0.25, m[7], fma_(-0.5, u6, fma_(0.5, u5, a)));
    f[3] = fma_(0.25, m[7], fma_(0.5, u4, fma_(-0.5, u3, a)));
    f[4] = fma_(-0.25, m[7], fma_(0.5, u6, fma_(-0.5, u5, a)));
    const double d = fma_(0.25, u2, fma_(0.5, u1, u0));    // diagonals
    const double p = fma_(0.25, u4, fma_(0.5, u3, d)), q = fma_(-0.25, u4, fma_(-0.5, u3, d));
    f[5] = fma_(0.25, m[8], fma_(0.25, u6, fma_(0.5, u5, p)));
    f[6] = fma_(-0.25, m[8], fma_(0.25, u6, fma_(0.5, u5, q)));
    f[7] = fma_(0.25, m[8], fma_(-0.25, u6, fma_(-0.5, u5, q)));
    f[8] = fma_(-0.25, m[8], fma_(-0.25, u6, fma_(-0.5, u5, p)));
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

__device__ __forceinline__ void collide(const KParams &kp, const double (&f)[9], double psi, double Sx, double Sy,
                                        double Fex, double Fey, double (&fb)[9], double &uxo, double &uyo)
{
    const double rho = density(f);
    const Divisor by_rho = divisor(rho);
    // m = M f, the terms in the order i = 0..8 (m_0 = rho, m_3 = j_x, m_5 = j_y)
    const double jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8];
    const double jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8];
    double m1 = -4.0 * f[0], m2 = 4.0 * f[0];
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
    const double m4 = fma_(2.0, f[3], -2.0 * f[1]) + f[5] - f[6] - f[7] + f[8];
    const double m6 = fma_(2.0, f[4], -2.0 * f[2]) + f[5] + f[6] - f[7] - f[8];
    const double m7 = f[1] - f[2] + f[3] - f[4], m8 = f[5] - f[6] + f[7] - f[8];

    const double Gpsi = kp.G * psi;
    const double Fix = -Gpsi * Sx, Fiy = -Gpsi * Sy;
    const double Fx = Fix + Fex, Fy = Fiy + Fey;
    const double ux = by_rho(fma_(0.5, Fx, jx)), uy = by_rho(fma_(0.5, Fy, jy));
    double meq[9];
    equilibrium_moments(rho, ux, uy, meq);
    const double Fxu = Fx * ux, Fyv = Fy * uy;
    const double Fm1 = 6.0 * (Fxu + Fyv), h7 = Fxu - Fyv;  // h7 = F_m7/2
    const double Fm8 = Fx * uy + Fy * ux;
    // Q_m with |F_int|^2 / (G psi^2) as written in the paper
    const Divisor by_Gpsi2 = divisor(Gpsi * psi);
    const double Fix2 = Fix * Fix, Fiy2 = Fiy * Fiy;
    const double X = by_Gpsi2(Fix2), Y = by_Gpsi2(Fiy2);
    const double Q1 = kp.q1c * (X + Y);
    const double Q7 = by_Gpsi2(kp.k1 * (Fix2 - Fiy2));
    const double Q8 = by_Gpsi2(kp.k1 * Fix * Fiy);
    double sp = kp.sp, sq = kp.sq;
    if (kp.var_tau) {
        double w = (rho - kp.rho_g) / (kp.rho_l - kp.rho_g);
        w = w < 0.0 ? 0.0 : (w > 1.0 ? 1.0 : w);
        const double nu = kp.nu_g + w * (kp.nu_l - kp.nu_g);
        const double tau = 3.0 * nu + 0.5;
        sp = 1.0 / tau;
        sq = 1.0 / (0.5 + kp.Lambda / (tau - 0.5));
    }
    // m_bar_k = m + F_m - s (m - m_eq + F_m/2) + s Q (Eq. lbe.col); s_0 = s_j = 1
    const double sQ1 = sp * Q1;
    double mb[9];
    mb[0] = rho;
    mb[1] = (m1 + Fm1) - sp * fma_(0.5, Fm1, m1 - meq[1]) + sQ1;
    const double c2 = (m2 - Fm1) - sp * fma_(-0.5, Fm1, m2 - meq[2]);
    mb[2] = kp.q2fac == -1.0 ? c2 - sQ1 : fma_(-0.5, sQ1, c2);
    mb[3] = (jx + Fx) - fma_(0.5, Fx, jx - meq[3]);
    mb[5] = (jy + Fy) - fma_(0.5, Fy, jy - meq[5]);
    mb[4] = (m4 - Fx) - sq * fma_(-0.5, Fx, m4 - meq[4]);
    mb[6] = (m6 - Fy) - sq * fma_(-0.5, Fy, m6 - meq[6]);
    if (kp.improved) {
        mb[4] += sq * ((kp.q4a * X - kp.q4b * Y) * ux);
        mb[6] += sq * ((kp.q4a * Y - kp.q4b * X) * uy);
    }
    mb[7] = fma_(2.0, h7, m7) - sp * ((m7 - meq[7]) + h7) + sp * Q7;
    mb[8] = (m8 + Fm8) - sp * fma_(0.5, Fm8, m8 - meq[8]) + sp * Q8;
    from_moments(mb, fb);
    uxo = ux;
    uyo = uy;
}

}  // namespace f64
}  // namespace lbm
