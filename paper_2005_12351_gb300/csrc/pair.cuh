// pair.cuh -- the FP64 terms of one source particle seen from one target
// (§2, Eq. (1) with the source moments S of §2):
//   phi_i += sum_{|a|=s} S_{j,a} D_a(R),  E_i -= sum_a S_{j,a} grad D_a(R),  R = x_i - x_j,
// written out per source order (s = 0, 1, 2); r = 0 contributes nothing.
// Shared by the direct sum, the P2P kernels and the Barnes-Hut walk, as is the
// P2P's reciprocal square root.
#pragma once

namespace fmm {

// 1/sqrt(x) for x > 0 in FP64 without the double-precision MUFU path:
//  1. x = m 4^k with m in [1, 4), by integer operations on the exponent;
//  2. an FP32 seed y_m = rsqrtf(m) (m rounded toward zero to float);
//  3. y0 = y_m 2^-k, assembled from the float's bits;
//  4. one third-order Householder step for f(y) = y^-2 - x:
//        e = 1 - x y0^2,   y = y0 + y0 e (1/2 + 3/8 e),
//     which leaves a relative error of about (5/16) e^3 ~ 2^-67 before the
//     final roundings (e ~ 2^-22 from the seed).  Five FP64 operations.
// x = 0 returns a finite value of no meaning (the callers mask r = 0).  A subnormal x (exponent field 0,
// x != 0: pairs closer than ~1.5e-154) takes CUDA's rsqrt instead: the
// exponent arithmetic above assumes a normal number.  The test is integer
// work only, so the FP64 pipe of the common path is unchanged.
__device__ __forceinline__ double rsqrt_hh(double x)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    if (__builtin_expect((hi & 0x7ff00000) == 0 && (hi | lo) != 0, 0)) return rsqrt(x);
    const int ex = ((hi >> 20) & 0x7ff) - 1023;                 // unbiased exponent
    const int k = ex >> 1;                                      // floor(ex / 2)
    const int mhi = (hi & 0x000fffff) | ((1023 + (ex - 2 * k)) << 20);   // m in [1, 4)
    // float with m's exponent and the top 23 mantissa bits
    const int fbits = ((mhi - (896 << 20)) << 3) | ((unsigned)lo >> 29);
    const float ym = rsqrtf(__int_as_float(fbits));
    const int yb = __float_as_int(ym);
    const int yhi = ((yb >> 3) + (896 << 20)) - (k << 20);
    const double y0 = __hiloint2double(yhi, yb << 29);
    const double t = x * y0;
    const double e = fma(-t, y0, 1.0);
    const double c = fma(e, 0.375, 0.5);
    const double u = y0 * e;
    return fma(u, c, y0);
}

template <int S, bool PHI, bool FIELD>
__device__ __forceinline__ void pair_fp64(double dx, double dy, double dz, const double *Sj,
                                          double &f, double &e0, double &e1, double &e2)
{
    const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
    const double rinv = r2 > 0.0 ? rsqrt(r2) : 0.0;
    const double rinv2 = rinv * rinv;
    if (S == 0) {
        const double q = Sj[0];
        if (PHI) f = fma(q, rinv, f);
        if (FIELD) {
            const double w = q * rinv * rinv2;
            e0 = fma(w, dx, e0); e1 = fma(w, dy, e1); e2 = fma(w, dz, e2);
        }
    } else if (S == 1) {
        const double rinv3 = rinv * rinv2;
        const double sr = fma(Sj[0], dx, fma(Sj[1], dy, Sj[2] * dz));
        if (PHI) f = fma(-sr, rinv3, f);
        if (FIELD) {
            const double w = 3.0 * sr * rinv3 * rinv2;
            e0 = fma(Sj[0], rinv3, fma(-w, dx, e0));
            e1 = fma(Sj[1], rinv3, fma(-w, dy, e1));
            e2 = fma(Sj[2], rinv3, fma(-w, dz, e2));
        }
    } else {
        const double rinv3 = rinv * rinv2, rinv5 = rinv3 * rinv2;
        // half-gradient of q: h = (grad q)/2 is not symmetric in the S layout, so form grad q
        const double gq0 = fma(2.0 * Sj[0], dx, fma(Sj[1], dy, Sj[2] * dz));
        const double gq1 = fma(Sj[1], dx, fma(2.0 * Sj[3], dy, Sj[4] * dz));
        const double gq2 = fma(Sj[2], dx, fma(Sj[4], dy, 2.0 * Sj[5] * dz));
        // q = (R . grad q) / 2 for a homogeneous quadratic
        const double q = 0.5 * fma(gq0, dx, fma(gq1, dy, gq2 * dz));
        const double tr = Sj[0] + Sj[3] + Sj[5];
        if (PHI) f += 3.0 * q * rinv5 - tr * rinv3;
        if (FIELD) {
            const double a = 3.0 * rinv5;
            const double w = fma(15.0 * q, rinv5 * rinv2, -3.0 * tr * rinv5);
            e0 = fma(w, dx, fma(-a, gq0, e0));
            e1 = fma(w, dy, fma(-a, gq1, e1));
            e2 = fma(w, dz, fma(-a, gq2, e2));
        }
    }
}

// Moments per particle of the orders SLO..SHI (graded order, shell by shell).
template <int SLO, int SHI>
struct Orders {
    static constexpr int n = ((SHI + 1) * (SHI + 2) * (SHI + 3) - SLO * (SLO + 1) * (SLO + 2)) / 6;
};

// A particle carrying every order SLO..SHI (§2 mixed systems): the sum of the
// pair terms of its shells, the moments of shell s starting after those of
// the lower shells.
template <int SLO, int SHI, bool PHI, bool FIELD>
__device__ __forceinline__ void pair_orders(double dx, double dy, double dz, const double *Sj,
                                            double &f, double &e0, double &e1, double &e2)
{
    pair_fp64<SLO, PHI, FIELD>(dx, dy, dz, Sj, f, e0, e1, e2);
    if constexpr (SHI >= SLO + 1)
        pair_fp64<SLO + 1, PHI, FIELD>(dx, dy, dz, Sj + (SLO + 1) * (SLO + 2) / 2, f, e0, e1, e2);
    if constexpr (SHI >= SLO + 2)
        pair_fp64<SLO + 2, PHI, FIELD>(dx, dy, dz, Sj + (SLO + 1) * (SLO + 2) / 2 + (SLO + 2) * (SLO + 3) / 2,
                                       f, e0, e1, e2);
}

}  // namespace fmm
