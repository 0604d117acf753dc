// Exponentially scaled modified Bessel functions of the kernel:
//     K0e(x) = e^x K0(x),     D(x) = e^x [K1(x) - K0(x)],
// the two functions in Eq. "SG force kernel exact" (D) and Eq. "grav.
// potential 2D" (K0e) of Rendon Restrepo et al. (2025), with X = d^2/8.
//
// CUDA's math library has no K0/K1, and FP64 units run at 1/64 of the FP32 rate
// here, so each function is one short polynomial (sg_bessel_tab.cuh):
//   x < 2^-20   ascending series (DLMF 10.31.1 and 10.31.2), FP64 only (rare);
//   x < 16      quarter-octave tables, FP64 12 and FP32 6 multiply-adds and the last sum;
//   x >= 16     polynomials in 1/x (the tails), FP64 9 or 10, FP32 4.
// (A quadrature of 24 reciprocal square roots and a Hankel series of 14
// divisions took their place before: 128 x 256 semi-spectral plan and solve 15.6 ms, now 2.1.)
#pragma once

#include <cuda_runtime.h>

#include "sg_bessel_tab.cuh"

namespace sg {

// the ascending series, x < 2
__device__ __forceinline__ void k0e_D_series(double x, double &k0e, double &D)
{
    // K0 = -(ln(x/2) + gamma) I0 + sum_{k>=1} H_k y^k / (k!)^2,
    // K1 = 1/x + ln(x/2) I1 - (x/4) sum_k (psi(k+1) + psi(k+2)) y^k / (k! (k+1)!),
    // y = x^2/4, psi(k+1) = H_k - gamma.
    const double gam = 0.57721566490153286061;
    const double y = 0.25 * x * x;
    const double L = log(0.5 * x);
    double t0 = 1.0, t1 = 1.0, H = 0.0;
    double I0 = 1.0, I1s = 1.0, S0 = 0.0;
    double S1 = 1.0 - 2.0 * gam;   // k = 0 term: psi(1) + psi(2) = 1 - 2 gamma
    for (int k = 1; k < 40; ++k) {
        t0 *= y / ((double)k * k);
        t1 *= y / ((double)k * (k + 1));
        H += 1.0 / k;
        I0 += t0;
        I1s += t1;
        S0 += H * t0;
        S1 += (2.0 * H + 1.0 / (k + 1) - 2.0 * gam) * t1;
        if (t0 < 1e-18 * I0) break;
    }
    const double K0 = -(L + gam) * I0 + S0;
    const double K1 = 1.0 / x + L * (0.5 * x) * I1s - 0.25 * x * S1;
    const double ex = exp(x);
    k0e = ex * K0;
    D = ex * (K1 - K0);
}

// K0e(x) and E(x) = x D(x) from the quarter-octave tables, 2^-20 <= x < 16
// (bessel_in_table).  The index and the argument come from the bits of x; a
// warp's lanes mostly share an entry, so the loads are broadcasts from L1.
__device__ __forceinline__ bool bessel_in_table(float x) { return x >= 0x1p-20f && x < 16.0f; }
__device__ __forceinline__ bool bessel_in_table(double x) { return x >= 0x1p-20 && x < 16.0; }
__device__ __forceinline__ void bessel_table(float x, float &k0e, float &E)
{
    const int b = __float_as_int(x);
    const int entry = (b >> 21) - 4 * (127 + BT_LO);
    const float4 *c = reinterpret_cast<const float4 *>(&BT_32[entry][0][0]);
    const float t = __int_as_float((b & 0x007FFFFF) | 0x3F800000) - __int_as_float((b & 0x00600000) | 0x3F900000);
    const float4 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2);
    const float4 l = __ldg(reinterpret_cast<const float4 *>(&BT_32L[entry][0]));
    // the value is c_0 + (the rest, an eighth of it at most): rounded once, as if
    // evaluated in 64 bits, within 0.2 of the last place
    const float v = 64.0f * t * t, T6 = fmaf(fmaf(fmaf(32.0f, v, -48.0f), v, 18.0f), v, -1.0f);
    const float k = fmaf(fmaf(fmaf(fmaf(c1.y, t, c1.x), t, c0.w), t, c0.z), t, c0.y);
    const float e = fmaf(fmaf(fmaf(fmaf(c2.w, t, c2.z), t, c2.y), t, c2.x), t, c1.w);
    k0e = c0.x + fmaf(k, t, fmaf(l.y, T6, l.x));
    E = c1.z + fmaf(e, t, fmaf(l.w, T6, l.z));
}
__device__ __forceinline__ void bessel_table(double x, double &k0e, double &E)
{
    const int hi = __double2hiint(x);
    const double *c = &BT_64[(hi >> 18) - 4 * (1023 + BT_LO)][0][0];
    const double t = __hiloint2double((hi & 0x000FFFFF) | 0x3FF00000, __double2loint(x)) -
                     __hiloint2double((hi & 0x000C0000) | 0x3FF20000, 0);
    double a = __ldg(c + 12), b = __ldg(c + 25);
#pragma unroll
    for (int k = 11; k >= 0; --k) {
        a = fma(a, t, __ldg(c + k));
        b = fma(b, t, __ldg(c + 13 + k));
    }
    k0e = a;
    E = b;
}
// The tails in z = 1/x <= 1/16: K0e = sqrt(pi z / 2) S0, E = sqrt(pi z / 2) Q / 2.
constexpr double BESSEL_ZTAIL = 0.0625;
__device__ __forceinline__ void bessel_tail(float z, float &S0, float &Q)
{
    S0 = BT_S0_32[4];
    Q = BT_Q_32[4];
#pragma unroll
    for (int k = 3; k >= 0; --k) {
        S0 = fmaf(S0, z, BT_S0_32[k]);
        Q = fmaf(Q, z, BT_Q_32[k]);
    }
}
__device__ __forceinline__ void bessel_tail(double z, double &S0, double &Q)
{
    S0 = BT_S0_64[9];
    Q = fma(BT_Q_64[10], z, BT_Q_64[9]);
#pragma unroll
    for (int k = 8; k >= 0; --k) {
        S0 = fma(S0, z, BT_S0_64[k]);
        Q = fma(Q, z, BT_Q_64[k]);
    }
}

// (K0e, D) at any x: table, tail or series (FP64).
__device__ __forceinline__ void k0e_D_short(double x, double &k0e, double &D)
{
    if (x >= 16.0) {
        double S0, Q;
        const double y = rsqrt(x), z = y * y, s = 1.2533141373155002512 * y;     // sqrt(pi / 2)
        bessel_tail(z, S0, Q);
        k0e = s * S0;
        D = 0.5 * s * z * Q;
    } else if (bessel_in_table(x)) {
        double E;
        bessel_table(x, k0e, E);
        D = E / x;
    } else {
        k0e_D_series(x, k0e, D);                   // x < 2^-20, or not a number
    }
}

// Pairs of one (target, source) row pair as a function of sg = sinh^2(Delta/2) +
// sin^2(psi/2) = s^2 / (4 r r'), with eta = H^2 / (r r'), X = sg / (2 eta):
//     P = A e^X K0(X) / (2 sqrt(pi) eta^1/2),   F = A D(X) / (8 sqrt(pi) eta^3/2).
struct RowPair { double ix, teta, cP, cF, tP, tF; };
__device__ __forceinline__ RowPair row_pair(double eta, double A)
{
    const double y = rsqrt(eta), c = A * 0.56418958354775628695 * y;       // 1 / sqrt(pi)
    return {0.5 / eta, 2.0 * eta, 0.5 * c, 0.25 * c, 0.5 * A, 0.125 * A};
}
// i1 = 1 / sqrt(sg)
__device__ __forceinline__ void row_pair_eval(const RowPair &c, double sg, double i1, double &P, double &F)
{
    const double X = sg * c.ix, isg = i1 * i1;
    if (X >= 16.0) {
        double S0, Q;
        bessel_tail(c.teta * isg, S0, Q);
        P = c.tP * i1 * S0;
        F = c.tF * i1 * isg * Q;
    } else if (bessel_in_table(X)) {
        double k0e, E;
        bessel_table(X, k0e, E);
        P = c.cP * k0e;
        F = c.cF * isg * E;
    } else {                                       // X < 2^-20, or not a number
        double k0e, D;
        k0e_D_series(X, k0e, D);
        P = c.cP * k0e;
        F = c.cF * isg * (D * X);
    }
}

}  // namespace sg
