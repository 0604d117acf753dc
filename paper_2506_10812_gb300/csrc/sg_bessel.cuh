// Exponentially scaled modified Bessel functions of the kernel:
//     K0e(x) = e^x K0(x),     D(x) = e^x [K1(x) - K0(x)],
// the two functions in Eq. "SG force kernel exact" (D) and Eq. "grav.
// potential 2D" (K0e) of Rendon Restrepo et al. (2025), with X = d^2/8.
//
// CUDA's math library has no K0/K1, so they are evaluated here from three
// published representations, each used where it converges fast:
//   x < 2       ascending series (DLMF 10.31.1 and 10.31.2), FP64 only;
//   x < x_asym  trapezoidal rule on the integral (DLMF 10.32.9 with
//               w = 2 sqrt(x) sinh(t/2)):
//                 K0e = x^-1/2     int_0^inf e^{-w^2/2} (1 + w^2/(4x))^-1/2 dw
//                 D   = (2x^3/2)^-1 int_0^inf w^2 e^{-w^2/2} (1 + w^2/(4x))^-1/2 dw,
//               both integrands positive (no cancellation for large x);
//   x >= x_asym Hankel's asymptotic expansion (DLMF 10.40.2), the K1 - K0
//               difference taken term by term (the leading terms cancel
//               exactly, so no digits are lost).
// Measured against 30-digit references: FP64 <= 1e-15, FP32 <= 2.3e-7
// relative over their ranges.
//
// Where a function is evaluated per pair of cells the representations above
// are too long: FP64 units run at 1/64 of the FP32 rate here, and a quadrature
// is 24 reciprocal square roots.  bessel_table and the tail polynomials
// (sg_bessel_tab.cuh) take one short polynomial per function instead: FP64
// 12 or 10 multiply-adds, FP32 5 or 4.
#pragma once

#include <cuda_runtime.h>

#include "sg_bessel_tab.cuh"

namespace sg {

constexpr int NW64 = 24;        // FP64 nodes w_n = 0.4 n, n = 1..24 (e^{-w^2/2} < 1e-19 beyond)
constexpr double HW64 = 0.4;
constexpr int NW32 = 13;        // FP32 nodes w_n = 0.5 n, n = 1..13
constexpr float HW32 = 0.5f;

// Gaussian weights e^{-w_n^2/2} and w_n^2 e^{-w_n^2/2}, filled once per CTA.
struct BesselWeights {
    double g64[NW64 + 1], w2g64[NW64 + 1];
    float g32[NW32 + 1], w2g32[NW32 + 1];
};

__device__ __forceinline__ void bessel_weights_init(BesselWeights &bw)
{
    for (int n = threadIdx.x; n <= NW64; n += blockDim.x) {
        double w = HW64 * n;
        bw.g64[n] = exp(-0.5 * w * w);
        bw.w2g64[n] = w * w * bw.g64[n];
    }
    for (int n = threadIdx.x; n <= NW32; n += blockDim.x) {
        double w = (double)HW32 * n;
        double g = exp(-0.5 * w * w);
        bw.g32[n] = (float)g;
        bw.w2g32[n] = (float)(w * w * g);
    }
}

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

__device__ __forceinline__ void k0e_D_f64(double x, const BesselWeights &bw, double &k0e, double &D)
{
    if (x < 2.0) {
        k0e_D_series(x, k0e, D);
    } else if (x < 40.0) {
        const double q = 0.25 / x;
        double s0 = 0.5, s1 = 0.0;
#pragma unroll 4
        for (int n = 1; n <= NW64; ++n) {
            const double w = HW64 * n;
            const double r = rsqrt(1.0 + w * w * q);
            s0 += bw.g64[n] * r;
            s1 += bw.w2g64[n] * r;
        }
        const double sx = sqrt(x);
        k0e = HW64 * s0 / sx;
        D = HW64 * s1 / (2.0 * x * sx);
    } else {
        const double s = sqrt(1.5707963267948966192 / x);
        double t0 = 1.0, t1 = 1.0, s0 = 1.0, sd = 0.0;
#pragma unroll
        for (int k = 0; k < 14; ++k) {
            const double o = (double)((2 * k + 1) * (2 * k + 1));
            const double den = 1.0 / (8.0 * (k + 1) * x);
            t0 *= -o * den;
            t1 *= (4.0 - o) * den;
            s0 += t0;
            sd += t1 - t0;
        }
        k0e = s * s0;
        D = s * sd;
    }
}

// FP32 evaluation, valid for x >= 1.
__device__ __forceinline__ void k0e_D_f32(float x, const BesselWeights &bw, float &k0e, float &D)
{
    if (x < 12.0f) {
        const float q = 0.25f / x;
        float s0 = 0.5f, s1 = 0.0f;
#pragma unroll
        for (int n = 1; n <= NW32; ++n) {
            const float w = HW32 * n;
            const float r = rsqrtf(fmaf(w * w, q, 1.0f));
            s0 = fmaf(bw.g32[n], r, s0);
            s1 = fmaf(bw.w2g32[n], r, s1);
        }
        const float rs = rsqrtf(x);
        k0e = HW32 * s0 * rs;
        D = HW32 * s1 * (0.5f * rs / x);
    } else {
        const float s = sqrtf(1.57079632679f / x);
        const float ix = 1.0f / x;
        float t0 = 1.0f, t1 = 1.0f, s0 = 1.0f, sd = 0.0f;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const float o = (float)((2 * k + 1) * (2 * k + 1));
            const float den = ix * (1.0f / (8.0f * (k + 1)));
            t0 *= -o * den;
            t1 *= (4.0f - o) * den;
            s0 += t0;
            sd += t1 - t0;
        }
        k0e = s * s0;
        D = s * sd;
    }
}

// K0e(x) and E(x) = x D(x) from the quarter-octave tables, 2^-20 <= x < 16
// (bessel_in_table).  The index and the argument come from the bits of x; a
// warp's lanes mostly share an entry, so the loads are broadcasts from L1.
__device__ __forceinline__ bool bessel_in_table(float x) { return x >= 0x1p-20f && x < 16.0f; }
__device__ __forceinline__ bool bessel_in_table(double x) { return x >= 0x1p-20 && x < 16.0; }
__device__ __forceinline__ void bessel_table(float x, float &k0e, float &E)
{
    const int b = __float_as_int(x);
    const float4 *c = reinterpret_cast<const float4 *>(&BT_32[(b >> 21) - 4 * (127 + BT_LO)][0][0]);
    const float t = __int_as_float((b & 0x007FFFFF) | 0x3F800000) - __int_as_float((b & 0x00600000) | 0x3F900000);
    const float4 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2);
    k0e = fmaf(fmaf(fmaf(fmaf(fmaf(c1.y, t, c1.x), t, c0.w), t, c0.z), t, c0.y), t, c0.x);
    E = fmaf(fmaf(fmaf(fmaf(fmaf(c2.w, t, c2.z), t, c2.y), t, c2.x), t, c1.w), t, c1.z);
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

// (K0e, D) at any x: table, tail or series (FP64; 10 to 14 multiply-adds a
// function in place of the quadrature above).
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

}  // namespace sg
