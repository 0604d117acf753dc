// Register-resident Stockham FFT for one CTA (float or double).
//
// A length-L transform (L = 16 T, L a power of two >= 16) is held by T
// threads, 16 elements each, in the "strided" layout: thread t holds
// x[t + T e] in register v[e].  Each Stockham pass of radix R reads exactly
// those registers (butterfly j = t + T q combines x[j + r L/R]), so a pass
// is: twiddle, radix-R DFT in registers, and (except after the last pass)
// one scatter/gather through a padded shared-memory buffer.  Passes are
// radix 16 with a final radix 2, 4 or 8; output is in natural order in the
// same strided layout, so a forward transform, a pointwise product and an
// inverse transform need no reordering at all.
//
// Twiddles come from a per-pass table (computed in FP64 on the host): the
// pass with stride Ns and radix R reads W_{Ns R}^{r k} = exp(-2 pi i r k / (Ns R))
// at (r - 1) Ns + k, so the threads of a warp (consecutive k) read
// consecutive entries; the passes' segments follow one another (Ns = 16,
// 256, ... for the radix-16 passes, then the final pass).  FP64 transforms take
// another set of roots per pass (fft_f64).
#pragma once

#include <cuda_runtime.h>

namespace sg {

template <typename R> struct cplx_of;
template <> struct cplx_of<float> { using type = float2; };
template <> struct cplx_of<double> { using type = double2; };
template <typename R> using cplx = typename cplx_of<R>::type;

template <typename T> __device__ __forceinline__ T mkc(decltype(T::x) a, decltype(T::x) b) { T c; c.x = a; c.y = b; return c; }
template <typename T> __device__ __forceinline__ T cadd(T a, T b) { return mkc<T>(a.x + b.x, a.y + b.y); }
template <typename T> __device__ __forceinline__ T csub(T a, T b) { return mkc<T>(a.x - b.x, a.y - b.y); }
template <typename T> __device__ __forceinline__ T cneg(T a) { return mkc<T>(-a.x, -a.y); }
template <typename T> __device__ __forceinline__ T cconj(T a) { return mkc<T>(a.x, -a.y); }
template <typename T> __device__ __forceinline__ T cmul_i(T a) { return mkc<T>(-a.y, a.x); }   // i a
template <typename T> __device__ __forceinline__ T cmul_mi(T a) { return mkc<T>(a.y, -a.x); }  // -i a
template <typename T> __device__ __forceinline__ T cscale(T a, decltype(T::x) s) { return mkc<T>(a.x * s, a.y * s); }
// a * b
template <typename T> __device__ __forceinline__ T cmul(T a, T b)
{
    return mkc<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
template <typename T> __device__ __forceinline__ T cmulc(T a, T b)
{
    return mkc<T>(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// acc + a * b
template <typename T> __device__ __forceinline__ T cfma(T a, T b, T acc)
{
    acc.x += a.x * b.x - a.y * b.y;
    acc.y += a.x * b.y + a.y * b.x;
    return acc;
}
// acc + a * b and acc + a * conj(b) as four multiply-adds (FP64, where every
// instruction counts; the compiler may not reassociate the form above into it.
// FP32 columns of length 4096 measured 0.6 % slower with it.)
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 acc)
{
    return mkc<double2>(fma(a.x, b.x, fma(-a.y, b.y, acc.x)), fma(a.x, b.y, fma(a.y, b.x, acc.y)));
}
__device__ __forceinline__ double2 cfmac(double2 a, double2 b, double2 acc)
{
    return mkc<double2>(fma(a.x, b.x, fma(a.y, b.y, acc.x)), fma(a.y, b.x, fma(-a.x, b.y, acc.y)));
}
template <bool FWD, typename T> __device__ __forceinline__ T twmul(T a, T w)
{
    return FWD ? cmul(a, w) : cmulc(a, w);
}

// cos(pi/8), sin(pi/8), cos(pi/4)
#define SG_C16 0.92387953251128675613
#define SG_S16 0.38268343236508977173
#define SG_C8 0.70710678118654752440

// a * exp(-+ 2 pi i P / 16)  (minus sign for the forward transform)
template <bool FWD, int P, typename T> __device__ __forceinline__ T w16(T a)
{
    using R = decltype(T::x);
    constexpr int p = P & 15;
    if constexpr (p == 0) {
        return a;
    } else if constexpr (p == 4) {
        return FWD ? cmul_mi(a) : cmul_i(a);
    } else if constexpr (p == 8) {
        return cneg(a);
    } else if constexpr (p == 12) {
        return FWD ? cmul_i(a) : cmul_mi(a);
    } else {
        constexpr double cs[16] = {1.0, SG_C16, SG_C8, SG_S16, 0.0, -SG_S16, -SG_C8, -SG_C16,
                                   -1.0, -SG_C16, -SG_C8, -SG_S16, 0.0, SG_S16, SG_C8, SG_C16};
        constexpr double sn[16] = {0.0, SG_S16, SG_C8, SG_C16, 1.0, SG_C16, SG_C8, SG_S16,
                                   0.0, -SG_S16, -SG_C8, -SG_C16, -1.0, -SG_C16, -SG_C8, -SG_S16};
        const R c = (R)cs[p];
        const R s = FWD ? (R)sn[p] : (R)(-sn[p]);
        // (a.x + i a.y)(c - i s)
        return mkc<T>(a.x * c + a.y * s, a.y * c - a.x * s);
    }
}

// ---- packed FP32 pairs (Blackwell add/sub/fma.f32x2): one instruction per
// complex add or subtract.  Results are bit-identical to the scalar forms
// (each lane is one correctly rounded operation; x * (+-1) is exact).
__device__ __forceinline__ float2 padd(float2 a, float2 b)
{
    float2 d;
    asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
        " add.rn.f32x2 rd, ra, rb;\n mov.b64 {%0, %1}, rd;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 psub(float2 a, float2 b)
{
    float2 d;
    asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
        " sub.rn.f32x2 rd, ra, rb;\n mov.b64 {%0, %1}, rd;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
// c + a * (sx, sy) with sx, sy = +-1
template <int SX, int SY>
__device__ __forceinline__ float2 pfma_sign(float2 a, float2 c)
{
    float2 d;
    asm("{\n .reg .b64 ra, rs, rc, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rs, {%6, %7};\n"
        " mov.b64 rc, {%4, %5};\n fma.rn.f32x2 rd, ra, rs, rc;\n mov.b64 {%0, %1}, rd;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(c.x), "f"(c.y), "f"((float)SX), "f"((float)SY));
    return d;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return padd(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return psub(a, b); }

template <bool FWD, typename T> __device__ __forceinline__ void dft2(T &a0, T &a1)
{
    T t = a0;
    a0 = cadd(t, a1);
    a1 = csub(t, a1);
}

// Packed radix 4: u = swap(a1 - a3) in scalar form, the +-i rotations as
// sign-vector FMAs (9 instructions instead of 16).
template <bool FWD> __device__ __forceinline__ void dft4(float2 &a0, float2 &a1, float2 &a2, float2 &a3)
{
    const float2 t0 = padd(a0, a2), t1 = psub(a0, a2), t2 = padd(a1, a3);
    const float2 u = make_float2(a1.y - a3.y, a1.x - a3.x);
    a0 = padd(t0, t2);
    a2 = psub(t0, t2);
    if (FWD) {   // t1 - i t3 = t1 + (u.x, -u.y),  t1 + i t3 = t1 + (-u.x, u.y)
        a1 = pfma_sign<1, -1>(u, t1);
        a3 = pfma_sign<-1, 1>(u, t1);
    } else {
        a1 = pfma_sign<-1, 1>(u, t1);
        a3 = pfma_sign<1, -1>(u, t1);
    }
}

template <bool FWD, typename T> __device__ __forceinline__ void dft4(T &a0, T &a1, T &a2, T &a3)
{
    T t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = csub(a1, a3);
    a0 = cadd(t0, t2);
    a2 = csub(t0, t2);
    if (FWD) {
        a1 = cadd(t1, cmul_mi(t3));
        a3 = cadd(t1, cmul_i(t3));
    } else {
        a1 = cadd(t1, cmul_i(t3));
        a3 = cadd(t1, cmul_mi(t3));
    }
}

// In-place 8-point DFT on a[OFF + S*n], n = 0..7 (natural order in and out).
template <bool FWD, int OFF, int S, typename T> __device__ __forceinline__ void dft8(T (&a)[16])
{
    // n = 2 n1 + n2, k = k1 + 4 k2: DFT4 over n1, twiddle W8^{n2 k1}, DFT2 over n2
    T b[8];
#pragma unroll
    for (int n = 0; n < 8; ++n) b[n] = a[OFF + S * n];
    dft4<FWD>(b[0], b[2], b[4], b[6]);
    dft4<FWD>(b[1], b[3], b[5], b[7]);
    // b[2 k1 + n2] now holds B[n2][k1]
    b[3] = w16<FWD, 2>(b[3]);
    b[5] = w16<FWD, 4>(b[5]);
    b[7] = w16<FWD, 6>(b[7]);
    dft2<FWD>(b[0], b[1]);
    dft2<FWD>(b[2], b[3]);
    dft2<FWD>(b[4], b[5]);
    dft2<FWD>(b[6], b[7]);
    // X[k1 + 4 k2] = b[2 k1 + k2]
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        a[OFF + S * k1] = b[2 * k1];
        a[OFF + S * (k1 + 4)] = b[2 * k1 + 1];
    }
}

// Second half of the 16-point DFT below (after its first radix-4 stage).
template <bool FWD, typename T> __device__ __forceinline__ void dft16_tail(T (&a)[16])
{
    // a[4 k1 + n2] = B[n2][k1]
    a[5] = w16<FWD, 1>(a[5]);
    a[6] = w16<FWD, 2>(a[6]);
    a[7] = w16<FWD, 3>(a[7]);
    a[9] = w16<FWD, 2>(a[9]);
    a[10] = w16<FWD, 4>(a[10]);
    a[11] = w16<FWD, 6>(a[11]);
    a[13] = w16<FWD, 3>(a[13]);
    a[14] = w16<FWD, 6>(a[14]);
    a[15] = w16<FWD, 9>(a[15]);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) dft4<FWD>(a[4 * k1], a[4 * k1 + 1], a[4 * k1 + 2], a[4 * k1 + 3]);
    // X[k1 + 4 k2] = a[4 k1 + k2]: transpose the 4x4 index
    T b[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) b[i] = a[i];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) a[k1 + 4 * k2] = b[4 * k1 + k2];
}

// In-place 16-point DFT on a[0..15] (natural order in and out).
template <bool FWD, typename T> __device__ __forceinline__ void dft16(T (&a)[16])
{
    // n = 4 n1 + n2, k = k1 + 4 k2: DFT4 over n1, twiddle W16^{n2 k1}, DFT4 over n2
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft4<FWD>(a[n2], a[4 + n2], a[8 + n2], a[12 + n2]);
    dft16_tail<FWD>(a);
}

// The same DFT when a[8..15] are zero (the radially zero-padded half of a
// forward column transform): each first-stage radix 4 has two inputs,
// X = x0 + x1, x0 -+ i x1, x0 - x1, x0 +- i x1 (4 packed instructions
// instead of 9).  Zero operands cannot be folded by the compiler (x + 0 is not
// x for x = -0), so the pruning is explicit.
template <bool FWD> __device__ __forceinline__ void dft16_half(float2 (&a)[16])
{
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
        const float2 x0 = a[n2], x1 = a[4 + n2];
        const float2 u = make_float2(x1.y, x1.x);
        a[n2] = padd(x0, x1);
        a[8 + n2] = psub(x0, x1);
        if (FWD) {   // x0 - i x1 = x0 + (u.x, -u.y),  x0 + i x1 = x0 + (-u.x, u.y)
            a[4 + n2] = pfma_sign<1, -1>(u, x0);
            a[12 + n2] = pfma_sign<-1, 1>(u, x0);
        } else {
            a[4 + n2] = pfma_sign<-1, 1>(u, x0);
            a[12 + n2] = pfma_sign<1, -1>(u, x0);
        }
    }
    dft16_tail<FWD>(a);
}
template <bool FWD, typename T> __device__ __forceinline__ void dft16_half(T (&a)[16])
{
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
        const T x0 = a[n2], x1 = a[4 + n2];
        a[n2] = cadd(x0, x1);
        a[8 + n2] = csub(x0, x1);
        a[4 + n2] = cadd(x0, FWD ? cmul_mi(x1) : cmul_i(x1));
        a[12 + n2] = cadd(x0, FWD ? cmul_i(x1) : cmul_mi(x1));
    }
    dft16_tail<FWD>(a);
}

// Padded shared-memory index: one extra slot every 16 elements makes the
// Stockham scatter (stride 16) and the strided gather conflict-free.
__device__ __forceinline__ int pidx(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int padded_len(int L) { return L + (L >> 4) + 1; }

// Scatter after a radix-16 pass with stride Ns, gather back the strided layout.
template <typename T>
__device__ __forceinline__ void exchange16(T (&v)[16], int t, int T_, int Ns, T *xb)
{
    const int k = t & (Ns - 1);
    const int base = (t - k) * 16 + k;     // (t / Ns) Ns 16 + k
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 16; ++r) xb[pidx(base + r * Ns)] = v[r];
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = xb[pidx(t + T_ * e)];
}

// Final Stockham pass of radix RL in {2, 4, 8} (Q = 16 / RL butterflies per
// thread; butterfly q combines registers q + r Q).  Lands in-register.
template <bool FWD, int RL, typename T>
__device__ __forceinline__ void final_pass(T (&v)[16], int t, int T_, int Ns, const T *__restrict__ tp)
{
    constexpr int Q = 16 / RL;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int k = (t + T_ * q) & (Ns - 1);
#pragma unroll
        for (int r = 1; r < RL; ++r) v[q + r * Q] = twmul<FWD>(v[q + r * Q], __ldg(&tp[(r - 1) * Ns + k]));
    }
    if constexpr (RL == 2) {
#pragma unroll
        for (int q = 0; q < Q; ++q) dft2<FWD>(v[q], v[q + Q]);
    } else if constexpr (RL == 4) {
#pragma unroll
        for (int q = 0; q < Q; ++q) dft4<FWD>(v[q], v[q + Q], v[q + 2 * Q], v[q + 3 * Q]);
    } else {
        dft8<FWD, 0, 2>(v);
        dft8<FWD, 1, 2>(v);
    }
}

// ---------------------------------------------------------------- FP64
// FP64 instructions bound these transforms (two lanes per clock and SM), so
// they are written for the fewest: every radix-2 butterfly takes its root with
// it.  A root is held as (c, t), w = c (1 + i t) (cosine and tangent, after Linzer and
// Feig's multiply-add transforms): (u, v) = b (1 + i t) takes two multiply-adds, a + c (u, v) and
// a - c (u, v) two each, six instructions and two roundings per value where a
// complex product and two sums are eight and three.  A right angle has no
// tangent: only the first level of a pass meets it (w^(R/2) at k = Ns/2), where
// b is rotated by register moves and the table holds the root 1 (bfly_first).
// (The tangent of the rounded right angle, 1.6e16, overflowed for inputs above 1e291.)
// All other tangents are below L / (2 pi), so that no input below 1e300 / L is
// lost.  A radix-16 pass is four such levels, the input twiddles w^r folded into them:
// level by level the roots are w^8; w^4 (and -i w^4); w^2 W8^k; w W16^k (k = 0,
// 1, and so on; the upper half of each level is -i times the lower), so that a
// pass reads 8 roots from its table, not 15, and is 192 instructions instead
// of 228; the first pass, with constants, 148 instead of 168.
// Table (pass_twiddles<double>): per pass of stride Ns, w = exp(-2 pi i k / (Ns R)),
// rows of Ns roots: radix 16: w^8, w^4, w^2, w^2 W8, w, w W16, w W8, w W16^3;
// radix 8: w^4, w^2, w, w W8; radix 4: w^2, w; radix 2: w; 1 where w^(R/2) is -i.
// (a, b) <- (a + w b, a - w b), w conjugated for the inverse transform
template <bool FWD> __device__ __forceinline__ void bfly(double2 &a, double2 &b, double2 w)
{
    const double t = FWD ? w.y : -w.y;
    const double u = fma(-t, b.y, b.x), v = fma(t, b.x, b.y);
    b = make_double2(fma(-w.x, u, a.x), fma(-w.x, v, a.y));
    a = make_double2(fma(w.x, u, a.x), fma(w.x, v, a.y));
}
// the first level of a pass: where `quarter`, the root is -i (the table's 1 times
// it).  Integer selects, not FP64 instructions: the pipe that bounds the transform
// is left alone.
template <bool FWD> __device__ __forceinline__ void bfly_first(double2 &a, double2 &b, double2 w, bool quarter)
{
    const double2 x = b;
    const int flip = quarter ? (int)0x80000000u : 0;
    b.x = quarter ? x.y : x.x;
    b.y = quarter ? x.x : x.y;
    double &n = FWD ? b.y : b.x;                      // -i (x, y) = (y, -x), i (x, y) = (-y, x)
    n = __hiloint2double(__double2hiint(n) ^ flip, __double2loint(n));
    bfly<FWD>(a, b, w);
}
// the same with the root -i w
template <bool FWD> __device__ __forceinline__ void bfly_mi(double2 &a, double2 &b, double2 w)
{
    b = FWD ? cmul_mi(b) : cmul_i(b);
    bfly<FWD>(a, b, w);
}
__device__ __forceinline__ void bfly_1(double2 &a, double2 &b)
{
    const double2 t = a;
    a = cadd(t, b);
    b = csub(t, b);
}
template <bool FWD> __device__ __forceinline__ void bfly_1mi(double2 &a, double2 &b)   // root -i
{
    const double2 t = a, u = FWD ? cmul_mi(b) : cmul_i(b);
    a = cadd(t, u);
    b = csub(t, u);
}
// bit-reversed registers to natural order (renaming only)
__device__ __forceinline__ void unreverse16(double2 (&v)[16])
{
    double2 b[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) b[i] = v[i];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[((i & 1) << 3) | ((i & 2) << 1) | ((i & 4) >> 1) | (i >> 3)] = b[i];
}
// first pass (all w = 1); HALF: v[8..15] are zero
template <bool FWD, bool HALF> __device__ __forceinline__ void dft16_f64(double2 (&v)[16])
{
    const double2 W8 = make_double2(SG_C8, -1.0), W16 = make_double2(SG_C16, -0.41421356237309504880),
                  W163 = make_double2(SG_S16, -2.41421356237309504880);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        if constexpr (HALF) v[r + 8] = v[r];
        else bfly_1(v[r], v[r + 8]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        bfly_1(v[r], v[r + 4]);
        bfly_1mi<FWD>(v[r + 8], v[r + 12]);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        bfly_1(v[r], v[r + 2]);
        bfly_1mi<FWD>(v[r + 4], v[r + 6]);
        bfly<FWD>(v[r + 8], v[r + 10], W8);
        bfly_mi<FWD>(v[r + 12], v[r + 14], W8);
    }
    bfly_1(v[0], v[1]);
    bfly_1mi<FWD>(v[2], v[3]);
    bfly<FWD>(v[4], v[5], W8);
    bfly_mi<FWD>(v[6], v[7], W8);
    bfly<FWD>(v[8], v[9], W16);
    bfly_mi<FWD>(v[10], v[11], W16);
    bfly<FWD>(v[12], v[13], W163);
    bfly_mi<FWD>(v[14], v[15], W163);
    unreverse16(v);
}
// a later radix-16 pass at this thread's k; tp0: its table
template <bool FWD>
__device__ __forceinline__ void pass16_f64(double2 (&v)[16], const double2 *__restrict__ tp0, int k, int Ns)
{
    const double2 *tp = tp0 + k;
    const bool quarter = 2 * k == Ns;
    const double2 w8 = __ldg(tp), w4 = __ldg(tp + Ns), w2 = __ldg(tp + 2 * Ns), w2a = __ldg(tp + 3 * Ns);
#pragma unroll
    for (int r = 0; r < 8; ++r) bfly_first<FWD>(v[r], v[r + 8], w8, quarter);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        bfly<FWD>(v[r], v[r + 4], w4);
        bfly_mi<FWD>(v[r + 8], v[r + 12], w4);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        bfly<FWD>(v[r], v[r + 2], w2);
        bfly_mi<FWD>(v[r + 4], v[r + 6], w2);
        bfly<FWD>(v[r + 8], v[r + 10], w2a);
        bfly_mi<FWD>(v[r + 12], v[r + 14], w2a);
    }
    const double2 w = __ldg(tp + 4 * Ns), wa = __ldg(tp + 5 * Ns), wb = __ldg(tp + 6 * Ns), wc = __ldg(tp + 7 * Ns);
    bfly<FWD>(v[0], v[1], w);
    bfly_mi<FWD>(v[2], v[3], w);
    bfly<FWD>(v[4], v[5], wb);
    bfly_mi<FWD>(v[6], v[7], wb);
    bfly<FWD>(v[8], v[9], wa);
    bfly_mi<FWD>(v[10], v[11], wa);
    bfly<FWD>(v[12], v[13], wc);
    bfly_mi<FWD>(v[14], v[15], wc);
    unreverse16(v);
}
// final pass of radix RL: butterfly q combines registers q + r Q
template <bool FWD, int RL>
__device__ __forceinline__ void final_f64(double2 (&v)[16], int t, int T_, int Ns, const double2 *__restrict__ tp0)
{
    constexpr int Q = 16 / RL;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int k = (t + T_ * q) & (Ns - 1);
        const double2 *tp = tp0 + k;
        const bool quarter = 2 * k == Ns;
        double2 *x = v + q;                           // element r at x[r Q]
        if constexpr (RL == 2) {
            bfly_first<FWD>(x[0], x[Q], __ldg(tp), quarter);
        } else if constexpr (RL == 4) {
            const double2 w2 = __ldg(tp), w = __ldg(tp + Ns);
            bfly_first<FWD>(x[0], x[2 * Q], w2, quarter);
            bfly_first<FWD>(x[Q], x[3 * Q], w2, quarter);
            bfly<FWD>(x[0], x[Q], w);
            bfly_mi<FWD>(x[2 * Q], x[3 * Q], w);
            const double2 y = x[Q];                   // order 0, 2, 1, 3
            x[Q] = x[2 * Q];
            x[2 * Q] = y;
        } else {
            const double2 w4 = __ldg(tp), w2 = __ldg(tp + Ns), w = __ldg(tp + 2 * Ns), wa = __ldg(tp + 3 * Ns);
#pragma unroll
            for (int r = 0; r < 4; ++r) bfly_first<FWD>(x[r * Q], x[(r + 4) * Q], w4, quarter);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                bfly<FWD>(x[r * Q], x[(r + 2) * Q], w2);
                bfly_mi<FWD>(x[(r + 4) * Q], x[(r + 6) * Q], w2);
            }
            bfly<FWD>(x[0], x[Q], w);
            bfly_mi<FWD>(x[2 * Q], x[3 * Q], w);
            bfly<FWD>(x[4 * Q], x[5 * Q], wa);
            bfly_mi<FWD>(x[6 * Q], x[7 * Q], wa);
            double2 y = x[Q];                         // order 0, 4, 2, 6, 1, 5, 3, 7
            x[Q] = x[4 * Q];
            x[4 * Q] = y;
            y = x[3 * Q];
            x[3 * Q] = x[6 * Q];
            x[6 * Q] = y;
        }
    }
}
// Full length-L FP64 transform, layout and contract of fft_reg below.
template <bool FWD, bool HALF = false>
__device__ __forceinline__ void fft_f64(double2 (&v)[16], int L, int T_, int t, double2 *xb,
                                        const double2 *__restrict__ twp)
{
    dft16_f64<FWD, HALF>(v);
    if (L == 16) return;
    int Ns = 16;
    const double2 *tp = twp;
    exchange16(v, t, T_, 1, xb);
    while (Ns * 16 <= L) {
        pass16_f64<FWD>(v, tp, t & (Ns - 1), Ns);
        tp += 8 * Ns;
        if (Ns * 16 == L) return;
        exchange16(v, t, T_, Ns, xb);
        Ns *= 16;
    }
    const int RL = L / Ns;
    if (RL == 8) final_f64<FWD, 8>(v, t, T_, Ns, tp);
    else if (RL == 4) final_f64<FWD, 4>(v, t, T_, Ns, tp);
    else final_f64<FWD, 2>(v, t, T_, Ns, tp);
}

// Full length-L transform (L = 16 T_, power of two) of the strided register
// layout v[e] = x[t + T_ e]; result X[t + T_ e] in v[e].  Forward: X[k] =
// sum x[n] exp(-2 pi i n k / L); inverse: the same with +i (unnormalised).
// xb: this transform's shared buffer of padded_len(L) elements.  Every thread
// of the CTA must call this together (it contains __syncthreads).
// twp: the per-pass twiddle table of length L (see pass_twiddle_count).
template <bool FWD, typename T>
__device__ __forceinline__ void fft_reg(T (&v)[16], int L, int T_, int t, T *xb, const T *__restrict__ twp)
{
    if constexpr (sizeof(T) == 16) {
        fft_f64<FWD>(v, L, T_, t, xb, twp);
        return;
    }
    dft16<FWD>(v);                              // pass Ns = 1: no twiddles
    if (L == 16) return;
    int Ns = 16;
    const T *tp = twp;
    exchange16(v, t, T_, 1, xb);
    while (Ns * 16 <= L) {
        const int k = t & (Ns - 1);
#pragma unroll
        for (int r = 1; r < 16; ++r) v[r] = twmul<FWD>(v[r], __ldg(&tp[(r - 1) * Ns + k]));
        dft16<FWD>(v);
        tp += 15 * Ns;
        if (Ns * 16 == L) return;
        exchange16(v, t, T_, Ns, xb);
        Ns *= 16;
    }
    const int RL = L / Ns;
    if (RL == 8) final_pass<FWD, 8>(v, t, T_, Ns, tp);
    else if (RL == 4) final_pass<FWD, 4>(v, t, T_, Ns, tp);
    else final_pass<FWD, 2>(v, t, T_, Ns, tp);
}

// ---------------------------------------------------------------------
// Compile-time-length variant (L >= 256): same passes and layout as
// fft_reg, but every stride is a constant, so the shared-memory and twiddle
// addresses are a per-thread base plus immediate offsets, and outputs the
// caller never reads are removed by the compiler.
//   pidx(16 t + r)           = 17 t + r                            (Ns = 1)
//   pidx(base + r Ns)        = base + (base >> 4) + r (Ns + Ns/16)   (Ns % 16 == 0)
//   pidx(t + T e)            = t + (t >> 4) + e (T + T/16)         (T % 16 == 0)
template <int Ns, int TT, typename T>
__device__ __forceinline__ void exchange_ct(T (&v)[16], int t, T *xb)
{
    T *w;
    constexpr int step = Ns == 1 ? 1 : Ns + Ns / 16;
    if constexpr (Ns == 1) {
        w = xb + 17 * t;
    } else {
        const int k = t & (Ns - 1);
        const int base = (t - k) * 16 + k;
        w = xb + base + (base >> 4);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 16; ++r) w[r * step] = v[r];
    __syncthreads();
    const T *rd = xb + t + (t >> 4);
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = rd[e * (TT + TT / 16)];
}

// Base twiddles of the compile-time pass with stride Ns, loaded before the
// exchange that precedes the pass so that their latency overlaps its
// barriers and shared-memory traffic:
//   radix-16 pass: W^{r k} (k = t mod Ns) for r = 1, 2, 3, 4, 8, 12; the
//   other nine are products of two loaded values (one extra rounding), which
//   spares the L1 data path 9 loads;
//   final radix-RL pass: for each of its Q = 16 / RL butterflies, r = 1..4
//   when RL = 8 (r = 5..7 as products of w4 and w1..w3), else r = 1..RL-1.
// FULL: every root is loaded and none is a product, the roundings of fft_reg.
constexpr int pass_tw_len(bool full) { return full ? 15 : 12; }
template <int L, int Ns, bool FULL, typename T>
__device__ __forceinline__ void load_pass_tw(const T *__restrict__ tp, int t, T (&b)[pass_tw_len(FULL)])
{
    constexpr int TT = L / 16;
    if constexpr (Ns * 16 <= L && FULL) {
        const T *p = tp + (t & (Ns - 1));
#pragma unroll
        for (int r = 0; r < 15; ++r) b[r] = __ldg(p + r * Ns);
    } else if constexpr (Ns * 16 <= L) {
        const T *p = tp + (t & (Ns - 1));
        b[0] = __ldg(p);
        b[1] = __ldg(p + Ns);
        b[2] = __ldg(p + 2 * Ns);
        b[3] = __ldg(p + 3 * Ns);
        b[4] = __ldg(p + 7 * Ns);
        b[5] = __ldg(p + 11 * Ns);
    } else {
        constexpr int RL = L / Ns, Q = 16 / RL, NL = RL == 8 && !FULL ? 4 : RL - 1;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const T *p = tp + ((t + TT * q) & (Ns - 1));
#pragma unroll
            for (int r = 0; r < NL; ++r) b[q * NL + r] = __ldg(p + r * Ns);
        }
    }
}

// The radix-16 butterflies of the compile-time passes, in registers; a
// policy with the same call operator (the tensor-core DFT engine) can stand
// in for it.
template <bool FWD> struct RegDft16 {
    template <typename T> __device__ __forceinline__ void operator()(T (&v)[16]) const { dft16<FWD>(v); }
    // first pass of a transform whose inputs v[8..15] are zero
    template <typename T> __device__ __forceinline__ void half(T (&v)[16]) const { dft16_half<FWD>(v); }
};

template <bool FWD, int L, int Ns, bool FULL, typename T, typename D16 = RegDft16<FWD>>
__device__ __forceinline__ void fft_ct_pass(T (&v)[16], int t, T *xb, const T *__restrict__ tp,
                                            const T (&b)[pass_tw_len(FULL)], D16 &&d16 = D16{})
{
    constexpr int TT = L / 16;
    if constexpr (Ns * 16 <= L) {
        if constexpr (FULL) {
#pragma unroll
            for (int r = 1; r < 16; ++r) v[r] = twmul<FWD>(v[r], b[r - 1]);
        } else {
            T w[16];
            w[1] = b[0];
            w[2] = b[1];
            w[3] = b[2];
            w[4] = b[3];
            w[8] = b[4];
            w[12] = b[5];
            w[5] = cmul(w[4], w[1]);
            w[6] = cmul(w[4], w[2]);
            w[7] = cmul(w[4], w[3]);
            w[9] = cmul(w[8], w[1]);
            w[10] = cmul(w[8], w[2]);
            w[11] = cmul(w[8], w[3]);
            w[13] = cmul(w[12], w[1]);
            w[14] = cmul(w[12], w[2]);
            w[15] = cmul(w[12], w[3]);
#pragma unroll
            for (int r = 1; r < 16; ++r) v[r] = twmul<FWD>(v[r], w[r]);
        }
        d16(v);
        if constexpr (Ns * 16 < L) {
            T nb[pass_tw_len(FULL)];
            load_pass_tw<L, Ns * 16, FULL>(tp + 15 * Ns, t, nb);
            exchange_ct<Ns, TT>(v, t, xb);
            fft_ct_pass<FWD, L, Ns * 16, FULL>(v, t, xb, tp + 15 * Ns, nb, d16);
        }
    } else {
        constexpr int RL = L / Ns, Q = 16 / RL;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if constexpr (RL == 8 && !FULL) {
                T w[8];
#pragma unroll
                for (int r = 1; r <= 4; ++r) w[r] = b[q * 4 + r - 1];
                w[5] = cmul(w[4], w[1]);
                w[6] = cmul(w[4], w[2]);
                w[7] = cmul(w[4], w[3]);
#pragma unroll
                for (int r = 1; r < 8; ++r) v[q + r * Q] = twmul<FWD>(v[q + r * Q], w[r]);
            } else {
#pragma unroll
                for (int r = 1; r < RL; ++r) v[q + r * Q] = twmul<FWD>(v[q + r * Q], b[q * (RL - 1) + r - 1]);
            }
        }
        if constexpr (RL == 2) {
#pragma unroll
            for (int q = 0; q < Q; ++q) dft2<FWD>(v[q], v[q + Q]);
        } else if constexpr (RL == 4) {
#pragma unroll
            for (int q = 0; q < Q; ++q) dft4<FWD>(v[q], v[q + Q], v[q + 2 * Q], v[q + 3 * Q]);
        } else {
            dft8<FWD, 0, 2>(v);
            dft8<FWD, 1, 2>(v);
        }
    }
}

// HALF: the inputs v[8..15] (x[L/2 ..]) are zero and the first pass skips them.
template <bool FWD, int L, bool HALF = false, bool FULL = false, typename T, typename D16 = RegDft16<FWD>>
__device__ __forceinline__ void fft_ct(T (&v)[16], int t, T *xb, const T *__restrict__ twp, D16 &&d16 = D16{})
{
    static_assert(L >= 256 && (L & (L - 1)) == 0, "compile-time FFT needs a power of two >= 256");
    if constexpr (HALF) d16.half(v);
    else d16(v);
    T b[pass_tw_len(FULL)];
    load_pass_tw<L, 16, FULL>(twp, t, b);
    exchange_ct<1, L / 16>(v, t, xb);
    fft_ct_pass<FWD, L, 16, FULL>(v, t, xb, twp, b, d16);
}

// Compile-time length when LC > 0 (FP32), runtime length L otherwise (the
// butterfly policy d16 applies to the compile-time lengths, the zero-half
// pruning HALF to those and to FP64; FULL: no derived roots, see load_pass_tw).
template <bool FWD, int LC, bool HALF = false, bool FULL = false, typename T, typename D16 = RegDft16<FWD>>
__device__ __forceinline__ void fft_any(T (&v)[16], int L, int T_, int t, T *xb, const T *__restrict__ twp,
                                        D16 &&d16 = D16{})
{
    if constexpr (sizeof(T) == 16) fft_f64<FWD, HALF>(v, L, T_, t, xb, twp);
    else if constexpr (LC >= 256) fft_ct<FWD, LC, HALF, FULL>(v, t, xb, twp, d16);
    else if constexpr (LC > 0) fft_reg<FWD>(v, LC, LC / 16, t, xb, twp);   // the same code with a constant length
    else fft_reg<FWD>(v, L, T_, t, xb, twp);
}

// The butterfly policies of a column pass: the forward and the inverse
// transforms' radix-16 DFTs (registers by default).
struct RegEngine {
    template <bool FWD> __device__ __forceinline__ RegDft16<FWD> d16() const { return {}; }
};

// Number of complex entries of the per-pass twiddle table of length L.
__host__ __device__ constexpr int pass_twiddle_count(int L)
{
    int n = 0, Ns = 16;
    while (Ns * 16 <= L) {
        n += 15 * Ns;
        Ns *= 16;
    }
    if (Ns < L) n += (L / Ns - 1) * Ns;
    return n > 0 ? n : 1;
}

}  // namespace sg
