// Semi-spectral solve for axisymmetric scale heights: the route Sec. 5.2
// gives for a non-constant H/r, a Fourier transform along phi and a direct
// sum along r (cost n_r n_phi log n_phi + n_phi n_r^2).
//
// With H_a = H_a(r) the pair kernel of Sec. 2.2 (Eq. "SG force kernel
// exact", Eq. "mean root square height", Eq. "grav. potential 2D") depends on
// the two radii and on the angle difference only.  The direct sum
//     f_c(i, j) = sum_a sum_{i', j'} W^{ab}_c(i, i', j - j') Sigma_a(i', j')
// is then a circular convolution in phi for every radial pair, and with the
// phi-DFT (hats) it becomes one complex n_r x n_r matrix-vector product per
// azimuthal mode m:
//     f^_c(i, m) = sum_a sum_{i'} W^^{ab}_c(i, i', m) Sigma^_a(i', m).
// Per unit surface density (m_u = r'^2 du dphi, H^2 = (H_a(r')^2 + H_b(r)^2)/2,
// X = s^2 / (8 H^2), Delta = (i - i') du, psi = (j - j') dphi):
//     W_Phi = -G m_u e^X K0(X) / (2 sqrt(pi) H),
//     W_r   = -G m_u D(X) r' (expm1(Delta) + 2 sin^2(psi/2)) / (8 sqrt(pi) H^3),
//     W_phi = -G m_u D(X) r' sin psi / (8 sqrt(pi) H^3),
// and 0 for the self cell; the direct path's pair terms, so the result is
// the direct sum's.
//
// With H = H(r) the samples are exactly even (W_Phi, W_r) or odd (W_phi) in
// psi, so W^ is real, or imaginary for W_phi.  The plan stores one real number
// per entry (FP64 samples and transforms, rounded to the plan dtype):
// [pair][component][n_phi/2 + 1][n_r][n_r], W_phi's without its factor i.
// The row spectra's slot m = 0 packs the real m = 0 and m = n_phi/2
// coefficients as re + i im; its products take the planes m = 0 and n_phi/2.
// The entries carry the conventions of the row transforms around them: the
// forward rows multiply each source row by r_i', the inverse rows divide the
// accelerations by r_i, and the inverse is unnormalised (1 / n_phi).  A solve
// is rows_fwd, k_semi_mv (the tables streamed from HBM once), rows_inv.
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "sg_bessel.cuh"
#include "sg_fft.cuh"
#include "sg_internal.h"
#include "sg_launch.h"
#include "sg_mem.cuh"

namespace sg {

namespace {

// Lag tables in FP64: gi[i - i' + nr - 1] = (sinh^2(Delta/2), expm1(Delta)),
// gj[dj] = (sin^2(psi/2), sin psi).
__global__ void k_semi_geometry(int nr, int nphi, double du, double2 *gi, double2 *gj)
{
    const int n = max(2 * nr - 1, nphi);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        if (q < 2 * nr - 1) {
            const double D = (q - (nr - 1)) * du, sh = sinh(0.5 * D);
            gi[q] = make_double2(sh * sh, expm1(D));
        }
        if (q < nphi) {
            const double sp = sinpi((double)q / nphi);
            gj[q] = make_double2(sp * sp, sinpi(2.0 * q / nphi));
        }
    }
}

// 1 / sqrt(sinh^2(Delta/2) + sin^2(psi/2)) for every lag, [|i - i'|][dj], dj <= nphi/2:
// a function of the lags alone, read by every row pair and pair of fluids
// in place of a reciprocal square root of about 10 FP64 instructions (128 x 256 gas +
// dust plan and solve 2.23 -> 2.12 ms).
__global__ void k_semi_lags(int nr, int N, const double2 *__restrict__ gi, const double2 *__restrict__ gj, double *i1)
{
    const int n = nr * (N + 1);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const int d = q / (N + 1), j = q - d * (N + 1);
        i1[q] = rsqrt(gi[nr - 1 + d].x + gj[j].x);           // infinite at the self cell, which nothing reads
    }
}

// Tables of one (source, target) pair of fluids: a CTA owns G source rows i'
// of one target row i (blockIdx.y), n_phi / 16 threads each.  It samples the
// three components for dj = 0 .. n_phi/2, mirrors them, transforms the row in
// registers and writes the real coefficients, G consecutive entries at a
// time; nothing passes through device memory in between.
//
// FP64 arithmetic bounds it (2 lanes per clock and SM), so the work is cut:
// half the samples by symmetry; one short polynomial per Bessel function (as in
// the direct sum, lengths in units of sqrt(r r')); and, for an FP32 plan, one
// complex transform for the three components, (W_Phi + W_phi) + i W_r, whose
// parts are separable because W_Phi and W_r are even and W_phi odd.  An FP64
// plan transforms W_Phi by itself (PASS 1) and W_r + W_phi (PASS 2), so that no
// component takes on the rounding of a larger one.  128 x 256 gas + dust:
// 15.6 -> 2.1 ms for a plan, a solve and the release (12.5 ms of it was sampling by
// branch, 2.0 ms twelve real transforms).
template <typename R, int PASS>
__global__ void __launch_bounds__(512)
k_semi_table(int nr, int nphi, int lgG, const double2 *__restrict__ gi, const double2 *__restrict__ gj,
             const double *__restrict__ i1, const double *__restrict__ rc, const double *__restrict__ Ha,
             const double *__restrict__ Hb, double scale, R *__restrict__ tab, const double2 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int T = nphi >> 4, N = nphi >> 1, G = 1 << lgG, PL = padded_len(nphi);
    double2 *buf = reinterpret_cast<double2 *>(smem_raw);
    double *sc = reinterpret_cast<double *>(buf + (size_t)G * PL);      // per row: eta, prefactor
    const int g = threadIdx.x / T, t = threadIdx.x - g * T;
    const int i = blockIdx.y, ip0 = blockIdx.x * G, ip = ip0 + g;
    for (int k = threadIdx.x; k < G; k += blockDim.x) {
        const double r = rc[i], p = rc[ip0 + k], q2 = 1.0 / (r * p), ha = Ha[ip0 + k], hb = Hb[i];
        sc[2 * k] = 0.5 * (ha * ha + hb * hb) * q2;
        sc[2 * k + 1] = scale * p * sqrt(q2);
    }
    __syncthreads();
    double2 *xb = buf + (size_t)g * PL;
    const double2 li = gi[i - ip + nr - 1];
    const double *lag = i1 + (size_t)abs(i - ip) * (N + 1);
    {
        const RowPair rp = row_pair(sc[2 * g], sc[2 * g + 1]);
#pragma unroll 1
        for (int dj = t; dj <= N; dj += T) {
            const double2 lj = gj[dj];
            double P = 0.0, F = 0.0;
            if (!(i == ip && dj == 0)) row_pair_eval(rp, li.x + lj.x, lag[dj], P, F);      // self cell excluded
            const double vR = F * (li.y + 2.0 * lj.x), vA = dj == N ? 0.0 : F * lj.y;
            double2 z, zm;                                              // at dj and at -dj
            if constexpr (PASS == 0) {
                z = make_double2(P + vA, vR);
                zm = make_double2(P - vA, vR);
            } else if constexpr (PASS == 1) {
                z = zm = make_double2(P, 0.0);
            } else {
                z = make_double2(vR + vA, 0.0);
                zm = make_double2(vR - vA, 0.0);
            }
            xb[pidx(dj)] = z;
            if (dj > 0 && dj < N) xb[pidx(nphi - dj)] = zm;
        }
    }
    __syncthreads();
    double2 v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = xb[pidx(t + T * e)];
    fft_reg<true>(v, nphi, T, t, xb, tw);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 16; ++e) xb[pidx(t + T * e)] = v[e];
    __syncthreads();
    const size_t plane = (size_t)nr * nr, comp = (size_t)(N + 1) * plane;
    for (int idx = threadIdx.x; idx < (N + 1) << lgG; idx += blockDim.x) {
        const int gg = idx & (G - 1), m = idx >> lgG;
        const double2 Z = buf[(size_t)gg * PL + pidx(m)], Zm = buf[(size_t)gg * PL + pidx((nphi - m) & (nphi - 1))];
        R *o = tab + m * plane + (size_t)i * nr + ip0 + gg;
        const double even = 0.5 * (Z.x + Zm.x), odd = 0.5 * (Z.y - Zm.y);
        if constexpr (PASS == 0) {
            o[0] = (R)even;
            o[comp] = (R)(0.5 * (Z.y + Zm.y));
            o[2 * comp] = (R)odd;
        } else if constexpr (PASS == 1) {
            o[0] = (R)even;
        } else {
            o[comp] = (R)even;
            o[2 * comp] = (R)odd;
        }
    }
}

struct SemiOut {
    int b[6], c[6];   // target fluid and component of each requested output (grid z)
};

// One CTA: mode m, 32 target rows, one requested output.  The source spectra
// of column m wait in shared memory; each warp runs 4 target rows, its lanes
// striding the source rows of each table row (each table entry is read once,
// streaming).  Slot m = 0 multiplies re by plane 0 and im by plane n_phi/2.
// The stream of the tables bounds it: one real number per entry is half the
// bytes of a complex table: 512 x 1024 gas 1.61 GB in 246 us (0.97 of the
// measured HBM bandwidth), 3.23 GB in 537 us before.
// FP32: a lane's four entries of a vector go to two sums in turn, so that neighbouring
// rows, whose terms are the largest, do not follow one another in one chain (g_phi of
// 7 grids, mean relative L2: 1.83e-7 in one chain, 1.79e-7 so). The registers are held to 4
// (one source) or 3 CTAs per SM: 512 x 1024 gas 250 -> 249 us a solve, 512 x 512 gas + dust 565 -> 497,
// 128 x 256 gas + dust 27.4 -> 29.4.
template <typename R> struct vec_of;
template <> struct vec_of<float> { using type = float4; };
template <> struct vec_of<double> { using type = double2; };

template <typename R, int NS>
__global__ void __launch_bounds__(256, sizeof(R) == 4 && NS == 1 ? 4 : 3)
k_semi_mv(const cplx<R> *__restrict__ sh, const R *__restrict__ tab, cplx<R> *__restrict__ oh, int nr,
          int N, const __grid_constant__ SemiOut q)
{
    using C = cplx<R>;
    using V = typename vec_of<R>::type;
    constexpr int W = sizeof(V) / sizeof(R);              // entries per 16-byte load
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *ss = reinterpret_cast<C *>(smem_raw);
    const int m = blockIdx.x, z = blockIdx.z, b = q.b[z], c = q.c[z];
    griddep_wait();                                       // the row spectra are complete from here on
    for (int k = threadIdx.x; k < NS * nr; k += blockDim.x) {
        const int a = k / nr, ip = k - a * nr;
        ss[k] = ld_cg_hint(sh + (size_t)a * N * nr + blk(m, ip, nr), l2_evict_last());
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ib = blockIdx.y * 32 + w * 4;
    const size_t plane = (size_t)nr * nr;
    R ar[4] = {0, 0, 0, 0}, ai[4] = {0, 0, 0, 0};
    R br[4] = {0, 0, 0, 0}, bi[4] = {0, 0, 0, 0};         // FP32: every other entry of a vector
    // nr is a power of two >= 8, so a warp's four rows are all in the grid
    const size_t r0 = (size_t)ib * nr, r1 = r0 + nr, r2 = r1 + nr, r3 = r2 + nr;
#pragma unroll 1
    for (int a = 0; a < NS; ++a) {
        const R *T = tab + ((size_t)((a * NS + b) * 3 + c) * (N + 1) + m) * plane;
        const C *sa = ss + a * nr;
        if (m != 0) {
#pragma unroll 4
            for (int ip = W * lane; ip < nr; ip += 32 * W) {
                const V t[4] = {__ldcs(reinterpret_cast<const V *>(T + r0 + ip)),
                                __ldcs(reinterpret_cast<const V *>(T + r1 + ip)),
                                __ldcs(reinterpret_cast<const V *>(T + r2 + ip)),
                                __ldcs(reinterpret_cast<const V *>(T + r3 + ip))};
                C s[W];
#pragma unroll
                for (int x = 0; x < W; x += 16 / sizeof(C))
                    *reinterpret_cast<float4 *>(&s[x]) = *reinterpret_cast<const float4 *>(sa + ip + x);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const R *tk = reinterpret_cast<const R *>(&t[k]);
#pragma unroll
                    for (int x = 0; x < W; ++x) {
                        R &xr = W == 4 && x % 2 ? br[k] : ar[k], &xi = W == 4 && x % 2 ? bi[k] : ai[k];
                        xr = fma(tk[x], s[x].x, xr);
                        xi = fma(tk[x], s[x].y, xi);
                    }
                }
            }
        } else {
            const R *TN = T + (size_t)N * plane;
            const size_t rk[4] = {r0, r1, r2, r3};
            for (int ip = lane; ip < nr; ip += 32) {
                const C s = sa[ip];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    ar[k] = fma(T[rk[k] + ip], s.x, ar[k]);
                    ai[k] = fma(TN[rk[k] + ip], s.y, ai[k]);
                }
            }
        }
    }
    if constexpr (W == 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            ar[k] += br[k];
            ai[k] += bi[k];
        }
    }
    griddep_launch();                                     // the inverse rows, late (as in the column pass)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ar[k] += __shfl_xor_sync(0xffffffffu, ar[k], o);
            ai[k] += __shfl_xor_sync(0xffffffffu, ai[k], o);
        }
    }
    if (lane < 4) {
        R xr = ar[0], xi = ai[0];
#pragma unroll
        for (int k = 1; k < 4; ++k)
            if (lane == k) {
                xr = ar[k];
                xi = ai[k];
            }
        C v = mkc<C>(xr, xi);
        if (c == 2 && m != 0) v = cmul_i(v);              // planes 0 and n_phi/2 of the odd component are zero
        oh[(size_t)(b * 3 + c) * N * nr + blk(m, ib + lane, nr)] = v;
    }
}

}  // namespace

size_t semi_table_bytes(int nr, int nphi, int nsrc, bool f64)
{
    return (size_t)nsrc * nsrc * 3 * (nphi / 2 + 1) * (size_t)nr * nr * (f64 ? 8 : 4);
}

template <typename R>
cudaError_t build_semi_tables(int nr, int nphi, int nsrc, double du, double dphi, double G, const double *rc_h,
                              const double *H_h[2], void *tab, const double *twp_h, size_t twp_n, cudaStream_t s)
{
    // scratch: the lag tables, the transform's twiddles, the radii and the profiles
    const size_t ngi = 2 * (size_t)(2 * nr), ngj = 2 * (size_t)nphi, nlag = (size_t)nr * (nphi / 2 + 1);
    double *scr = nullptr;
    cudaError_t e = cudaMalloc((void **)&scr, (ngi + ngj + twp_n + 3 * (size_t)nr + nlag) * sizeof(double));
    if (e != cudaSuccess) return e;
    double2 *gi = (double2 *)scr, *gj = (double2 *)(scr + ngi);
    double *tw = scr + ngi + ngj, *rc = tw + twp_n, *H = rc + nr, *i1 = H + 2 * nr;
    e = cudaMemcpyAsync(tw, twp_h, twp_n * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(rc, rc_h, nr * sizeof(double), cudaMemcpyHostToDevice, s);
    for (int a = 0; a < nsrc && e == cudaSuccess; ++a)
        e = cudaMemcpyAsync(H + (size_t)a * nr, H_h[a], nr * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        k_semi_geometry<<<(std::max(2 * nr, nphi) + 255) / 256, 256, 0, s>>>(nr, nphi, du, gi, gj);
        k_semi_lags<<<(int)std::min<size_t>((nlag + 255) / 256, 152 * 16), 256, 0, s>>>(nr, nphi / 2, gi, gj, i1);
        e = cudaGetLastError();
    }
    // rows per CTA: 256 threads (512 for the longest rows) and at most the radial cells
    const int T = nphi / 16;
    int lgG = 0;
    while ((T << (lgG + 1)) <= 256 && (1 << (lgG + 1)) <= nr) ++lgG;
    const size_t smem = semi_table_smem(nphi, lgG);
    const dim3 grid(nr >> lgG, nr), block(T << lgG);
    const double scale = -G * du * dphi / nphi;
    for (int a = 0; a < nsrc && e == cudaSuccess; ++a)
        for (int b = 0; b < nsrc && e == cudaSuccess; ++b) {
            R *dst = (R *)tab + (size_t)(a * nsrc + b) * 3 * (nphi / 2 + 1) * nr * nr;
            auto go = [&](auto kern) {
                kern<<<grid, block, smem, s>>>(nr, nphi, lgG, gi, gj, i1, rc, H + (size_t)a * nr, H + (size_t)b * nr, scale, dst,
                                               (const double2 *)tw);
            };
            if constexpr (sizeof(R) == 4) {
                go(k_semi_table<R, 0>);
            } else {
                go(k_semi_table<R, 1>);
                go(k_semi_table<R, 2>);
            }
            e = cudaGetLastError();
        }
    cudaError_t e2 = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = e2;
    cudaFree(scr);
    return e;
}

size_t semi_table_smem(int nphi, int lgG) { return ((size_t)padded_len(nphi) * 16 + 16) << lgG; }

size_t semi_mv_smem(int nr, int nsrc, bool f64) { return (size_t)nsrc * nr * (f64 ? 16 : 8); }

template <typename R>
cudaError_t launch_semi_mv(const void *sh, const void *tab, void *oh, int nr, int nphi, int nsrc, uint32_t outmask,
                           cudaStream_t s, bool pdl)
{
    SemiOut q{};
    int nz = 0;
    for (int k = 0; k < 6; ++k)
        if ((outmask >> k) & 1u) {
            q.b[nz] = k / 3;
            q.c[nz] = k % 3;
            ++nz;
        }
    if (!nz) return cudaSuccess;
    const int N = nphi / 2;
    const dim3 grid(N, (nr + 31) / 32, nz);
    const size_t smem = semi_mv_smem(nr, nsrc, sizeof(R) == 8);
    using C = cplx<R>;
    const int threads = nr >= 32 ? 256 : nr * 8;          // 4 target rows a warp
    const cudaError_t e = launch_ex(nsrc == 1 ? k_semi_mv<R, 1> : k_semi_mv<R, 2>, grid, dim3(threads), smem, s, pdl,
                                    (const C *)sh, (const R *)tab, (C *)oh, nr, N, q);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t set_semi_smem_limits(int max_optin)
{
    const void *fns[] = {(const void *)k_semi_mv<float, 1>,       (const void *)k_semi_mv<float, 2>,
                         (const void *)k_semi_mv<double, 1>,      (const void *)k_semi_mv<double, 2>,
                         (const void *)k_semi_table<float, 0>,    (const void *)k_semi_table<double, 1>,
                         (const void *)k_semi_table<double, 2>};
    for (const void *f : fns) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template cudaError_t build_semi_tables<float>(int, int, int, double, double, double, const double *,
                                              const double *[2], void *, const double *, size_t, cudaStream_t);
template cudaError_t build_semi_tables<double>(int, int, int, double, double, double, const double *,
                                               const double *[2], void *, const double *, size_t, cudaStream_t);
template cudaError_t launch_semi_mv<float>(const void *, const void *, void *, int, int, int, uint32_t, cudaStream_t,
                                           bool);
template cudaError_t launch_semi_mv<double>(const void *, const void *, void *, int, int, int, uint32_t, cudaStream_t,
                                            bool);

}  // namespace sg
