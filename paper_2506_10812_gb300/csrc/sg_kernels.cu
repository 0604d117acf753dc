// FFT-convolution path of the thin-disc self-gravity solver (Sec. 5.2 and
// App. C of Rendon Restrepo et al. 2025) for sm_103a.
//
// Data flow of one solve (constant aspect ratios, nr x nphi grid, L = 2 nr,
// N = nphi / 2, H = nr):
//   rows_fwd  each source Sigma_a [nr][nphi], scaled by r_i (see below) and
//             with its row mean removed -> row R2C (length nphi) -> packed
//             spectra (column m = 0 holds the real m = 0 and m = nphi/2
//             coefficients as re + i im) stored column-major;
//   cols      per column m: zero-padded length-L forward FFT of every
//             source, products with the kernel spectra (staged in shared
//             memory by TMA bulk copies, all at kernel start or one
//             (target, component) step at a time) summed over sources (Sec.
//             5.2 multi-fluid sums), inverse FFT of every requested (target,
//             component), rows 0..nr-1 written back;
//   rows_inv  per output row: packed C2R (length nphi) and the epilogue.
// The column pass and the inverse rows launch as programmatic dependents of
// the kernel before them (launch_ex; griddep_wait before reading its output).
//
// Layout of the [N][rows] intermediates (sg_mem.cuh, BW = 1): column-major,
// element (m, i) at m rows + i, so the column pass moves contiguous columns
// and a row transform that owns 2 or 4 consecutive rows moves a 16- or
// 32-byte slice of every column.  (The column-blocked variant BW = 4, element (m, i) at
// ((m / 4) rows + i) 4 + m % 4, gives the row transforms whole 128-byte
// lines but makes every column access a stride-4 vector; on the 2048 x 4096
// disc it makes the column pass 44 % slower and the row transforms 14 %
// faster.)
//
// Radial scaling: the lattice kernels carry e^{-3 Delta / 2}, which makes
// the convolution output span (r_out / r_in)^{3/2} across the grid while
// FP32 FFT rounding is uniform in absolute terms.  With
// e^{-alpha Delta} = (r' / r)^alpha the convolution is rewritten exactly as
//     sum_i' Sigma(i') K(i - i') = r_i^-alpha sum_i' [Sigma(i') r_i'^alpha] [e^{alpha Delta} K](i - i'),
// alpha = 1: the sources are multiplied by r_i' in rows_fwd, the kernel
// tables by e^Delta, and the accelerations by 1/r_i in rows_inv (the
// potential's own r_i prefactor cancels the 1/r_i).  Removing each row's
// mean before the row FFT (and adding nphi * mean back to the m = 0
// coefficient) is exact by linearity and keeps the small m != 0 modes of a
// nearly axisymmetric disc from inheriting the rounding of the mean.
//
// The kernel spectra (built once per plan by tab_eval -> rows_fwd<double>
// -> tabcols) already carry -G du dphi / (L nphi), the FFT normalisation.
#include <math.h>
#include <stdint.h>

#include <mutex>
#include <type_traits>
#include <utility>

#include "sg_bessel.cuh"
#include "sg_cols.cuh"
#include "sg_fft.cuh"
#include "sg_internal.h"
#include "sg_launch.h"
#include "sg_mem.cuh"

namespace sg {



bool cols_staging_steps(int nr, int nsrc, bool f64, int staging)
{
    return staging < 0 ? cols_steps_default(nsrc, f64, 2 * nr) : staging != 0 && !f64;
}

size_t col_smem_bytes(int nr, int nsrc, bool f64, int staging)
{
    const size_t esz = f64 ? 16 : 8;
    const int L = 2 * nr;
    const size_t xb = align16((size_t)padded_len(L) * esz);
    // per step: one (target, component) step of kernel spectra staged at a
    // time, source spectra in registers
    if (cols_staging_steps(nr, nsrc, f64, staging)) return 16 + xb + (size_t)nsrc * tab_pitch(nr) * esz;
    const size_t tb = (size_t)nsrc * 3 * tab_pitch(nr) * esz;
    const size_t spec = nsrc == 2 ? (size_t)2 * L * esz : 0;   // gas + dust spectra live in shared memory
    return 16 + xb + tb + spec;
}

size_t tabcol_smem_bytes(int L, bool) { return (size_t)padded_len(L) * 16; }

// ----------------------------------------------------------- kernel table
// A CTA owns KR lattice rows and up to 256 lags j <= nphi/2: the rows' constants are
// computed once in shared memory, a thread keeps its lag's sine and walks
// the rows, and each value is written at j and, mirrored (exactly even, or
// odd for the azimuthal component), at nphi - j.  FP64 instructions bound it:
// about 45 a sample and half the samples, where every sample used to compute
// its exponentials, sines and a quadrature (preparing a 1024 x 2048 gas + dust plan
// and its input 12.4 -> 7.3 ms, a 2048 x 4096 gas one 18.2 -> 12.6).
constexpr int KR = 32;
__global__ void __launch_bounds__(256)
k_tab_eval(int nr, int nphi, double du, double ha, double hb, double scale, double alpha,
           double *p0, double *p1, double *p2, float *q0, float *q1, float *q2)
{
    __shared__ RowPair rp[KR];
    __shared__ double sh2[KR], em1[KR];
    const int L = 2 * nr, k0 = blockIdx.y * KR;
    for (int x = threadIdx.x; x < KR && k0 + x < L; x += blockDim.x) {
        const int k = k0 + x, di = (k < nr) ? k : k - L;
        const double Dl = di * du, sh = sinh(0.5 * Dl);                  // Delta = u - u'
        const double hab2 = 0.5 * (ha * ha * exp(-Dl) + hb * hb * exp(Dl));
        sh2[x] = sh * sh;
        em1[x] = expm1(Dl);
        rp[x] = row_pair(hab2, scale * exp((alpha - 1.5) * Dl));
    }
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const double sp = sinpi((double)j / nphi), sp2 = sp * sp, spsi = sinpi(2.0 * j / nphi);   // sin(psi / 2), sin(psi)
    __syncthreads();
    if (2 * j > nphi) return;
    const bool mirror = j > 0 && 2 * j < nphi;
    const int kn = min(KR, L - k0);
    for (int x = 0; x < kn; ++x) {
        const int k = k0 + x;
        double vP = 0.0, vR = 0.0, vA = 0.0;
        if (k != nr && !(k == 0 && j == 0)) {
            double F;
            const double sg = sh2[x] + sp2;
            row_pair_eval(rp[x], sg, rsqrt(sg), vP, F);
            vR = F * (em1[x] + 2.0 * sp2);
            vA = F * spsi;
        }
        const size_t a = (size_t)k * nphi + j, b = (size_t)k * nphi + (nphi - j);
        if (p0) {
            p0[a] = vP;
            if (mirror) p0[b] = vP;
        }
        if (p1) {
            p1[a] = vR;
            if (mirror) p1[b] = vR;
        }
        if (p2) {
            p2[a] = vA;
            if (mirror) p2[b] = -vA;
        }
        if (q0) {
            q0[a] = (float)vP;
            if (mirror) q0[b] = (float)vP;
        }
        if (q1) {
            q1[a] = (float)vR;
            if (mirror) q1[b] = (float)vR;
        }
        if (q2) {
            q2[a] = (float)vA;
            if (mirror) q2[b] = (float)-vA;
        }
    }
}

cudaError_t launch_tab_eval(int nr, int nphi, double du, double ha, double hb, double scale,
                            double alpha, double *o64[3], float *o32[3], cudaStream_t s)
{
    const int lags = nphi / 2 + 1, threads = lags < 256 ? (lags + 31) / 32 * 32 : 256;
    const dim3 grid((lags + threads - 1) / threads, (2 * nr + KR - 1) / KR);
    k_tab_eval<<<grid, threads, 0, s>>>(nr, nphi, du, ha, hb, scale, alpha, o64[0], o64[1], o64[2], o32[0], o32[1],
                                        o32[2]);
    return cudaGetLastError();
}

// All-at-once column kernel of a plan shape (ST = 0; per-step kernels in
// sg_cols_steps.cu).
template <typename R>
using ColsKernel = void (*)(const cplx<R> *, const cplx<R> *, cplx<R> *, int, int, uint32_t, const cplx<R> *,
                            unsigned int *, int);
template <typename R>
ColsKernel<R> cols_kernel_all(int nsrc, int L)
{
    if constexpr (sizeof(R) == 4) {
        if (nsrc == 1) {
            if (L == 4096) return k_cols<R, 1, 4096, false>;
            if (L == 2048) return k_cols<R, 1, 2048, false>;
            if (L == 1024) return k_cols<R, 1, 1024, false>;
            if (L == 512) return k_cols<R, 1, 512, false>;
            if (L == 256) return k_cols<R, 1, 256, false>;
            if (L == 128) return k_cols<R, 1, 128, false>;
            if (L == 64) return k_cols<R, 1, 64, false>;
        } else {
            if (L == 4096) return k_cols<R, 2, 4096, false>;
            if (L == 2048) return k_cols<R, 2, 2048, false>;
            if (L == 1024) return k_cols<R, 2, 1024, false>;
            if (L == 512) return k_cols<R, 2, 512, false>;
            if (L == 256) return k_cols<R, 2, 256, false>;
            if (L == 128) return k_cols<R, 2, 128, false>;
            if (L == 64) return k_cols<R, 2, 64, false>;
        }
    }
    if (nsrc == 1) return k_cols<R, 1, 0, false>;
    return k_cols<R, 2, 0, false>;
}

template <typename R>
cudaError_t launch_cols(const void *sh, const void *tab, void *oh, int nr, int nphi, int nsrc,
                        uint32_t outmask, const void *tw_col, unsigned int *flag, cudaStream_t s, int ncols, bool pdl,
                        bool discard, int staging)
{
    const bool f64 = sizeof(R) == 8;
    const int N = nphi / 2, T = (2 * nr) / 16;
    const bool steps = cols_staging_steps(nr, nsrc, f64, staging);
    const size_t smem = col_smem_bytes(nr, nsrc, f64, steps ? 1 : 0);
    const int nq = __builtin_popcount(outmask);
    const bool split = ncols <= 0 && cols_split(N, T, nq, f64);
    const dim3 grid = split ? dim3(N, nq) : dim3((ncols > 0 && ncols < N ? ncols : N) - 1 + nq);
    // whole 128-byte lines per source column (a column read by every output's
    // CTA, column 0 or a split launch's, is not discarded)
    const bool dc = discard && !split && BW == 1 && ((size_t)nr * 2 * sizeof(R)) % 128 == 0 && ((uintptr_t)sh & 127u) == 0;
    ColsKernel<R> kern;
    if constexpr (sizeof(R) == 4) kern = steps ? cols_kernel_steps(nsrc, 2 * nr) : cols_kernel_all<R>(nsrc, 2 * nr);
    else kern = cols_kernel_all<R>(nsrc, 2 * nr);
    const cudaError_t err = launch_ex(kern, grid, dim3(T), smem, s, pdl, (const cplx<R> *)sh,
                                      (const cplx<R> *)tab, (cplx<R> *)oh, nr, N, outmask,
                                      (const cplx<R> *)tw_col, flag, dc ? 1 : 0);
    return err != cudaSuccess ? err : cudaGetLastError();
}

// ------------------------------------------- table column FFT + packing
// spec: [nphi/2][L] row spectra of one real table (FP64, sg_mem.cuh layout);
// tab: [nphi/2 + 1][P] kernel spectrum columns (slot k = S(k), 0 <= k <= H).
template <typename R>
__global__ void __launch_bounds__(512)
k_tabcols(const double2 *__restrict__ spec, cplx<R> *__restrict__ tab, int L, int N, int odd,
          const double2 *__restrict__ tw)
{
    using C = cplx<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *xb = reinterpret_cast<double2 *>(smem_raw);
    const int T = L >> 4, H = L >> 1, t = threadIdx.x, m = blockIdx.x;
    const int P = H + 2;
    double2 v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = spec[blk(m, t + T * e, L)];
    fft_reg<true>(v, L, T, t, xb, tw);
    // the spectrum goes back to the (now free) exchange buffer, padded index
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 16; ++e) xb[pidx(t + T * e)] = v[e];
    __syncthreads();
    auto sp = [&](int k) { return xb[pidx(k & (L - 1))]; };
    // stored spectrum S = i T for the odd (sin psi) component, T otherwise;
    // S(0) and S(H) are real by symmetry and stored with a zero imaginary part
    auto S = [&](double2 x) { return odd ? cmul_i(x) : x; };
    auto put = [&](C *col, int k, double2 x) {
        if (k == 0 || k == H) x.y = 0.0;
        col[k] = mkc<C>((R)x.x, (R)x.y);
    };
    for (int k = t; k <= H; k += T) {
        if (m != 0) {
            put(tab + (size_t)m * P, k, S(sp(k)));
        } else {
            // unpack columns 0 and nphi/2 from the packed column
            const double2 X = sp(k), Xn = cconj(sp(L - k));
            put(tab, k, S(cscale(cadd(X, Xn), 0.5)));
            put(tab + (size_t)N * P, k, S(cscale(cmul_mi(csub(X, Xn)), 0.5)));
        }
    }
    if (t == 0) {
        tab[(size_t)m * P + H + 1] = mkc<C>(0, 0);
        if (m == 0) tab[(size_t)N * P + H + 1] = mkc<C>(0, 0);
    }
}

template <typename R>
cudaError_t launch_tabcols(const void *spec, void *tab, int L, int nphi, bool odd,
                           const void *tw_col64, cudaStream_t s)
{
    const int N = nphi / 2;
    k_tabcols<R><<<N, L / 16, tabcol_smem_bytes(L, true), s>>>(
        (const double2 *)spec, (cplx<R> *)tab, L, N, odd ? 1 : 0, (const double2 *)tw_col64);
    return cudaGetLastError();
}

// Raise every kernel's dynamic shared-memory limit to the device maximum
// (the launch's own request still sets the occupancy), so plans of any size
// can share the kernels.
cudaError_t set_smem_limits(int max_optin)
{
    const void *fns[] = {(const void *)k_cols<float, 1, 0, false>,    (const void *)k_cols<float, 1, 4096, false>,
                         (const void *)k_cols<float, 1, 2048, false>, (const void *)k_cols<float, 1, 1024, false>,
                         (const void *)k_cols<float, 1, 512, false>,  (const void *)k_cols<float, 1, 256, false>,
                         (const void *)k_cols<float, 2, 0, false>,    (const void *)k_cols<float, 2, 4096, false>,
                         (const void *)k_cols<float, 2, 2048, false>, (const void *)k_cols<float, 2, 1024, false>,
                         (const void *)k_cols<float, 2, 512, false>,  (const void *)k_cols<float, 2, 256, false>,
                         (const void *)k_cols<float, 1, 128, false>,  (const void *)k_cols<float, 1, 64, false>,
                         (const void *)k_cols<float, 2, 128, false>,  (const void *)k_cols<float, 2, 64, false>,
                         (const void *)k_cols<double, 1, 0, false>,   (const void *)k_cols<double, 2, 0, false>,
                         (const void *)k_tabcols<float>,              (const void *)k_tabcols<double>};
    for (const void *fn : fns) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = set_cols_steps_smem_limits(max_optin);
    return e != cudaSuccess ? e : set_row_smem_limits(max_optin);
}

template cudaError_t launch_cols<float>(const void *, const void *, void *, int, int, int, uint32_t, const void *,
                                        unsigned int *, cudaStream_t, int, bool, bool, int);
template cudaError_t launch_cols<double>(const void *, const void *, void *, int, int, int, uint32_t, const void *,
                                         unsigned int *, cudaStream_t, int, bool, bool, int);
template cudaError_t launch_tabcols<float>(const void *, void *, int, int, bool, const void *, cudaStream_t);
template cudaError_t launch_tabcols<double>(const void *, void *, int, int, bool, const void *, cudaStream_t);
}  // namespace sg
