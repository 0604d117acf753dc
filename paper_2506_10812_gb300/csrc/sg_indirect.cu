// Indirect term (Sec. 5.4, App. E of Rendon Restrepo et al. 2025): the
// star's pull by each source fluid a reduces to two global sums,
//     A_a = sqrt(2) G sum_cells m_a K_a cos phi',   B_a = the same with sin phi',
//     K_a = (1/sqrt(pi)) H_a^-2 (d_a/4) e^{d_a^2/4} [K1 - K0](d_a^2/4),  d_a = r'/H_a,
// m_a = Sigma_a r'^2 du dphi, and the indirect potential's gradient is
// (A cos phi + B sin phi) e_r + (-A sin phi + B cos phi) e_phi.
//
// For a constant aspect ratio h_a, K_a r'^2 = D(1/(4 h_a^2)) / (4 sqrt(pi) h_a^3)
// is one number, so the per-cell work is a weighted sum of Sigma; with a
// scale-height field the factor is evaluated per cell (FP64 Bessel).  The
// reduction is FP64 and deterministic: per-block partial sums, then one
// block adds them in a fixed order.
//
// FP64 additions bound it (2 lanes per clock and SM: 7 us for the 4.2 M cells
// of a 1024 x 2048 gas + dust disc, whose bytes take 2.5 us), so a thread does
// one per cell and little else: it keeps VEC columns and walks the rows, the
// cosines and sines come in once per column and block from a table laid out
// with the plan, FP32 values widen in integer arithmetic, and one block per SM
// keeps the per-block reductions few.  The final sums run in parallel over the
// blocks, launched as a programmatic dependent.  1024 x 2048 gas + dust: 66 ->
// 14 us of device time (a 64-bit division per cell, FP64 conversions and a serial
// sum over the blocks before); 2048 x 4096 gas 98 -> 22.
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "sg_bessel.cuh"
#include "sg_internal.h"
#include "sg_launch.h"
#include "sg_mem.cuh"

namespace sg {

constexpr int IT = 512;            // threads per block
constexpr int IBLOCKS = 152;       // blocks, at most: one per SM

// doubles of a plan's indirect-term buffer: the blocks' partial sums and the
// table (cos, sin) of the cell centres' azimuths
size_t indirect_doubles(int nphi) { return (size_t)IBLOCKS * 2 + 2 * (size_t)nphi; }

__global__ void k_indirect_angles(int nphi, double2 *cs)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nphi; j += gridDim.x * blockDim.x) {
        double sj, cj;
        sincospi(2.0 * ((double)j + 0.5) / nphi, &sj, &cj);
        cs[j] = make_double2(cj, sj);
    }
}
cudaError_t launch_indirect_angles(int nphi, double *buf, cudaStream_t s)
{
    k_indirect_angles<<<std::min((nphi + 127) / 128, 1024), 128, 0, s>>>(nphi, (double2 *)(buf + IBLOCKS * 2));
    return cudaGetLastError();
}

template <typename R, int VEC> struct __align__(VEC * sizeof(R)) Cells { R v[VEC]; };

// sum[x] += q.v[x].  FP32 -> FP64 by moving the exponent and mantissa fields
// (the conversion instruction shares the FP64 units): one branch for the
// vector, as zeros, denormals, infinities and NaN take the instruction.
template <int VEC> __device__ __forceinline__ void add_cells(double (&sum)[VEC], const Cells<double, VEC> &q)
{
#pragma unroll
    for (int x = 0; x < VEC; ++x) sum[x] += q.v[x];
}
template <int VEC> __device__ __forceinline__ void add_cells(double (&sum)[VEC], const Cells<float, VEC> &q)
{
    unsigned b[VEC];
    bool normal = true;
#pragma unroll
    for (int x = 0; x < VEC; ++x) {
        b[x] = __float_as_uint(q.v[x]);
        normal &= (b[x] & 0x7fffffffu) - 0x00800000u < 0x7f000000u;
    }
    if (normal) {
#pragma unroll
        for (int x = 0; x < VEC; ++x)
            sum[x] += __hiloint2double((int)((b[x] & 0x80000000u) | (((b[x] & 0x7fffffffu) >> 3) + 0x38000000u)),
                                       (int)(b[x] << 29));
    } else {
#pragma unroll
        for (int x = 0; x < VEC; ++x) sum[x] += (double)q.v[x];
    }
}

// blockDim = (CX, IT / CX): CX groups of VEC columns, the rest row slots.
// blockIdx.z is the fluid, so that one block's loop is one stream (both
// fluids in one loop: 57 against 44 us at 2048 x 4096).  partial: [fluid][block][cos, sin].
template <typename R, int VEC, bool FIELDS>
__global__ void __launch_bounds__(IT, 1)
k_indirect_partial(int nr, int nphi, const R *__restrict__ s0, const R *__restrict__ s1,
                   const R *__restrict__ H0, const R *__restrict__ H1, const R *__restrict__ rcen,
                   const double2 *__restrict__ cs, double2 *partial)
{
    using V = Cells<R, VEC>;
    __shared__ double col[IT * VEC];               // column sums, [row slot][column]
    __shared__ double red[IT][2];
    griddep_launch();                              // the final sums may set up
    const int CX = blockDim.x, RY = blockDim.y, tx = threadIdx.x, ty = threadIdx.y, tid = ty * CX + tx;
    const int ncols = CX * VEC;
    const R *__restrict__ sig = blockIdx.z ? s1 : s0;
    const R *__restrict__ Hf = blockIdx.z ? H1 : H0;
    double ac = 0.0, as = 0.0;                     // this thread's columns
    for (int c0 = blockIdx.x * ncols; c0 < nphi; c0 += gridDim.x * ncols) {
        const int j = c0 + tx * VEC;
        double sum[VEC];
#pragma unroll
        for (int x = 0; x < VEC; ++x) sum[x] = 0.0;
        if (j < nphi) {
            const int step = gridDim.y * RY;
            int i = blockIdx.y * RY + ty;
            if (FIELDS && Hf) {
                for (; i < nr; i += step) {
                    const size_t c = (size_t)i * nphi + j;
                    const V q = *reinterpret_cast<const V *>(sig + c), h = *reinterpret_cast<const V *>(Hf + c);
                    const double r = (double)rcen[i];
#pragma unroll
                    for (int x = 0; x < VEC; ++x) {
                        // per-cell factor r'^2 K_a
                        const double H = (double)h.v[x];
                        double k0e, D;
                        k0e_D_short(0.25 * r * r / (H * H), k0e, D);
                        sum[x] += (double)q.v[x] * (r * r * (0.56418958354775628695 / (H * H)) * (0.25 * r / H) * D);
                    }
                }
            } else {
                const R *p = sig + (size_t)i * nphi + j;
                const size_t ps = (size_t)step * nphi;
                for (; i + 3 * step < nr; i += 4 * step, p += 4 * ps) {          // four rows in flight
                    const V q0 = *reinterpret_cast<const V *>(p), q1 = *reinterpret_cast<const V *>(p + ps),
                            q2 = *reinterpret_cast<const V *>(p + 2 * ps),
                            q3 = *reinterpret_cast<const V *>(p + 3 * ps);
                    add_cells(sum, q0);
                    add_cells(sum, q1);
                    add_cells(sum, q2);
                    add_cells(sum, q3);
                }
                for (; i < nr; i += step, p += ps) add_cells(sum, *reinterpret_cast<const V *>(p));
            }
        }
        __syncthreads();
#pragma unroll
        for (int x = 0; x < VEC; ++x) col[ty * ncols + tx * VEC + x] = sum[x];
        __syncthreads();
        for (int x = tid; x < ncols && c0 + x < nphi; x += IT) {
            double v = 0.0;
            for (int y = 0; y < RY; ++y) v += col[y * ncols + x];
            const double2 w = cs[c0 + x];
            ac += v * w.x;
            as += v * w.y;
        }
    }
    red[tid][0] = ac;
    red[tid][1] = as;
    __syncthreads();
    // two warps, one per sum: 16 threads' values each, then across the lanes
    if (tid < 64) {
        const int k = tid >> 5, lane = tid & 31;
        double v = 0.0;
        for (int y = lane; y < IT; y += 32) v += red[y][k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0)
            reinterpret_cast<double *>(
                partial + (size_t)blockIdx.z * gridDim.x * gridDim.y + blockIdx.y * gridDim.x + blockIdx.x)[k] = v;
    }
}

// out[2 a + k] = sqrt(2) G du dphi C_a sum_blocks partial; C_a = 1 with a
// scale-height field (already in the partials), else D(1/(4 h_a^2)) / (4 sqrt(pi) h_a^3).
// nblocks: the blocks of one fluid.  One warp per sum.
__global__ void __launch_bounds__(128)
k_indirect_final(int nblocks, int nsrc, const double *__restrict__ partial, double h0, double h1, int field0,
                 int field1, double scale, double *out)
{
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31, a = k >> 1;
    double C = 1.0;
    if (!(a ? field1 : field0)) {
        const double h = a ? h1 : h0;
        double k0e, D;
        k0e_D_short(0.25 / (h * h), k0e, D);
        C = D * 0.56418958354775628695 / (4.0 * h * h * h);
    }
    griddep_wait();                                // the partial sums are complete from here on
    double s = 0.0;
    if (a < nsrc)
        for (int b = lane; b < nblocks; b += 32) s += __ldcg(&partial[((size_t)a * nblocks + b) * 2 + (k & 1)]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0 && k < 2 * nsrc) out[k] = scale * C * s;
}

template <typename R>
cudaError_t launch_indirect(int nr, int nphi, int nsrc, const R *s0, const R *s1, const R *H0, const R *H1,
                            double h0, double h1, const R *rcen, double G, double du, double dphi, double *buf,
                            double *out, cudaStream_t s)
{
    // 16-byte loads where every row of every array starts on one
    constexpr int VW = 16 / sizeof(R);
    const uintptr_t all = (uintptr_t)s0 | (uintptr_t)s1 | (uintptr_t)H0 | (uintptr_t)H1;
    const int vec = nphi % VW == 0 && (all & 15u) == 0 ? VW : 1;
    const int groups = (nphi + vec - 1) / vec;
    int cx = 64;                                   // column groups a block: 64, fewer for short rows
    while (cx > 1 && cx / 2 >= groups) cx /= 2;
    const int per = IBLOCKS / nsrc;                // blocks a fluid
    const int gx = std::min((groups + cx - 1) / cx, per);
    const int gy = std::max(1, std::min(per / gx, (nr + IT / cx - 1) / (IT / cx)));
    const dim3 grid(gx, gy, nsrc), block(cx, IT / cx);
    const double2 *cs = (const double2 *)(buf + IBLOCKS * 2);
    auto go = [&](auto kern) {
        kern<<<grid, block, 0, s>>>(nr, nphi, s0, s1, H0, H1, rcen, cs, (double2 *)buf);
    };
    const bool fields = H0 || H1;
    if (vec == 1) {
        if (fields) go(k_indirect_partial<R, 1, true>);
        else go(k_indirect_partial<R, 1, false>);
    } else {
        if (fields) go(k_indirect_partial<R, VW, true>);
        else go(k_indirect_partial<R, VW, false>);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_ex(k_indirect_final, dim3(1), dim3(128), 0, s, true, gx * gy, nsrc, (const double *)buf, h0, h1,
                     (int)(H0 != nullptr), (int)(H1 != nullptr), 1.4142135623730950488 * G * du * dphi, out);
}

template cudaError_t launch_indirect<float>(int, int, int, const float *, const float *, const float *, const float *,
                                            double, double, const float *, double, double, double, double *,
                                            double *, cudaStream_t);
template cudaError_t launch_indirect<double>(int, int, int, const double *, const double *, const double *,
                                             const double *, double, double, const double *, double, double, double,
                                             double *, double *, cudaStream_t);

}  // namespace sg
