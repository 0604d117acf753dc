// Direct O(N^2) pair sum with position-dependent scale heights (Sec. 2.2):
//     g_b(r) = -G sum_a sum_{cells r' != r} m_a(r') K_ab(r, r') e_s,
//     Phi_b(r) = -G sum_a sum_{cells r' != r} m_a(r') e^X K0(X) / (2 sqrt(pi) H_ab),
// m_a = Sigma_a r'^2 du dphi, H_ab^2 = (H_a(r')^2 + H_b(r)^2) / 2 (Eq. "mean
// root square height"), X = s^2 / (8 H_ab^2).  This is the parity path of
// the library and the only one valid for non-constant H/r.
//
// The pair geometry is taken from the integer index differences
// (di, dj) = (i - i', j - j'), with Delta = di du and psi = dj dphi:
//     s^2            = 4 r r' [sinh^2(Delta/2) + sin^2(psi/2)],
//     e_r . (r - r') = r' [expm1(Delta) + 2 sin^2(psi/2)],
//     e_phi . (r - r') = r' sin psi,
// using per-lag tables built in FP64, so FP32 keeps full relative precision
// for the nearest neighbours (no cancellation in r - r').
//
// Bound and decomposition.  The sum is bound by the FP pipes (FP64: 1/64 of the
// FP32 lane rate), so the kernel is built to leave few operations per pair.  A
// pair's geometry depends on the row pair and on dj alone, its scale height on
// the two cells.  With lengths in units of sqrt(r r') (sigma = s^2 / (r r'),
// eta = H^2 / (r r')) and z = 1/X = 4 (eta_a + eta_b) / sigma,
//     Phi term = m / s S0(z),   force term = m / s^3 (r - r') Q(z),
// S0 and Q the tails of the Bessel functions (1 at z = 0: the Newtonian
// limit).  So a CTA owns KT x blockDim targets of one row and walks the source
// rows; per source row it tabulates, for a tile of lags dj, (4 / sigma,
// sigma^-1/2 and the two sigma^-3/2 weights) once for all its targets, stages
// the window of sources the tile meets, and then runs over dj: the lag's
// entry is one broadcast, a target's source is at a fixed distance (conflict-
// free), and a pair with z <= 1/16 costs 24 operations (FP32; 36 in FP64)
// instead of a Bessel evaluation by branch (about 360).  Lags that may hold a larger z (a bound from the
// tile's largest scale heights; they lie around dj = 0) take the table
// polynomials instead; every lane of a warp is on the same lag, so the two paths do not diverge.
// (One thick cell sends its window's lags that way for all the CTA's targets: 128 x 256 gas
// 1.2 ms with smooth heights, 6.0 with heights of 10^U(-2, 1) r, where it took 970 by branch.)
// Every term is added with Kahan's compensation, 12 of the 24 operations.  (Sums of 16 lags
// without it took 15 operations, 3.75 and 6.89 ms below, but left 0.56 units in the last place
// where a compensated sum leaves 0.30.)  Measured (solve): 128 x 256 gas + dust FP32
// 112.6 -> 4.62 ms (0.93 Tpair/s; 24 operations at the FMA pipes' 37 Tlane/s would be 2.8 ms), 61 x 150
// gas FP64 227 -> 8.74 ms (9.6 Gpair/s of the 16 that 36 operations allow), against one thread per
// target with the Bessel functions by branch; errors against 64 bits 1.2e-7 (1.8e-7 then) and 3.6e-15 (3.5e-15).
//
// The source rows are split over the CTAs of a cluster, whose partial sums
// are added through distributed shared memory in rank order (no workspace, the
// same bits every time).
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <mutex>

#include "sg.h"
#include "sg_bessel.cuh"
#include "sg_direct_tile.h"
#include "sg_internal.h"

namespace sg {

namespace cg = cooperative_groups;

template <typename R> struct pair_of;
template <> struct pair_of<float> { using type = float2; };
template <> struct pair_of<double> { using type = double2; };

template <typename R> struct Acc {
    R s = 0, c = 0;
    __device__ __forceinline__ void add(R v)   // Kahan-compensated sum
    {
        R y = v - c;
        R t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ void add(R a, R b)   // the same for a b, its rounding included
    {
        R y = fma(a, b, -c);
        R t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

constexpr int DLT = kDirectLagTile, DMAXT = kDirectMaxThreads;

template <typename R> struct __align__(16) LagFar { R iz, w1, wr, wp; };   // 4 / sigma, and the weights
template <typename R> struct __align__(2 * sizeof(R)) Duo { R x, y; };

// x times a constant held in two parts (the second is 0 in FP64): its rounding would
// be one relative error, up to 6e-8, that all pairs share
template <typename R> __device__ __forceinline__ R times(R x, Duo<R> c) { return fma(x, c.x, x * c.y); }

// shared memory of a CTA of T threads and KT targets each; the partial sums
// overlay the tables at the end
template <typename R> constexpr size_t direct_smem(int T, int KT)
{
    const size_t tab = DLT * (sizeof(LagFar<R>) + sizeof(Duo<R>)) + (size_t)(T * KT + DLT) * sizeof(Duo<R>);
    const size_t red = (size_t)6 * T * KT * sizeof(R);
    return tab > red ? tab : red;
}

// 1 / sqrt(x) to rounding (the FP32 instruction alone is off by 2 ulp)
__device__ __forceinline__ float rsqrt_r(float x)
{
    const float y = rsqrtf(x), e = fmaf(-x * y, y, 1.0f);
    return fmaf(0.5f * y, e, y);
}
__device__ __forceinline__ double rsqrt_r(double x) { return rsqrt(x); }

// x / (2 sqrt(pi)), the common factor of a pair's terms, without the constant's own
// rounding, which all pairs would share.  With w = m / (2 sqrt(pi) H) a pair is
//     Phi term = w K0e,   force term = w E 2 / s^2 (r - r'),
// one power of 1/H (its cube, in D = E / X, carried three times its rounding).
__device__ __forceinline__ float over_2_sqrt_pi(float x)
{
    constexpr double c = 0.5 * 0.56418958354775628695;
    constexpr float hi = (float)c, lo = (float)(c - (double)hi);
    return fmaf(x, hi, x * lo);
}
__device__ __forceinline__ double over_2_sqrt_pi(double x) { return x * (0.5 * 0.56418958354775628695); }

// One pair by its own scale height: (K0e, E) at z = 1 / X, any z.
template <typename R>
__device__ __forceinline__ void pair_bessel(R z, R &k0e, R &E)
{
    if (z <= (R)BESSEL_ZTAIL) {
        R S0, Q;
        bessel_tail(z, S0, Q);
        const R s = sqrt((R)1.5707963267948966192 * z);
        k0e = s * S0;
        E = (R)0.5 * s * Q;
        return;
    }
    const R X = (R)1 / z;
    if (bessel_in_table(X)) {
        bessel_table(X, k0e, E);
    } else {                                   // X < 2^-20, or not a number
        double a, b;
        k0e_D_series((double)X, a, b);
        k0e = (R)a;
        E = (R)(b * (double)X);
    }
}

template <typename R, int KT>
__global__ void __launch_bounds__(DMAXT)
k_direct(int nr, int nphi, int nchunk, R G, const R *__restrict__ sig_g, const R *__restrict__ sig_d,
         const R *__restrict__ Hg, const R *__restrict__ Hd, R h_g, R h_d, int tgt, R *phi, R *gr,
         R *gphi, const typename pair_of<R>::type *__restrict__ geo_i,
         const typename pair_of<R>::type *__restrict__ geo_j, const R *__restrict__ rcen, Duo<R> cell,
         unsigned int *flag)
{
    using P2 = typename pair_of<R>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LagFar<R> *lagF = reinterpret_cast<LagFar<R> *>(smem_raw);
    Duo<R> *lagN = reinterpret_cast<Duo<R> *>(lagF + DLT);       // (e_r, e_phi) geometry over r'
    Duo<R> *win = lagN + DLT;                                    // (mass / sqrt(r r'), eta_a)
    __shared__ unsigned s_bmax, s_amax[2];                       // largest |H_b| / r and eta_a, as their bits
    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int t = threadIdx.x, T = blockDim.x, TJ = KT * T, lane = t & 31;
    const int unit = blockIdx.x / S, i = unit / nchunk, j0 = (unit - i * nchunk) * TJ;
    const R r = rcen[i];
    const R *Hb_f = tgt == 0 ? Hg : Hd;
    const R hb = tgt == 0 ? h_g : h_d;
    R Hb[KT];
    if (t == 0) {
        s_bmax = 0u;
        s_amax[0] = 0u;
    }
    __syncthreads();
    {
        float mx = 0.f;
        bool nan = false;
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            const int j = min(j0 + t + k * T, nphi - 1);        // past the row: a copy of its last target
            Hb[k] = Hb_f ? Hb_f[(size_t)i * nphi + j] : hb * r;
            const float h = fabsf((float)(Hb[k] / r));
            nan |= h != h;
            mx = fmaxf(mx, h);
        }
        const unsigned m = __reduce_max_sync(0xffffffffu, nan ? 0x7fc00000u : __float_as_uint(mx));
        if (lane == 0) atomicMax(&s_bmax, m);
    }
    Acc<R> agr[KT], agp[KT], aph[KT];
    int tile = 0;
    const int nsrc_fluids = sig_d ? 2 : 1;
    for (int a = 0; a < nsrc_fluids; ++a) {
        const R *sig = a == 0 ? sig_g : sig_d;
        const R *Ha_f = a == 0 ? Hg : Hd;
        const R ha = a == 0 ? h_g : h_d;
        for (int i2 = rank; i2 < nr; i2 += S) {
            const R rr = rcen[i2];
            const P2 gi = geo_i[i - i2 + nr - 1];                // (sinh^2(D/2), expm1(D))
            const R q = (R)1 / sqrt(r * rr);
            R eb[KT];
#pragma unroll
            for (int k = 0; k < KT; ++k) {
                const R h = Hb[k] * q;
                eb[k] = h * h;
            }
            bool flat = false;
#pragma unroll
            for (int k = 0; k < KT; ++k) flat |= eb[k] == (R)0;
            for (int d0 = 0; d0 < nphi; d0 += DLT, ++tile) {
                const int nlag = min(DLT, nphi - d0);
                // the previous tile is done with.  A pair of two zero heights has no
                // kernel (NaN, as in the short rows' kernel), which the tails at z = 0, the
                // Newtonian limit, would hide: such a tile takes the pair by pair path.
                const bool flats = __syncthreads_or(flat);
                if (t == 0) s_amax[(tile + 1) & 1] = 0u;
                // target slot x and lag d of the tile meet the source at window slot x - d + DLT - 1
                float mx = 0.f;
                bool nan = false;
                for (int w = DLT - nlag + t; w < TJ + DLT - 1; w += T) {
                    int jj = (j0 - d0 + w - (DLT - 1)) % nphi;
                    if (jj < 0) jj += nphi;
                    const size_t src = (size_t)i2 * nphi + jj;
                    const R h = (Ha_f ? Ha_f[src] : ha * rr) * q, e = h * h;
                    win[w] = {times(G * sig[src] * rr * rr, cell) * q, e};
                    const float ef = (float)e;
                    nan |= ef != ef || (flats && e == (R)0);
                    mx = fmaxf(mx, ef);
                }
                const unsigned m = __reduce_max_sync(0xffffffffu, nan ? 0x7fc00000u : __float_as_uint(mx));
                if (lane == 0) atomicMax(&s_amax[tile & 1], m);
                for (int l = t; l < nlag; l += T) {
                    const P2 gj = geo_j[d0 + l];                 // (sin^2(psi/2), sin psi)
                    const R sg = (R)4 * (gi.x + gj.x);
                    const R er = gi.y + (R)2 * gj.x;
                    const R i1 = (R)1 / sqrt(sg), i3 = i1 / sg;
                    lagF[l] = {(R)4 / sg, i1, i3 * er, i3 * gj.y};
                    lagN[l] = {er, gj.y};
                }
                __syncthreads();
                // [lo, hi): the lags whose pairs all have z <= 1/16 and whose
                // weights are ordinary numbers; 4 / sigma falls towards dj = nphi / 2
                int lo = 0, hi = nlag;
                {
                    const float hq = __uint_as_float(s_bmax) * (float)(r * q);
                    const float lim = 1.001f * (__uint_as_float(s_amax[tile & 1]) + hq * hq);
                    for (int l0 = 0; l0 < nlag; l0 += 32) {
                        const int l = l0 + lane;
                        bool near = false;
                        if (l < nlag) {
                            const float iz = (float)lagF[l].iz;
                            near = !(iz * lim <= (float)BESSEL_ZTAIL && iz < 1e20f && iz > 1e-20f);
                        }
                        const bool first = 2 * (d0 + l) <= nphi;
                        const unsigned nf = __ballot_sync(0xffffffffu, near && first);
                        const unsigned ns = __ballot_sync(0xffffffffu, near && !first);
                        if (nf) lo = l0 + 32 - __clz(nf);
                        if (ns) hi = min(hi, l0 + __ffs(ns) - 1);
                    }
                }
                const Duo<R> *wt = win + t + DLT - 1;
#pragma unroll 4
                for (int d = lo; d < hi; ++d) {
                    const LagFar<R> L = lagF[d];
#pragma unroll
                    for (int k = 0; k < KT; ++k) {
                        const Duo<R> s = wt[k * T - d];
                        R S0, Q;
                        bessel_tail((s.y + eb[k]) * L.iz, S0, Q);
                        aph[k].add(s.x, S0 * L.w1);
                        Q *= s.x;
                        agr[k].add(Q, L.wr);
                        agp[k].add(Q, L.wp);
                    }
                }
#pragma unroll 1
                for (int d = 0; d < nlag; ++d) {
                    if (d == lo && lo < hi) d = hi;
                    if (d >= nlag) break;
                    if (i2 == i && d0 + d == 0) continue;        // self cell excluded
                    const R iz = lagF[d].iz, hz = (R)0.5 * iz;
                    const Duo<R> g = lagN[d];
#pragma unroll
                    for (int k = 0; k < KT; ++k) {
                        const Duo<R> s = wt[k * T - d];
                        const R eta = s.y + eb[k], z = eta * iz;
                        R k0e, E;
                        pair_bessel(z, k0e, E);
                        const R w = over_2_sqrt_pi(s.x * rsqrt_r((R)0.5 * eta));
                        const R f = w * hz * E;                    // G m K / s
                        agr[k].add(f * g.x);
                        agp[k].add(f * g.y);
                        aph[k].add(w * k0e);
                    }
                }
            }
        }
    }
    // partial sums of the cluster's ranks, in rank order, each with its compensation
    Duo<R> *red = reinterpret_cast<Duo<R> *>(smem_raw);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < KT; ++k) {
        red[t + k * T] = {aph[k].s, -aph[k].c};
        red[TJ + t + k * T] = {agr[k].s, -agr[k].c};
        red[2 * TJ + t + k * T] = {agp[k].s, -agp[k].c};
    }
    cluster.sync();
    const R inv_r = (R)1 / r;
    bool bad = false;
    for (int x = rank * T + t; x < 3 * TJ; x += S * T) {
        const int c = x / TJ, j = j0 + x - c * TJ;
        if (j >= nphi) continue;
        Acc<R> v;
        for (int p = 0; p < S; ++p) {
            const Duo<R> s = *cluster.map_shared_rank(red + x, p);
            v.add(s.x);
            v.add(s.y);
        }
        const R o = c == 0 ? -v.s : -v.s * inv_r;
        R *out = c == 0 ? phi : c == 1 ? gr : gphi;
        if (out) out[(size_t)i * nphi + j] = o;
        bad |= !isfinite(o);
    }
    if (flag && bad) atomicOr(flag, 1u);
    cluster.sync();                                              // no CTA leaves while another reads its sums
}

// Short rows (nphi < kDirectRowMin): one thread per target over all sources,
// the pair terms in the same variables.  A row kernel's warp would own one row
// pair's few pairs and spend its time on the tables.  The line: at nphi = 8 the
// rows take 0.042 against 0.164 ms (50 rows) and 5.98 against 5.45 (2000 rows),
// at nphi = 4 0.054 against 0.165 (100 rows) but 12.8 against 4.1 (3000 rows).
constexpr int DT = 256;   // targets per CTA and sources per shared-memory tile
template <typename R>
__global__ void __launch_bounds__(DT)
k_direct_short(int nr, int nphi, R G, const R *__restrict__ sig_g, const R *__restrict__ sig_d,
               const R *__restrict__ Hg, const R *__restrict__ Hd, R h_g, R h_d, int tgt, R *phi, R *gr,
               R *gphi, const typename pair_of<R>::type *__restrict__ geo_i,
               const typename pair_of<R>::type *__restrict__ geo_j, const R *__restrict__ rcen, Duo<R> cell,
               unsigned int *flag)
{
    using P2 = typename pair_of<R>::type;
    __shared__ R s_r[DT], s_m[DT], s_H2[DT];
    __shared__ int s_i[DT], s_j[DT];
    const int ncell = nr * nphi;
    const int tid = blockIdx.x * DT + threadIdx.x;
    const bool valid = tid < ncell;
    const int i = valid ? tid / nphi : 0;
    const int j = valid ? tid - i * nphi : 0;
    const R r = rcen[i];
    const R *Hb_f = tgt == 0 ? Hg : Hd;
    const R hb = tgt == 0 ? h_g : h_d;
    const R Hb = valid ? (Hb_f ? Hb_f[tid] : hb * r) : (R)1;
    const R Hb2 = Hb * Hb;
    Acc<R> agr, agp, aph;
    const int nsrc_fluids = sig_d ? 2 : 1;
    for (int a = 0; a < nsrc_fluids; ++a) {
        const R *sig = a == 0 ? sig_g : sig_d;
        const R *Ha_f = a == 0 ? Hg : Hd;
        const R ha = a == 0 ? h_g : h_d;
        for (int s0 = 0; s0 < ncell; s0 += DT) {
            __syncthreads();
            const int src = s0 + threadIdx.x;
            if (src < ncell) {
                const int ii = src / nphi, jj = src - (src / nphi) * nphi;
                const R rr = rcen[ii];
                const R Ha = Ha_f ? Ha_f[src] : ha * rr;
                s_r[threadIdx.x] = rr;
                s_m[threadIdx.x] = times(G * sig[src] * rr * rr, cell);
                s_H2[threadIdx.x] = Ha * Ha;
                s_i[threadIdx.x] = ii;
                s_j[threadIdx.x] = jj;
            }
            __syncthreads();
            const int cnt = min(DT, ncell - s0);
            if (!valid) continue;
            for (int q = 0; q < cnt; ++q) {
                if (s0 + q == tid) continue;                 // self cell excluded
                const int di = i - s_i[q];
                int dj = j - s_j[q];
                if (dj < 0) dj += nphi;
                const P2 gi = geo_i[di + nr - 1];            // (sinh^2(D/2), expm1(D))
                const P2 gj = geo_j[dj];                     // (sin^2(psi/2), sin psi)
                const R rr = s_r[q];
                const R s2 = (R)4 * r * rr * (gi.x + gj.x);
                const R H2 = (R)0.5 * (s_H2[q] + Hb2);
                const R z = (R)8 * H2 / s2;
                R k0e, E;
                pair_bessel(z, k0e, E);
                const R w = over_2_sqrt_pi(s_m[q] * rsqrt_r(H2));
                const R f = w * ((R)2 * rr / s2) * E;        // G m K r' / s
                agr.add(f * (gi.y + (R)2 * gj.x));
                agp.add(f * gj.y);
                aph.add(w * k0e);
            }
        }
    }
    if (!valid) return;
    if (phi) phi[tid] = -aph.s;
    if (gr) gr[tid] = -agr.s;
    if (gphi) gphi[tid] = -agp.s;
    if (flag && !(isfinite(aph.s) && isfinite(agr.s) && isfinite(agp.s))) atomicOr(flag, 1u);
}
constexpr int kDirectRowMin = 8;

template <typename R>
cudaError_t launch_direct(int nr, int nphi, double r_in, double du, double G, const R *sig_g,
                          const R *sig_d, const R *Hg, const R *Hd, double h_g, double h_d, int tgt,
                          R *phi, R *gr, R *gphi, const R *geo_i, const R *geo_j, const R *rcen,
                          unsigned int *flag, cudaStream_t s)
{
    (void)r_in;
    using P2 = typename pair_of<R>::type;
    const double dphi = 2.0 * M_PI / nphi, area = du * dphi;
    const Duo<R> cell = {(R)area, (R)(area - (double)(R)area)};
    if (nphi < kDirectRowMin) {
        const int ncell = nr * nphi;
        k_direct_short<R><<<(ncell + DT - 1) / DT, DT, 0, s>>>(
            nr, nphi, (R)G, sig_g, sig_d, Hg, Hd, (R)h_g, (R)h_d, tgt, phi, gr, gphi, (const P2 *)geo_i,
            (const P2 *)geo_j, rcen, cell, flag);
        return cudaGetLastError();
    }
    const DirectTile d = direct_tile(nr, nphi, sizeof(R) == 8);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)d.S;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nr * d.nchunk * d.S));
    cfg.blockDim = dim3((unsigned)(32 * d.W));
    cfg.dynamicSmemBytes = direct_smem<R>(32 * d.W, d.KT);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    auto go = [&](auto kern) {
        return cudaLaunchKernelEx(&cfg, kern, nr, nphi, d.nchunk, (R)G, sig_g, sig_d, Hg, Hd, (R)h_g, (R)h_d, tgt, phi,
                                  gr, gphi, (const P2 *)geo_i, (const P2 *)geo_j, rcen, cell, flag);
    };
    cudaError_t e;
    if (d.KT == 1) e = go(k_direct<R, 1>);
    else if (d.KT == 2) e = go(k_direct<R, 2>);
    else if constexpr (sizeof(R) == 4) e = go(k_direct<R, 4>);
    else e = cudaErrorInvalidConfiguration;
    return e != cudaSuccess ? e : cudaGetLastError();
}

template cudaError_t launch_direct<float>(int, int, double, double, double, const float *, const float *,
                                          const float *, const float *, double, double, int, float *,
                                          float *, float *, const float *, const float *, const float *,
                                          unsigned int *, cudaStream_t);
template cudaError_t launch_direct<double>(int, int, double, double, double, const double *, const double *,
                                           const double *, const double *, double, double, int, double *,
                                           double *, double *, const double *, const double *,
                                           const double *, unsigned int *, cudaStream_t);

}  // namespace sg

// ---------------------------------------------------------------------------
// Allocation-free direct sum (sg_direct_noalloc in sg.h).
//
// Some callers cannot let a library allocate device memory: host codes whose
// device memory is owned by their own allocator or a fixed pool (a library
// cudaMalloc would bypass their accounting or fragment the pool), and time
// loops that must never enter the CUDA allocator.  sg_direct_noalloc serves
// them with the direct pair sum of a plan of the DIRECT method, without a
// plan: the per-lag geometry tables that a plan keeps in its own device
// memory live instead in the fixed array below, compiled into this library.
// Every GPU that loads the library holds the array until the process exits.

namespace {

constexpr int kNoAllocMaxNr = 1024;     // largest nr the array can serve
constexpr int kNoAllocMaxNphi = 4096;   // largest nphi
// FP64 layout (FP32 uses the first half of each part):
//   [0, 32768)       lag table over di: (sinh^2(D/2), expm1(D)), 2 (2 nr - 1) reals
//   [32768, 98304)   lag table over dj: (sin^2(psi/2), sin psi), 2 nphi reals
//   [98304, 106496)  cell-centre radii, nr reals
constexpr size_t kNoAllocGeoJ = 32768, kNoAllocRcen = 98304, kNoAllocBytes = 106496;
static_assert(2 * (2 * kNoAllocMaxNr - 1) * sizeof(double) <= kNoAllocGeoJ, "geo_i part too small");
static_assert(2 * kNoAllocMaxNphi * sizeof(double) <= kNoAllocRcen - kNoAllocGeoJ, "geo_j part too small");
static_assert(kNoAllocMaxNr * sizeof(double) <= kNoAllocBytes - kNoAllocRcen, "rcen part too small");

}  // namespace

static __device__ __align__(256) unsigned char g_sg_noalloc_scratch[kNoAllocBytes];

namespace sg {

// Fill the three geometry tables for one grid (FP64 arithmetic).
template <typename R>
__global__ void k_direct_geometry(int nr, int nphi, double r_in, double du, R *geo_i, R *geo_j, R *rcen)
{
    const int n = max(2 * nr - 1, max(nphi, nr));
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        if (q < 2 * nr - 1) {
            const double D = (q - (nr - 1)) * du, sh = sinh(0.5 * D);
            geo_i[2 * q] = (R)(sh * sh);
            geo_i[2 * q + 1] = (R)expm1(D);
        }
        if (q < nphi) {
            const int jj = (2 * q <= nphi) ? q : nphi - q;
            const double sg = (2 * q <= nphi) ? 1.0 : -1.0;
            const double sp = sinpi((double)jj / nphi);
            geo_j[2 * q] = (R)(sp * sp);
            geo_j[2 * q + 1] = (R)(sg * sinpi(2.0 * jj / nphi));
        }
        if (q < nr) rcen[q] = (R)(r_in * exp((q + 0.5) * du));
    }
}

// Load every kernel that a call may launch (CUDA loads a kernel at its first use,
// which may take device memory): the grid's size chooses among them.
static cudaError_t load_direct_kernels()
{
    const void *kernels[] = {(const void *)k_direct<float, 1>,        (const void *)k_direct<float, 2>,
                             (const void *)k_direct<float, 4>,        (const void *)k_direct<double, 1>,
                             (const void *)k_direct<double, 2>,       (const void *)k_direct_short<float>,
                             (const void *)k_direct_short<double>,    (const void *)k_direct_geometry<float>,
                             (const void *)k_direct_geometry<double>};
    for (const void *k : kernels) {
        cudaFuncAttributes a;
        const cudaError_t e = cudaFuncGetAttributes(&a, k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace sg

namespace {

// The array's device address, looked up once per CUDA context.  A context is
// identified by its unique id (cuCtxGetId: never reused within a process), so
// a primary context that cudaDeviceReset tore down and the runtime created
// again gets a fresh lookup instead of the old, dangling address.
struct NoAllocSlot {
    unsigned long long ctx_id;
    void *ptr;
};
std::mutex g_noalloc_mutex;
NoAllocSlot g_noalloc[64] = {};

using CtxGetCurrentFn = CUresult (*)(CUcontext *);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long *);

// Unique id of the calling thread's current context; 0 when none is current.
unsigned long long current_ctx_id()
{
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<CtxGetCurrentFn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<CtxGetIdFn>(f);
    });
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (!get_current || !get_id || get_current(&c) != CUDA_SUCCESS || !c || get_id(c, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// Device address of the array in the current context: the lookup runs on the
// first call in each context (it also makes the device's primary context
// current when none is, and loads the kernels), later calls reuse it.
cudaError_t noalloc_scratch(void **out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    NoAllocSlot &slot = g_noalloc[dev];
    const unsigned long long id = current_ctx_id();
    if (id == 0 || id != slot.ctx_id || !slot.ptr) {
        void *ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_sg_noalloc_scratch);
        if (e == cudaSuccess) e = sg::load_direct_kernels();
        if (e != cudaSuccess) return e;
        slot.ptr = ptr;
        slot.ctx_id = current_ctx_id();            // nonzero once the lookup made a context current
    }
    *out = slot.ptr;
    return cudaSuccess;
}

template <typename R>
sg_status direct_noalloc_t(const sg_params *p, void *scratch, const void *sg_, const void *sd_,
                           void *const outs[6], int nsrc, cudaStream_t s)
{
    const double du = std::log(p->r_out / p->r_in) / p->nr;
    R *geo_i = (R *)scratch;
    R *geo_j = (R *)((char *)scratch + kNoAllocGeoJ);
    R *rcen = (R *)((char *)scratch + kNoAllocRcen);
    // every entry the sum reads is rewritten here first, so nothing from an
    // earlier call is used
    const int n = std::max(2 * p->nr - 1, std::max(p->nphi, p->nr));
    sg::k_direct_geometry<R><<<(n + 255) / 256, 256, 0, s>>>(p->nr, p->nphi, p->r_in, du, geo_i, geo_j, rcen);
    cudaError_t e = cudaGetLastError();
    for (int b = 0; b < nsrc && e == cudaSuccess; ++b) {
        if (!(outs[3 * b] || outs[3 * b + 1] || outs[3 * b + 2])) continue;
        e = sg::launch_direct<R>(p->nr, p->nphi, p->r_in, du, p->G, (const R *)sg_, nsrc == 2 ? (const R *)sd_ : nullptr,
                                 (const R *)p->H_g_field, (const R *)p->H_d_field, p->h_g, p->h_d, b, (R *)outs[3 * b],
                                 (R *)outs[3 * b + 1], (R *)outs[3 * b + 2], geo_i, geo_j, rcen, nullptr, s);
    }
    if (e != cudaSuccess) {
        fprintf(stderr, "sg_direct_noalloc: %s\n", cudaGetErrorString(e));
        return SG_ERR_CUDA;
    }
    return SG_OK;
}

}  // namespace

extern "C" sg_status sg_direct_noalloc(const sg_params *p, const void *sigma_g, const void *sigma_d, void *phi_g,
                                       void *gr_g, void *gphi_g, void *phi_d, void *gr_d, void *gphi_d, void *stream)
{
    if (!p || !sigma_g) return SG_ERR_ARG;
    if (p->method != SG_METHOD_DIRECT || (p->dtype != SG_F32 && p->dtype != SG_F64)) return SG_ERR_ARG;
    if (!(std::isfinite(p->r_in) && std::isfinite(p->r_out) && p->r_in > 0 && p->r_out > p->r_in) ||
        !std::isfinite(p->G) || p->nr < 1 || p->nphi < 1)
        return SG_ERR_ARG;
    if (p->nr > kNoAllocMaxNr || p->nphi > kNoAllocMaxNphi) {
        fprintf(stderr, "sg_direct_noalloc: grid %d x %d exceeds the fixed scratch (nr <= %d, nphi <= %d)\n", p->nr,
                p->nphi, kNoAllocMaxNr, kNoAllocMaxNphi);
        return SG_ERR_UNSUPPORTED;
    }
    // the parameter sets sg_plan_create accepts for a DIRECT plan
    if (!(std::isfinite(p->h_g) && (p->h_g > 0 || p->H_g_field))) return SG_ERR_ARG;
    const int nsrc = (p->h_d > 0 || p->H_d_field) ? 2 : 1;
    if (nsrc == 2 && (!std::isfinite(p->h_d) || !sigma_d)) return SG_ERR_ARG;
    // an error left pending by the caller's own work is theirs: report it
    // without consuming it, and launch nothing
    const cudaError_t pending = cudaPeekAtLastError();
    if (pending != cudaSuccess) {
        fprintf(stderr, "sg_direct_noalloc: a CUDA error is already pending (%s); nothing launched\n",
                cudaGetErrorString(pending));
        return SG_ERR_CUDA;
    }
    void *scratch = nullptr;
    cudaError_t e = noalloc_scratch(&scratch);
    if (e != cudaSuccess) {
        fprintf(stderr, "sg_direct_noalloc: scratch or kernels: %s\n", cudaGetErrorString(e));
        return SG_ERR_CUDA;
    }
    void *outs[6] = {phi_g, gr_g, gphi_g, phi_d, gr_d, gphi_d};
    cudaStream_t s = (cudaStream_t)stream;
    return p->dtype == SG_F64 ? direct_noalloc_t<double>(p, scratch, sigma_g, sigma_d, outs, nsrc, s)
                              : direct_noalloc_t<float>(p, scratch, sigma_g, sigma_d, outs, nsrc, s);
}

