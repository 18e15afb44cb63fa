// Observables of the state: norm (Sec. 2: conserved by the unitary
// evolution), position moments and the energy <psi|H|psi> of the
// tight-binding Hamiltonian H = -J * (nearest-neighbour hops) + diag(V).
//
// FP32 grids: every product is formed exactly (two_prod) and each thread
// accumulates in double-float (hi + lo floats, ~48 significant bits) on the
// FP32 pipe; the per-thread sums are converted to FP64 once and combined
// across threads and blocks with Neumaier's compensated update.  (This
// GB300 runs FP64 at ~1/67 of the FP32 rate, so per-site FP64 work would
// make the reduction several times slower than one pass over HBM.)
// FP64 grids: every term in FP64; each thread sums a run of 4 sites in
// plain FP64 and adds the run into Neumaier-compensated per-thread sums.
// Either way the block writes FP64 partials and a final block sums them.
#include <algorithm>

#include "common.cuh"
#include "ffloat.cuh"
#include "internal.h"
#include "walk.cuh"

namespace ts {

namespace {

constexpr int kThreads = 256;

struct Neu {
    double s, c;
    __device__ __forceinline__ void add(double v)
    {
        double t = s + v;
        c += (fabs(s) >= fabs(v)) ? ((s - t) + v) : ((v - t) + s);
        s = t;
    }
    __device__ __forceinline__ double val() const { return s + c; }
};

// Merge two compensated sums (a += b).
__device__ __forceinline__ void neu_merge(Neu &a, const Neu &b)
{
    a.add(b.s);
    a.c += b.c;
}

// Sum a quantity over the block: lane l of one warp adds the values of
// threads l, l + 32, ... (a value is v.x + v.y, v.y its low part), then the
// lanes' sums are merged.
template <typename V2>
__device__ __forceinline__ Neu warp_sum(const V2 *v, int lane)
{
    Neu a = {0.0, 0.0};
#pragma unroll
    for (int i = 0; i < kThreads / 32; ++i) {
        const V2 x = v[lane + 32 * i];
        a.add((double)x.x);
        a.c += (double)x.y;
    }
    return a;
}

__device__ __forceinline__ Neu warp_merge(Neu a)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        Neu b;
        b.s = __shfl_down_sync(0xffffffffu, a.s, off);
        b.c = __shfl_down_sync(0xffffffffu, a.c, off);
        neu_merge(a, b);
    }
    return a;
}

// Block-level compensated reduction of NQ per-thread sums into partials, one
// warp per quantity.  The FP64 units bound it (64 cycles per warp-wide
// operation and scheduler): so shared, a block takes about 90 of them per
// quantity; with every warp merging all quantities over its lanes first it took
// 270 (a whole ts_observe at 128^2: 117 -> 42 us; 2048^2: 217 -> 79 us).
template <int NQ, typename V2>
__device__ __forceinline__ void block_reduce_write(const V2 (&acc)[NQ], double *__restrict__ partials)
{
    __shared__ V2 sh[NQ][kThreads];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NQ; ++q) sh[q][threadIdx.x] = acc[q];
    __syncthreads();
    constexpr int stride = NQ > OBS_Q ? NQ : OBS_Q;
    for (int q = warp; q < NQ; q += kThreads / 32) {
        const Neu a = warp_merge(warp_sum(sh[q], lane));
        if (lane == 0) partials[(int64_t)blockIdx.x * stride + q] = a.val();
    }
}

// FP32 state: exact products, double-float per-thread sums.  A thread takes
// chunks of 4 consecutive sites of one row (x0 a multiple of 4; the row
// pitch is a multiple of 32 floats, so the float4 loads stay inside the
// row's padding and columns >= nx are masked).
template <bool NORM_ONLY>
__global__ void __launch_bounds__(kThreads)
observe_f32_kernel(const float *__restrict__ re, const float *__restrict__ im,
                   const float *__restrict__ vp, int nx, int ny, int64_t pitch,
                   double *__restrict__ partials)
{
    grid_dep_sync();
    constexpr int NQ = NORM_ONLY ? 1 : OBS_Q;
    FF acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = ff_make(0.f);

    const int chunks_per_row = (nx + 3) / 4;
    const int64_t nchunks = (int64_t)chunks_per_row * ny;
    for (Walk w(chunks_per_row, blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
                (int64_t)gridDim.x * blockDim.x);
         w.i < nchunks; w.next()) {
        const int y = (int)w.y;
        const int x0 = (int)w.x * 4;
        const int64_t o = (int64_t)y * pitch + x0;
        const float4 r4 = *reinterpret_cast<const float4 *>(re + o);
        const float4 m4 = *reinterpret_cast<const float4 *>(im + o);
        const float r[4] = {r4.x, r4.y, r4.z, r4.w}, m[4] = {m4.x, m4.y, m4.z, m4.w};
        FF P = ff_make(0.f), XP = ff_make(0.f), X2P = ff_make(0.f), KIN = ff_make(0.f),
           VP = ff_make(0.f);
        if constexpr (NORM_ONLY) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (x0 + u < nx)
                    P = ff_add(P, ff_add(two_prod(r[u], r[u]), two_prod(m[u], m[u])));
            }
            acc[0] = ff_add(acc[0], P);
        } else {
            const float4 v4 = *reinterpret_cast<const float4 *>(vp + o);
            const float v[4] = {v4.x, v4.y, v4.z, v4.w};
            float rd[4] = {0.f, 0.f, 0.f, 0.f}, md[4] = {0.f, 0.f, 0.f, 0.f};
            if (y + 1 < ny) {
                const float4 a = *reinterpret_cast<const float4 *>(re + o + pitch);
                const float4 b = *reinterpret_cast<const float4 *>(im + o + pitch);
                rd[0] = a.x; rd[1] = a.y; rd[2] = a.z; rd[3] = a.w;
                md[0] = b.x; md[1] = b.y; md[2] = b.z; md[3] = b.w;
            }
            const float r_next = (x0 + 4 < nx) ? re[o + 4] : 0.f;
            const float m_next = (x0 + 4 < nx) ? im[o + 4] : 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (x0 + u >= nx) break;
                const FF p = ff_add(two_prod(r[u], r[u]), two_prod(m[u], m[u]));
                P = ff_add(P, p);
                XP = ff_add(XP, ff_mul_f(p, (float)u));
                X2P = ff_add(X2P, ff_mul_f(p, (float)(u * u)));
                VP = ff_add(VP, ff_mul_f(p, v[u]));
                // bonds to the right and downward neighbours
                const float rr = (u < 3) ? r[u + 1] : r_next, mr = (u < 3) ? m[u + 1] : m_next;
                if (x0 + u + 1 < nx) {
                    KIN = ff_add(KIN, two_prod(r[u], rr));
                    KIN = ff_add(KIN, two_prod(m[u], mr));
                }
                if (y + 1 < ny) {
                    KIN = ff_add(KIN, two_prod(r[u], rd[u]));
                    KIN = ff_add(KIN, two_prod(m[u], md[u]));
                }
            }
            const float fx0 = (float)x0, fy = (float)y;   // exact: sides <= 2^20
            acc[0] = ff_add(acc[0], P);
            // sum x p = x0 P + sum u p ; sum x^2 p = x0^2 P + 2 x0 (sum u p) + sum u^2 p
            const FF Px0 = ff_mul_f(P, fx0);
            acc[1] = ff_add(acc[1], ff_add(Px0, XP));
            acc[2] = ff_add(acc[2], ff_mul_f(P, fy));
            acc[3] = ff_add(acc[3], ff_add(ff_add(ff_mul_f(Px0, fx0), ff_mul_f(XP, 2.f * fx0)), X2P));
            acc[4] = ff_add(acc[4], ff_mul_f(ff_mul_f(P, fy), fy));
            acc[5] = ff_add(acc[5], KIN);
            acc[6] = ff_add(acc[6], VP);
        }
    }
    float2 sums[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) sums[q] = make_float2(acc[q].hi, acc[q].lo);
    block_reduce_write<NQ>(sums, partials);
}

// <phi|psi>: exact products, double-float per-thread sums, FP64 combine.
__global__ void __launch_bounds__(kThreads)
inner_f32_kernel(const float *__restrict__ ar, const float *__restrict__ ai,
                 const float *__restrict__ br, const float *__restrict__ bi, int nx, int ny,
                 int64_t pitch, double *__restrict__ partials)
{
    grid_dep_sync();
    FF sr = ff_make(0.f), si = ff_make(0.f);
    const int chunks_per_row = (nx + 3) / 4;
    const int64_t nchunks = (int64_t)chunks_per_row * ny;
    for (Walk w(chunks_per_row, blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
                (int64_t)gridDim.x * blockDim.x);
         w.i < nchunks; w.next()) {
        const int y = (int)w.y;
        const int x0 = (int)w.x * 4;
        const int64_t o = (int64_t)y * pitch + x0;
        const float4 a4 = *reinterpret_cast<const float4 *>(ar + o);
        const float4 b4 = *reinterpret_cast<const float4 *>(ai + o);
        const float4 c4 = *reinterpret_cast<const float4 *>(br + o);
        const float4 d4 = *reinterpret_cast<const float4 *>(bi + o);
        const float pr[4] = {a4.x, a4.y, a4.z, a4.w}, pi[4] = {b4.x, b4.y, b4.z, b4.w};
        const float qr[4] = {c4.x, c4.y, c4.z, c4.w}, qi[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (x0 + u >= nx) break;
            // conj(p) q = (pr qr + pi qi) + i (pr qi - pi qr)
            sr = ff_add(sr, ff_add(two_prod(pr[u], qr[u]), two_prod(pi[u], qi[u])));
            si = ff_add(si, ff_add(two_prod(pr[u], qi[u]), two_prod(-pi[u], qr[u])));
        }
    }
    const float2 sums[2] = {make_float2(sr.hi, sr.lo), make_float2(si.hi, si.lo)};
    block_reduce_write<2>(sums, partials);
}

// Observables in FP64 (2-D or 3-D grids; slab z = rows z*ny .. z*ny + ny - 1):
// runs of 4 sites are summed plainly and added into Neumaier-compensated
// per-thread sums.  The FP64 units bound it, so a run sums p, u p and u^2 p
// (u = 0 .. 3) and expands x = x0 + u, y and z once per run, and the kinetic
// sum takes its factor -2 J in the final pass (a whole ts_observe at 2047 x 1536: 355 -> 190 us, at 256^3 1856 -> 1215 us).
template <typename T, bool NORM_ONLY, bool THREE>
__global__ void __launch_bounds__(kThreads)
observe_kernel(const T *__restrict__ re, const T *__restrict__ im, const T *__restrict__ vp,
               int nx, int ny, int nz, int64_t pitch, double *__restrict__ partials)
{
    grid_dep_sync();
    constexpr int NQ = NORM_ONLY ? 1 : THREE ? OBS_Q3 : OBS_Q;
    Neu acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = {0.0, 0.0};

    const int64_t rows = (int64_t)ny * nz;
    const int64_t slab = (int64_t)ny * pitch;
    const int chunks_per_row = (nx + 3) / 4;
    const int64_t nchunks = (int64_t)chunks_per_row * rows;
    for (Walk w(chunks_per_row, blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
                (int64_t)gridDim.x * blockDim.x);
         w.i < nchunks; w.next()) {
        const int64_t row = w.y;
        const int x0 = (int)w.x * 4;
        const int z = THREE ? (int)(row / ny) : 0, y = (int)(row - (int64_t)z * ny);
        const int64_t o = row * pitch + x0;
        const bool down = y + 1 < ny, below = THREE && z + 1 < nz;
        double P = 0.0, XP = 0.0, X2P = 0.0, KIN = 0.0, VP = 0.0;
        double r = (double)re[o], m = (double)im[o];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (x0 + u >= nx) break;
            const double p = fma(r, r, m * m);
            P += p;
            if constexpr (!NORM_ONLY) {
                if (u == 1) {
                    XP += p;
                    X2P += p;
                } else if (u > 1) {
                    XP = fma((double)u, p, XP);
                    X2P = fma((double)(u * u), p, X2P);
                }
                VP = fma((double)vp[o + u], p, VP);
                if (down)
                    KIN = fma(r, (double)re[o + pitch + u], fma(m, (double)im[o + pitch + u], KIN));
                if (below)
                    KIN = fma(r, (double)re[o + slab + u], fma(m, (double)im[o + slab + u], KIN));
            }
            if (x0 + u + 1 < nx) {
                const double rn = (double)re[o + u + 1], mn = (double)im[o + u + 1];
                if constexpr (!NORM_ONLY) KIN = fma(r, rn, fma(m, mn, KIN));
                r = rn;
                m = mn;
            }
        }
        acc[0].add(P);
        if constexpr (!NORM_ONLY) {
            const double fx = (double)x0, fy = (double)y;
            acc[1].add(fma(fx, P, XP));
            acc[2].add(fy * P);
            acc[3].add(fma(fx, fma(fx, P, 2.0 * XP), X2P));
            acc[4].add(fy * fy * P);
            acc[5].add(KIN);
            acc[6].add(VP);
            if constexpr (THREE) {
                const double fz = (double)z;
                acc[7].add(fz * P);
                acc[8].add(fz * fz * P);
            }
        }
    }
    double2 sums[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) sums[q] = make_double2(acc[q].s, acc[q].c);
    block_reduce_write<NQ>(sums, partials);
}

// The blocks' partials: one warp per quantity.  Quantity 5 is the kinetic sum,
// which takes its factor here.
__global__ void __launch_bounds__(kThreads)
observe_finalize_kernel(const double *__restrict__ partials, int nblocks, int nq, int stride,
                        double kin_factor, double *__restrict__ result)
{
    grid_dep_sync();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int q = warp; q < nq; q += kThreads / 32) {
        Neu a = {0.0, 0.0};
        for (int b = lane; b < nblocks; b += 32) a.add(partials[(int64_t)b * stride + q]);
        a = warp_merge(a);
        if (lane == 0) result[q] = q == 5 ? kin_factor * a.val() : a.val();
    }
}

// Blocks of a reduction over nchunks runs of 4 sites.  More blocks per SM hide
// the loads but add block reductions, which the FP64 units take one after the
// other: FP32 grids get 1, 2 from 8 and 4 from 64 runs per thread and SM-filling
// block (observables at 1001 x 777: 54, 58, 80 us with 1, 2, 4; at 8192^2: 636,
// 436, 428 us; norm at 8192^2: 372, 217, 153 us), FP64 kernels, bound by those
// units in any case, 1 (2047 x 1536: 189, 191, 213 us).
int reduce_blocks(int64_t nchunks, bool fp64)
{
    const int64_t per = (nchunks + kThreads - 1) / kThreads, sms = num_sms();
    const int64_t most = fp64 ? sms : per >= 64 * sms ? 4 * sms : per >= 8 * sms ? 2 * sms : sms;
    return (int)std::max<int64_t>(1, std::min({per, most, (int64_t)OBS_MAX_BLOCKS}));
}

}  // namespace

cudaError_t launch_observe(const void *re, const void *im, const void *vplane, bool f64, int nx,
                           int ny, int64_t pitch, double J, bool norm_only, double *partials,
                           double *result, cudaStream_t st)
{
    const int nblocks = reduce_blocks((int64_t)((nx + 3) / 4) * ny, f64);
    if (f64) {
        const double *r = (const double *)re, *m = (const double *)im, *v = (const double *)vplane;
        if (norm_only)
            launch_pdl(observe_kernel<double, true, false>, nblocks, kThreads, 0, st, r, m, v, nx,
                       ny, 1, pitch, partials);
        else
            launch_pdl(observe_kernel<double, false, false>, nblocks, kThreads, 0, st, r, m, v, nx,
                       ny, 1, pitch, partials);
    } else {
        const float *r = (const float *)re, *m = (const float *)im, *v = (const float *)vplane;
        if (norm_only)
            launch_pdl(observe_f32_kernel<true>, nblocks, kThreads, 0, st, r, m, v, nx, ny, pitch,
                       partials);
        else
            launch_pdl(observe_f32_kernel<false>, nblocks, kThreads, 0, st, r, m, v, nx, ny, pitch,
                       partials);
    }
    launch_pdl(observe_finalize_kernel, 1, kThreads, 0, st, partials, nblocks,
               norm_only ? 1 : OBS_Q, OBS_Q, -2.0 * J, result);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_observe3(const void *re, const void *im, const void *vplane, bool f64, int nx,
                            int ny, int nz, int64_t pitch, double J, double *partials,
                            double *result, cudaStream_t st)
{
    const int nblocks = reduce_blocks((int64_t)((nx + 3) / 4) * ny * nz, true);
    if (f64)
        launch_pdl(observe_kernel<double, false, true>, nblocks, kThreads, 0, st, (const double *)re,
                   (const double *)im, (const double *)vplane, nx, ny, nz, pitch, partials);
    else
        launch_pdl(observe_kernel<float, false, true>, nblocks, kThreads, 0, st, (const float *)re,
                   (const float *)im, (const float *)vplane, nx, ny, nz, pitch, partials);
    launch_pdl(observe_finalize_kernel, 1, kThreads, 0, st, partials, nblocks, OBS_Q3, OBS_Q3,
               -2.0 * J, result);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_inner(const float *phi_re, const float *phi_im, const float *psi_re,
                         const float *psi_im, int nx, int ny, int64_t pitch, double *partials,
                         double *result, cudaStream_t st)
{
    const int nblocks = reduce_blocks((int64_t)((nx + 3) / 4) * ny, false);
    launch_pdl(inner_f32_kernel, nblocks, kThreads, 0, st, phi_re, phi_im, psi_re, psi_im, nx, ny,
               pitch, partials);
    launch_pdl(observe_finalize_kernel, 1, kThreads, 0, st, partials, nblocks, 2, OBS_Q, 1.0,
               result);
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace ts
