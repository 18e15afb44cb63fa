// Fused second-order Trotter-Suzuki steps for FP64 grids: one step per launch.
//
// What bounds it: the FP64 units.  A scheduler of this GPU issues one warp-wide
// DFMA in 64 cycles (76 when all four of an SM do), and a single warp with a
// chain of dependent DFMAs already keeps it busy, so the only things that
// count are the number of DFMAs and an even share of them for each scheduler.
//  - Scaled rotations (see pair_s in scaled.cuh): 2 DFMA per site and sweep
//    instead of 3.  With six sweeps and the phase a step takes 16 DFMA per site
//    (22 with lifting sweeps).  The scale stays in the state from launch to
//    launch and the tail takes it out: the host carries the growth of the bulk
//    and of the edges, from which each launch's edge coefficients follow.
//  - One pass over memory per step (48 B per site, far from a bound) instead of
//    seven (240 B).
//
// The steps, with X and Y factors commuting and the sweeps of neighbouring
// steps merged, are cut behind the X group:
//   Xe Xo | Ye Yo P Yo (Xo Xe Xo) | Ye Yo P Yo (Xo Xe Xo) | ... | Ye
// A launch takes one part: in y it needs only two rows more on either side.
// A warp owns a strip of 32 C columns, C per lane, and walks down a range of h
// rows; its lanes' columns 3 .. 32 C - 4 are stored.  The rows above and below
// cost 24 DFMA per column and range, against 16 h.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "internal.h"
#include "scaled.cuh"

namespace ts {

namespace {

constexpr int kWarps = 4;   // per block: one per scheduler

template <int C>
struct Row {
    double re[C], im[C];
};

// a, b <- a + i ta b, b + i tb a
__device__ __forceinline__ void pair64(double &ar, double &ai, double &br, double &bi, double ta,
                                       double tb)
{
    const double r = ar, m = ai;
    ar = fma(-ta, bi, ar);
    ai = fma(ta, br, ai);
    br = fma(-tb, m, br);
    bi = fma(tb, r, bi);
}

__device__ __forceinline__ void take64(double &ar, double &ai, double br, double bi, double t)
{
    ar = fma(-t, bi, ar);
    ai = fma(t, br, ai);
}

// what the lane's columns receive in one X sweep ([column][lane])
template <int C>
__device__ __forceinline__ void x_even64(Row<C> &v, const double (*e)[32], int lane)
{
    if constexpr (C == 1) {
        const double pr = __shfl_xor_sync(FULL, v.re[0], 1), pi = __shfl_xor_sync(FULL, v.im[0], 1);
        take64(v.re[0], v.im[0], pr, pi, e[0][lane]);
    } else {
#pragma unroll
        for (int i = 0; i < C; i += 2)
            pair64(v.re[i], v.im[i], v.re[i + 1], v.im[i + 1], e[i][lane], e[i + 1][lane]);
    }
}

template <int C>
__device__ __forceinline__ void x_odd64(Row<C> &v, const double (*o)[32], int lane)
{
    if constexpr (C == 1) {
        const int src = (lane & 1) ? lane + 1 : lane - 1;
        const double pr = __shfl_sync(FULL, v.re[0], src & 31);
        const double pi = __shfl_sync(FULL, v.im[0], src & 31);
        take64(v.re[0], v.im[0], pr, pi, o[0][lane]);
    } else {
        const double nr = __shfl_down_sync(FULL, v.re[0], 1), ni = __shfl_down_sync(FULL, v.im[0], 1);
        const double pr = __shfl_up_sync(FULL, v.re[C - 1], 1);
        const double pi = __shfl_up_sync(FULL, v.im[C - 1], 1);
#pragma unroll
        for (int i = 1; i + 1 < C; i += 2)
            pair64(v.re[i], v.im[i], v.re[i + 1], v.im[i + 1], o[i][lane], o[i + 1][lane]);
        take64(v.re[C - 1], v.im[C - 1], nr, ni, o[C - 1][lane]);
        take64(v.re[0], v.im[0], pr, pi, o[0][lane]);
    }
}

__device__ __forceinline__ void pair_coef64(int kind, const Sweep64 &s, double &first,
                                            double &second)
{
    first = kind == PAIR_BULK ? s.t : kind == PAIR_LOW ? s.lo : kind == PAIR_HIGH ? s.hi : 0.0;
    second = kind == PAIR_BULK ? s.t : kind == PAIR_LOW ? s.hi : kind == PAIR_HIGH ? s.lo : 0.0;
}

template <int C>
__device__ __forceinline__ void y_pair64(Row<C> &a, Row<C> &b, const Sweep64 &s, int y, int ny)
{
    double ta, tb;
    pair_coef64(pair_kind(y, ny), s, ta, tb);
#pragma unroll
    for (int i = 0; i < C; ++i) pair64(a.re[i], a.im[i], b.re[i], b.im[i], ta, tb);
}

// One row of the lane's columns (zeros off the grid; xg is even or C is 1).
template <int C>
__device__ __forceinline__ void load_row(double (&v)[C], const double *__restrict__ plane, int y,
                                         int xg, const Step64 &p)
{
    const double *src = plane + (int64_t)y * p.pitch + xg;
    const bool row = y >= 0 && y < p.ny;
    if constexpr (C == 1) {
        v[0] = row && xg >= 0 && xg < p.nx ? src[0] : 0.0;
    } else {
#pragma unroll
        for (int i = 0; i < C; i += 2) {
            double2 d = make_double2(0.0, 0.0);
            if (row && xg + i >= 0 && xg + i < p.nx) d = *reinterpret_cast<const double2 *>(src + i);
            v[i] = d.x;
            v[i + 1] = xg + i + 1 < p.nx ? d.y : 0.0;   // (a row's padding holds anything)
        }
    }
}

template <int C>
__global__ void __launch_bounds__(32 * kWarps)
step64_kernel(const __grid_constant__ Step64 p)
{
    __shared__ double coef[kWarps][3][C][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int item = blockIdx.x * kWarps + warp;
    const int sx = item % p.n_strips, rr = item / p.n_strips;
    const int Y0 = rr * p.rows;
    if (Y0 >= p.ny) return;
    const int Y1 = min(Y0 + p.rows, (p.ny + 1) / 2 * 2);
    const int XL = sx * (32 * C - 6) - 4, xg = XL + C * lane;
    // the X sweeps' coefficients: odd, even, odd
    double (*xc)[C][32] = coef[warp];
#pragma unroll
    for (int i = 0; i < C; ++i) {
        // column xg + i is the first (even) or second member of its even pair
        const int x = xg + i, me = x & 1;
        double a, b;
        pair_coef64(pair_kind(x - me, p.nx), p.xe, a, b);
        xc[1][i][lane] = me ? b : a;
        const int od = me ? x : x - 1;   // its odd pair's first column
        pair_coef64(pair_kind(od, p.nx), p.xo1, a, b);
        xc[0][i][lane] = me ? a : b;
        pair_coef64(pair_kind(od, p.nx), p.xo2, a, b);
        xc[2][i][lane] = me ? a : b;
    }
    grid_dep_sync();

    Row<C> a, b, c = {};      // rows y, y + 1 of this pair, y - 1
    double g0[C], s0[C], g1[C], s1[C];   // the table of rows y - 1, y
    load_row<C>(a.re, p.in_re, Y0 - 2, xg, p);
    load_row<C>(a.im, p.in_im, Y0 - 2, xg, p);
    load_row<C>(b.re, p.in_re, Y0 - 1, xg, p);
    load_row<C>(b.im, p.in_im, Y0 - 1, xg, p);
    for (int y = Y0 - 2; y <= Y1; y += 2) {
        // the next pair and the table of the rows it completes
        Row<C> na, nb;
        double h0[C], u0[C], h1[C], u1[C];
        if (y < Y1) {
            load_row<C>(na.re, p.in_re, y + 2, xg, p);
            load_row<C>(na.im, p.in_im, y + 2, xg, p);
            load_row<C>(nb.re, p.in_re, y + 3, xg, p);
            load_row<C>(nb.im, p.in_im, y + 3, xg, p);
            load_row<C>(h0, p.pg, y + 1, xg, p);
            load_row<C>(u0, p.ps, y + 1, xg, p);
            load_row<C>(h1, p.pg, y + 2, xg, p);
            load_row<C>(u1, p.ps, y + 2, xg, p);
        }
        y_pair64<C>(a, b, p.ye, y, p.ny);
        if (y >= Y0) {
            y_pair64<C>(c, a, p.yo1, y - 1, p.ny);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                phase1(c.re[i], c.im[i], g0[i], s0[i]);
                phase1(a.re[i], a.im[i], g1[i], s1[i]);
            }
            y_pair64<C>(c, a, p.yo2, y - 1, p.ny);
            auto out = [&](Row<C> &v, int row) {
                if (row < Y0 || row >= Y1 || row >= p.ny) return;   // the whole warp
                x_odd64<C>(v, xc[0], lane);
                x_even64<C>(v, xc[1], lane);
                if (!p.last) x_odd64<C>(v, xc[2], lane);
                const int64_t o = (int64_t)row * p.pitch + xg;
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    const int k = C * lane + i;   // column of the strip
                    if (k >= 3 && k < 32 * C - 3 && xg + i >= 0 && xg + i < p.nx) {
                        p.out_re[o + i] = v.re[i];
                        p.out_im[o + i] = v.im[i];
                    }
                }
            };
            out(c, y - 1);
            out(a, y);
        }
        c = b;
        a = na;
        b = nb;
#pragma unroll
        for (int i = 0; i < C; ++i) {
            g0[i] = h0[i];
            s0[i] = u0[i];
            g1[i] = h1[i];
            s1[i] = u1[i];
        }
    }
}

// The last even Y sweep and the scale: u <- (scale of the site) times what the
// sweep leaves, from one pair of planes to another or in place.
__global__ void __launch_bounds__(256)
tail64_kernel(const __grid_constant__ Step64 p)
{
    grid_dep_sync();
    for (int q = blockIdx.y; 2 * q < p.ny; q += gridDim.y) {
        const int y = 2 * q;
        const bool two = y + 1 < p.ny;
        double ta, tb;
        pair_coef64(pair_kind(y, p.ny), p.ye, ta, tb);
        const double sa = p.sy[edge_kind(y, p.ny)], sb = p.sy[edge_kind(y + 1, p.ny)];
        for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < p.nx; x += gridDim.x * blockDim.x) {
            const int64_t o = (int64_t)y * p.pitch + x, o1 = o + p.pitch;
            const double sc = p.sx[edge_kind(x, p.nx)];
            double ar = p.in_re[o], ai = p.in_im[o], br = 0.0, bi = 0.0;
            if (two) {
                br = p.in_re[o1];
                bi = p.in_im[o1];
            }
            pair64(ar, ai, br, bi, ta, tb);
            p.out_re[o] = ar * (sc * sa);
            p.out_im[o] = ai * (sc * sa);
            if (two) {
                p.out_re[o1] = br * (sc * sb);
                p.out_im[o1] = bi * (sc * sb);
            }
        }
    }
}

}  // namespace

// Columns per lane and rows per range.  A range of h rows takes (16 h + 24) C
// warp-wide DFMAs per warp, one warp per scheduler in a block; an SM's blocks
// share its units two at a time, and a block that runs alone takes 1.3 times as
// long, since nothing covers its shuffles and loads (2047 x 1536, C = 4: h = 44,
// one block per SM, 136 us per step; h = 22, two, 107 us; h = 16, three, 128 us;
// h = 12, four, 123 us).  The FP64 units alone would need 97 us there.
void plan_step64(Step64 &p, int num_sms, int &cols, int &blocks)
{
    double best = 0.0;
    cols = 0;
    for (int C : {1, 2, 4}) {
        const int strips = (p.nx + 1 + 32 * C - 7) / (32 * C - 6);
        const int pairs = (p.ny + 1) / 2;
        for (int hp = 1; hp <= pairs; hp = hp < 64 ? hp + 1 : hp * 9 / 8) {
            const int64_t items = (int64_t)strips * ((pairs + hp - 1) / hp);
            const int64_t nb = (items + kWarps - 1) / kWarps;
            const int64_t rounds = (nb + num_sms - 1) / num_sms;
            const double t = ((double)rounds + (rounds & 1 ? 0.3 : 0.0)) * (32.0 * hp + 24.0) * C;
            if (cols == 0 || t < best * 0.999) {
                best = t;
                cols = C;
                p.n_strips = strips;
                p.rows = 2 * hp;
                blocks = (int)nb;
            }
        }
    }
}

cudaError_t launch_step64(const Step64 &p, int cols, int blocks, cudaStream_t st)
{
    cudaError_t e = cudaErrorInvalidValue;
    switch (cols) {
    case 1: e = launch_pdl(step64_kernel<1>, blocks, 32 * kWarps, 0, st, p); break;
    case 2: e = launch_pdl(step64_kernel<2>, blocks, 32 * kWarps, 0, st, p); break;
    case 4: e = launch_pdl(step64_kernel<4>, blocks, 32 * kWarps, 0, st, p); break;
    }
    count_launches(1);
    return e;
}

cudaError_t launch_tail64(const Step64 &p, cudaStream_t st)
{
    const int pairs = (p.ny + 1) / 2;
    const dim3 grid((p.nx + 255) / 256, std::min(pairs, 65535));
    const cudaError_t e = launch_pdl(tail64_kernel, grid, 256, 0, st, p);
    count_launches(1);
    return e;
}

}  // namespace ts
