// Register-level pieces of the fused FP32 kernels with scaled rotations
// (fused.cu, tile.cu): a warp holds 128 columns of a row, lane l columns
// 4l .. 4l + 3 as float4 re and im.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"
#include "mbar.cuh"

namespace ts {

constexpr uint32_t FULL = 0xffffffffu;

// Scaled rotations (see pair_s): a warp's coefficients in shared memory, written
// once per segment.  recv has what the columns of a lane receive in each X
// sweep, by the kind of lane: only the lanes at the grid's two edges differ
// from the rest, so a sweep reads 16 bytes, mostly the same ones for the whole
// warp, and strips at the edges cost what the others do.  (With selects instead
// of the table, for edge strips alone, those strips took 1.4 times as long and
// held up the launch.)  lohi, h and f serve the rows at the edges.  Sweep
// k < K + 1 is even sweep k, sweep K + 1 + m odd sweep m.
// Kept small: 2.4 KB is what the fourth-order and the adjoint kernels have
// beside their rings for 8 blocks per SM.  The modes are those of fused.cu.
constexpr int LANE_CLASSES = 5;   // see lane_class
template <int K, int MODE>
struct EdgeTab {
    static constexpr int SWEEPS = 3 * K + 1, CLASSES = LANE_CLASSES;
    static constexpr int SLABS = MODE == 6 ? 2 : 1;   // slabs z and z + 1
    float4 recv[SWEEPS][CLASSES];
    float4 bulk[MODE == 7 ? SWEEPS : 1];   // (-t, -t, t, t) of the sweep's bulk pairs
    float4 hrow[SLABS][CLASSES];   // h and f of the columns of a lane, bulk rows
    float4 frow[MODE == 5 ? K : 1][CLASSES];
    float2 lohi[SWEEPS];
    float h[13 * SLABS];           // per slab: 3 x 3 (rows by columns), the 4 of the bulk
    float f[MODE == 5 ? 9 * K : 1];
};

// Four columns of one row of one state, held by one lane.
struct Frag {
    float4 re, im;
};

__device__ __forceinline__ Frag zero_frag()
{
    Frag f;
    f.re = make_float4(0.f, 0.f, 0.f, 0.f);
    f.im = f.re;
    return f;
}

// Scaled rotations (SC kernels).  A pair rotation divided by its cosine,
//   a' = a + i t b,  b' = b + i t a,   t = tan(theta),
// takes one FMA per real component: 4 per pair against the lifting form's 6
// (and the versine form's 8).  A sweep so applied leaves every paired site
// 1/cos(theta) too large; all sites share that factor, so it commutes with
// every later factor and the launch takes it out once, at the end, by
// a -= h a with h = 1 - (product of the cosines).  A site at the grid's edge
// that a sweep leaves unpaired does not grow: beside its neighbours it is then
// rho = cos(theta) times too small, so its later pairs take the coefficients
// t rho_a / rho_b (into a) and t rho_b / rho_a (into b), and it has its own h.
// These values are the same along an edge and depend on the sweep's place in
// the launch only (ScaledEdge, computed in FP64 from the rounded t).
__device__ __forceinline__ void pair_s(float &ar, float &ai, float &br, float &bi, float ta,
                                       float tb)
{
    const float r = ar, m = ai;
    ar = fmaf(-ta, bi, ar);
    ai = fmaf(ta, br, ai);
    br = fmaf(-tb, m, br);
    bi = fmaf(tb, r, bi);
}

// what a lane's columns receive from their partners in an X sweep
struct Recv {
    float c0, c1, c2, c3;
};

__device__ __forceinline__ void x_even_s(Frag &f, const Recv &e)
{
    pair_s(f.re.x, f.im.x, f.re.y, f.im.y, e.c0, e.c1);
    pair_s(f.re.z, f.im.z, f.re.w, f.im.w, e.c2, e.c3);
}

__device__ __forceinline__ void x_odd_s(Frag &f, const Recv &o)
{
    const float nr = __shfl_down_sync(FULL, f.re.x, 1);
    const float ni = __shfl_down_sync(FULL, f.im.x, 1);
    const float pr = __shfl_up_sync(FULL, f.re.w, 1);
    const float pi = __shfl_up_sync(FULL, f.im.w, 1);
    pair_s(f.re.y, f.im.y, f.re.z, f.im.z, o.c1, o.c2);
    f.re.w = fmaf(-o.c3, ni, f.re.w);
    f.im.w = fmaf(o.c3, nr, f.im.w);
    f.re.x = fmaf(-o.c0, pi, f.re.x);
    f.im.x = fmaf(o.c0, pr, f.im.x);
}

// How a pair lies on the grid, and what its members receive at a sweep whose
// bulk coefficient is t: at an edge the edge member takes lo, its partner hi.
// (A pair with both members on an edge, a side of two sites, is a bulk pair.)
enum : int { PAIR_OFF = 0, PAIR_BULK = 1, PAIR_LOW = 2, PAIR_HIGH = 3 };

__device__ __forceinline__ int pair_kind(int a, int n)
{
    return a < 0 || a + 1 >= n      ? PAIR_OFF
           : n == 2                 ? PAIR_BULK
           : a == 0                 ? PAIR_LOW
           : a + 2 == n             ? PAIR_HIGH
                                    : PAIR_BULK;
}

__device__ __forceinline__ void pair_coef(int kind, float t, float lo, float hi, float &first,
                                          float &second)
{
    first = kind == PAIR_BULK ? t : kind == PAIR_LOW ? lo : kind == PAIR_HIGH ? hi : 0.f;
    second = kind == PAIR_BULK ? t : kind == PAIR_LOW ? hi : kind == PAIR_HIGH ? lo : 0.f;
}

// A site's place along an axis of n sites, for the tables of ScaledEdge:
// 0 bulk, 1 the first site, 2 the last.
__device__ __forceinline__ int edge_kind(int i, int n) { return i == 0 ? 1 : i == n - 1 ? 2 : 0; }

// Packed forms (Cfg<K>::PACKED): the column halves (x, y) and (z, w) of a
// lane's float4 are register pairs, and __ffma2_rn applies one FMA to both
// elements with the rounding of fmaf, so the results are bit for bit those of
// the scalar forms with half the FMA instructions.  Used where the members
// of every pair sit in the same column (Y sweeps, the phase).

__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 join2(float2 lo, float2 hi)
{
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// phase1 on two columns at once: r - g r + s m, m - g m - s r
__device__ __forceinline__ void phase2(float2 &r, float2 &m, float2 g, float2 s)
{
    const float2 ng = make_float2(-g.x, -g.y), ns = make_float2(-s.x, -s.y);
    const float2 nr = __ffma2_rn(s, m, __ffma2_rn(ng, r, r));
    m = __ffma2_rn(ns, r, __ffma2_rn(ng, m, m));
    r = nr;
}

// Scaled Y (or Z) pair rotation of two rows; a receives ta, b receives tb.
template <bool PACKED>
__device__ __forceinline__ void y_pair_s(Frag &a, Frag &b, float ta, float tb)
{
    if constexpr (PACKED) {
        const float2 na = make_float2(-ta, -ta), pa = make_float2(ta, ta);
        const float2 nb = make_float2(-tb, -tb), pb = make_float2(tb, tb);
        auto half = [&](float2 &ar, float2 &ai, float2 &br, float2 &bi) {
            const float2 r = ar, m = ai;
            ar = __ffma2_rn(na, bi, ar);
            ai = __ffma2_rn(pa, br, ai);
            br = __ffma2_rn(nb, m, br);
            bi = __ffma2_rn(pb, r, bi);
        };
        float2 ar = lo2(a.re), ai = lo2(a.im), br = lo2(b.re), bi = lo2(b.im);
        float2 cr = hi2(a.re), ci = hi2(a.im), dr = hi2(b.re), di = hi2(b.im);
        half(ar, ai, br, bi);
        half(cr, ci, dr, di);
        a.re = join2(ar, cr);
        a.im = join2(ai, ci);
        b.re = join2(br, dr);
        b.im = join2(bi, di);
    } else {
        pair_s(a.re.x, a.im.x, b.re.x, b.im.x, ta, tb);
        pair_s(a.re.y, a.im.y, b.re.y, b.im.y, ta, tb);
        pair_s(a.re.z, a.im.z, b.re.z, b.im.z, ta, tb);
        pair_s(a.re.w, a.im.w, b.re.w, b.im.w, ta, tb);
    }
}

// The same for a bulk pair with t = (-t, -t, t, t), packed.
__device__ __forceinline__ void y_pair_bulk(Frag &a, Frag &b, float4 t)
{
    const float2 n = make_float2(t.x, t.y), p = make_float2(t.z, t.w);
    auto half = [&](float2 &ar, float2 &ai, float2 &br, float2 &bi) {
        const float2 r = ar, m = ai;
        ar = __ffma2_rn(n, bi, ar);
        ai = __ffma2_rn(p, br, ai);
        br = __ffma2_rn(n, m, br);
        bi = __ffma2_rn(p, r, bi);
    };
    float2 ar = lo2(a.re), ai = lo2(a.im), br = lo2(b.re), bi = lo2(b.im);
    float2 cr = hi2(a.re), ci = hi2(a.im), dr = hi2(b.re), di = hi2(b.im);
    half(ar, ai, br, bi);
    half(cr, ci, dr, di);
    a.re = join2(ar, cr);
    a.im = join2(ai, ci);
    b.re = join2(br, dr);
    b.im = join2(bi, di);
}

// a -= h a, h per column
__device__ __forceinline__ void unscale(Frag &f, float4 h)
{
    const float2 n0 = make_float2(-h.x, -h.y), n1 = make_float2(-h.z, -h.w);
    const float2 r0 = lo2(f.re), r1 = hi2(f.re), m0 = lo2(f.im), m1 = hi2(f.im);
    f.re = join2(__ffma2_rn(n0, r0, r0), __ffma2_rn(n1, r1, r1));
    f.im = join2(__ffma2_rn(n0, m0, m0), __ffma2_rn(n1, m1, m1));
}

template <bool PACKED>
__device__ __forceinline__ void phase4(Frag &f, float4 g, float4 s)
{
    if constexpr (PACKED) {
    float2 r0 = lo2(f.re), m0 = lo2(f.im), r1 = hi2(f.re), m1 = hi2(f.im);
    phase2(r0, m0, lo2(g), lo2(s));
    phase2(r1, m1, hi2(g), hi2(s));
    f.re = join2(r0, r1);
    f.im = join2(m0, m1);
    } else {
    phase1(f.re.x, f.im.x, g.x, s.x);
    phase1(f.re.y, f.im.y, g.y, s.y);
    phase1(f.re.z, f.im.z, g.z, s.z);
    phase1(f.re.w, f.im.w, g.w, s.w);
    }
}

__device__ __forceinline__ unsigned col_places(int xg, int nx)
{
    unsigned v = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) v |= (unsigned)edge_kind(xg + i, nx) << (2 * i);
    return v;
}

// Lanes with the same class receive the same coefficients in every sweep:
// 0 off the grid, 1 inside, 2 holds the first column, 3 the last, 4 beside the
// lane whose first column is the last one.  (nx >= SCALED_MIN_SIDE: no lane is two of
// these.)
__device__ __forceinline__ int lane_class(int xg, int nx)
{
    const bool L = xg == 0, R = xg < nx && nx <= xg + 4, B = xg + 5 == nx;
    return xg < 0 || xg >= nx ? 0 : L ? 2 : R ? 3 : B ? 4 : 1;
}

// Zeros for the columns past the grid's last one in a lane that starts on the
// grid (xg < nx): a row's padding holds anything.
__device__ __forceinline__ void cut_padding(float4 &v, int xg, int nx)
{
    if (xg + 1 >= nx) v.y = 0.f;
    if (xg + 2 >= nx) v.z = 0.f;
    if (xg + 3 >= nx) v.w = 0.f;
}

// the entries of a 3 x 3 edge table (rows by columns) for one row of the lane
__device__ __forceinline__ float4 edge4(const float *tab, int row, int ny, unsigned cols)
{
    const float *t = tab + 3 * edge_kind(row, ny);
    return make_float4(t[cols & 3], t[cols >> 2 & 3], t[cols >> 4 & 3], t[cols >> 6 & 3]);
}

// h of one row of the lane: as edge4, and in the bulk each column's own (entries
// 9 .. 12 of the table)
__device__ __forceinline__ float4 edge_h(const float *tab, int row, int ny, unsigned cols)
{
    const float *t = tab + 3 * edge_kind(row, ny);
    auto at = [&](int i) {
        const int k = cols >> 2 * i & 3;
        return t[k == 0 && t == tab ? 9 + i : k];
    };
    return make_float4(at(0), at(1), at(2), at(3));
}

// asynchronous 16-byte copies to shared memory
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src)
                 : "memory");
}

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// (zeros unless `in`)
__device__ __forceinline__ void cp_async16_zfill(void *dst, const void *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src),
                 "r"(in ? 16 : 0)
                 : "memory");
}

}  // namespace ts
