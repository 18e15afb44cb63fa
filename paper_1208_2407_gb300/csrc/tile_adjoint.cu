// Backward adjoint steps on tiles held in registers (FP32, scaled rotations):
// the tiles of tile.cu for two states, psi and the costate lambda, that step
// back together, with G's terms conj(lambda~) m formed at every phase point (see
// adjoint.cu and mode 5 of fused.cu, whose sweeps, coefficients and order of
// sums these are).
//
// What bounds it: one launch's latency and then the shared-memory pipe.  A block
// of 12 warps holds 48 rows of 128 columns, 4 rows of both states per warp in
// registers (64 registers), the phase table and the running sums of G in shared
// memory (96 KB).  On small grids the streams' backward kernel spends most of
// its row pairs on pipeline fill (1024^2, depth 3: 4 row pairs of 10 are its
// own).
#include <algorithm>

#include "common.cuh"
#include "ffloat.cuh"
#include "internal.h"
#include "per_device.h"
#include "scaled.cuh"

namespace ts {

namespace {

constexpr int R = 4, W = 12, ROWS = R * W;
constexpr int MAX_K = FUSED_ADJ_MAX_K, SWEEPS = 3 * MAX_K + 1, CLASSES = LANE_CLASSES;

struct Shared {
    float4 recv[SWEEPS][CLASSES];   // as EdgeTab in scaled.cuh
    float4 hrow[CLASSES], frow[MAX_K][CLASSES];
    float2 lohi[SWEEPS];
    float h[13], f[MAX_K][9];
    // first and last row of each warp (psi re, im, lambda re, im), two buffers
    float4 ex[2][W][2][4][32];
    float4 tab[ROWS][2][32];   // gamma_V, s_V
    float4 sum[ROWS][2][32];   // the rows' terms of G so far (re, im)
};

struct Two {
    Frag a, b;   // psi, lambda
};

__device__ __forceinline__ float4 neg4(float4 v) { return make_float4(-v.x, -v.y, -v.z, -v.w); }

// conj(l) m, as adj_term in fused.cu
__device__ __forceinline__ Frag term(const Frag &l, const Frag &m)
{
    auto neg = [](float2 v) { return make_float2(-v.x, -v.y); };
    auto re = [](float2 lr, float2 li, float2 mr, float2 mi) {
        return __ffma2_rn(lr, mr, __fmul2_rn(li, mi));
    };
    auto im = [&](float2 lr, float2 li, float2 mr, float2 mi) {
        return __ffma2_rn(lr, mi, __fmul2_rn(neg(li), mr));
    };
    Frag t;
    t.re = join2(re(lo2(l.re), lo2(l.im), lo2(m.re), lo2(m.im)),
                 re(hi2(l.re), hi2(l.im), hi2(m.re), hi2(m.im)));
    t.im = join2(im(lo2(l.re), lo2(l.im), lo2(m.re), lo2(m.im)),
                 im(hi2(l.re), hi2(l.im), hi2(m.re), hi2(m.im)));
    return t;
}

__device__ __forceinline__ float4 fma4(float4 f, float4 b, float4 a)
{
    return join2(__ffma2_rn(lo2(f), lo2(b), lo2(a)), __ffma2_rn(hi2(f), hi2(b), hi2(a)));
}

struct Ctx {
    int K, yw, ny, warp, lane, cls;
    unsigned cols;
    float te_end, te_mid, to_a, to_b;
};

template <bool EDGE>
__device__ __forceinline__ void steps(Two (&st)[R], const Ctx &c, Shared &sh)
{
    const int K = c.K;
    auto even_x = [&](int k) {
        const float4 v = sh.recv[k][c.cls];
        const Recv e = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int r = 0; r < R; ++r) {
            x_even_s(st[r].a, e);
            x_even_s(st[r].b, e);
        }
    };
    auto odd_x = [&](int m) {
        const float4 v = sh.recv[K + 1 + m][c.cls];
        const Recv o = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int r = 0; r < R; ++r) {
            x_odd_s(st[r].a, o);
            x_odd_s(st[r].b, o);
        }
    };
    auto y_pair = [&](Two &a, Two &b, int y, int i, float t) {
        float ta = t, tb = t;
        if constexpr (EDGE) {
            const float2 lh = sh.lohi[i];
            pair_coef(pair_kind(y, c.ny), t, lh.x, lh.y, ta, tb);
        }
        y_pair_s<true>(a.a, b.a, ta, tb);
        y_pair_s<true>(a.b, b.b, ta, tb);
    };
    auto even_y = [&](int k, float t) {
#pragma unroll
        for (int r = 0; r < R; r += 2) y_pair(st[r], st[r + 1], c.yw + r, k, t);
    };
    Two top, bot;   // the rows above and below this warp's
    auto odd_y = [&](int m, float t) {
        y_pair(top, st[0], c.yw - 1, K + 1 + m, t);
#pragma unroll
        for (int r = 1; r < R - 1; r += 2) y_pair(st[r], st[r + 1], c.yw + r, K + 1 + m, t);
        y_pair(st[R - 1], bot, c.yw + R - 1, K + 1 + m, t);
    };
    const float4 (*tab)[2][32] = sh.tab + R * c.warp;
    float4 (*sum)[2][32] = sh.sum + R * c.warp;
    auto phase = [&](Two &v, int r) {   // backward: exp(+i V dt), sine -s_V
        const float4 g = tab[r][0][c.lane], s = neg4(tab[r][1][c.lane]);
        phase4<true>(v.a, g, s);
        phase4<true>(v.b, g, s);
    };
    even_x(0);
    odd_x(0);
    even_y(0, c.te_end);
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
        // (a buffer is written again two steps later: the barrier between
        // follows every read of it)
        float4 (*ex)[2][4][32] = sh.ex[k & 1];
        auto put = [&](int side, const Two &v) {
            ex[c.warp][side][0][c.lane] = v.a.re;
            ex[c.warp][side][1][c.lane] = v.a.im;
            ex[c.warp][side][2][c.lane] = v.b.re;
            ex[c.warp][side][3][c.lane] = v.b.im;
        };
        auto get = [&](int warp, int side) {
            Two v;
            v.a.re = ex[warp][side][0][c.lane];
            v.a.im = ex[warp][side][1][c.lane];
            v.b.re = ex[warp][side][2][c.lane];
            v.b.im = ex[warp][side][3][c.lane];
            return v;
        };
        put(0, st[0]);
        put(1, st[R - 1]);
        if (k == 0) cp_async_wait_all();   // this thread's part of the table
        __syncthreads();
        top = bot = Two{zero_frag(), zero_frag()};
        if (c.warp > 0) top = get(c.warp - 1, 1);
        if (c.warp < W - 1) bot = get(c.warp + 1, 0);
        odd_y(2 * k, c.to_a);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const Frag t = term(st[r].b, st[r].a);
            const float4 f = EDGE ? edge4(sh.f[k], c.yw + r, c.ny, c.cols) : sh.frow[k][c.cls];
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            sum[r][0][c.lane] = fma4(f, t.re, k ? sum[r][0][c.lane] : z);
            sum[r][1][c.lane] = fma4(f, t.im, k ? sum[r][1][c.lane] : z);
        }
        if (c.warp > 0) phase(top, -1);
#pragma unroll
        for (int r = 0; r < R; ++r) phase(st[r], r);
        if (c.warp < W - 1) phase(bot, R);
        odd_y(2 * k + 1, c.to_b);
        if (k < K - 1) {
            odd_x(2 * k + 1);
            even_x(k + 1);
            odd_x(2 * k + 2);
            even_y(k + 1, c.te_mid);
        }
    }
    even_y(K, c.te_end);
    odd_x(2 * K - 1);
    even_x(K);
}

__global__ void __launch_bounds__(32 * W, 1)
tile_adjoint_kernel(const TileAdjoint p, const __grid_constant__ ScaledEdge ed,
                    const float te_end, const float te_mid, const float to_a, const float to_b,
                    int K, int n_strips)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Shared &sh = *reinterpret_cast<Shared *>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sx = blockIdx.x % n_strips, ty = blockIdx.x / n_strips;
    const int halo = depth_halo(K);
    const int y0 = ty * (ROWS - 4 * K);
    const int XL = sx * strip_valid(halo), xg = XL + 4 * lane;
    const unsigned cols = col_places(xg, p.nx);
    const Ctx c = {K, y0 + R * warp, p.ny, warp, lane, lane_class(xg, p.nx), cols,
                   te_end, te_mid, to_a, to_b};
    // the edge values (as in tile.cu)
    for (int i = threadIdx.x; i < 3 * K + 1; i += 32 * W)
        sh.lohi[i] = i <= K ? make_float2(ed.elo[i], ed.ehi[i])
                            : make_float2(ed.olo[i - K - 1], ed.ohi[i - K - 1]);
    if (threadIdx.x < 13)
        sh.h[threadIdx.x] = threadIdx.x < 9 ? ed.h[threadIdx.x] : ed.hb[0][threadIdx.x - 9];
    if (threadIdx.x < 9 * K) sh.f[threadIdx.x / 9][threadIdx.x % 9] = ed.f[threadIdx.x / 9][threadIdx.x % 9];
    __syncthreads();
    for (int i = warp; i < 3 * K + 1; i += W) {
        const float2 lh = sh.lohi[i];
        float4 v;
        float other;
        if (i <= K) {
            const float t = i == 0 || i == K ? te_end : te_mid;
            pair_coef(pair_kind(xg, p.nx), t, lh.x, lh.y, v.x, v.y);
            pair_coef(pair_kind(xg + 2, p.nx), t, lh.x, lh.y, v.z, v.w);
        } else {
            const float t = (i - K - 1) & 1 ? to_b : to_a;
            pair_coef(pair_kind(xg + 1, p.nx), t, lh.x, lh.y, v.y, v.z);
            pair_coef(pair_kind(xg + 3, p.nx), t, lh.x, lh.y, v.w, other);
            pair_coef(pair_kind(xg - 1, p.nx), t, lh.x, lh.y, other, v.x);
        }
        sh.recv[i][c.cls] = v;   // the same value from every lane of the class
    }
    if (warp == 0) sh.hrow[c.cls] = edge_h(sh.h, -1, p.ny, cols);
    if (warp >= 1 && warp <= K) sh.frow[warp - 1][c.cls] = edge4(sh.f[warp - 1], -1, p.ny, cols);
    __syncthreads();
    grid_dep_sync();

    // the states, and the table into shared memory (zeros off the grid)
    Two st[R];
    const bool col = xg < p.nx;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int y = c.yw + r;
        const bool in = col && y < p.ny;
        const int64_t o = in ? (int64_t)y * p.pitch + xg : 0;
        auto load = [&](const float *plane) {
            float4 v = in ? *reinterpret_cast<const float4 *>(plane + o) : z;
            cut_padding(v, xg, p.nx);
            return v;
        };
        st[r].a.re = load(p.in[0]);
        st[r].a.im = load(p.in[1]);
        st[r].b.re = load(p.in[2]);
        st[r].b.im = load(p.in[3]);
        cp_async16_zfill(&sh.tab[R * warp + r][0][lane], p.pg + o, in);
        cp_async16_zfill(&sh.tab[R * warp + r][1][lane], p.ps + o, in);
    }
    cp_async_commit();
    // the table's padding, as in tile.cu; a lane reads only the columns that it
    // (in this or a neighbouring warp) has copied
    if (xg < p.nx && xg + 4 > p.nx) {
        cp_async_wait_all();
        for (int r = 0; r < R; ++r)
            for (int i = 0; i < 2; ++i) cut_padding(sh.tab[R * warp + r][i][lane], xg, p.nx);
    }

    const bool edge = y0 <= 0 || y0 + ROWS >= p.ny;   // the same for the whole block
    if (edge)
        steps<true>(st, c, sh);
    else
        steps<false>(st, c, sh);

    grid_dep_launch();
    const bool store = col && (4 * lane >= halo || sx == 0) &&
                       (4 * lane < FUSED_BOX_COLS - halo || XL + FUSED_BOX_COLS >= p.nx);
    const bool first = ty == 0, last = y0 + ROWS >= p.ny;
    bool mine[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int t = R * warp + r;
        mine[r] = store && (t >= 2 * K || first) && (t < ROWS - 2 * K || last) && y0 + t < p.ny;
    }
    // G's rows, all loads before the first store (one wait for them, not eight)
    float4 g[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            g[r][i] = mine[r] ? *reinterpret_cast<const float4 *>(
                                    p.g[i] + (int64_t)(c.yw + r) * p.pitch + xg)
                              : z;
    const float4 hb = sh.hrow[c.cls];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float4 h = edge ? edge_h(sh.h, c.yw + r, p.ny, cols) : hb;
        unscale(st[r].a, h);
        unscale(st[r].b, h);
        if (!mine[r]) continue;
        const int64_t o = (int64_t)(c.yw + r) * p.pitch + xg;
        *reinterpret_cast<float4 *>(p.out[0] + o) = st[r].a.re;
        *reinterpret_cast<float4 *>(p.out[1] + o) = st[r].a.im;
        *reinterpret_cast<float4 *>(p.out[2] + o) = st[r].b.re;
        *reinterpret_cast<float4 *>(p.out[3] + o) = st[r].b.im;
    }
    // G += the rows' terms, in double-float (as adj_commit in fused.cu)
    auto acc = [](float &hi, float &lo, float v) {
        FF s = two_sum(hi, v);
        s.lo += lo;
        s = fast_two_sum(s.hi, s.lo);
        hi = s.hi;
        lo = s.lo;
    };
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (!mine[r]) continue;
        const int64_t o = (int64_t)(c.yw + r) * p.pitch + xg;
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            const float4 v = sh.sum[R * warp + r][i / 2][lane];
            float4 hi = g[r][i], lo = g[r][i + 1];
            acc(hi.x, lo.x, v.x);
            acc(hi.y, lo.y, v.y);
            acc(hi.z, lo.z, v.z);
            acc(hi.w, lo.w, v.w);
            *reinterpret_cast<float4 *>(p.g[i] + o) = hi;
            *reinterpret_cast<float4 *>(p.g[i + 1] + o) = lo;
        }
    }
}

}  // namespace

static int tile_blocks_of(int K, int nx, int ny)
{
    const int rows = ROWS - 4 * K;
    return strip_count(nx, depth_halo(K)) * (ny <= ROWS ? 1 : (ny - 4 * K + rows - 1) / rows);
}

// Up to two rounds of one block per SM at depths 3 and 4, one at depth 2, none
// at depth 1: a launch spends 7 us on its loads and stores (72 B per site) and
// 2.5 us per step and round.  Us per step, tiles and streams: 512^2 depth 1 10.2
// and 7.9, depth 2 6.4 and 7.9, depth 3 5.0 and 6.8; 1024^2 depth 2 11.4 and
// 10.6, depth 3 8.8 and 9.2; 1500^2 (4 rounds) depth 3 20.3 and 13.5.
bool tile_adjoint_serves(int K, int nx, int ny)
{
    return K >= 2 && K <= MAX_K && tile_blocks_of(K, nx, ny) <= (K == 2 ? 1 : 2) * num_sms();
}

cudaError_t launch_tile_adjoint(int K, const TileAdjoint &p, const ScaledCoef &c, cudaStream_t st)
{
    if (K < 1 || K > MAX_K) return cudaErrorInvalidValue;
    static PerDevice<cudaError_t> attr;
    cudaError_t e = attr.get([] {
        return cudaFuncSetAttribute(tile_adjoint_kernel,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(Shared));
    });
    if (e != cudaSuccess) return e;
    e = launch_pdl(tile_adjoint_kernel, tile_blocks_of(K, p.nx, p.ny), 32 * W, sizeof(Shared), st, p,
                   c.edge, c.te_end, c.te_mid, c.to_a, c.to_b, K,
                   strip_count(p.nx, depth_halo(K)));
    count_launches(1);
    return e;
}

}  // namespace ts
