// Fused second-order Trotter-Suzuki steps on tiles held in registers (FP32,
// scaled rotations).
//
// The warp streams of fused.cu walk down a strip: a warp's row pairs depend on
// one another, and a grid of a few hundred rows gives each warp a short chain
// that is mostly pipeline fill, run at one instruction in four cycles.  Here a
// block holds a tile of 128 columns by R W rows in registers, R = 4 or 8 rows
// per warp with their phase tables, and applies each sweep to all of them at
// once.  The sweeps,
// their order and their coefficients are those of the warp streams at the same
// depth K, so the results are bit for bit the same.
//
// What bounds it: the latency of one launch.  A step takes 0.9 us however few
// rows a warp holds (512^2: 6.8 us per launch of depth 4, 2.4 us of it the
// launch, the loads and the stores; 14.7 us with warp streams); one to three
// warps per scheduler issue one instruction in 2 to 3.5 cycles.  The table in
// shared memory instead of registers was 10 % slower up to 1500^2 (at 1024^2
// alone, where 12 warps of 8 rows then make one round, it gained 12 %).
//
// X sweeps stay in a row (shuffles at the lanes' borders).  Even Y pairs lie in
// a warp; odd ones also join the last row of a warp and the first of the next.
// Between two even Y sweeps come odd sweep, phase, odd sweep, all on the same
// pairs: each warp takes a copy of the neighbouring rows (through shared
// memory, one barrier per step) and applies the three to them as well.
//
// A tile reads 2K halo rows and roundup(2K, 4) halo columns per side, where the
// grid goes on, and stores the rest.  Rows and columns off the grid are zeros whose pairs have
// coefficient zero.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "per_device.h"
#include "scaled.cuh"

namespace ts {

namespace {

constexpr int SWEEPS = 3 * TILE_MAX_K + 1, CLASSES = LANE_CLASSES;

// One grid of a launch.
struct TileGrid {
    const float *in_re, *in_im, *pg, *ps;
    float *out_re, *out_im;
    int nx, ny;
    int64_t pitch;
    float te_end, te_mid, to_a, to_b;
};

template <int R, int W>
struct TileShared {
    // tables of the rows above and below a warp: in registers, but for the shapes
    // of 8 rows and more than 8 warps (168 registers: they would spill)
    static constexpr bool TABS = R == 8 && W > 8;
    float4 recv[SWEEPS][CLASSES];   // as EdgeTab in scaled.cuh
    float4 hrow[CLASSES];
    float2 lohi[SWEEPS];
    float h[13];
    // first and last row of each warp (re, im), two buffers
    float4 ex[2][W][2][2][32];
    float4 tab[TABS ? W : 1][2][2][32];
};

// What every step of a tile needs besides the rows.
struct TileCtx {
    int K, yw, ny, warp, lane, cls;
    float te_end, te_mid, to_a, to_b;
};

template <int R, int W, bool EDGE>
__device__ __forceinline__ void tile_steps(Frag (&st)[R], const float4 (&tg)[R + 2],
                                           const float4 (&tv)[R + 2], const TileCtx &c,
                                           TileShared<R, W> &sh)
{
    const int K = c.K;
    auto even_x = [&](int k) {
        const float4 v = sh.recv[k][c.cls];
        const Recv e = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int r = 0; r < R; ++r) x_even_s(st[r], e);
    };
    auto odd_x = [&](int m) {
        const float4 v = sh.recv[K + 1 + m][c.cls];
        const Recv o = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int r = 0; r < R; ++r) x_odd_s(st[r], o);
    };
    // the pair of rows (y, y + 1); i: the sweep's entry in lohi
    auto y_pair = [&](Frag &a, Frag &b, int y, int i, float t) {
        float ta = t, tb = t;
        if constexpr (EDGE) {
            const float2 lh = sh.lohi[i];
            pair_coef(pair_kind(y, c.ny), t, lh.x, lh.y, ta, tb);
        }
        y_pair_s<true>(a, b, ta, tb);
    };
    auto even_y = [&](int k, float t) {
#pragma unroll
        for (int r = 0; r < R; r += 2) y_pair(st[r], st[r + 1], c.yw + r, k, t);
    };
    Frag top, bot;   // the rows above and below this warp's
    auto odd_y = [&](int m, float t) {
        y_pair(top, st[0], c.yw - 1, K + 1 + m, t);
#pragma unroll
        for (int r = 1; r < R - 1; r += 2) y_pair(st[r], st[r + 1], c.yw + r, K + 1 + m, t);
        y_pair(st[R - 1], bot, c.yw + R - 1, K + 1 + m, t);
    };
    even_x(0);
    odd_x(0);
    even_y(0, c.te_end);
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
        // (a buffer is written again two steps later: the barrier between
        // follows every read of it)
        float4 (*ex)[2][2][32] = sh.ex[k & 1];
        ex[c.warp][0][0][c.lane] = st[0].re;
        ex[c.warp][0][1][c.lane] = st[0].im;
        ex[c.warp][1][0][c.lane] = st[R - 1].re;
        ex[c.warp][1][1][c.lane] = st[R - 1].im;
        __syncthreads();
        top = bot = zero_frag();
        if (c.warp > 0) {
            top.re = ex[c.warp - 1][1][0][c.lane];
            top.im = ex[c.warp - 1][1][1][c.lane];
        }
        if (c.warp < W - 1) {
            bot.re = ex[c.warp + 1][0][0][c.lane];
            bot.im = ex[c.warp + 1][0][1][c.lane];
        }
        odd_y(2 * k, c.to_a);
        auto phase_out = [&](Frag &f, int i) {   // the row above (0) or below (1)
            if constexpr (TileShared<R, W>::TABS)
                phase4<true>(f, sh.tab[c.warp][i][0][c.lane], sh.tab[c.warp][i][1][c.lane]);
            else
                phase4<true>(f, tg[i * (R + 1)], tv[i * (R + 1)]);
        };
        phase_out(top, 0);
#pragma unroll
        for (int r = 0; r < R; ++r) phase4<true>(st[r], tg[r + 1], tv[r + 1]);
        phase_out(bot, 1);
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

// K steps of the tile (sx, ty) of grid g: ed has the edge values at depth K.
template <int R, int W>
__device__ __forceinline__ void run_tile(const TileGrid &g, const ScaledEdge *ed, int K, int sx,
                                         int ty, TileShared<R, W> &sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int halo = depth_halo(K);
    const int rows = R * W - 4 * K;              // rows stored per tile
    const int y0 = ty * rows;                    // the tile's first row (even)
    const int XL = sx * strip_valid(halo), xg = XL + 4 * lane;   // the lane's first column
    TileCtx c = {K, y0 + R * warp, g.ny, warp, lane, lane_class(xg, g.nx),
                 g.te_end, g.te_mid, g.to_a, g.to_b};

    // the edge values (see run_segment in fused.cu), one warp per sweep in turn;
    // they come from the kernel's parameters, so they need not wait for the
    // kernel before
    const unsigned cols = col_places(xg, g.nx);
    for (int i = threadIdx.x; i < 3 * K + 1; i += 32 * W)
        sh.lohi[i] = i <= K ? make_float2(ed->elo[i], ed->ehi[i])
                            : make_float2(ed->olo[i - K - 1], ed->ohi[i - K - 1]);
    if (threadIdx.x < 13)
        sh.h[threadIdx.x] = threadIdx.x < 9 ? ed->h[threadIdx.x] : ed->hb[0][threadIdx.x - 9];
    __syncthreads();
    for (int i = warp; i < 3 * K + 1; i += W) {
        const float2 lh = sh.lohi[i];
        float4 v;
        float other;
        if (i <= K) {
            const float t = i == 0 || i == K ? g.te_end : g.te_mid;
            pair_coef(pair_kind(xg, g.nx), t, lh.x, lh.y, v.x, v.y);
            pair_coef(pair_kind(xg + 2, g.nx), t, lh.x, lh.y, v.z, v.w);
        } else {
            const float t = (i - K - 1) & 1 ? g.to_b : g.to_a;
            pair_coef(pair_kind(xg + 1, g.nx), t, lh.x, lh.y, v.y, v.z);
            pair_coef(pair_kind(xg + 3, g.nx), t, lh.x, lh.y, v.w, other);
            pair_coef(pair_kind(xg - 1, g.nx), t, lh.x, lh.y, other, v.x);
        }
        sh.recv[i][c.cls] = v;   // the same value from every lane of the class
    }
    if (warp == 0) sh.hrow[c.cls] = edge_h(sh.h, -1, g.ny, cols);
    __syncthreads();
    grid_dep_sync();

    // the state and the table (the rows above and below take part in the phase)
    Frag st[R];
    float4 tg[R + 2], tv[R + 2];
    const bool col = xg >= 0 && xg < g.nx;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = -1; r <= R; ++r) {
        const int y = c.yw + r;
        const bool in = col && y >= 0 && y < g.ny;
        const int64_t o = (int64_t)y * g.pitch + xg;
        if (r >= 0 && r < R) {
            st[r].re = in ? *reinterpret_cast<const float4 *>(g.in_re + o) : z;
            st[r].im = in ? *reinterpret_cast<const float4 *>(g.in_im + o) : z;
        }
        tg[r + 1] = in ? *reinterpret_cast<const float4 *>(g.pg + o) : z;
        tv[r + 1] = in ? *reinterpret_cast<const float4 *>(g.ps + o) : z;
    }
    // a lane across the grid's last column: its further columns are padding,
    // which holds anything, in the table too (NaN there would reach the last
    // column: a pair that the grid's edge cuts takes 0 times its partner)
    if (xg < g.nx && xg + 4 > g.nx) {
#pragma unroll
        for (int r = -1; r <= R; ++r) {
            if (r >= 0 && r < R) {
                cut_padding(st[r].re, xg, g.nx);
                cut_padding(st[r].im, xg, g.nx);
            }
            cut_padding(tg[r + 1], xg, g.nx);
            cut_padding(tv[r + 1], xg, g.nx);
        }
    }
    if constexpr (TileShared<R, W>::TABS) {   // (read by the lane that writes it)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            sh.tab[warp][i][0][lane] = tg[i * (R + 1)];
            sh.tab[warp][i][1][lane] = tv[i * (R + 1)];
        }
    }
    const bool edge = y0 <= 0 || y0 + R * W >= g.ny;   // the same for the whole block
    if (edge)
        tile_steps<R, W, true>(st, tg, tv, c, sh);
    else
        tile_steps<R, W, false>(st, tg, tv, c, sh);

    grid_dep_launch();
    const bool store = col && (4 * lane >= halo || sx == 0) &&
                       (4 * lane < FUSED_BOX_COLS - halo || XL + FUSED_BOX_COLS >= g.nx);
    const bool first = ty == 0, last = y0 + R * W >= g.ny;   // tiles at the grid's top and bottom
    const float4 hb = sh.hrow[c.cls];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int t = R * warp + r, y = y0 + t;
        unscale(st[r], edge ? edge_h(sh.h, y, g.ny, cols) : hb);
        if (store && (t >= 2 * K || first) && (t < R * W - 2 * K || last) && y < g.ny) {
            const int64_t o = (int64_t)y * g.pitch + xg;
            *reinterpret_cast<float4 *>(g.out_re + o) = st[r].re;
            *reinterpret_cast<float4 *>(g.out_im + o) = st[r].im;
        }
    }
}

// Block b of a grid's launch takes tile (b mod strips, b / strips).
template <int R, int W>
__global__ void __launch_bounds__(32 * W, R == 4 && W == 8 ? 2 : 1)
tile_kernel(const TileGrid g, const __grid_constant__ ScaledEdge ed, int K, int n_strips)
{
    extern __shared__ __align__(16) unsigned char smem[];
    run_tile<R, W>(g, &ed, K, blockIdx.x % n_strips, blockIdx.x / n_strips,
                   *reinterpret_cast<TileShared<R, W> *>(smem));
}

// Many grids in one launch: tab[i].begin is grid i's first block.
template <int R, int W>
__global__ void __launch_bounds__(32 * W, R == 4 && W == 8 ? 2 : 1)
tile_multi_kernel(const EpochEntry *__restrict__ tab, int n_grids, int K, int flip)
{
    extern __shared__ __align__(16) unsigned char smem[];
    grid_dep_sync();   // the table and the descriptors are in device memory
    int lo = 0, hi = n_grids - 1;
    while (lo < hi) {   // the last entry whose first block is <= blockIdx.x
        const int mid = (lo + hi + 1) >> 1;
        if (tab[mid].begin <= blockIdx.x)
            lo = mid;
        else
            hi = mid - 1;
    }
    const EpochEntry e = tab[lo];
    const GridDesc *d = e.desc;
    const int cur = e.cur0 ^ flip;
    const ScaledCoef &c = d->sc[K - 1];
    const TileGrid g = {d->re[cur], d->im[cur], d->pg, d->ps, d->re[cur ^ 1], d->im[cur ^ 1],
                        d->nx, d->ny, d->pitch, c.te_end, c.te_mid, c.to_a, c.to_b};
    const int strips = strip_count(d->nx, depth_halo(K)), b = (int)(blockIdx.x - e.begin);
    run_tile<R, W>(g, &c.edge, K, b % strips, b / strips, *reinterpret_cast<TileShared<R, W> *>(smem));
}

template <int R, int W>
cudaError_t launch_one(int K, const TileLaunch &a, int blocks, int strips, cudaStream_t st)
{
    const ScaledCoef &c = *a.sc;
    const TileGrid g = {a.in_re, a.in_im, a.pg, a.ps, a.out_re, a.out_im, a.nx, a.ny, a.pitch,
                        c.te_end, c.te_mid, c.to_a, c.to_b};
    constexpr int smem = (int)sizeof(TileShared<R, W>);
    static PerDevice<cudaError_t> attr;
    cudaError_t e = attr.get([] {
        return cudaFuncSetAttribute(tile_kernel<R, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    smem);
    });
    if (e != cudaSuccess) return e;
    e = launch_pdl(tile_kernel<R, W>, blocks, 32 * W, smem, st, g, c.edge, K, strips);
    count_launches(1);
    return e;
}

template <int R, int W>
cudaError_t prepare_multi()
{
    static PerDevice<cudaError_t> attr;
    return attr.get([] {
        return cudaFuncSetAttribute(tile_multi_kernel<R, W>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(TileShared<R, W>));
    });
}

template <int R, int W>
cudaError_t launch_many(int K, const EpochEntry *tab, int n, int blocks, int flip, cudaStream_t st)
{
    cudaError_t e = prepare_multi<R, W>();
    if (e == cudaSuccess)
        e = launch_pdl(tile_multi_kernel<R, W>, blocks, 32 * W, sizeof(TileShared<R, W>), st, tab, n,
                       K, flip);
    count_launches(1);
    return e;
}

// The tile shapes: rows per warp and warps per block.
struct Shape {
    int r, w;
};
constexpr Shape shapes[TILE_SHAPES] = {{4, 8}, {4, 10}, {8, 8}, {8, 10}};

int64_t tiles_of(int K, const Shape &s, int nx, int ny)
{
    // rows of tiles as strips of columns: the first and the last store their
    // halo at the grid's edge
    const int rows = s.r * s.w - 4 * K;
    const int64_t down = ny <= s.r * s.w ? 1 : (ny - 4 * K + rows - 1) / rows;
    return strip_count(nx, depth_halo(K)) * down;
}

}  // namespace

int num_sms()
{
    static PerDevice<int> n;
    return n.get([] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            v = 1;
        return v;
    });
}

int tile_blocks(int K, int shape, int nx, int ny) { return (int)tiles_of(K, shapes[shape], nx, ny); }

// Tiles or warp streams?  Tiles of 64 rows in at most 1, 2, 2 and 3 rounds of one
// block per SM at depths 1 to 4.  A tile recomputes its halo (at depth 4 three
// quarters of its rows and 7/8 of its columns are stored), so once the SMs are full
// the streams win; at a smaller depth sooner, since a launch has less work to set
// against its loads.  Measured, us per launch, tiles / streams:
//   depth 4: 512^2 6.7 / 14.7, 1024^2 12.2 / 19.1 (1 round of 80 rows), 1300^2 21.1 /
//     22.4 (3), 1500^2 22.2 / 25.0 (3), 1600^2 28.2 / 26.2 (4), 2048^2 43 / 33 (6);
//   depth 3: 1300^2 13.7 / 16.6 (2), 1400^2 18.6 / 18.1 (3), 1600^2 23.5 / 19.6 (4);
//   depth 2: 1400^2 11.7 / 13.9 (2), 1500^2 14.8 / 15.6 and 1024 x 2048 17.3 / 14.8
//     (3), 1700^2 18.8 / 17.6 (4);
//   depth 1: 900^2 4.9 / 6.4 (1), 1024^2 7.2 / 7.2 and 1500^2 10.6 / 10.1 (2 and 3).
//
// Which shape?  The least of time = 1.3 + rounds (g + s K) us, fitted to
// launches from 128^2 to 1500^2 at depths 1 to 4; two blocks of the first shape
// share an SM, a second round costs it half.  The last shape, 80 rows, has three
// warps on two of the schedulers and is worth it where it makes one round of what
// tiles of 64 rows make two: 1024^2 at depth 4 14.9 -> 12.2 us (13.2 with 12
// warps), 1000^2 14.4 -> 12.1, 1024^2 at depth 3 12.3 -> 10.4.
int tile_shape(int K, int n, const int *nx, const int *ny, bool multi)
{
    if (K < 1 || K > TILE_MAX_K) return -1;
    static const double g[TILE_SHAPES] = {1.1, 1.1, 1.8, 3.65}, s[TILE_SHAPES] = {0.9, 1.06, 1.28, 1.8};
    const int64_t sms = num_sms();
    int best = -1;
    double best_us = 0.0;
    for (int i : {2, 3, 1, 0}) {   // tiles of 64 rows first: they decide
        if (i == 3 && multi) continue;   // (spills in that kernel)
        int64_t tiles = 0;
        for (int k = 0; k < n; ++k) tiles += tiles_of(K, shapes[i], nx[k], ny[k]);
        if (i == 2 && tiles > (K + 2) / 2 * sms) return -1;
        double rounds = (double)((tiles + sms - 1) / sms);
        if (i == 0 && rounds > 1.0) rounds *= 0.75;
        const double us = rounds * (g[i] + s[i] * K);
        if (best < 0 || us < best_us) {
            best = i;
            best_us = us;
        }
    }
    return best;
}

cudaError_t launch_tile(int K, int shape, const TileLaunch &a, cudaStream_t st)
{
    if (K < 1 || K > TILE_MAX_K || !a.sc) return cudaErrorInvalidValue;
    const int strips = strip_count(a.nx, depth_halo(K));
    const int blocks = tile_blocks(K, shape, a.nx, a.ny);
    switch (shape) {
    case 0: return launch_one<4, 8>(K, a, blocks, strips, st);
    case 1: return launch_one<4, 10>(K, a, blocks, strips, st);
    case 2: return launch_one<8, 8>(K, a, blocks, strips, st);
    case 3: return launch_one<8, 10>(K, a, blocks, strips, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t tile_multi_prepare()
{
    num_sms();
    cudaError_t e = prepare_multi<4, 8>();
    if (e == cudaSuccess) e = prepare_multi<4, 10>();
    if (e == cudaSuccess) e = prepare_multi<8, 8>();
    return e;
}

cudaError_t launch_tile_multi(int K, int shape, const EpochEntry *tab, int n, int blocks, int flip,
                              cudaStream_t st)
{
    if (K < 1 || K > TILE_MAX_K || n < 1 || blocks < 1) return cudaErrorInvalidValue;
    switch (shape) {
    case 0: return launch_many<4, 8>(K, tab, n, blocks, flip, st);
    case 1: return launch_many<4, 10>(K, tab, n, blocks, flip, st);
    case 2: return launch_many<8, 8>(K, tab, n, blocks, flip, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace ts
