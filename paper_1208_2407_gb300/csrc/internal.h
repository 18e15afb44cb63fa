// Internal interface between the C-ABI layer (api.cu) and the kernel files.
// Not installed; the public boundary is include/trotter.h.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#ifdef __CUDACC__
#define TS_HD __host__ __device__
#else
#define TS_HD
#endif

struct ts_grid;

namespace ts {

// Error bits written by kernels into the grid's device error word.
enum : int { ERRBIT_WAIT_TIMEOUT = 1, ERRBIT_BAD_CONFIG = 2 };

// Number of FP64 quantities the observables reduction produces per block.
constexpr int OBS_Q = 7;
constexpr int OBS_Q3 = 9;   // 3-D grids: the 7 quantities plus sum z p and sum z^2 p
constexpr int OBS_MAX_BLOCKS = 1024;

// --- conversions, tables, plain path (plain.cu) ---------------------------
// dense (nx*ny, src type) -> pitched plane of dst type
cudaError_t launch_convert_in(const void *src, bool src_f64, void *dst, bool dst_f64,
                              int nx, int ny, int64_t pitch, cudaStream_t st);
// pitched plane -> dense
cudaError_t launch_convert_out(const void *src, bool src_f64, void *dst, bool dst_f64,
                               int nx, int ny, int64_t pitch, cudaStream_t st);
// the same for two arrays (re, im) in one launch
cudaError_t launch_convert_in2(const void *src0, const void *src1, bool src_f64, void *dst0,
                               void *dst1, bool dst_f64, int nx, int ny, int64_t pitch,
                               cudaStream_t st);
// (launch_convert_out2 writes nothing if *err is not 0 when it runs)
cudaError_t launch_convert_out2(const void *src0, const void *src1, bool src_f64, void *dst0,
                                void *dst1, bool dst_f64, int nx, int ny, int64_t pitch,
                                const int *err, cudaStream_t st);
// V (dense FP64) -> (gamma_V, s_V, V) pitched planes of the grid's type
cudaError_t launch_phase_table(const double *V, void *pg, void *ps, void *vplane, bool f64,
                               int nx, int ny, int64_t pitch, double dt, cudaStream_t st);
// one sweep along x (axis 0) or y (axis 1) of the given parity, in place;
// (g, s) versine coefficients, or with lift (FP64 only) (tan(theta/2), s)
cudaError_t launch_plain_sweep(void *re, void *im, bool f64, int nx, int ny, int64_t pitch,
                               int axis, int parity, double g, double s, cudaStream_t st,
                               bool lift = false);
// the diagonal phase exp(-i V dt) from the stored table, in place
cudaError_t launch_plain_phase(void *re, void *im, const void *pg, const void *ps, bool f64,
                               int nx, int ny, int64_t pitch, cudaStream_t st);
// psi <- psi exp(-i adt V1) (the drive term of a time-dependent potential),
// in place; V1 is a pitched plane of the grid's dtype.
cudaError_t launch_plain_drive(void *re, void *im, const void *v1, bool f64, int nx, int ny,
                               int64_t pitch, double adt, cudaStream_t st);

// --- failure path of the bounded waits (selftest.cu) ----------------------
// One warp waits on an mbarrier that nothing completes; after limit_ns the
// wait gives up and ERRBIT_WAIT_TIMEOUT is or-ed into *err, as in the fused
// kernels.
cudaError_t launch_wait_timeout_check(int *err, uint64_t limit_ns, cudaStream_t st);

// --- three-dimensional lattices (lattice3d.cu) ----------------------------
// A 3-D grid of nx x ny x nz sites keeps slab z (rows z*ny .. z*ny + ny - 1
// of every plane) right after slab z - 1, so the 2-D kernels see a grid of
// ny*nz rows.  X sweeps, the phase and the tables need nothing else.
// One Y sweep inside every slab (pairs (y, y+1), y of the given parity
// counted from the slab's first row), in place.
cudaError_t launch_plain_sweep_y3(void *re, void *im, bool f64, int nx, int ny, int nz,
                                  int64_t pitch, int parity, double g, double s,
                                  cudaStream_t st, bool lift = false);
// One Z sweep: pairs of slabs (z, z+1), z of the given parity, in place.
cudaError_t launch_plain_sweep_z(void *re, void *im, bool f64, int nx, int ny, int nz,
                                 int64_t pitch, int parity, double g, double s, cudaStream_t st,
                                 bool lift = false);

// --- observables (reduce.cu) ----------------------------------------------
// partials: OBS_MAX_BLOCKS * OBS_Q doubles; result: OBS_Q doubles.
// norm_only computes only sum |psi|^2 (result[0]).
cudaError_t launch_observe(const void *re, const void *im, const void *vplane, bool f64,
                           int nx, int ny, int64_t pitch, double J, bool norm_only,
                           double *partials, double *result, cudaStream_t st);

// The same for a 3-D grid: OBS_Q3 quantities (sum p, sum x p, sum y p,
// sum x^2 p, sum y^2 p, kinetic, potential, sum z p, sum z^2 p), bonds along
// x, y (inside slabs) and z; partials hold OBS_MAX_BLOCKS * OBS_Q3 doubles.
cudaError_t launch_observe3(const void *re, const void *im, const void *vplane, bool f64,
                            int nx, int ny, int nz, int64_t pitch, double J, double *partials,
                            double *result, cudaStream_t st);

// <phi|psi> = sum conj(phi) psi over two FP32 pitched states: result[0] real,
// result[1] imaginary part (exact products, double-float then FP64 sums).
cudaError_t launch_inner(const float *phi_re, const float *phi_im, const float *psi_re,
                         const float *psi_im, int nx, int ny, int64_t pitch, double *partials,
                         double *result, cudaStream_t st);

// --- fused temporally blocked path (fused.cu) -----------------------------
constexpr int FUSED_MAX_K = 8;
constexpr int FUSED_LIFT_MAX_K = 4;   // ... of the lifting form (deeper ones run slower)
constexpr int FUSED_ADJ_MAX_K = 4;
// Scaled rotations (see pair_s in fused.cu): what the pairs with a member on
// an edge of the grid receive in even sweep k and odd sweep m (the edge member
// lo, its partner hi), h = 1 - scale of a launch for a site at place (z, y, x),
// entry 9 z + 3 y + x with 0 bulk, 1 the first site of the axis, 2 the last,
// and (adjoint) the squared scale at phase k, entry 3 y + x.  In the bulk of x
// and y, column i mod 4 takes hb[z][i] instead of h[9 z]: the two floats around
// h, mixed so that their mean is nearer to it than one float is (the rounding of
// h is the same at every site and launch, and would show in the norm).
struct ScaledEdge {
    float elo[FUSED_MAX_K + 1], ehi[FUSED_MAX_K + 1];
    float olo[2 * FUSED_MAX_K], ohi[2 * FUSED_MAX_K];
    float h[27];
    float hb[3][4];
    float f[FUSED_ADJ_MAX_K][9];
};
// The bulk coefficients (tangents) of a launch: even sweeps 0 and K, the even
// sweeps between, odd sweeps before and after a phase; fourth-order steps:
// the even sweeps that join a and b substeps and the odd sweeps of b.
struct ScaledCoef {
    float te_end, te_mid, to_a, to_b, te_ab, to_sub;
    ScaledEdge edge;
};

struct FusedLaunch {
    const CUtensorMap *tm_state;   // (re, im) planes of the input pair, 3-D map
    const CUtensorMap *tm_phase;   // (gamma_V, s_V) planes, 3-D map
    const CUtensorMap *tm_b = nullptr;   // launch_fused_u4: the b substep's table
    float *out_re, *out_im;
    int nx, ny;
    int64_t pitch;
    // rotation at theta: lifting form (t1 = tan(theta/2), s1 = sin theta) and
    // versine form (g1 = 1 - cos theta, s1); at 2 theta: lifting (t2, s2)
    float t1, s1, g1, t2, s2;
    int *err;
    // launch_fused_adjoint: the costate's output planes (out_re, out_im take
    // psi) and G as double-float planes
    float *out2_re = nullptr, *out2_im = nullptr;
    float *g_rh = nullptr, *g_rl = nullptr, *g_ih = nullptr, *g_il = nullptr;
    // time-dependent potential (launch_fused_drive only): a_n dt of step k
    float adt[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    // the fused fourth-order step (launch_fused_u4): t1..s2 above are the
    // a substep's; the b substep's lifting (tb, sb) and versine (gb) forms,
    // and the merged angle a + b in lifting form (tab, sab)
    float tb = 0, sb = 0, gb = 0, tab = 0, sab = 0;
    // not null: scaled rotations with these coefficients (the rest is unused)
    const ScaledCoef *sc = nullptr;
};
static_assert(sizeof(FusedLaunch::adt) / sizeof(float) == FUSED_MAX_K, "one a_n dt per step");
constexpr int FUSED_BOX_COLS = 128;   // columns a warp strip loads (box width)
// Strips over nx columns at a halo of `halo` columns: strip s loads columns
// s valid - shift .. s valid - shift + 127, valid = 128 - 2 halo, and stores all
// but the halo; the first stores its first columns and the last its last ones
// too, since beyond the grid's edge there is nothing to be wrong about.  shift is
// 0, or halo (launch_k in fused.cu).
TS_HD constexpr int strip_valid(int halo) { return FUSED_BOX_COLS - 2 * halo; }
TS_HD constexpr int strip_count(int64_t nx, int halo, int shift = 0)
{
    return nx + shift <= FUSED_BOX_COLS
               ? 1
               : (int)((nx + shift - 2 * halo + strip_valid(halo) - 1) / strip_valid(halo));
}
// A grid whose sweep over memory (24 bytes per site) passes L2 many times over.
TS_HD constexpr bool far_beyond_l2(int64_t nx, int64_t ny) { return 24 * nx * ny > 800000000; }
TS_HD constexpr int depth_halo(int K) { return (2 * K + 3) / 4 * 4; }   // of K steps, in whole lanes
constexpr int FUSED_BOX_ROWS = 2;     // rows per pipeline slot (box height)
cudaError_t launch_fused(int K, const FusedLaunch &a, cudaStream_t st);
// K (1..FUSED_ADJ_MAX_K) backward adjoint steps U^dagger (pass the
// coefficients at -theta) on two states at once: tm_state maps four planes
// (psi re, im, lambda re, im), psi goes to (out_re, out_im) and lambda to
// (out2_re, out2_im).  At each step's phase point G += conj(lambda~) m, with
// lambda~ = B^dagger lambda_s and m = B^dagger psi_s.
cudaError_t launch_fused_adjoint(int K, const FusedLaunch &a, cudaStream_t st);
// K (1..4) steps with the time-dependent potential V0 + a_n V1: tm_phase
// maps three planes (gamma_V, s_V, V1) and adt[k] = a_n dt of step k.
constexpr int FUSED_DRIVE_MAX_K = 4;
cudaError_t launch_fused_drive(int K, const FusedLaunch &a, cudaStream_t st);
// One fourth-order step U4 = a a b a a in one launch (five substeps, depth
// 5): tm_phase maps the a substep's table, tm_b the b substep's.
cudaError_t launch_fused_u4(const FusedLaunch &a, cudaStream_t st);
// One 3-D step Xe Xo Ye Yo Ze Zo P Zo Ze Yo Ye Xo Xe over an nx x ny x nz
// FP32 grid in one HBM round trip: a.ny is the rows of one slab, tm_state
// and tm_phase map all ny * nz rows (slab after slab), out_re, out_im take
// the result.  Needs (nz + 32) * ny < 2^31.
cudaError_t launch_fused3d(const FusedLaunch &a, int nz, cudaStream_t st);

// --- fused FP64 steps (fused64.cu) -----------------------------------------
// A scaled sweep: the bulk tangent, and what a pair with a member on an edge
// receives (the edge member lo, its partner hi).
struct Sweep64 {
    double t, lo, hi;
};
// One launch Ye Yo P Yo (Xo Xe Xo), the last of a run without its second Xo;
// or the tail: Ye and the scale (sx, sy by place: 0 bulk, 1 first, 2 last).
struct Step64 {
    const double *in_re, *in_im, *pg, *ps;
    double *out_re, *out_im;
    int nx, ny;
    int64_t pitch;
    Sweep64 ye, yo1, yo2, xo1, xe, xo2;
    double sx[3], sy[3];
    int last;
    int n_strips, rows;   // set by plan_step64: strips, rows per range (even)
};
// Set the split; cols (columns per lane) and blocks go to launch_step64.
void plan_step64(Step64 &p, int num_sms, int &cols, int &blocks);
cudaError_t launch_step64(const Step64 &p, int cols, int blocks, cudaStream_t st);
cudaError_t launch_tail64(const Step64 &p, cudaStream_t st);

// --- fused steps on tiles held in registers (tile.cu) ---------------------
constexpr int TILE_MAX_K = 4;
struct TileLaunch {
    const float *in_re, *in_im, *pg, *ps;   // state and phase table
    float *out_re, *out_im;
    int nx, ny;
    int64_t pitch;
    const ScaledCoef *sc;   // of depth K
};
// The tile shape for a launch of depth K over n grids with scaled rotations,
// or -1 where the warp streams are faster (or K > TILE_MAX_K).  multi: for
// launch_tile_multi.
constexpr int TILE_SHAPES = 4;
int num_sms();   // of the current device
int tile_shape(int K, int n, const int *nx, const int *ny, bool multi);
// Blocks of one grid at that shape.
int tile_blocks(int K, int shape, int nx, int ny);
// K steps (1..TILE_MAX_K): what launch_fused with scaled rotations gives at
// that depth, bit for bit.
cudaError_t launch_tile(int K, int shape, const TileLaunch &a, cudaStream_t st);

// --- backward adjoint steps on tiles (tile_adjoint.cu) --------------------
struct TileAdjoint {
    const float *in[4];   // psi re, im, lambda re, im
    float *out[4];
    float *g[4];          // G: re hi, re lo, im hi, im lo
    const float *pg, *ps;
    int nx, ny;
    int64_t pitch;
};
// whether a launch of depth K is faster on tiles than on warp streams
bool tile_adjoint_serves(int K, int nx, int ny);
// What launch_fused_adjoint does at depth K (1..FUSED_ADJ_MAX_K) with scaled
// rotations (c: coefficients at -theta).
cudaError_t launch_tile_adjoint(int K, const TileAdjoint &p, const ScaledCoef &c, cudaStream_t st);

// Device-resident description of one FP32 grid for the multi-grid launch
// (written once per grid set-up; read by the kernel with generic loads, its
// tensor maps by TMA).
struct GridDesc {
    CUtensorMap tm_state[2];   // (re, im) of pair 0 / pair 1
    CUtensorMap tm_phase;      // (gamma_V, s_V)
    float *re[2], *im[2];      // planes of pair 0 / pair 1
    int nx, ny;
    int64_t pitch;
    float t1, s1, g1, t2, s2;  // rotation coefficients (see FusedLaunch)
    ScaledCoef sc[FUSED_MAX_K];   // scaled rotations, by depth - 1
    const float *pg, *ps;      // the phase table's planes
};

// One grid of an epoch: its descriptor, where its work starts in the
// launch's plan (its first warp in an aligned plan, its first row-pair unit
// in an even one), its warps per strip (aligned plans), and which pair holds
// its state at flip = 0.
struct EpochEntry {
    const GridDesc *desc;
    int64_t begin;
    int cur0;
    int strip_warps;
};

// How one multi-grid launch splits its work over warps.
struct MultiPlan {
    int warps;       // warps launched
    int64_t units;   // row-pair units of all grids (strips x row pairs)
    bool aligned;    // strip-aligned (per-grid warps per strip) or even split
    int shape;       // >= 0: a launch of tiles of that shape instead (units: its blocks)
};

// Set the multi-grid kernel's attributes for depth K (call outside stream capture).
cudaError_t fused_multi_prepare(int K);
// Plan one multi-grid launch at depth K over n grids (sides nx[i] x ny[i])
// and fill tab[i].begin and tab[i].strip_warps (the caller sets desc and
// cur0).  The strip-aligned split (every strip of a grid on the same row
// ranges, so neighbouring strips share halo columns through L2) is taken
// when its longest warp is within 10 % of the even split's; mixes of many
// small grids get the even split.  warps == 0 on an error.
MultiPlan fused_multi_plan(int K, bool scaled, int n, const int *nx, const int *ny,
                           EpochEntry *tab);
// K steps for every grid of a device epoch table planned by
// fused_multi_plan; the input pair of grid i is tab[i].cur0 ^ flip.
// A plan with a tile shape runs as tiles (tile.cu), which report no error.
cudaError_t tile_multi_prepare();
cudaError_t launch_tile_multi(int K, int shape, const EpochEntry *tab, int n, int blocks, int flip,
                              cudaStream_t st);
cudaError_t launch_fused_multi(int K, bool scaled, const EpochEntry *tab, int n_grids,
                               const MultiPlan &plan, int flip, int *err, cudaStream_t st);

// Build a 3-D FP32 tensor map over `planes` consecutive pitched planes
// (nx x ny each, `plane_bytes` apart) for the fused path.  Its boxes span
// 128 columns, 2 rows and `box_planes` planes (1 to 4; 0: all `planes`), so
// one box load fetches the same rows of those planes.  Returns false (and a
// message) if the driver entry point is unavailable or the encode call fails.
bool make_pair_tensor_map(CUtensorMap *tm, const void *base, int nx, int ny, int64_t pitch,
                          size_t plane_bytes, const char **why, int planes = 2,
                          int box_planes = 0);

// Thread-local count of kernel launches issued by this library.
void count_launches(int64_t n);

#ifdef __CUDACC__
// Launch a kernel of this library as a programmatic dependent of the kernel
// before it in the stream.  Every kernel here calls grid_dep_sync (common.cuh)
// before it touches memory, which waits until that kernel has completed, so
// the stream's work keeps the order of plain launches.  Why: plain launches of
// one stream start on a grid of 2.05 us on this machine (a kernel of 2.1 us
// repeats every 4.1 us, one of 4.9 us every 8.2 us); dependent ones follow
// 0.4 to 0.7 us after the kernel before, whatever its length: 6 us launches
// become 4.6 us (depth 1 at 256^2), 27.3 us ones 25.2 us (depth 3 at 2048^2).
// The register tiles (tile.cu, tile_adjoint.cu) let their successor start early, before
// their stores (griddepcontrol.launch_dependents): its blocks then wait in grid_dep_sync
// until the stores are visible.  That is safe because every kernel launched here
// calls grid_dep_sync before its first access to global memory; a kernel without
// that call must not be launched by launch_pdl.  The other kernels do not: blocks
// that become resident during the tail cost more than they hide there, 2 to 10 % up
// to 1024^2 and 40 % for depth 3 at 2048^2.
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

// Record a message for ts_last_error() and return `status` (api.cu).
int set_error(int status, const char *fmt, ...);

// Drop the adjoint record of a grid that is being destroyed (adjoint.cu).
void forget_adjoint(const ::ts_grid *g);

}  // namespace ts
