// The grid handle behind the opaque ts_grid of include/trotter.h (internal).
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cuda.h>
#include <vector>

#include "../../include/trotter.h"
#include "internal.h"

namespace ts {
// Kinetic rotation coefficients of one angle theta (FP64, rounded once where
// used): versine form (g1 = 1 - cos theta, s1 = sin theta), lifting form
// (t1 = tan(theta/2), s1) and the merged angle 2 theta (t2 = tan theta,
// s2 = sin 2 theta).
struct RotCoef {
    double g1, s1, t1, s2, t2;
};
RotCoef rot_coef(double theta);

// Scaled rotations (fused.cu) serve |theta| <= this, per substep.  A launch
// takes its scale out by a -= h a; the rounding of h is what they add to the
// norm.  The tangents and the edge ratios stay far from their poles.  Larger
// angles take the lifting form.
constexpr double SCALED_MAX_THETA = 0.075;
// ... on grids of at least this many columns and rows.  In the bulk four columns mix
// two floats h, so that the norm of a |psi|^2 spread evenly over columns mod 4 drifts by
// at most 5e-10 per step at depths 1, 2 and 4, 9e-10 at the others, 8e-10 per fourth-order
// step and 1e-9 per 3-D step; the lines at the edges take one float, up to 2e-9 per step for
// the sites on them, which shows where they are a large part of all (sides of 1 to 4:
// 1e-9 to 2e-9 per step over theta, 4e-10 to 5e-10 in the lifting form; 16^2 6e-10
// and 8e-10).
constexpr int SCALED_MIN_SIDE = 8;
inline bool scaled_angle(double theta, int64_t nx, int64_t ny)
{
    return std::fabs(theta) <= SCALED_MAX_THETA && nx >= SCALED_MIN_SIDE && ny >= SCALED_MIN_SIDE;
}
// Whether a launch of K plain steps takes them.  Depth 2 on the largest grids does
// not: its warps wait for HBM, and those of neighbouring strips drift apart and read
// their shared columns twice, which the lifting form's slower, evener pace avoids
// (us per step, scaled and lifting: 4096^2 32.0 and 34.1, 6000^2 79 and 66, 8192^2
// 134 and 125, 16384^2 550 and 522).
inline bool runs_scaled(double theta, int K, int64_t nx, int64_t ny)
{
    return scaled_angle(theta, nx, ny) && !(K == 2 && far_beyond_l2(nx, ny));
}
// Coefficients of a launch of K substeps with kinetic half angles sub[i].
void scaled_coef(const double *sub, int K, int64_t nx, int64_t ny, int64_t nz, ScaledCoef &c);
}  // namespace ts

// One grid: a slab of seven planes (re, im of ping-pong pairs 0 and 1,
// gamma_V, s_V, V) plus reduction scratch; see ts_grid_layout.
struct ts_grid {
    ts_layout L;
    size_t esize;
    unsigned char *slab;
    bool owns_slab;
    int cur;                 // 0: planes 0/1 hold the state, 1: planes 2/3
    double dt, theta, J;
    double g1, s1, t1, s2, t2;   // rotation coefficients (FP64): theta and 2 theta
    int order;                   // 2: U2(dt) per step; 4: U4(dt) (ts_set_potential_order)
    ts::RotCoef sub[2];          // order 4: substeps p dt and (1 - 4p) dt
    unsigned char *tab_b;        // order 4: (gamma_V, s_V) at (1 - 4p) dt, library-owned;
                                 // planes 4/5 then hold the table at p dt
    CUtensorMap tm_phase_b;
    // time-dependent potential V0 + a_n V1 (ts_set_drive): a library-owned
    // slab of three planes (copies of gamma_V, s_V, then V1), its tensor map,
    // the amplitudes a_n and the index of the next one
    unsigned char *drive_slab;
    CUtensorMap tm_drive;
    std::vector<double> drive_a;
    int64_t drive_pos;
    bool driven;
    double *partials, *result;
    int *err;
    bool served;               // a server's grid: launches report in the server's word, not in err
    cudaEvent_t host_copied;   // host-input copies done (created on first use)
    // a batch whose grids take several kernels runs a group of them here, beside
    // the caller's stream (created by the first such batch that this grid leads)
    cudaStream_t side;
    cudaEvent_t fork, join;
    bool tmaps_ok;
    CUtensorMap tm_state[2], tm_phase;   // (re, im) of pair 0 / 1; (gamma_V, s_V)
    ts::GridDesc *desc_dev;              // the same, for multi-grid launches (in the slab)
    ts::GridDesc desc_host;
    double sc_theta;                     // the angle of desc_host.sc
    bool desc_written;                   // desc_dev holds desc_host ...
    double desc_theta;                   // ... of this angle

    void *plane(int i) const { return slab + (size_t)i * L.plane_bytes; }
    void *re() const { return plane(2 * cur); }
    void *im() const { return plane(2 * cur + 1); }
    void *re_other() const { return plane(2 * (cur ^ 1)); }
    void *im_other() const { return plane(2 * (cur ^ 1) + 1); }
    void *pg() const { return plane(4); }
    void *ps() const { return plane(5); }
    void *vp() const { return plane(6); }
    void *drive_v1() const { return drive_slab + 2 * L.plane_bytes; }
    void *pg_b() const { return tab_b; }
    void *ps_b() const { return tab_b + L.plane_bytes; }
    bool f64() const { return L.dtype == TS_F64; }
    // rows of every plane: ny per slab, nz slabs (3-D grids; nz = 1 in 2-D)
    int64_t rows() const { return L.ny * L.nz; }
    bool is3d() const { return L.nz > 1; }
};


namespace ts {
// Fill a grid handle for a caller-provided slab (tensor maps included) with
// no device work; ts_create_grid adds the zero-fill (api.cu).
ts_status grid_setup(const ts_layout &L, void *slab, bool owns_slab, ts_grid **out);
// Byte offset of the scratch area (partials, result, error word, descriptor).
size_t grid_scratch_offset(const ts_layout &L);
// Rotation coefficients for (dt, theta) (api.cu).
void grid_set_coefficients(ts_grid *g, double dt, double theta);
// Write the grid's multi-grid descriptor (tensor maps, planes, coefficients)
// into its slab on stream st (api.cu).
void grid_write_desc(ts_grid *g, cudaStream_t st);
// Evolve n FP32 grids (|theta| <= pi/4, with `scaled` scaled_angle of each)
// together with the multi-grid kernel at depth K (api.cu).
cudaError_t evolve_multi(ts_grid *const *gs, const int64_t *steps, int n, int K, bool scaled,
                         cudaStream_t st);
// Launches of grids with scaled rotations and of grids in the lifting form run side
// by side (on two streams) up to this many sites in all, where they leave parts of
// the GPU idle; beyond that one after the other.  Half of the grids scaled, us per
// step, in turn and side by side: 4 x 128^2 5.3 and 3.2, 4 x 512^2 7.1 and 5.4, 16 x
// 512^2 14.0 and 13.1, 16 x 1024^2 31.0 and 31.3, 16 mixed sizes (13 M sites) 37.9
// and 41.4.  (Planned for a part of the GPU each, they lost up to 45 %: registers
// keep few warps of one kernel beside the other's.)
constexpr double SIDE_BY_SIDE_MAX_SITES = 1e7;
}  // namespace ts
