// gals_internal.h -- host-side interface between the C ABI and the kernel launchers.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gals_device.cuh"
#include "per_device.h"

namespace gals {

// Launch `kern` on s; dependent: as a programmatic dependent of the kernel before it (see
// pdl_wait), so that its launch overlaps that kernel.  For chains of small kernels, us per
// step: a 64^2 step called by itself (coefficients, step, clock) 11.5 -> 8.4, 3D graphs of
// 20^3 7 -> 4.7, 64 x 60 x 50 9.2 -> 8.0; steps of many waves of blocks lose nothing.
template <class... P, class... A>
cudaError_t launch_kernel(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool dependent,
                          const A &...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

struct StepLaunch {
    const float *in;     // state at t (all planes, plane stride geom.plane)
    float *out;          // state at t + dt
    Geom geom;
    VelParams vp;
    const StageCoef *coef; // this step's stage coefficients (filled by launch_coef_table)
    double dt;
    int trace;           // TR_EULER / TR_RK3
    int cross_in;        // CROSS_PLANE: read mixed derivatives; CROSS_RECON: rebuild from psi
    int write_cross;     // 1: also write the mixed-derivative planes of the new state
    // TMA maps of `in`, [short 2D tiles][4 or (3D: 8) planes with the stored mixed derivatives:
    // 1, phi and psi only: 0]
    const CUtensorMap *tmap[2][2];
    const CUtensorMap *tmap_cross; // 3D FULL: TMA map of `out` with the reconstruction box
    int *err;            // device error word (kErrTmaTimeout on a lost tile copy)
    // the band of nodes to update along the last axis (2D rows, 3D z-levels), [lo, hi);
    // hi == 0: all.  lo must be a multiple of band_unit(dim), hi too unless it is n.
    int band_lo, band_hi;
    bool dependent;      // launch_kernel's
};

// Persistent 2D time loop (FULL layout, approach A): nsteps steps from buffer cur in one
// launch; ctl holds 4 + run2d_tiles(geom) ints, zero before the launch (ticket counter,
// abort word, per-tile step flags).  Feet must stay within run2d_max_cells(axis) cells of
// their node.
struct RunLaunch {
    float *buf[2];
    int cur;
    Geom geom;
    VelParams vp;
    const StageCoef *coef;     // stage coefficients of the launch's steps
    double dt;
    int trace;                 // TR_EULER / TR_RK3 / TR_HEUN
    const CUtensorMap *tmap[2]; // FULL-box TMA maps of buf[0], buf[1]
    int *err;
    int *ctl;
    int nsteps;
};
int run2d_tiles(const Geom &g);
int run2d_max_cells(int axis);
cudaError_t launch_step2d_run(const RunLaunch &a, cudaStream_t s);

// A run of steps on a small 2D grid in one launch of one cluster (step2d_small.cu).  Rule
// (small2d_fits): at most kSmallNodes nodes in rows of at most kSmallColumns, and the
// blocks' shared memory; a run of at least kSmallSteps steps.  At every size up to the limit
// it is the faster way (128 x 96: 1.8 us per step against 7.2 for the banded launches;
// 512 x 24: 2.4 against 6.7).  It does not stop being faster there: 128 x 97 takes 7.2, and the
// shared memory would hold four times the nodes.  The limit is the interface's: larger grids keep
// the launches per step and band that gals_last_step_launches is specified to count.  A run of
// fewer than 8 steps gains
// little, its coefficient and clock kernels being most of it (5.3 us per step at 8 steps
// against 9.9 at 7 of a first launch per step).
constexpr int kSmallNodes = 12288, kSmallColumns = 512, kSmallSteps = 8;
constexpr int kSmallMaxBytes = 96 * 1024;
struct SmallLaunch {
    const float *in;       // state at the run's start (all planes)
    float *out;            // state at its end; may be `in`
    Geom geom;
    VelParams vp;
    const StageCoef *coef; // stage coefficients of the run's steps
    double dt;
    int trace;             // TR_EULER / TR_RK3 / TR_HEUN
    int cell;              // approach B
    int planes;            // the first step reads the stored mixed derivatives
    int write_cross;       // write the mixed-derivative plane of the end state
    int nsteps;
};
bool small2d_fits(const Geom &g);
// done: false if the current device cannot place the cluster (nothing is queued then)
cudaError_t launch_step2d_small(const SmallLaunch &a, cudaStream_t s, bool *done);

// Granularity of StepLaunch bands: the 2D tile height, the 3D tile depth.
int band_unit(int dim);

// Box of the 2D step kernels' staged tile (tall or short) for np planes; rows of a tall tile.
void tile_box2d(int is_short, int np, uint32_t box[3]);
int tile_rows2d();
// Box (x, y, z, planes) of the 3D step kernel's staged tile.
void tile_box3d(int cross_recon, uint32_t box[4]);
// Box (x, y, z, planes) of the 3D reconstruction kernel's staged psi_y, psi_z.
void recon_box3d(uint32_t box[4]);
// Encode a tiled TMA map of FP32 data: rank dims (innermost first), byte strides of
// dims 1..rank-1, box extents; zero fill outside the tensor.
cudaError_t make_tile_map(CUtensorMap *map, const float *base, int rank, const uint64_t *dims,
                          const uint64_t *strides_bytes, const uint32_t *box);

// Kernel launchers; return the launch error (cudaSuccess if launched).
cudaError_t launch_step2d(const StepLaunch &a, cudaStream_t s);
cudaError_t launch_step3d(const StepLaunch &a, cudaStream_t s);
// Rebuild the mixed-derivative planes of `buf` from its gradient planes (approach A).
cudaError_t launch_recon(int dim, const Geom &g, float *buf, cudaStream_t s);
// table[s] = stage coefficients of step s (t = t_dev[0] + s*dt), s < nsteps
cudaError_t launch_coef_table(StageCoef *table, const VelParams &vp, const double *t_dev,
                              double dt, int nsteps, cudaStream_t s, bool dependent = false);
// t_dev[0] += nsteps * dt
cudaError_t launch_advance_time(double *t_dev, int nsteps, double dt, cudaStream_t s, bool dependent = false);
// the device clock set to t, in stream order (no host staging, the caller does not block)
cudaError_t launch_set_time(double *t_dev, double t, cudaStream_t s);
// Velocity kinds supported per dimension.
bool vel_supported(int dim, int kind);

// Value, unit normal and curvature of the interpolant at npts points (curvature.cu);
// pts: npts * dim FP64 coordinates on the device; any output may be null.
cudaError_t launch_eval_points(int dim, const Geom &g, const double lo[3], const double h[3],
                               const float *state, const double *pts, int64_t npts, bool cell_b,
                               float *H, float *normal, float *kappa, cudaStream_t s);

// Diagnostics (diag.cu)
struct DiagOut {
    unsigned long long n_neg, n_sym, nonfinite;
    unsigned int emax_phi_bits, emax_psi_bits;  // non-negative floats as ordered integers
    double l2_phi_sum;
    unsigned int dense, pad;                 // warps with many undecided cells
    unsigned long long pre_neg, pre_sym;     // what the pass that finds them counts
};
// The diagnostics' launches with `nparts` blocks (one FP64 partial each; diag_partials_needed()
// unless the caller has a reason).  Scratch: nparts doubles, a DiagOut, kDiagList words.
// cell_a / cell_b: the interpolant of a / b takes its mixed derivatives by approach B.
constexpr unsigned kDiagList = 4096;
int diag_partials_needed();
cudaError_t launch_diag(int dim, const Geom &g, const float *a, const float *b, int q, DiagOut *counters,
                        double *partials, int nparts, unsigned *list, cudaStream_t s, bool cell_a = false,
                        bool cell_b = false);

}  // namespace gals
