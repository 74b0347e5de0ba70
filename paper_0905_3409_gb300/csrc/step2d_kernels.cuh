// step2d_kernels.cuh -- the single-grid 2D GALS step kernels and their launchers, instantiated
// per velocity kind in step2d_*.cu.
//
// The per-tile work (trace, Hermite, write-back, fused phi_xy) is step2d_tile.cuh and
// step2d_walk.cuh; this file maps one thread block to one tile of the grid.
#pragma once

#ifndef GALS_2D_TY
#define GALS_2D_TY 14
#endif
#ifndef GALS_2D_MINB
#define GALS_2D_MINB 5
#endif
#ifndef GALS_2D_HY
#define GALS_2D_HY 1
#endif
#ifndef GALS_WALK_MINB
#define GALS_WALK_MINB 5
#endif
#ifndef GALS_SHORT_BLOCKS
#define GALS_SHORT_BLOCKS 850
#endif
#ifndef GALS_2D_OV
#define GALS_2D_OV 1
#endif

#include "step2d_kinds.h"
#include "step2d_walk.cuh"

namespace gals {

namespace {

using namespace t2;
constexpr int TY = GALS_2D_TY;  // output tile rows (even)
constexpr int HYT = GALS_2D_HY; // staged halo rows above and below the tile
constexpr bool OVX = GALS_2D_OV; // overlapped tiles where phi_xy is written (see tile_step2d)
constexpr int TWS = OVX ? TW + 4 : TW;  // staged columns of the single-grid kernels
using GT = Geo<TY, HYT, TWS>;
constexpr int TYS = 2;          // tile rows on grids too small to fill the chip with tall tiles
constexpr int64_t kShortTileBlocks = GALS_SHORT_BLOCKS;

// A field of many plane waves is bound by its hardware sines and cosines alone, a tile's copy and
// set-up being nothing beside them: short tiles on any grid, because a step's few waves of
// tall ones leave the last one part empty (2048^2: 2516 tiles on 760 places).  256 waves: 2048^2 1.60 -> 1.49 ms
// per step, 1000^2 476 -> 371 us, 700^2 with 512 707 -> 377; the floor of the sines and
// cosines is 1.28 ms at 2048^2.  With 16 and 32 waves both shapes take the same time.  Grids
// of more rows than a launch of short tiles holds (65535 tiles along y) keep the tall ones,
// whose number the grid's size limit is made for; the rule looks at the whole grid, so that
// every band of a step decides alike.
constexpr int kShortWaves = 64;
constexpr int kMaxShortRows = 65535 * TYS;

template <int WC> constexpr bool overlapped() { return OVX && WC; }
template <int WC> constexpr int tile_stride() { return overlapped<WC>() ? TX - 2 : TX; }

// Steps that write phi_xy.
template <int TY, int TR, int VK, int CR, int WC>
__global__ void __launch_bounds__(TX, GALS_2D_MINB)
k_step2d(const float *__restrict__ in, float *__restrict__ out, Geom g, VelParams vp,
         const StageCoef *__restrict__ coef, float dt, const __grid_constant__ CUtensorMap tmap,
         int *__restrict__ err, int row0)
{
    extern __shared__ __align__(128) float tile[];
    __shared__ __align__(16) Smem<TY, WC> sm;
    if (threadIdx.x == 0) mbar_init(&sm.bar, 1);
    pdl_wait();
    __syncthreads();
    tile_step2d<TY, TR, VK, CR, WC, HYT, false, TWS, overlapped<WC>()>(
        in, out, g, vp, coef, dt, &tmap, err, blockIdx.x * tile_stride<WC>(), row0 + blockIdx.y * TY, tile, sm, 0);
}

// Steps that do not.
template <int TY, int TR, int VK, int CR>
__global__ void __launch_bounds__(TX, GALS_WALK_MINB)
k_walk2d(const float *__restrict__ in, float *__restrict__ out, Geom g, VelParams vp,
         const StageCoef *__restrict__ coef, float dt, const __grid_constant__ CUtensorMap tmap,
         int *__restrict__ err, int row0, int row_end)
{
    extern __shared__ __align__(128) float tile[];
    __shared__ __align__(16) WalkSmem<TY> sm;
    if (threadIdx.x == 0) mbar_init(&sm.bar, 1);
    pdl_wait();
    __syncthreads();
    tile_walk2d<TY, TR, VK, CR, HYT, TWS>(in, out, g, vp, coef, dt, &tmap, err, blockIdx.x * TX,
                                          row0 + blockIdx.y * TY, row_end, tile, sm, 0);
}

// ---------------------------------------------------------------- persistent time loop
//
// All steps of one call in one launch (FULL layout, approach A).  Work items are
// (step, tile) pairs numbered step-major; a block takes the next item from a ticket counter
// and, for step s > 0, first waits until the 3 x 3 tiles around its own have finished step
// s - 1 (a per-tile flag holds the number of steps a tile has finished in this launch).
// With feet at most TY - 2 rows and TX - 2 columns from their node those are every tile
// whose output the step reads (the staged tile, global gathers) and every tile that still
// reads the region the step overwrites (the ping-pong buffer of step s - 1's input), so
// the order of the per-step launches is kept where it matters and nowhere else: blocks
// move on to the next step while the last tiles of the previous one drain.  Items are
// handed out in increasing order and a block waits only for smaller items, so the launch
// finishes whatever the number of resident blocks.  Every wait is bounded; a wait that
// runs out sets the launch's abort word and the error word, and every block returns.
constexpr int kErrRunTimeout = 3;
constexpr uint32_t kSpinLimit = 1u << 22;  // flag polls (~0.2 us each) before giving up

__device__ __forceinline__ int ld_acquire_gpu(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_gpu(int *p, int v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <int TR, int VK>
__global__ void __launch_bounds__(TX, GALS_2D_MINB)
k_step2d_run(float *__restrict__ buf0, float *__restrict__ buf1, Geom g, VelParams vp,
             const StageCoef *__restrict__ coef, float dt, const __grid_constant__ CUtensorMap tmap0,
             const __grid_constant__ CUtensorMap tmap1, int *__restrict__ err, int *__restrict__ ctl,
             int nsteps, int cur)
{
    extern __shared__ __align__(128) float tile[];
    __shared__ __align__(16) Smem<TY, 1> sm;
    __shared__ int s_item;
    const int tid = threadIdx.x;
    if (tid == 0) mbar_init(&sm.bar, 1);
    const int ntx = (g.n0 + TX - 1) / TX, nty = (g.n1 + TY - 1) / TY, ntiles = ntx * nty;
    const int total = ntiles * nsteps;  // < 2^31 - 2^20 (host)
    int *ticket = ctl, *abort_word = ctl + 1, *flags = ctl + 4;
    // thread 0 draws the block's next item one item ahead, so that the draw's latency
    // hides behind a tile (a block waits only for items smaller than the one it holds,
    // and it finishes its current item before the drawn one: no cycle of waits)
    int next = 0;
    if (tid == 0) next = atomicAdd(ticket, 1);
    uint32_t parity = 0;
    for (;;) {
        if (tid == 0) s_item = next;
        __syncthreads();
        const int t = s_item;
        if (t >= total) break;
        const int st = t / ntiles, tt = t - st * ntiles, bx = tt % ntx, by = tt / ntx;
        // wait until the 3 x 3 tiles around this one have finished step st - 1: one flag
        // per thread of the first warp, in parallel
        bool lost = false;
        if (st > 0 && tid < 9) {
            const int nx = bx + tid % 3 - 1, ny = by + tid / 3 - 1;
            if (nx >= 0 && nx < ntx && ny >= 0 && ny < nty) {
                const int *f = flags + ny * ntx + nx;
                for (uint32_t it = 0; ld_acquire_gpu(f) < st; ++it) {
                    if (it >= kSpinLimit || *(volatile int *)abort_word) {
                        lost = true;
                        break;
                    }
                    __nanosleep(64);
                }
            }
        }
        if (__syncthreads_or(lost)) {
            if (tid == 0 && atomicExch(abort_word, 1) == 0) atomicExch(err, kErrRunTimeout);
            break;
        }
        const int b = (cur + st) & 1;
        if (tid == 0) {
            // the tile copy is an async-proxy read of data other blocks wrote through the
            // generic proxy (acquired above, ordered before this thread by the barrier)
            asm volatile("fence.proxy.async.global;" ::: "memory");
        }
        const bool ok = tile_step2d<TY, TR, VK, CROSS_PLANE, 1, HYT, true, TWS>(
            b ? buf1 : buf0, b ? buf0 : buf1, g, vp, coef + st, dt, b ? &tmap1 : &tmap0, err,
            bx * TX, by * TY, tile, sm, parity, [&]() { next = atomicAdd(ticket, 1); });
        parity ^= 1u;
        if (!ok) {  // block-uniform: the staged copy was lost
            if (tid == 0) atomicExch(abort_word, 1);
            break;
        }
        __syncthreads();  // every store of the tile is issued before thread 0 publishes it
        if (tid == 0) {
            __threadfence();
            st_release_gpu(flags + tt, st + 1);
        }
    }
}

// Whether the grid has too few tall tiles to occupy the chip (whole grid, so that every band
// of a step decides alike): a short tile then does in one row pair per thread what a tall
// one does in seven, on seven times the blocks, its trace hidden behind the tile's copy.
// The line, 850 tall tiles, lies between the largest grid measured faster with short ones (747)
// and the smallest measured faster with tall ones (1023); a full wave of them, five blocks on
// each of 152 SMs, is 760.  Us per step, short against tall tiles: vortex 200 x 172 2.8 against 6.8, 1021 x 777 (448 tall
// tiles) 6.8 against 8.9, 1150^2 (747) 10.9 against 12.0, 1300^2 (1023) 14.5 against 13.7,
// 2048^2 34.1 against 27.5; rotation 1150^2 9.2 against 9.5, 1300^2 12.1 against 11.0.
bool short_tiles(const Geom &g)
{
    const int64_t blocks = (int64_t)((g.n0 + TX - 1) / TX) * ((g.n1 + TY - 1) / TY);
    return blocks < kShortTileBlocks;
}

// Whether the steps that write no phi_xy walk their tiles: not the tall tiles of the Fourier
// field, whose tables leave no registers for the carried rows (4096^2: 241 us per step
// walked, spilling, against 236), and not those of approach B, whose cells share less
// (2048^2: 0 to 2 % slower walked but for the RK3 trace).
template <int TYT, int VK, int CR, int WC> constexpr bool walked()
{
    return !WC && (TYT == TYS || (VK != VK_FOURIER2D && CR != CROSS_CELL));
}

template <int TYT, int TR, int VK, int CR, int WC>
cudaError_t launch_ty(const StepLaunch &a, cudaStream_t s)
{
    constexpr int NP = CR == CROSS_PLANE ? 4 : 3;
    constexpr int bytes = Geo<TYT, HYT, TWS>::bytes(NP);
    static PerDevice ready;  // one attribute call per instantiation and device (not a stream op)
    cudaError_t e = ready.once([] {
        if constexpr (!walked<TYT, VK, CR, WC>()) return allow_dynamic_smem(k_step2d<TYT, TR, VK, CR, WC>, bytes);
        else return allow_dynamic_smem(k_walk2d<TYT, TR, VK, CR>, bytes);
    });
    if (e != cudaSuccess) return e;
    // rows of the band (all by default)
    const int row0 = a.band_lo, row1 = a.band_hi > 0 ? a.band_hi : a.geom.n1;
    if (row1 <= row0) return cudaSuccess;
    const dim3 grid((a.geom.n0 + tile_stride<WC>() - 1) / tile_stride<WC>(), (row1 - row0 + TYT - 1) / TYT);
    const CUtensorMap &map = *a.tmap[TYT == TYS][NP - 3];
    if constexpr (!walked<TYT, VK, CR, WC>())
        return launch_kernel(k_step2d<TYT, TR, VK, CR, WC>, grid, dim3(TX), bytes, s, a.dependent, a.in, a.out, a.geom,
                             a.vp, a.coef, (float)a.dt, map, a.err, row0);
    else
        return launch_kernel(k_walk2d<TYT, TR, VK, CR>, grid, dim3(TX), bytes, s, a.dependent, a.in, a.out, a.geom,
                             a.vp, a.coef, (float)a.dt, map, a.err, row0, row1);
}

template <int TR, int VK, int CR, int WC>
cudaError_t launch_t(const StepLaunch &a, cudaStream_t s)
{
    const bool is_short = short_tiles(a.geom) ||
                          (VK == VK_WAVES2D && a.vp.nwaves >= kShortWaves && a.geom.n1 <= kMaxShortRows);
    return is_short ? launch_ty<TYS, TR, VK, CR, WC>(a, s) : launch_ty<TY, TR, VK, CR, WC>(a, s);
}

template <int TR, int VK>
cudaError_t launch_cr(const StepLaunch &a, cudaStream_t s)
{
    if (a.cross_in == CROSS_CELL) return launch_t<TR, VK, CROSS_CELL, 0>(a, s);  // approach B
    if (a.write_cross)
        return a.cross_in == CROSS_PLANE ? launch_t<TR, VK, CROSS_PLANE, 1>(a, s)
                                         : launch_t<TR, VK, CROSS_RECON, 1>(a, s);
    return a.cross_in == CROSS_PLANE ? launch_t<TR, VK, CROSS_PLANE, 0>(a, s)
                                     : launch_t<TR, VK, CROSS_RECON, 0>(a, s);
}

template <int VK>
cudaError_t launch_tr(const StepLaunch &a, cudaStream_t s)
{
    if (a.trace == TR_HEUN) return launch_cr<TR_HEUN, VK>(a, s);
    return a.trace == TR_EULER ? launch_cr<TR_EULER, VK>(a, s) : launch_cr<TR_RK3, VK>(a, s);
}

template <int TR, int VK>
cudaError_t launch_run_t(const RunLaunch &a, cudaStream_t s)
{
    auto kern = k_step2d_run<TR, VK>;
    static PerDevice fit;  // per instantiation
    int blocks_per_sm = 0;
    cudaError_t e = fit.get(&blocks_per_sm, [&](int *nb) {
        cudaError_t a = allow_dynamic_smem(kern, GT::bytes(4));
        if (a == cudaSuccess) a = cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, kern, TX, GT::bytes(4));
        if (*nb < 1) *nb = 1;
        return a;
    });
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t items = (int64_t)run2d_tiles(a.geom) * a.nsteps;
    const int64_t want = (int64_t)blocks_per_sm * (sms > 0 ? sms : 1);
    const int grid = (int)(want < items ? want : items);
    kern<<<grid, TX, GT::bytes(4), s>>>(a.buf[0], a.buf[1], a.geom, a.vp, a.coef, (float)a.dt, *a.tmap[0],
                                        *a.tmap[1], a.err, a.ctl, a.nsteps, a.cur);
    return cudaGetLastError();
}

template <int VK>
cudaError_t launch_run_tr(const RunLaunch &a, cudaStream_t s)
{
    if (a.trace == TR_HEUN) return launch_run_t<TR_HEUN, VK>(a, s);
    return a.trace == TR_EULER ? launch_run_t<TR_EULER, VK>(a, s) : launch_run_t<TR_RK3, VK>(a, s);
}

}  // namespace

// every step of a velocity kind, and its persistent runs
template <int VK> cudaError_t step2d_kind(const StepLaunch &a, cudaStream_t s) { return launch_tr<VK>(a, s); }
template <int VK> cudaError_t run2d_kind(const RunLaunch &a, cudaStream_t s) { return launch_run_tr<VK>(a, s); }

}  // namespace gals
