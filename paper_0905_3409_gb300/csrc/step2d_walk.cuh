// step2d_walk.cuh -- one 2D GALS step over one tile for the steps that write no phi_xy plane
// (approach A between the steps of a run, the COMPACT layout, approach B).
//
// A thread owns one column of the tile and walks down its two halves at once: the lanes of
// its paired arithmetic are rows r and r + rows/2.  While the feet stay in the same column of
// cells and move down one cell per row -- everywhere but at the zero lines of a velocity
// component, at CFL up to 1 -- the lower corners of a foot's cell are the upper corners of
// the next one, so a row costs one new row of corner data per lane (8 loads and one paired
// central difference per corner) where each foot used to load its own two rows (16 loads,
// its own range checks, index arithmetic and scalar differences).  With rows r and r + 1 as
// the lanes, as in tile_step2d, the shared row would have to be copied into the other lane.
// 4096^2 vortex, GB300: 107.8 us per step against 119.4 for tile_step2d's non-writing form
// (rotation 2048^2 20.1 against 23.6); issue and dependency latency bound both.
// Anything else (a new column or a skipped row, a cell outside the staged tile or at the
// box's ends) reloads both rows by gather_lane; the arithmetic is the same, and so are the
// bits.
#pragma once

#include <climits>

#include "step2d_tile.cuh"

namespace gals {
namespace t2 {

// Rows per iteration of the walk.  Two, so that the carried rows change names instead of
// registers (4096^2 vortex 107.8 us per step against 112.8 with one and 118.1 with all
// seven); one for the fields evaluated from tables, whose loads the compiler would keep live
// over two rows (16-mode Fourier field: 584 us against 241).
template <int VK> constexpr int walk_unroll() { return VK == VK_FOURIER2D || VK == VK_WAVES2D ? 1 : 2; }

// static shared memory of a walked tile (the staged tile is dynamic)
template <int TY> struct WalkSmem {
    StageCoefPair scp;
    float fsum[12][TY];               // FOURIER2D stage 1: row sums of the tile's rows
    uint64_t bar;
};

// One row (two corners x 4 data, both lanes) of the foot cells from the staged tile; tA, tB
// point at the left corner's phi of each lane's row.
template <int CR, int PS>
__device__ __forceinline__ void walk_row(const float *tA, const float *tB, float i2h0, F2 c0[4], F2 c1[4])
{
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        c0[p] = make_float2(tA[p * PS], tB[p * PS]);
        c1[p] = make_float2(tA[p * PS + 1], tB[p * PS + 1]);
    }
    if (CR == CROSS_PLANE) {
        c0[3] = make_float2(tA[3 * PS], tB[3 * PS]);
        c1[3] = make_float2(tA[3 * PS + 1], tB[3 * PS + 1]);
    }
    if (CR == CROSS_RECON) {
        // dcentral of both lanes at once
        const F2 wm = make_float2(tA[2 * PS - 1], tB[2 * PS - 1]), wp = make_float2(tA[2 * PS + 2], tB[2 * PS + 2]);
        c0[3] = mul2(sub2(c1[2], wm), bc(i2h0));
        c1[3] = mul2(sub2(wp, c0[2]), bc(i2h0));
    }
}

// One tile step: columns x0 .. x0 + TX - 1, rows y0 .. y0 + min(TY, row_end - y0) - 1; the
// other arguments as tile_step2d's.
template <int TY, int TR, int VK, int CR, int HYV, int W, bool COH = false, class Hook = NoHook>
__device__ __forceinline__ bool tile_walk2d(const float *__restrict__ in, float *__restrict__ out, const Geom &g,
                                            const VelParams &vp, const StageCoef *__restrict__ coef, float dt,
                                            const CUtensorMap *tmap, int *__restrict__ err, int x0, int y0,
                                            int row_end, float *tile, WalkSmem<TY> &sm, uint32_t parity,
                                            Hook after_issue = Hook())
{
    constexpr int NP = CR == CROSS_PLANE ? 4 : 3;
    constexpr int PS = Geo<TY, HYV, W>::PS;
    constexpr bool LATE = TY == 2;  // one pair per thread: trace it while the tile is on its way
    const int tid = threadIdx.x;
#ifdef GALS_CHECKED
    const uint32_t polls = g.wait_polls;
    if (tid == 0 && !g.skip_copy) {
#else
    constexpr uint32_t polls = kWaitLimit;
    if (tid == 0) {
#endif
        mbar_arrive_expect_tx(&sm.bar, Geo<TY, HYV, W>::bytes(NP));
        tma_load_3d(tile, tmap, x0 - HX, y0 - HYV, 0, &sm.bar);
        after_issue();
    }
    const StageCoef &sc = *coef;
    const StageCoefPair *scp = &sm.scp;
    const int rows = min(TY, row_end - y0), half = (rows + 1) >> 1;
    if (VK == VK_FOURIER2D && TR != TR_GIVEN) {
        for (int e = tid; e < 3 * 3 * 16; e += TX) {
            const int tab = e / 48, rest = e % 48, st = rest / 16, kl = rest % 16;
            const float v = tab == 0 ? __ldg(&coef->A[st][kl])
                          : (tab == 1 ? __ldg(&coef->Al[st][kl]) : __ldg(&coef->All[st][kl]));
            F2 *dst = tab == 0 ? &sm.scp.A[st][kl] : (tab == 1 ? &sm.scp.Al[st][kl] : &sm.scp.All[st][kl]);
            *dst = bc(v);
        }
        for (int e = tid; e < TY * 4; e += TX) {
            const int r = e >> 2, k = (e & 3) + 1;
            const float yr = node_pos(g.lo1, min(y0 + r, g.n1 - 1), g.h1);
            float ux, vx, w;
            fourier_row(sc, yr, k, ux, vx, w);
            sm.fsum[k - 1][r] = ux;
            sm.fsum[4 + k - 1][r] = vx;
            sm.fsum[8 + k - 1][r] = w;
        }
        __syncthreads();
    }
    const int i = x0 + tid;
    const float xs = node_pos(g.lo0, i, g.h0);
    const F2 x = bc(xs);
    const VCol cx = (VK == VK_VORTEX2D) ? vortex_col(xs, sc.mod[0]) : VCol{0.f, 0.f, 0.f, 0.f, 0.f};
    FCol fcol;
    if (VK == VK_FOURIER2D && TR != TR_GIVEN) fcol = fourier_col(xs);

    F2 y, dx, dy, J[4];
    Sep2 ry = Sep2{bc(0.f), bc(0.f), bc(0.f)};
    V2p a1;
    int j0 = 0, j1 = 0;
    auto trace = [&](int r) {
        j0 = y0 + r;
        j1 = min(j0 + half, g.n1 - 1);
        y = make_float2(node_pos(g.lo1, j0, g.h1), node_pos(g.lo1, j1, g.h1));
        if (TR == TR_GIVEN) {
            const int64_t o0 = (int64_t)j0 * g.pitch + i, o1 = (int64_t)j1 * g.pitch + i;
            const float *tb = vp.given;
            const int64_t P = vp.given_plane;
            dx = make_float2(__ldg(tb + o0), __ldg(tb + o1));
            dy = make_float2(__ldg(tb + P + o0), __ldg(tb + P + o1));
#pragma unroll
            for (int e = 0; e < 4; ++e) J[e] = make_float2(__ldg(tb + (2 + e) * P + o0), __ldg(tb + (2 + e) * P + o1));
            return;
        }
        if (VK == VK_VORTEX2D) ry = sep_factors2(y);
        a1 = VK == VK_FOURIER2D ? fourier_stage1_pair<TY>(fcol, sm.fsum, r, r + half)
                                : stage1_pair<VK>(vp, sc, scp, x, y, cx, ry);
        trace2d_pair<TR, VK>(a1, vp, sc, scp, x, y, dt, dx, dy, J);
    };

    // the corner rows carried down (c[2], c[3] of the last row are c[0], c[1] of the next), the
    // cell column and upper row each lane must meet to use them, and where its next row lies
    F2 c[4][4];
    int kA = 0, kB = 0, lA = INT_MIN, lB = INT_MIN;
    const float *tA = tile, *tB = tile;
    const int kmin = max(x0 - HX + 1, 1), kmax = min(x0 - HX + W - 3, g.n0 - 3);
    const int lmin = y0 - HYV, lmax = y0 - HYV + Geo<TY, HYV, W>::TH - 2;  // staged cells
    auto gather = [&](int k0, int l0, int k1, int l1) {
        if (TY > 2 && k0 == kA && l0 == lA && k1 == kB && l1 == lB && l0 <= lmax && l1 <= lmax) {
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                c[0][a] = c[2][a];
                c[1][a] = c[3][a];
            }
#ifdef GALS_CHECKED
            tA = tile + GALS_CHK(g, (int)(tA - tile), PS - 2);
            tB = tile + GALS_CHK(g, (int)(tB - tile), PS - 2);
#endif
            walk_row<CR, PS>(tA, tB, g.i2h0, c[2], c[3]);
        } else {
            float ca[4][4], cb[4][4];
            gather_lane<TY, CR == CROSS_CELL ? CROSS_NONE : CR, HYV, COH, W, false>(in, g, tile, x0, y0, k0, l0, ca);
            gather_lane<TY, CR == CROSS_CELL ? CROSS_NONE : CR, HYV, COH, W, false>(in, g, tile, x0, y0, k1, l1, cb);
#pragma unroll
            for (int v = 0; v < 4; ++v)
#pragma unroll
                for (int a = 0; a < (CR == CROSS_CELL ? 3 : 4); ++a) c[v][a] = make_float2(ca[v][a], cb[v][a]);
            kA = k0;
            kB = k1;
            const bool ok = k0 >= kmin && k0 <= kmax && k1 >= kmin && k1 <= kmax && l0 >= lmin && l1 >= lmin &&
                            l0 < lmax && l1 < lmax;
            lA = ok ? l0 : INT_MIN;
            lB = ok ? l1 : INT_MIN;
            if (ok) {
                tA = tile + ((l0 - y0 + HYV + 1) * W + k0 - x0 + HX);
                tB = tile + ((l1 - y0 + HYV + 1) * W + k1 - x0 + HX);
            }
        }
        lA += 1;  // INT_MIN + 1 matches no row either
        lB += 1;
        tA += W;
        tB += W;
    };
    auto finish = [&](int r) {
        F2 phi, px, py;
        node2d_feet<TR, VK>(g, vp, sc, scp, dt, i, j0, i, j1, x, y, dx, dy, J, cx, ry,
                            [&](int k0, int l0, int k1, int l1, F2 cc[4][4]) {
                                gather(k0, l0, k1, l1);
#pragma unroll
                                for (int v = 0; v < 4; ++v)
#pragma unroll
                                    for (int a = 0; a < 4; ++a) cc[v][a] = c[v][a];
                                if (CR == CROSS_CELL) cross_cell2d_pair(cc, g.ih0, g.ih1);
                            }, phi, px, py, VK == VK_FOURIER2D ? &a1 : nullptr);
        const int o = GALS_CHK(g, j0 * g.pitch + i, plane_extent(g));
        out[o] = phi.x;
        out[g.plane + o] = px.x;
        out[2 * g.plane + o] = py.x;
        if (r + half < rows) {
            const int o1 = GALS_CHK(g, o + half * g.pitch, plane_extent(g));
            out[o1] = phi.y;
            out[g.plane + o1] = px.y;
            out[2 * g.plane + o1] = py.y;
        }
    };

    if (LATE && i < g.n0) trace(0);
    // bounded wait for the tile; a block-uniform verdict so no thread is left at a barrier
    if (!mbar_wait_block(&sm.bar, parity, polls)) {
        if (tid == 0) {
            atomicExch(err, kErrTmaTimeout);
            mbar_wait_bounded(&sm.bar, parity, polls);  // let a late copy land before giving up
        }
        return false;
    }
    if (i < g.n0) {
        if (LATE) {
            finish(0);
        } else {
#pragma unroll walk_unroll<VK>()
            for (int r = 0; r < half; ++r) {
                trace(r);
                finish(r);
            }
        }
    }
    return true;
}

}  // namespace t2
}  // namespace gals
