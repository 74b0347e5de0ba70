// step3d.cu -- the 3D GALS step kernel and the 3D mixed-derivative reconstruction.
//
// One thread per two grid nodes of a z-column, in paired FP32 (FFMA2): trace back with the
// 3x3 Jacobian (Sec. 5.1, superconsistent Shu-Osher RK3) -> locate the foot cell -> stream
// the cell's 4 x-lines (2 corners x 8 data) from the TMA-staged tile -> tricubic Hermite
// value and gradient (Sec. 2.3) -> phi+ = H, psi+ = J^T grad H.
// Mixed derivatives (Sec. 2.3, approach A): phi_xy = Dx psi_y, phi_xz = Dx psi_z,
// phi_yz = Dy psi_z, phi_xyz = Dx Dy psi_z, read from their planes (FULL) or rebuilt
// from psi windows around the cell (COMPACT) with the same stencils.
#include "step3d_common.cuh"


namespace gals {

namespace {

using namespace t3;

// Output tile per block: TX x TY nodes in x, y and TZ in z (each thread walks TZ nodes in z).
constexpr int TX = 32, TY = 4, TZ = 4;
constexpr int HX = 4;                  // halo (x rounded to 16 bytes for TMA)
template <int CR> struct Tile3 {
    // psi_z y-window needs one more row (CROSS_RECON); CROSS_CELL shares that tile's map
    static constexpr int HZ = 1;
    static constexpr int HY = CR == CROSS_PLANE ? 1 : 2;
    static constexpr int NP = CR == CROSS_PLANE ? 8 : 4;
    static constexpr int W = TX + 2 * HX, H = TY + 2 * HY, D = TZ + 2 * HZ;
    static constexpr int PS = W * H * D;
    static constexpr int BYTES = NP * PS * 4;
    // CROSS_RECON: phi_yz of the staged nodes is a fifth plane behind them
    static constexpr int SMEM = BYTES + (CR == CROSS_RECON ? PS * 4 : 0);
};

// phi_yz = Dy psi_z at every staged node of the rows a foot's cell can use, four nodes of a row
// at a time (approach A with one-sided ends at the box; nodes outside it hold anything).
__device__ __forceinline__ void stage_yz(float *tile, const Geom &g, int y0)
{
    using T = Tile3<CROSS_RECON>;
    // a thread keeps its place in the level: rows 1 .. H - 2 of the tile, Q quadruples each
    constexpr int Q = T::W / 4, R = T::H - 2, N = Q * R, L = TX * TY / N;
    static_assert(T::W % 4 == 0 && L >= 1, "rows of whole quadruples, a level per pass or more");
    const int tid = threadIdx.x + TX * threadIdx.y;
    if (tid >= L * N) return;
    const int q = tid % Q, r = tid / Q % R + 1, j = y0 - T::HY + r;
    for (int z = tid / N; z < T::D; z += L) {
        const int o = (z * T::H + r) * T::W + 4 * q;
        const float4 *p = reinterpret_cast<const float4 *>(tile + 3 * T::PS + o);
        constexpr int S = T::W / 4;             // a row further
        float4 v;
        if (j == 0) {
            const float4 a = p[0], b = p[S], c = p[2 * S];
            v = make_float4(dfirst(a.x, b.x, c.x, g.i2h1), dfirst(a.y, b.y, c.y, g.i2h1),
                            dfirst(a.z, b.z, c.z, g.i2h1), dfirst(a.w, b.w, c.w, g.i2h1));
        } else if (j == g.n1 - 1) {
            const float4 a = p[0], b = p[-S], c = p[-2 * S];
            v = make_float4(dlast(a.x, b.x, c.x, g.i2h1), dlast(a.y, b.y, c.y, g.i2h1),
                            dlast(a.z, b.z, c.z, g.i2h1), dlast(a.w, b.w, c.w, g.i2h1));
        } else {
            const float4 a = p[S], b = p[-S];
            v = make_float4(dcentral(a.x, b.x, g.i2h1), dcentral(a.y, b.y, g.i2h1), dcentral(a.z, b.z, g.i2h1),
                            dcentral(a.w, b.w, g.i2h1));
        }
        *reinterpret_cast<float4 *>(tile + 4 * T::PS + o) = v;
    }
}

// Two nodes per thread, (i, j, kz) and (i, j, kz+1), in paired FP32: trace with the 3x3
// Jacobian, cell location, tricubic Hermite value and gradient from the staged tile,
// phi+ = H and psi+ = J^T grad H.  Feet whose cell data lie outside the staged tile
// (large CFL) read global memory instead.
// At most 128 registers (4 blocks per SM; a few words spill), measured faster than 166
// registers at 3 blocks per SM.
// CROSS_RECON (COMPACT, and FULL between the steps of a run where step_launch chooses it)
// stages phi and psi only: phi_yz is differenced once per staged node into shared memory and
// the x-differences are taken, both feet at once, as a cell's lines are read.  It replaces
// the reconstruction pass (66 us of a 256^3 step) by 115 instructions per node; us per step,
// against the windows of 16 psi_z per line it used to rebuild phi_yz from / FULL's two
// passes: 256^3 deformation 344 against 447 / 351, rotation 306 against 406 / 311, 101^3
// deformation 33.2 against 39.8 / 37.4.  Tiles of 2, 6 or 8 levels (363, 354, 356) and a halo
// of two cells (397) were slower, as was a branch for the one-sided ends per difference (373).
// WIDE (CROSS_RECON on grids that put at most two blocks on an SM, step3d_wide): twice the
// registers, and feet outside the tile both at once, all their values from global memory (a
// choice per value cost 30 us of 150).  There a step is the latency of one block; us per step with
// one foot after the other / the windows of both before that / now: 48^3 constant at CFL 2
// 12.5 / 9.2 / 7.5, rotation at CFL 6 15.9 / 12.9 / 9.9, deformation at CFL 0.5 7.7 / 7.6 / 6.3;
// 33 x 30 x 28 deformation 6.2 / 5.8 / 5.6.  At 390 blocks (64 x 60 x 50) it loses: rotation at
// CFL 2 18.0 against 14.9.
template <int TR, int VK, int CR, bool WIDE>
__global__ void __launch_bounds__(TX *TY, CR == CROSS_CELL ? 1 : (WIDE ? 2 : 4))
k_step3d(const float *__restrict__ in, float *__restrict__ out, Geom g, VelParams vp,
         const StageCoef *__restrict__ coef, float dt, const __grid_constant__ CUtensorMap tmap,
         int *__restrict__ err, int zlo)
{
    using T = Tile3<CR>;
    extern __shared__ __align__(128) float tile[];
    __shared__ __align__(8) uint64_t bar;
    // CROSS_RECON keeps the Jacobian here while the interpolant is evaluated (18 registers)
    constexpr bool JS = CR == CROSS_RECON && TR != TR_HEUN && VK == VK_DEFORM3D;
    __shared__ F2 Jsh[JS ? 9 : 1][JS ? TX * TY : 1];
    const int tid = threadIdx.x + TX * threadIdx.y;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = zlo + blockIdx.z * TZ;
    if (tid == 0) mbar_init(&bar, 1);
    pdl_wait();
    __syncthreads();
    if (tid == 0) {
        mbar_arrive_expect_tx(&bar, T::BYTES);
        tma_load_4d(tile, &tmap, x0 - HX, y0 - T::HY, z0 - T::HZ, 0, &bar);
    }
    const StageCoef &sc = *coef;
    // threads past a ragged edge trace a clamped node and store nothing
    const bool valid = x0 + (int)threadIdx.x < g.n0 && y0 + (int)threadIdx.y < g.n1;
    const int i = min(x0 + (int)threadIdx.x, g.n0 - 1), j = min(y0 + (int)threadIdx.y, g.n1 - 1);
    const float x = g.lo0 + (float)i * g.h0;
    const float y = g.lo1 + (float)j * g.h1;
    const Pre3 pre = pre3<VK>(x, y);
    const int64_t P = g.plane;
    const int64_t zstride = (int64_t)g.n1 * g.pitch;
    const int zend = min(z0 + TZ, g.n2);
    const F2 X = bc(x), Y = bc(y);
    for (int kz = z0; kz < zend; kz += 2) {
        const bool two = kz + 1 < zend;
        const int kz1 = two ? kz + 1 : kz;
        const F2 Z = make_float2(g.lo2 + (float)kz * g.h2, g.lo2 + (float)kz1 * g.h2);
        F2 d[3], J[9];
        auto trace = [&]() {
            if (kz + 2 >= zend) pdl_release();
            trace3d_pair<TR, VK>(stage1_pair<VK>(vp, sc, pre, X, Y, Z), vp, sc, X, Y, Z, dt, d, J);
            if (JS)
#pragma unroll
                for (int e = 0; e < 9; ++e) Jsh[e][tid] = J[e];
        };
        // CROSS_RECON: the first trace while the tile is on its way (33 x 30 x 28 deformation 6.2 ->
        // 5.7 us per step, large grids the same)
        if (CR == CROSS_RECON) trace();
        if (kz == z0) {
            if (!mbar_wait_block(&bar, 0)) {
                if (tid == 0) {
                    atomicExch(err, kErrTmaTimeout);
                    mbar_wait_bounded(&bar, 0);
                }
                return;
            }
            if (CR == CROSS_RECON) {
                stage_yz(tile, g, y0);
                __syncthreads();
            }
        }
        if (CR != CROSS_RECON) trace();

        int k0, l0, m0, k1, l1, m1;
        float xi0, eta0, zeta0, xi1, eta1, zeta1;
        locate(i, d[0].x * g.ih0, g.n0, k0, xi0);
        locate(j, d[1].x * g.ih1, g.n1, l0, eta0);
        locate(kz, d[2].x * g.ih2, g.n2, m0, zeta0);
        locate(i, d[0].y * g.ih0, g.n0, k1, xi1);
        locate(j, d[1].y * g.ih1, g.n1, l1, eta1);
        locate(kz1, d[2].y * g.ih2, g.n2, m1, zeta1);
        const Basis2 bx = basis_pair(make_float2(xi0, xi1), g.h0, g.ih0);
        const Basis2 by = basis_pair(make_float2(eta0, eta1), g.h1, g.ih1);
        const Basis2 bz = basis_pair(make_float2(zeta0, zeta1), g.h2, g.ih2);

        // a cell is served from the tile if every value its line reads is staged
        auto in_tile = [&](int k, int l, int m) {
            const int tx = k - x0 + HX, ty = l - y0 + T::HY, tz = m - z0 + T::HZ;
            return CR != CROSS_RECON
                ? (tx >= 0 && tx <= T::W - 2 && ty >= 0 && ty <= T::H - 2 && tz >= 0 && tz <= T::D - 2)
                : (tx >= 1 && tx <= T::W - 3 && ty >= 1 && ty <= T::H - 3 && tz >= 0 && tz <= T::D - 2);
        };
        auto lds = [&](int a, int zz, int yy, int xx) {
            return tile[GALS_CHK(g, a * T::PS + ((zz - z0 + T::HZ) * T::H + yy - y0 + T::HY) * T::W + xx - x0 + HX,
                                 T::NP * T::PS)];
        };
        auto ldg = [&](int a, int zz, int yy, int xx) {
#ifdef GALS_CHECKED
            return __ldg(in + a * P + GALS_CHK(g, (int64_t)zz * zstride + (int64_t)yy * g.pitch + xx, plane_extent(g)));
#else
            return __ldg(in + a * P + (int64_t)zz * zstride + (int64_t)yy * g.pitch + xx);
#endif
        };
        const bool in0 = in_tile(k0, l0, m0), in1 = in_tile(k1, l1, m1);
        F2 H, gr[3];
        if (CR == CROSS_CELL) {
            // approach B: the cell's 8 vertices x (phi, psi) per foot, mixed derivatives from them
            auto ld0 = [&](int a, int zz, int yy, int xx) { return in0 ? lds(a, zz, yy, xx) : ldg(a, zz, yy, xx); };
            auto ld1 = [&](int a, int zz, int yy, int xx) { return in1 ? lds(a, zz, yy, xx) : ldg(a, zz, yy, xx); };
            float q0[8][4], q1[8][4], c0[8][4], c1[8][4];
#pragma unroll
            for (int v = 0; v < 8; ++v)
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    q0[v][a] = ld0(a, m0 + (v >> 2), l0 + ((v >> 1) & 1), k0 + (v & 1));
                    q1[v][a] = ld1(a, m1 + (v >> 2), l1 + ((v >> 1) & 1), k1 + (v & 1));
                }
            cross_cell3d([&](int v, int a) { return q0[v][a]; }, g.ih0, g.ih1, g.ih2, c0);
            cross_cell3d([&](int v, int a) { return q1[v][a]; }, g.ih0, g.ih1, g.ih2, c1);
            hermite3d_pair(bx, by, bz, [&](int G, int B, int C, F2 lo[4], F2 hi[4]) {
                const int v = 2 * B + 4 * C;
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const int p = group_plane(G, a), e = p < 4 ? p : p - 4;
                    lo[a] = p < 4 ? make_float2(q0[v][e], q1[v][e]) : make_float2(c0[v][e], c1[v][e]);
                    hi[a] = p < 4 ? make_float2(q0[v + 1][e], q1[v + 1][e]) : make_float2(c0[v + 1][e], c1[v + 1][e]);
                }
            }, H, gr);
        } else if (CR == CROSS_RECON && in0 && in1) {
            // phi_xy, phi_xz, phi_xyz of the cell's corners by x-differences of psi_y, psi_z and
            // the staged phi_yz, both feet at once; one-sided where the cell touches the box
            const float *p0 = tile + (((m0 - z0 + T::HZ) * T::H + l0 - y0 + T::HY) * T::W + k0 - x0 + HX);
            const float *p1 = tile + (((m1 - z0 + T::HZ) * T::H + l1 - y0 + T::HY) * T::W + k1 - x0 + HX);
#ifdef GALS_CHECKED
            // the reads below: planes 0 .. 4, rows and levels up to one further, columns -1 .. 2
            p0 = tile + 1 + GALS_CHK(g, (int)(p0 - tile) - 1, T::PS - (T::H + 1) * T::W - 3);
            p1 = tile + 1 + GALS_CHK(g, (int)(p1 - tile) - 1, T::PS - (T::H + 1) * T::W - 3);
#endif
            // bits: a foot's cell at the first column (1, 2) or the last one (4, 8)
            const int edge = (k0 == 0) | (k1 == 0) << 1 | (k0 == g.n0 - 2) << 2 | (k1 == g.n0 - 2) << 3;
            auto line = [&](int G, int B, int C, F2 lo[4], F2 hi[4], bool ends) {
                const int o = (C * T::H + B) * T::W;
                auto ld = [&](int a, int q) { return make_float2(p0[a * T::PS + o + q], p1[a * T::PS + o + q]); };
                // data v and v + 1 of the group from plane a (psi_y, psi_z, phi_yz) and its Dx
                auto dx = [&](int a, int v) {
                    const F2 um = ld(a, -1), u0 = ld(a, 0), u1 = ld(a, 1), up = ld(a, 2);
                    F2 d0 = mul2(sub2(u1, um), bc(g.i2h0)), d1 = mul2(sub2(up, u0), bc(g.i2h0));
                    if (ends) {
                        if (edge & 1) d0.x = dfirst(u0.x, u1.x, up.x, g.i2h0);
                        if (edge & 2) d0.y = dfirst(u0.y, u1.y, up.y, g.i2h0);
                        if (edge & 4) d1.x = dlast(u1.x, u0.x, um.x, g.i2h0);
                        if (edge & 8) d1.y = dlast(u1.y, u0.y, um.y, g.i2h0);
                    }
                    lo[v] = u0; hi[v] = u1;
                    lo[v + 1] = d0; hi[v + 1] = d1;
                };
                if (G == 0) {
                    lo[0] = ld(0, 0); hi[0] = ld(0, 1);
                    lo[1] = ld(1, 0); hi[1] = ld(1, 1);
                    dx(2, 2);
                } else {
                    dx(3, 0);
                    dx(4, 2);
                }
            };
            // (a branch per difference cost 24 instructions per node)
            if (__any_sync(__activemask(), edge))
                hermite3d_pair(bx, by, bz, [&](int G, int B, int C, F2 lo[4], F2 hi[4]) { line(G, B, C, lo, hi, true); }, H, gr);
            else
                hermite3d_pair(bx, by, bz, [&](int G, int B, int C, F2 lo[4], F2 hi[4]) { line(G, B, C, lo, hi, false); }, H, gr);
        } else if (CR == CROSS_RECON && !WIDE) {
            // a foot outside the tile: both from global memory, a foot's two lanes the same, so that
            // this path's windows do not set the kernel's registers; one at a time where two would
            // all the same (256^3, us per step: constant at CFL 2 574 one at a time, 503 both; RK3
            // deformation 348 against 354)
            constexpr int kFeet = VK == VK_DEFORM3D && TR == TR_RK3 ? 1 : 2;
#pragma unroll kFeet
            for (int e = 0; e < 2; ++e) {
                const int k = e ? k1 : k0, l = e ? l1 : l0, m = e ? m1 : m0;
                auto dup = [&](const F2 &v) { return bc(e ? v.y : v.x); };
                const Basis2 ex{dup(bx.S), dup(bx.dS), dup(bx.hG0), dup(bx.hG1), dup(bx.dG0), dup(bx.dG1)};
                const Basis2 ey{dup(by.S), dup(by.dS), dup(by.hG0), dup(by.hG1), dup(by.dG0), dup(by.dG1)};
                const Basis2 ez{dup(bz.S), dup(bz.dS), dup(bz.hG0), dup(bz.hG1), dup(bz.dG0), dup(bz.dG1)};
                F2 He, ge[3];
                hermite3d_pair(ex, ey, ez, [&](int G, int B, int C, F2 lo[4], F2 hi[4]) {
                    float a0[8], b0[8];
                    cell_line<CR>(ldg, g, k, l, m, B, C, a0, b0);
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        lo[a] = bc(a0[group_plane(G, a)]);
                        hi[a] = bc(b0[group_plane(G, a)]);
                    }
                }, He, ge);
                if (e) {
                    H.y = He.y;
#pragma unroll
                    for (int a = 0; a < 3; ++a) gr[a].y = ge[a].y;
                } else {
                    H = He;
#pragma unroll
                    for (int a = 0; a < 3; ++a) gr[a] = ge[a];
                }
            }
        } else if (in0 && in1) {
            hermite3d_lines(bx, by, bz, [&](int B, int C, F2 lo[8], F2 hi[8]) {
                float a0[8], b0[8], a1[8], b1[8];
                cell_line<CR>(lds, g, k0, l0, m0, B, C, a0, b0);
                cell_line<CR>(lds, g, k1, l1, m1, B, C, a1, b1);
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    lo[a] = make_float2(a0[a], a1[a]);
                    hi[a] = make_float2(b0[a], b1[a]);
                }
            }, H, gr);
        } else {
            // (WIDE: both feet from global memory, without the choice per value)
            auto ld0 = [&](int a, int zz, int yy, int xx) { return !WIDE && in0 ? lds(a, zz, yy, xx) : ldg(a, zz, yy, xx); };
            auto ld1 = [&](int a, int zz, int yy, int xx) { return !WIDE && in1 ? lds(a, zz, yy, xx) : ldg(a, zz, yy, xx); };
            hermite3d_lines(bx, by, bz, [&](int B, int C, F2 lo[8], F2 hi[8]) {
                float a0[8], b0[8], a1[8], b1[8];
                cell_line<CR>(ld0, g, k0, l0, m0, B, C, a0, b0);
                cell_line<CR>(ld1, g, k1, l1, m1, B, C, a1, b1);
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    lo[a] = make_float2(a0[a], a1[a]);
                    hi[a] = make_float2(b0[a], b1[a]);
                }
            }, H, gr);
        }
        F2 psi[3];
        if (TR == TR_HEUN) {
            // CIR gradient update (Sec. 4): Dv at the foot at time t, Dv at the node at t + dt
            const V3p Df = vel3d_pair<VK>(vp, sc, 1, fma2(d[0], bc(1.f), X), fma2(d[1], bc(1.f), Y),
                                           fma2(d[2], bc(1.f), Z));
            const V3p Dn = stage1_pair<VK>(vp, sc, pre, X, Y, Z);
            heun_psi3(Df, Dn, dt, gr, psi);
        } else {
            if (JS)
#pragma unroll
                for (int e = 0; e < 9; ++e) J[e] = Jsh[e][tid];
#pragma unroll
            for (int a = 0; a < 3; ++a)  // (J^T grad H)_a = sum_b J[b][a] dH/dx_b
                psi[a] = fma2(J[a], gr[0], fma2(J[3 + a], gr[1], mul2(J[6 + a], gr[2])));
        }
        if (!valid) continue;
        const int64_t o = GALS_CHK(g, (int64_t)kz * zstride + (int64_t)j * g.pitch + i, plane_extent(g));
        out[o] = H.x;
#pragma unroll
        for (int a = 0; a < 3; ++a) out[(a + 1) * P + o] = psi[a].x;
        if (two) {
#ifdef GALS_CHECKED
            const int64_t o1 = GALS_CHK(g, o + zstride, plane_extent(g));
            out[o1] = H.y;
#pragma unroll
            for (int a = 0; a < 3; ++a) out[(a + 1) * P + o1] = psi[a].y;
#else
            out[o + zstride] = H.y;
#pragma unroll
            for (int a = 0; a < 3; ++a) out[(a + 1) * P + o + zstride] = psi[a].y;
#endif
        }
    }
}

// Mixed derivatives at every node from psi_y, psi_z (approach A, one-sided ends):
// phi_xy = Dx psi_y, phi_xz = Dx psi_z, phi_yz = Dy psi_z, phi_xyz = Dx (Dy psi_z).
// One thread per (x, y) column walks RZ z-slices; every stencil operand is a direct
// read-only load (neighbours' reads hit L1), with no barriers, so all loads of a slice are
// in flight together.  The stencil functions are the ones the step kernels use, so the
// results are identical.
constexpr int RX = 32, RY = 8, RZ = 4;

__global__ void __launch_bounds__(RX *RY) k_recon3d(const float *__restrict__ py,
                                                     const float *__restrict__ pz,
                                                     float *__restrict__ cross, Geom g)
{
    const int i = blockIdx.x * RX + threadIdx.x, j = blockIdx.y * RY + threadIdx.y;
    if (i >= g.n0 || j >= g.n1) return;
    const int64_t P = g.plane;
    const int z0 = blockIdx.z * RZ, zend = min(z0 + RZ, g.n2);
#pragma unroll
    for (int dz = 0; dz < RZ; ++dz) {
        const int kz = z0 + dz;
        if (kz >= zend) break;
        const int64_t row = ((int64_t)kz * g.n1) * g.pitch;
        const float *ly = py + row, *lz = pz + row;
        auto Y = [&](int xx, int yy) { return __ldg(ly + (int64_t)yy * g.pitch + xx); };
        auto Z = [&](int xx, int yy) { return __ldg(lz + (int64_t)yy * g.pitch + xx); };
        const float fxy = dline(i, g.n0, g.i2h0, [&](int q) { return Y(q, j); });
        const float fxz = dline(i, g.n0, g.i2h0, [&](int q) { return Z(q, j); });
        const float fyz = dline(j, g.n1, g.i2h1, [&](int r) { return Z(i, r); });
        const float fxyz = dline(i, g.n0, g.i2h0, [&](int q) {
            return dline(j, g.n1, g.i2h1, [&](int r) { return Z(q, r); });
        });
        const int64_t o = row + (int64_t)j * g.pitch + i;
        cross[o] = fxy;
        cross[P + o] = fxz;
        cross[2 * P + o] = fyz;
        cross[3 * P + o] = fxyz;
    }
}

// The same reconstruction after a FULL step, with psi_y and psi_z of a block's nodes
// (x-halo 4 for 16-byte TMA rows, y-halo 2 for the one-sided ends) staged in shared memory
// by one TMA copy: a block of 32 x 8 threads covers QZ z-slices.
constexpr int QX = 32, QY = 8, QZ = 4, QHX = 4, QHY = 2;
constexpr int QW = QX + 2 * QHX, QH = QY + 2 * QHY;

__global__ void __launch_bounds__(QX *QY)
k_recon3d_tma(float *__restrict__ buf, Geom g, const __grid_constant__ CUtensorMap map,
              int *__restrict__ err, int zq0)
{
    __shared__ __align__(128) float t[2][QZ][QH][QW];  // psi_y, psi_z
    __shared__ __align__(8) uint64_t bar;
    const int tid = threadIdx.x + QX * threadIdx.y;
    // slabs zq0 .. zq0 + gridDim.z - 1, in reverse: the step kernel wrote the last slabs
    // last, so their psi_y, psi_z are the ones most likely still in L2
    const int x0 = blockIdx.x * QX, y0 = blockIdx.y * QY;
    const int z0 = (zq0 + (int)gridDim.z - 1 - (int)blockIdx.z) * QZ;
    if (tid == 0) mbar_init(&bar, 1);
    pdl_wait();
    __syncthreads();
    if (tid == 0) {
        mbar_arrive_expect_tx(&bar, (uint32_t)sizeof(t));
        tma_load_4d(&t[0][0][0][0], &map, x0 - QHX, y0 - QHY, z0, 2, &bar);
    }
    if (!mbar_wait_block(&bar, 0)) {
        if (tid == 0) {
            atomicExch(err, kErrTmaTimeout);
            mbar_wait_bounded(&bar, 0);
        }
        return;
    }
    const int i = x0 + threadIdx.x, j = y0 + threadIdx.y;
    if (i >= g.n0 || j >= g.n1) return;
    const int64_t P = g.plane;
    const int nz = min(QZ, g.n2 - z0);
    if (x0 >= 1 && x0 + QX <= g.n0 - 1 && y0 >= 1 && y0 + QY <= g.n1 - 1) {
        // every node of the block is interior in x and y: central differences only (the
        // same operations dline performs there)
        const int tx = threadIdx.x + QHX, ty = threadIdx.y + QHY;
        int64_t o = ((int64_t)z0 * g.n1 + j) * g.pitch + i;
        const int64_t zs = (int64_t)g.n1 * g.pitch;
        for (int dz = 0; dz < nz; ++dz, o += zs) {
            const float(*Y)[QW] = t[0][dz];
            const float(*Z)[QW] = t[1][dz];
            buf[4 * P + o] = dcentral(Y[ty][tx + 1], Y[ty][tx - 1], g.i2h0);
            buf[5 * P + o] = dcentral(Z[ty][tx + 1], Z[ty][tx - 1], g.i2h0);
            buf[6 * P + o] = dcentral(Z[ty + 1][tx], Z[ty - 1][tx], g.i2h1);
            buf[7 * P + o] = dcentral(dcentral(Z[ty + 1][tx + 1], Z[ty - 1][tx + 1], g.i2h1),
                                      dcentral(Z[ty + 1][tx - 1], Z[ty - 1][tx - 1], g.i2h1), g.i2h0);
        }
        return;
    }
    for (int dz = 0; dz < nz; ++dz) {
        auto Y = [&](int q, int r) { return t[0][dz][r - y0 + QHY][q - x0 + QHX]; };
        auto Z = [&](int q, int r) { return t[1][dz][r - y0 + QHY][q - x0 + QHX]; };
        const int64_t o = ((int64_t)(z0 + dz) * g.n1 + j) * g.pitch + i;
        buf[4 * P + o] = dline(i, g.n0, g.i2h0, [&](int q) { return Y(q, j); });
        buf[5 * P + o] = dline(i, g.n0, g.i2h0, [&](int q) { return Z(q, j); });
        buf[6 * P + o] = dline(j, g.n1, g.i2h1, [&](int r) { return Z(i, r); });
        buf[7 * P + o] = dline(i, g.n0, g.i2h0, [&](int q) {
            return dline(j, g.n1, g.i2h1, [&](int r) { return Z(q, r); });
        });
    }
}

// Whether a step has at most two blocks for each of the chip's 152 SMs (whole grid, so that every
// band decides alike).
bool step3d_wide(const Geom &g)
{
    return (int64_t)((g.n0 + TX - 1) / TX) * ((g.n1 + TY - 1) / TY) * ((g.n2 + TZ - 1) / TZ) <= 2 * 152;
}

template <int TR, int VK, int CR, bool WIDE = false>
cudaError_t launch_t(const StepLaunch &a, cudaStream_t s, int z0, int z1)
{
    using T = Tile3<CR>;
    static PerDevice ready;
    cudaError_t e = ready.once([] { return allow_dynamic_smem(k_step3d<TR, VK, CR, WIDE>, T::SMEM); });
    if (e != cudaSuccess) return e;
    dim3 block(TX, TY);
    dim3 grid((a.geom.n0 + TX - 1) / TX, (a.geom.n1 + TY - 1) / TY, (z1 - z0 + TZ - 1) / TZ);
    const CUtensorMap &map = *a.tmap[0][CR == CROSS_PLANE];
    return launch_kernel(k_step3d<TR, VK, CR, WIDE>, grid, block, T::SMEM, s, a.dependent, a.in, a.out, a.geom, a.vp, a.coef,
                         (float)a.dt, map, a.err, z0);
}

template <int TR, int VK>
cudaError_t launch_cr(const StepLaunch &a, cudaStream_t s, int z0, int z1)
{
    if (a.cross_in == CROSS_CELL) return launch_t<TR, VK, CROSS_CELL>(a, s, z0, z1);
    if (a.cross_in == CROSS_PLANE) return launch_t<TR, VK, CROSS_PLANE>(a, s, z0, z1);
    return step3d_wide(a.geom) ? launch_t<TR, VK, CROSS_RECON, true>(a, s, z0, z1)
                               : launch_t<TR, VK, CROSS_RECON>(a, s, z0, z1);
}

template <int VK>
cudaError_t launch_tr(const StepLaunch &a, cudaStream_t s, int z0, int z1)
{
    if (a.trace == TR_HEUN) return launch_cr<TR_HEUN, VK>(a, s, z0, z1);
    return a.trace == TR_EULER ? launch_cr<TR_EULER, VK>(a, s, z0, z1)
                               : launch_cr<TR_RK3, VK>(a, s, z0, z1);
}

// step kernel over the z-levels [z0, z1)
cudaError_t launch_step_tiles(const StepLaunch &a, cudaStream_t s, int z0, int z1)
{
    switch (a.vp.kind) {
    case VK_CONST: return launch_tr<VK_CONST>(a, s, z0, z1);
    case VK_ROTATION: return launch_tr<VK_ROTATION>(a, s, z0, z1);
    case VK_DEFORM3D: return launch_tr<VK_DEFORM3D>(a, s, z0, z1);
    default: return cudaErrorInvalidValue;
    }
}

// reconstruction of the z-slabs [zq0, zq0 + nzq) of the new state
cudaError_t launch_recon_slabs(const StepLaunch &a, cudaStream_t s, int zq0, int nzq)
{
    dim3 grid((a.geom.n0 + QX - 1) / QX, (a.geom.n1 + QY - 1) / QY, nzq);
    return launch_kernel(k_recon3d_tma, grid, dim3(QX, QY), 0, s, a.dependent, a.out, a.geom, *a.tmap_cross, a.err, zq0);
}

}  // namespace

cudaError_t launch_step3d(const StepLaunch &a, cudaStream_t s)
{
    // z-levels of the band (all by default); the reconstruction of a level needs the new
    // psi_y, psi_z of that level only
    static_assert(TZ == 4 && QZ == 4, "bands are whole tiles of both kernels");
    const int z0 = a.band_lo, z1 = a.band_hi > 0 ? a.band_hi : a.geom.n2;
    if (z1 <= z0) return cudaSuccess;
    cudaError_t e = launch_step_tiles(a, s, z0, z1);
    if (e != cudaSuccess || !a.write_cross) return e;
    return launch_recon_slabs(a, s, z0 / QZ, (z1 - z0 + QZ - 1) / QZ);
}

void recon_box3d(uint32_t box[4])
{
    box[0] = QW; box[1] = QH; box[2] = QZ; box[3] = 2;
}

void tile_box3d(int cross_recon, uint32_t box[4])
{
    if (cross_recon) {
        using T = Tile3<CROSS_RECON>;
        box[0] = T::W; box[1] = T::H; box[2] = T::D; box[3] = T::NP;
    } else {
        using T = Tile3<CROSS_PLANE>;
        box[0] = T::W; box[1] = T::H; box[2] = T::D; box[3] = T::NP;
    }
}

cudaError_t launch_recon3d(const Geom &g, float *buf, cudaStream_t s)
{
    dim3 block(RX, RY);
    dim3 grid((g.n0 + RX - 1) / RX, (g.n1 + RY - 1) / RY, (g.n2 + RZ - 1) / RZ);
    k_recon3d<<<grid, block, 0, s>>>(buf + 2 * g.plane, buf + 3 * g.plane, buf + 4 * g.plane, g);
    return cudaGetLastError();
}

}  // namespace gals
