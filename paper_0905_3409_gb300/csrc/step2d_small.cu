// step2d_small.cu -- all steps of a run on a small 2D grid in one launch of one thread-block
// cluster, with the state kept in the cluster's shared memory.
//
// What bounds a small grid is latency, not work: a step of a 64^2 grid is 4096 nodes, and as
// one launch (or two bands) per step it took 6.8 us, of which the chip worked for well
// under one.  Here the rows of the grid are dealt out to up to 16 blocks of a cluster
// (distributed shared memory), each thread advances one pair of rows of one column per
// step, a foot's cell is read from the block that owns its row (any distance: no halo and
// no bound on the feet), and one cluster barrier separates the steps, whose two state
// buffers alternate.  Steps after the first rebuild a cell's mixed derivatives from the
// psi_y window around it (the stencils of the plane, so the same bits); the last step's
// phi_xy plane is written at the end.  The per-node arithmetic is that of the tile step.
// A node's data lie together in shared memory: with a plane each, the gathers were 24 more
// load and address instructions per pair and the 64^2 step 0.1 us longer.
// Measured (GB300, 256-step calls, us per step, against the banded graph of launches):
// 64^2 vortex 1.18 against 6.8, 128 x 96 1.78 against 7.2 (128 x 97); 16-mode Fourier field
// 1.96 and 3.15 against 12.0 (128 x 97).  It is a chain of dependent instructions at one
// to four warps per scheduler; of a 64^2 step the barrier and its fence are about 600 of
// 2450 cycles.
#include "step2d_tile.cuh"

namespace gals {

namespace {

using namespace t2;

constexpr int kSmallThreads = 512;   // at most (128 registers a thread)
constexpr int kSmallCluster = 16;    // blocks of the cluster, where the device schedules them

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// address of `local` (this block's shared memory) in block `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}

__device__ __forceinline__ float ld_cluster(uint32_t a)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ float4 ld_cluster4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}

// What a step reads from its coefficients, double-buffered: the next step's are copied
// asynchronously while this one runs (a plain load into shared memory stalled every thread's
// step by the latency of L2).
struct SmallCoef {
    StageCoef sc;        // mod and wamp only
    StageCoefPair scp;   // FOURIER2D tables
};

__device__ __forceinline__ void copy_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

template <int VK>
__device__ __forceinline__ void load_coef(SmallCoef &dst, const StageCoef *__restrict__ c)
{
    const int tid = threadIdx.x;
    if (tid < 3) copy_async4(&dst.sc.mod[tid], &c->mod[tid]);
    if (VK == VK_WAVES2D && tid < 2)
        copy_async4(reinterpret_cast<float *>(&dst.sc.wamp) + tid, reinterpret_cast<const float *>(&c->wamp) + tid);
    if (VK == VK_FOURIER2D)  // both halves of a pair hold the coefficient
        for (int e = tid; e < 6 * 48; e += blockDim.x) {
            const int half = e & 1, tab = e / 96, q = e % 96 / 2, st = q / 16, kl = q % 16;
            const float *src = tab == 0 ? &c->A[st][kl] : (tab == 1 ? &c->Al[st][kl] : &c->All[st][kl]);
            F2 *d = tab == 0 ? &dst.scp.A[st][kl] : (tab == 1 ? &dst.scp.Al[st][kl] : &dst.scp.All[st][kl]);
            copy_async4(reinterpret_cast<float *>(d) + half, src);
        }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// before the barrier that publishes them
__device__ __forceinline__ void wait_coef() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A thread's pair of nodes: column i, rows j0 = row0 + r and j1, and what of the stage-1
// velocity depends on the position only.
template <int VK> struct SmallPair {
    int i, r, j0, j1;
    F2 x, y;
    float A, B;   // VORTEX2D column factors
    Sep2 ry;      // and row factors
    __device__ __forceinline__ void set(const Geom &g, int row0, int i_, int r_)
    {
        i = i_;
        r = r_;
        j0 = row0 + r;
        j1 = min(j0 + 1, g.n1 - 1);
        x = bc(node_pos(g.lo0, i, g.h0));
        y = make_float2(node_pos(g.lo1, j0, g.h1), node_pos(g.lo1, j1, g.h1));
        if (VK == VK_VORTEX2D) {
            sincos_turn(x.x, &A, &B);
            ry = sep_factors2(y);
        }
    }
};

// Block r of the cluster owns rows [r R, (r + 1) R) (R even).  Shared memory of a block:
// two buffers of R x n0 nodes (phi, psi_x, psi_y, and phi_xy in the buffer that the first
// step reads, if `planes`), a node's data together: one 16-byte load per corner.
// CR: CROSS_RECON (approach A) or CROSS_CELL.
template <int TR, int VK, int CR>
__global__ void __launch_bounds__(kSmallThreads)
k_step2d_small(const float *in, float *out, Geom g, VelParams vp, const StageCoef *__restrict__ coef,
               float dt, int nsteps, int R, int planes, int write_cross)
{
    extern __shared__ __align__(16) float4 smem[];
    __shared__ SmallCoef sc[2];
    const int tid = threadIdx.x, n0 = g.n0, PS = R * n0;
    const int row0 = (int)cluster_rank() * R;
    const int rows = max(0, min(R, g.n1 - row0));
    for (int e = tid; e < rows * n0; e += blockDim.x) {
        const int r = e / n0, i = e - r * n0;
        const int64_t o = (int64_t)(row0 + r) * g.pitch + i;
        smem[e] = make_float4(in[o], in[g.plane + o], in[2 * g.plane + o], planes ? in[3 * g.plane + o] : 0.f);
    }
    load_coef<VK>(sc[0], coef);
    wait_coef();
    cluster_sync();

    const int npairs = (rows + 1) / 2 * n0;  // rows past the block's are not stored
    const float invR = 1.f / (float)R;
    SmallPair<VK> P;
    if (tid < npairs) P.set(g, row0, tid % n0, tid / n0 * 2);
    for (int s = 0; s < nsteps; ++s) {
        const float4 *src = smem + (s & 1) * PS;
        float4 *dst = smem + (1 - (s & 1)) * PS;
        const uint32_t src_u = smem_u32(src);
        const bool plane_now = planes && s == 0;
        const SmallCoef &cf = sc[s & 1];
        if (s + 1 < nsteps) load_coef<VK>(sc[(s + 1) & 1], coef + s + 1);
        // the cell (k, l) of one lane from the blocks that own its two rows
        auto gather = [&](int k, int l, float c[4][4]) {
#pragma unroll
            for (int B = 0; B < 2; ++B) {
                const int lr = l + B - row0;
                float4 a0, a1;
                float w0 = 0.f, w3 = 0.f;
                const int kl = k > 0 ? -1 : 0, kr = k + 2 < n0 ? 2 : 1;
                if (lr >= 0 && lr < R) {
                    const float4 *t = src + GALS_CHK(g, lr * n0 + k, PS - 1);
                    a0 = t[0];
                    a1 = t[1];
                    if (CR == CROSS_RECON) {
                        w0 = t[kl].z;
                        w3 = t[kr].z;
                    }
                } else {
                    const int rank = (int)(((float)(l + B) + 0.5f) * invR);  // exact: rows are few
                    const uint32_t t = map_rank(src_u, (uint32_t)rank) +
                                       16u * (uint32_t)GALS_CHK(g, (l + B - rank * R) * n0 + k, PS - 1);
                    a0 = ld_cluster4(t);
                    a1 = ld_cluster4(t + 16u);
                    if (CR == CROSS_RECON) {
                        w0 = ld_cluster(t + (uint32_t)(16 * kl + 8));
                        w3 = ld_cluster(t + (uint32_t)(16 * kr + 8));
                    }
                }
                c[2 * B][0] = a0.x; c[2 * B][1] = a0.y; c[2 * B][2] = a0.z;
                c[2 * B + 1][0] = a1.x; c[2 * B + 1][1] = a1.y; c[2 * B + 1][2] = a1.z;
                if (CR == CROSS_RECON) {
                    const float w[4] = {w0, a0.z, a1.z, w3};
                    c[2 * B][3] = plane_now ? a0.w : cross_from_window<0>(w, k, n0, g.i2h0);
                    c[2 * B + 1][3] = plane_now ? a1.w : cross_from_window<1>(w, k + 1, n0, g.i2h0);
                }
            }
            if (CR == CROSS_CELL) cross_cell2d(c, g.ih0, g.ih1);
        };
        for (int p = tid; p < npairs; p += blockDim.x) {
            if (npairs > blockDim.x) P.set(g, row0, p % n0, p / n0 * 2);
            const VCol cx = (VK == VK_VORTEX2D) ? vortex_col_from(P.A, P.B, cf.sc.mod[0]) : VCol{0.f, 0.f, 0.f, 0.f, 0.f};
            F2 dx, dy, J[4], phi, px, py;
            trace2d_pair<TR, VK>(stage1_pair<VK>(vp, cf.sc, &cf.scp, P.x, P.y, cx, P.ry), vp, cf.sc, &cf.scp, P.x,
                                 P.y, dt, dx, dy, J);
            node2d_foot<TR, VK>(g, vp, cf.sc, &cf.scp, dt, P.i, P.j0, P.i, P.j1, P.x, P.y, dx, dy, J, cx, P.ry,
                                gather, phi, px, py, nullptr);
            float4 *t = dst + GALS_CHK(g, P.r * n0 + P.i, PS);
            t[0] = make_float4(phi.x, px.x, py.x, 0.f);
            if (P.r + 1 < rows) t[n0] = make_float4(phi.y, px.y, py.y, 0.f);
        }
        wait_coef();
        cluster_sync();  // every block's rows of the new state are in place and the old ones read
    }

    const float4 *fin = smem + (nsteps & 1) * PS;
    for (int e = tid; e < rows * n0; e += blockDim.x) {
        const int r = e / n0, i = e - r * n0;
        const int64_t o = (int64_t)(row0 + r) * g.pitch + i;
        const float4 v = fin[e];
        out[o] = v.x;
        out[g.plane + o] = v.y;
        out[2 * g.plane + o] = v.z;
        if (write_cross) {
            const float4 *line = fin + r * n0;
            out[3 * g.plane + o] = dline(i, n0, g.i2h0, [&](int q) { return line[q].z; });
        }
    }
}

// Rows per block: even, and at most `cluster` blocks.
int rows_per_block(int n1, int cluster) { return (n1 + 2 * cluster - 1) / (2 * cluster) * 2; }

size_t small_bytes(const Geom &g, int R) { return sizeof(float4) * 2 * (size_t)R * g.n0; }

template <int TR, int VK, int CR>
cudaError_t launch_t(const SmallLaunch &a, cudaStream_t s, bool *done)
{
    auto kern = k_step2d_small<TR, VK, CR>;
    static PerDevice fit;  // per instantiation
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cfg.stream = s;
    // 16 blocks where the device can place them, else 8, else (0) no cluster at all
    int cluster = 0;
    cudaError_t e = fit.get(&cluster, [&](int *out) {
        const bool smem = allow_dynamic_smem(kern, kSmallMaxBytes) == cudaSuccess;
        const bool large = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        cfg.blockDim = dim3(kSmallThreads);
        cfg.dynamicSmemBytes = kSmallMaxBytes;
        *out = large ? kSmallCluster : 8;
        for (int nc = 0; smem && *out >= 8; *out /= 2) {
            at.val.clusterDim.x = *out;
            cfg.gridDim = dim3(*out);
            if (cudaOccupancyMaxActiveClusters(&nc, kern, &cfg) == cudaSuccess && nc >= 1) break;
        }
        cudaGetLastError();  // of what this device does not have
        if (!smem || *out < 8) *out = 0;
        return cudaSuccess;
    });
    if (e != cudaSuccess || cluster == 0) return e;
    *done = true;
    const int R = rows_per_block(a.geom.n1, cluster);
    const int pairs = (R / 2) * a.geom.n0;
    at.val.clusterDim.x = cluster;
    cfg.gridDim = dim3(cluster);
    cfg.blockDim = dim3(std::min(kSmallThreads, (pairs + 31) / 32 * 32));
    cfg.dynamicSmemBytes = small_bytes(a.geom, R);
    return cudaLaunchKernelEx(&cfg, kern, a.in, a.out, a.geom, a.vp, a.coef, (float)a.dt, a.nsteps, R, a.planes,
                              a.write_cross);
}

template <int TR, int VK>
cudaError_t launch_cr(const SmallLaunch &a, cudaStream_t s, bool *done)
{
    return a.cell ? launch_t<TR, VK, CROSS_CELL>(a, s, done) : launch_t<TR, VK, CROSS_RECON>(a, s, done);
}

template <int VK>
cudaError_t launch_tr(const SmallLaunch &a, cudaStream_t s, bool *done)
{
    if (a.trace == TR_HEUN) return launch_cr<TR_HEUN, VK>(a, s, done);
    return a.trace == TR_EULER ? launch_cr<TR_EULER, VK>(a, s, done) : launch_cr<TR_RK3, VK>(a, s, done);
}

}  // namespace

bool small2d_fits(const Geom &g)
{
    // the shared memory of the 8-block cluster, the larger of the two cases
    return g.n0 <= kSmallColumns && (int64_t)g.n0 * g.n1 <= kSmallNodes &&
           small_bytes(g, rows_per_block(g.n1, 8)) <= (size_t)kSmallMaxBytes;
}

cudaError_t launch_step2d_small(const SmallLaunch &a, cudaStream_t s, bool *done)
{
    *done = false;
    switch (a.vp.kind) {
    case VK_CONST: return launch_tr<VK_CONST>(a, s, done);
    case VK_ROTATION: return launch_tr<VK_ROTATION>(a, s, done);
    case VK_VORTEX2D: return launch_tr<VK_VORTEX2D>(a, s, done);
    case VK_PSEUDO1D: return launch_tr<VK_PSEUDO1D>(a, s, done);
    case VK_FOURIER2D: return launch_tr<VK_FOURIER2D>(a, s, done);
    case VK_WAVES2D: return launch_tr<VK_WAVES2D>(a, s, done);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace gals
