// mlp_infer.cu -- tensor-core (tcgen05 + TMEM) inference of the flow-map surrogate and the
// surrogate trace of one GALS step.
//
// A block holds all 16-bit weights (120 KB with the bias slabs) in shared memory and runs
// NWG = 3 groups of 4 warps, each with its own 128-point tile in flight, so that one tile's
// epilogue overlaps another tile's matrix products.  Per layer and group, one elected
// thread issues tcgen05.mma (M = 128 points, N = 128 units (16 for the output layer),
// K = 16 per instruction, FP16 operands from shared memory, FP32 accumulator in TMEM, 128
// columns per group) and commits them to the group's mbarrier; after a bounded wait each
// thread reads its accumulator row back with tcgen05.ld (the bias is one more K-slab of the
// product), applies SiLU on FP16 pairs and stores the FP16 activations as the next layer's
// A operand.  (GALS_MLP_F16=0 builds the former BF16 operands, SiLU in FP32 with tanh on
// FP16 pairs.)  Operands use the no-swizzle K-major core-matrix layout: 8 rows
// x 16 bytes per core matrix, core matrices adjacent in K `lbo` bytes apart and adjacent
// in M/N 128 bytes apart.  The trace kernel turns the outputs into the foot displacement
// and the Jacobian of the backward map; a fifth warp per group checks a few nodes of every
// tile against the exact RK3 trace (Sec. 5.1), and the group recomputes the whole tile with
// RK3 when the check fails.
#include <cuda_fp16.h>

#include "mlp_internal.h"
#include "tc.cuh"
#include "tma.cuh"

#ifndef GALS_MLP_F16
#define GALS_MLP_F16 1
#endif

namespace gals {
namespace mlp {

using namespace tc;

namespace {

constexpr bool kF16 = GALS_MLP_F16;  // operand type of every inference product

__device__ __forceinline__ uint16_t to_op(float v)
{
    return kF16 ? __half_as_ushort(__float2half_rn(v)) : __bfloat16_as_ushort(__float2bfloat16(v));
}
__device__ __forceinline__ uint32_t pack_op(float a, float b) { return kF16 ? pack_f16(a, b) : pack_bf16(a, b); }
__host__ __device__ constexpr uint32_t idesc_op(int M, int N) { return kF16 ? idesc_f16(M, N) : idesc_bf16(M, N); }

constexpr int NWG = 3;               // tile groups (tiles in flight) per block
constexpr int GT = 128;              // threads per tile group: one per accumulator row
                                     // (four warps, one per TMEM lane quarter)
constexpr int NT = GT * NWG;         // threads per block
constexpr int ROWS = 128;            // points per tile (= M of the products, = TMEM lanes)
constexpr uint32_t TMEM_COLS = NWG <= 2 ? 256 : 512;  // power of two >= NWG * 128
constexpr int kErrMmaTimeout = 2;

struct Smem {
    uint16_t w[W_TOTAL];                 // packed operands (weights, bias slabs, ones block)
    __align__(1024) uint16_t act[NWG][ROWS * HID];  // A operand of each group's tile
    uint64_t bar[NWG];
    uint32_t tmem;                       // TMEM base address from tcgen05.alloc
    int fail[NWG];
};

__device__ __forceinline__ void wg_sync(int g)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(GT) : "memory");
}
// named barrier of the tile group that also ORs a flag over its threads
__device__ __forceinline__ int wg_sync_or(int g, int flag)
{
    int r;
    asm volatile(
        "{\n .reg .pred q, o;\n setp.ne.s32 q, %1, 0;\n bar.red.or.pred o, %2, %3, q;\n"
        " selp.s32 %0, 1, 0, o;\n}\n"
        : "=r"(r)
        : "r"(flag), "r"(1 + g), "n"(GT)
        : "memory");
    return r;
}

// SiLU of two pre-activations given as h = z/2 (FP32): silu(z) = z (1 + tanh(z/2)) / 2
// = h + h tanh(h), returned as an operand pair.  FP16 operands: h rounded to FP16, tanh on
// the FP16 pair (one MUFU operation for two values, relative error about 1e-3) and one
// FP16 fused multiply-add, whose result is the next layer's operand pair as it stands
// (FP16 carries 3 more mantissa bits than BF16).  BF16 operands: the multiply-add in FP32
// and the result rounded to BF16.
__device__ __forceinline__ uint32_t silu2_op(float2 h)
{
    const __half2 hh = __floats2half2_rn(h.x, h.y);
    uint32_t tr;
    asm("tanh.approx.f16x2 %0, %1;" : "=r"(tr) : "r"(*reinterpret_cast<const uint32_t *>(&hh)));
    if (kF16) {
        const __half2 y = __hfma2(hh, *reinterpret_cast<const __half2 *>(&tr), hh);
        return *reinterpret_cast<const uint32_t *>(&y);
    }
    const float2 t = __half22float2(*reinterpret_cast<const __half2 *>(&tr));
    const float2 y = __ffma2_rn(h, t, h);
    return pack_bf16(y.x, y.y);
}

// ---- block setup / teardown ----

// Weights and biases into shared memory, barriers, TMEM allocation (warp 0).
__device__ void block_setup(Smem &sm, const InferParams &ip)
{
    const uint4 *src = reinterpret_cast<const uint4 *>(ip.w);
    uint4 *dst = reinterpret_cast<uint4 *>(sm.w);
    for (int e = threadIdx.x; e < (int)(W_TOTAL * 2 / 16); e += blockDim.x) dst[e] = src[e];
    if (threadIdx.x < NWG) {
        mbar_init(&sm.bar[threadIdx.x], 1);
        sm.fail[threadIdx.x] = 0;
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&sm.tmem)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}

__device__ void block_teardown(Smem &sm)
{
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(TMEM_COLS)
                     : "memory");
}

// Per-thread state of the tile engine.  Tile group g owns TMEM columns 128g..128g+127;
// warp q of the group reads TMEM lane quarter q (rows 32q..32q+31).
struct Wg {
    int g;            // tile group
    int r;            // thread's row = TMEM lane
    uint32_t tcol;    // TMEM address of the group's accumulator, lane 0
    uint32_t tlane;   // this warp's TMEM lane base, in address units
    uint32_t phase;   // parity of the group's mbarrier
};

__device__ __forceinline__ Wg make_wg(const Smem &sm)
{
    Wg w;
    w.g = threadIdx.x / GT;
    w.r = threadIdx.x % GT;
    w.tcol = sm.tmem + (uint32_t)(128 * w.g);
    w.tlane = (uint32_t)((w.r & ~31) << 16);
    w.phase = 0u;
    return w;
}

// Row r's network input (x, y, phase in [-1, 1], then 1 for the bias, K padded to 16 with
// zeros) as the first layer's A operand; then the group barrier that publishes it to the
// tensor core.
__device__ __forceinline__ void stage_input(Smem &sm, const Wg &w, float a, float b, float c)
{
    char *base = reinterpret_cast<char *>(sm.act[w.g]) + (w.r >> 3) * 128 + (w.r & 7) * 16;
    *reinterpret_cast<uint4 *>(base) = make_uint4(pack_op(a, b), pack_op(c, 1.f), 0u, 0u);
    *reinterpret_cast<uint4 *>(base + 2048) = make_uint4(0u, 0u, 0u, 0u);
    fence_async_smem();
    wg_sync(w.g);
}

// The network on the warpgroup's staged tile: out[0..5] = outputs of row r (+ 2 padding).
// Returns false (after recording the error) if a product did not complete in time.
__device__ bool run_tile(Smem &sm, Wg &w, int *err, float out[8])
{
    const int g = w.g;
    const char *act = reinterpret_cast<const char *>(sm.act[g]);
    const char *wts = reinterpret_cast<const char *>(sm.w);
    const bool leader = threadIdx.x % GT == 0;
    for (int L = 0; L < NLAYER; ++L) {
        if (leader) {
            tc_fence_after();
            if (L == 0) {
                umma(w.tcol, sdesc(act, 2048, 128), sdesc(wts + 2 * W1_OFF, 2048, 128),
                     idesc_op(128, 128), 0u);
            } else if (L < NLAYER - 1) {
                const char *W = wts + 2 * (W2_OFF + (int64_t)(L - 1) * 128 * 128);
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    umma(w.tcol, sdesc(act + s * 4096, 2048, 128), sdesc(W + s * 4096, 2048, 128),
                         idesc_op(128, 128), s > 0 ? 1u : 0u);
                umma(w.tcol, sdesc(wts + 2 * ONES_OFF, 2048, 128),
                     sdesc(wts + 2 * (WB_OFF + (int64_t)(L - 1) * 128 * 16), 2048, 128), idesc_op(128, 128), 1u);
            } else {
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    umma(w.tcol, sdesc(act + s * 4096, 2048, 128), sdesc(wts + 2 * W5_OFF + s * 512, 256, 128),
                         idesc_op(128, 16), s > 0 ? 1u : 0u);
                umma(w.tcol, sdesc(wts + 2 * ONES_OFF, 2048, 128), sdesc(wts + 2 * W5B_OFF, 256, 128),
                     idesc_op(128, 16), 1u);
            }
            umma_commit(&sm.bar[g]);
        }
        // one warp polls the barrier; the others sleep in the group barrier below
        const bool ok = (threadIdx.x % GT) < 32 ? mbar_wait_bounded(&sm.bar[g], w.phase) : true;
        w.phase ^= 1u;
        if (wg_sync_or(g, !ok)) {
            if (leader) atomicExch(err, kErrMmaTimeout);
            return false;
        }
        tc_fence_after();
        const uint32_t ta = w.tcol + w.tlane;
        if (L < NLAYER - 1) {
            // SiLU of h = z/2 (the accumulator), BF16 activations of row r as the next
            // layer's A operand (K = 128)
            char *arow = reinterpret_cast<char *>(sm.act[g]) + (w.r >> 3) * 128 + (w.r & 7) * 16;
            // one 32-column TMEM load per wait: two per wait held 64 accumulator values live
            // and pushed the trace kernel past its register cap (spills)
            constexpr int NU = 1;
#pragma unroll 1
            for (int c = 0; c < 4; c += NU) {
                uint32_t v[NU][32];
#pragma unroll
                for (int u = 0; u < NU; ++u) tmem_ld32_nowait(ta + 32 * (c + u), v[u]);
                tmem_wait_ld();
#pragma unroll
                for (int u = 0; u < NU; ++u)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t p[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int k = 8 * q + 2 * e;
                            p[e] = silu2_op(make_float2(__uint_as_float(v[u][k]), __uint_as_float(v[u][k + 1])));
                        }
                        *reinterpret_cast<uint4 *>(arow + (4 * (c + u) + q) * 2048) =
                            make_uint4(p[0], p[1], p[2], p[3]);
                    }
            }
            tc_fence_before();
            fence_async_smem();
            wg_sync(g);
        } else {
            uint32_t v[8];
            tmem_ld8(ta, v);
#pragma unroll
            for (int k = 0; k < 8; ++k) out[k] = __uint_as_float(v[k]);
            tc_fence_before();
        }
    }
    return true;
}

// After an abort: bounded wait for the products still in flight, before TMEM is freed.
__device__ void drain(Smem &sm, const Wg &w, bool aborted)
{
    if (aborted) mbar_wait_bounded(&sm.bar[w.g], w.phase ^ 1u);
}

__global__ void __launch_bounds__(NT, 1)
k_infer_points(InferParams ip, const float *__restrict__ Xn, float *__restrict__ Y, int n, int *err)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    block_setup(sm, ip);
    Wg w = make_wg(sm);
    bool aborted = false;
    const int ntiles = (n + ROWS - 1) / ROWS;
    for (int tile = blockIdx.x * NWG + w.g; tile < ntiles; tile += gridDim.x * NWG) {
        const int p = tile * ROWS + w.r;
        const int64_t pc = min(p, n - 1);
        stage_input(sm, w, Xn[3 * pc], Xn[3 * pc + 1], Xn[3 * pc + 2]);
        float o[8];
        if (!run_tile(sm, w, err, o)) { aborted = true; break; }
        if (p < n)
            for (int c = 0; c < OUT; ++c) Y[6 * (int64_t)p + c] = o[c];
        wg_sync(w.g);  // act[g] is rewritten by the next tile's inputs
    }
    drain(sm, w, aborted);
    block_teardown(sm);
}

__device__ __forceinline__ uint32_t tile_hash(uint32_t a, uint32_t b)
{
    uint32_t h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u;
    h ^= h >> 15;
    h *= 0xC2B2AE3Du;
    return h ^ (h >> 13);
}

// named barrier id: the tile group arrives (or waits), its checking warp waits (or arrives)
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(GT + 32) : "memory"); }
__device__ __forceinline__ void pair_arrive(int id)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(GT + 32) : "memory");
}
constexpr int kBarWritten = 1 + NWG, kBarChecked = 1 + 2 * NWG;
constexpr int NTT = NT + 32 * NWG;  // threads per block of the trace kernel

// Whether one of the tile's sampled nodes (first, first + stride, ...; for a cheap field all of
// them, one per lane) is off the exact RK3 trace: warp-wide; value(q, e): the network's values
// of the tile's node q, delta and J.
template <int VK, class V>
__device__ __forceinline__ bool tile_fails(const InferParams &ip, const Geom &g, const VelParams &vp,
                                           const StageCoef &coef, float dtf, V value, int tile, int tiles_x,
                                           int kstep, const Check &chk, int first, int stride)
{
    const int lane = threadIdx.x & 31;
    const int j = tile / tiles_x, x0 = (tile % tiles_x) * ROWS, width = min(ROWS, g.n0 - x0);
    const float yy = g.lo1 + (float)j * g.h1;
    bool bad = false;
    // a costly field: each node's trace by the whole warp (modes split over the lanes)
    constexpr bool WARP = VK == VK_WAVES2D;
    for (int jj = WARP ? first : lane; jj < chk.samples; jj += WARP ? stride : 32) {
        const int q = (int)(tile_hash((uint32_t)tile, (uint32_t)kstep + 977u * jj) % (uint32_t)width);
        const float xq = g.lo0 + (float)(x0 + q) * g.h0;
        float dr[2], Jr[4], m[6];
#pragma unroll
        for (int e = 0; e < 6; ++e) m[e] = value(q, e);
        if (WARP) trace2d_waves_warp(vp, coef, xq, yy, dtf, dr[0], dr[1], Jr);
        else trace2d<TR_RK3, VK>(vp, coef, xq, yy, dtf, dr[0], dr[1], Jr);
        const float ex = fmaxf(fabsf(m[0] - dr[0]) * g.ih0, fabsf(m[1] - dr[1]) * g.ih1);
        float eJ = 0.f;
        for (int e = 0; e < 4; ++e) eJ = fmaxf(eJ, fabsf(m[2 + e] - Jr[e]));
        bad = bad || !(ex <= chk.tol_x) || !(eJ <= chk.tol_J);
    }
    return __any_sync(0xffffffffu, bad);
}

// Surrogate trace of one step over the grid: tile = 128 consecutive nodes of a row; VK
// is the field of the exact trace the residual check and the fallback run.  Latency bounds the
// kernel (12 warps of network, MUFU and tensor pipes a third busy), and the check of 4 nodes
// is one long FP32 chain on 4 lanes that used to hold up the tile's other threads: now a
// fifth warp of the group checks a tile, read back from the trace planes, while the group
// runs the next one, and the group recomputes a tile that failed one tile later.  2048^2,
// 16 modes, a whole step: 794 -> 733 us with 4 nodes, 809 -> 766 with 128 nodes a tile (four
// rounds of the warp), 876 -> 842 where every tile fails; 500^2 70.5 -> 68.
//
// A costly field keeps the check in the group, a sample per warp with its modes over the
// lanes: one warp alone falls behind the network.  2048^2, us per step in the group / aside:
// 256 waves, 4 nodes 926 / 811, 16 nodes 1397 / 2259, every tile failing 3443 / 3996; 1024
// waves, 4 nodes 1382 / 2262.  The rule looks at the kind of field alone: with few waves and
// nodes aside gains up to 1.14 times, with more of either it costs up to 1.64.
template <int VK> constexpr bool aside() { return VK != VK_WAVES2D; }

template <int VK>
__global__ void __launch_bounds__(aside<VK>() ? NTT : NT, 1)
k_mlp_trace(InferParams ip, Geom g, VelParams vp, const StageCoef *__restrict__ coef,
            const double *__restrict__ t_dev, int kstep, double dt, float *trace, Check chk)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    block_setup(sm, ip);
    const float dtf = (float)dt;
    const int tiles_x = (g.n0 + ROWS - 1) / ROWS;
    const int ntiles = tiles_x * g.n1;
    if (aside<VK>() && threadIdx.x >= NT) {
        const int gg = (threadIdx.x - NT) >> 5;
        const bool lead = (threadIdx.x & 31) == 0;
        for (int tile = blockIdx.x * NWG + gg; tile < ntiles; tile += gridDim.x * NWG) {
            pair_sync(kBarWritten + gg);
            if (sm.fail[gg] < 0) break;  // the group gave up
            const float *at = trace + (int64_t)(tile / tiles_x) * g.pitch + (tile % tiles_x) * ROWS;
            auto value = [&](int q, int e) { return at[e * g.plane + q]; };
            const bool fail = tile_fails<VK>(ip, g, vp, *coef, dtf, value, tile, tiles_x, kstep, chk, 0, 1);
            if (lead) {
                sm.fail[gg] = fail;
                atomicAdd(chk.tiles, 1ull);
                if (fail) atomicAdd(chk.fallbacks, 1ull);
            }
            pair_arrive(kBarChecked + gg);
        }
    } else {
        Wg w = make_wg(sm);
        bool aborted = false;
        const double t = t_dev[0] + (double)kstep * dt;
        const float phase = (float)(t - floor(t));
        int prev = -1;
        auto store = [&](int j, int i, const float (&d)[2], const float (&J)[4]) {
            const int64_t o = (int64_t)j * g.pitch + i;
            trace[o] = d[0];
            trace[g.plane + o] = d[1];
#pragma unroll
            for (int e = 0; e < 4; ++e) trace[(2 + e) * g.plane + o] = J[e];
        };
        auto finish = [&](int tile) {  // the check's verdict on a tile written earlier
            pair_sync(kBarChecked + w.g);
            const int j = tile / tiles_x, i = (tile % tiles_x) * ROWS + w.r;
            if (sm.fail[w.g] && i < g.n0) {
                float d[2], J[4];
                trace2d<TR_RK3, VK>(vp, *coef, g.lo0 + (float)i * g.h0, g.lo1 + (float)j * g.h1, dtf, d[0], d[1], J);
                store(j, i, d, J);
            }
        };
        for (int tile = blockIdx.x * NWG + w.g; tile < ntiles; tile += gridDim.x * NWG) {
            const int j = tile / tiles_x, i = (tile % tiles_x) * ROWS + w.r;
            {
                const float x = g.lo0 + (float)min(i, g.n0 - 1) * g.h0, y = g.lo1 + (float)j * g.h1;
                stage_input(sm, w, 2.f * x - 1.f, 2.f * y - 1.f, 2.f * phase - 1.f);
            }
            float y[8];
            if (!run_tile(sm, w, chk.err, y)) { aborted = true; break; }
            float d[2], J[4];
            d[0] = y[0] * ip.scale[0] * g.h0;
            d[1] = y[1] * ip.scale[1] * g.h1;
            J[0] = 1.f + dtf * y[2] * ip.scale[2];
            J[1] = dtf * y[3] * ip.scale[3];
            J[2] = dtf * y[4] * ip.scale[4];
            J[3] = 1.f + dtf * y[5] * ip.scale[5];
            if (!aside<VK>()) {
                float *outs = reinterpret_cast<float *>(sm.act[w.g]);  // free after the products
#pragma unroll
                for (int e = 0; e < 6; ++e) outs[w.r * 8 + e] = e < 2 ? d[e] : J[e - 2];
                wg_sync(w.g);
                auto value = [&](int q, int e) { return outs[q * 8 + e]; };
                const bool fail = wg_sync_or(w.g, tile_fails<VK>(ip, g, vp, *coef, dtf, value, tile, tiles_x, kstep,
                                                                 chk, w.r >> 5, GT / 32));
                if (fail && i < g.n0)
                    trace2d<TR_RK3, VK>(vp, *coef, g.lo0 + (float)i * g.h0, g.lo1 + (float)j * g.h1, dtf, d[0], d[1], J);
                if (i < g.n0) store(j, i, d, J);
                if (w.r == 0) {
                    atomicAdd(chk.tiles, 1ull);
                    if (fail) atomicAdd(chk.fallbacks, 1ull);
                }
                continue;
            }
            if (i < g.n0) store(j, i, d, J);
            if (prev >= 0) finish(prev);
            pair_arrive(kBarWritten + w.g);
            prev = tile;
        }
        if (aside<VK>() && prev >= 0) finish(prev);
        if (aside<VK>() && aborted) {  // the checking warp waits for the tile that did not come
            wg_sync(w.g);
            sm.fail[w.g] = -1;
            pair_arrive(kBarWritten + w.g);
        }
        drain(sm, w, aborted);
    }
    block_teardown(sm);
}

// FP32 master parameters -> packed 16-bit operands in the core-matrix layout (see
// mlp_internal.h): hidden layers and their biases halved, biases as K-slab columns.
__global__ void k_pack(const float *__restrict__ p, uint16_t *__restrict__ w)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < 128 * 16) {  // W1/2 (inputs 0..2), b1/2 (column 3), zeros
        const int r = e / 16, c = e % 16;
        const float v = c < IN ? p[woff(0) + r * IN + c] : (c == IN ? p[boff(0) + r] : 0.f);
        w[W1_OFF + cm_off(128, r, c) / 2] = to_op(0.5f * v);
    }
    if (e < 3 * 128 * 128) {  // W2/2..W4/2: 128 x 128
        const int L = e / (128 * 128), rem = e % (128 * 128), r = rem / 128, c = rem % 128;
        w[W2_OFF + (int64_t)L * 128 * 128 + cm_off(128, r, c) / 2] = to_op(0.5f * p[woff(1 + L) + rem]);
    }
    if (e < 16 * 128) {  // W5: 16 x 128, rows 6..15 zero
        const int r = e / 128, c = e % 128;
        w[W5_OFF + cm_off(16, r, c) / 2] = to_op(r < OUT ? p[woff(4) + r * 128 + c] : 0.f);
    }
    if (e < 3 * 128 * 16) {  // hidden bias slabs: b/2 in column 0
        const int L = e / (128 * 16), rem = e % (128 * 16), r = rem / 16, c = rem % 16;
        w[WB_OFF + (int64_t)L * 128 * 16 + cm_off(128, r, c) / 2] =
            to_op(c == 0 ? 0.5f * p[boff(1 + L) + r] : 0.f);
    }
    if (e < 16 * 16) {  // output bias slab: b5 in column 0
        const int r = e / 16, c = e % 16;
        w[W5B_OFF + cm_off(16, r, c) / 2] = to_op(c == 0 && r < OUT ? p[boff(4) + r] : 0.f);
    }
    if (e < 128 * 16) {  // ones block
        const int r = e / 16, c = e % 16;
        w[ONES_OFF + cm_off(128, r, c) / 2] = to_op(c == 0 ? 1.f : 0.f);
    }
}

int sm_count()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

static_assert(sizeof(Smem) <= 227 * 1024, "shared memory budget");
static_assert(W_TOTAL * 2 % 16 == 0, "weights are copied in 16-byte chunks");
static_assert(W2_OFF * 2 % 16 == 0 && W5_OFF * 2 % 16 == 0 && WB_OFF * 2 % 16 == 0 &&
                  W5B_OFF * 2 % 16 == 0 && ONES_OFF * 2 % 16 == 0,
              "operands start on 16-byte boundaries");

}  // namespace

cudaError_t pack_infer(const float *params, InferParams &ip, cudaStream_t s)
{
    k_pack<<<(3 * 128 * 128 + 255) / 256, 256, 0, s>>>(params, ip.w);
    return cudaGetLastError();
}

cudaError_t infer_points(const InferParams &ip, const float *Xn, float *Y, int n, int *err, cudaStream_t s)
{
    static PerDevice ready;
    cudaError_t e = ready.once([] { return allow_dynamic_smem(k_infer_points, (int)sizeof(Smem)); });
    if (e != cudaSuccess) return e;
    const int tiles = (n + ROWS - 1) / ROWS, sms = sm_count();
    const int blocks = (tiles + NWG - 1) / NWG;
    k_infer_points<<<blocks < sms ? blocks : sms, NT, sizeof(Smem), s>>>(ip, Xn, Y, n, err);
    return cudaGetLastError();
}

cudaError_t launch_mlp_trace(const InferParams &ip, const Geom &g, const VelParams &vp,
                             const StageCoef *coef, const double *t_dev, int kstep, double dt,
                             float *trace, const Check &chk, cudaStream_t s)
{
    static PerDevice ready;
    cudaError_t e = ready.once([] {
        const cudaError_t a = allow_dynamic_smem(k_mlp_trace<VK_FOURIER2D>, (int)sizeof(Smem));
        return a != cudaSuccess ? a : allow_dynamic_smem(k_mlp_trace<VK_WAVES2D>, (int)sizeof(Smem));
    });
    if (e != cudaSuccess) return e;
    const int ntiles = ((g.n0 + ROWS - 1) / ROWS) * g.n1, sms = sm_count();
    const int blocks = (ntiles + NWG - 1) / NWG;
    auto kern = vp.kind == VK_WAVES2D ? k_mlp_trace<VK_WAVES2D> : k_mlp_trace<VK_FOURIER2D>;
    const int threads = vp.kind == VK_WAVES2D ? NT : NTT;  // aside()
    kern<<<blocks < sms ? blocks : sms, threads, sizeof(Smem), s>>>(ip, g, vp, coef, t_dev, kstep, dt, trace, chk);
    return cudaGetLastError();
}

}  // namespace mlp
}  // namespace gals
