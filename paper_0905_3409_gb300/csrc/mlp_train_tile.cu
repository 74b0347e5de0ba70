// mlp_train_tile.cu -- one optimizer step of the flow-map surrogate in two launches: forward and
// backward pass of a chunk of samples in one block on the tensor cores, then the sum of the
// blocks' gradients and the Adam update.
//
// The general path (mlp_train.cu) is about fifty launches a step, each reading and writing
// n x 128 FP32 matrices; a step of 16384 samples took 570 us of which the products need a
// few.  Here a block owns one split-K chunk of the weight gradients (at most 128 samples, one
// TMEM lane each) and keeps its activations in shared memory from the forward to the
// backward pass: the BF16 activations of the four hidden layers are the A operands of the
// forward products and, read with the other dimension leading (MN-major descriptors), the
// B operands of dW = G^T A; layer l's gradient G_l takes the place of its activations.  The
// pre-activations Z (FP32) wait in a scratch in L2, the weights arrive as one bulk copy per
// layer (packed BF16, written by the Adam kernel) while the previous layer's epilogue runs.
// Operands, accumulation order (K in slabs of 16 samples or units from the chunk's start),
// element functions and the order of every sum are the general path's, so the gradients are
// the same bits.  Measured: see launch_train_tiles.
#include "mlp_internal.h"
#include "tc.cuh"

namespace gals {
namespace mlp {

using namespace tc;

namespace {

constexpr int TT = 256;                 // threads: two warps per TMEM lane quarter
constexpr int kErrTrainTimeout = 5;
constexpr uint32_t ACC = 0, ACCW = 128; // TMEM columns: forward / dA accumulator, two for dW
constexpr int SLD = 33;                 // row stride of the staged gradient columns

struct TrainSmem {
    __align__(1024) uint16_t act[4][128 * HID];  // A_1..A_4, later G_1..G_4 (samples x units)
    uint16_t w[HID * HID];                       // the current layer's weights (units x inputs)
    uint16_t x[128 * 16];                        // inputs, K padded to 16
    uint16_t g5[128 * 16];                       // output gradient
    float stage[2][128 * SLD];                   // FP32 gradient columns for the bias sums
    float bias[2][HID];
    uint64_t bar, wbar;
    uint32_t tmem;
};
static_assert(sizeof(TrainSmem) <= 227 * 1024, "shared memory budget");

// packed BF16 weights: core-matrix operands (units x inputs) of each layer
__host__ __device__ constexpr int64_t wt_off(int l)
{
    return l == 0 ? 0 : (l < 4 ? 2048 + (int64_t)(l - 1) * 16384 : 2048 + 3 * 16384);
}
__host__ __device__ constexpr uint32_t wt_bytes(int l) { return l == 0 || l == 4 ? 4096u : 32768u; }
constexpr int64_t WT_TOTAL = wt_off(4) + 2048;

// position of parameter e (flat order) in the packed weights, -1 for a bias
__device__ __forceinline__ int packed_at(int e)
{
    if (e < (int)boff(0)) return (int)(cm_off(128, e / IN, e % IN) / 2);
    if (e >= (int)woff(4)) {
        const int q = e - (int)woff(4);
        return q < OUT * HID ? (int)wt_off(4) + (int)(cm_off(16, q / HID, q % HID) / 2) : -1;
    }
    if (e < (int)woff(1)) return -1;
    const int l = 1 + (e - (int)woff(1)) / (HID * HID + HID), q = (e - (int)woff(1)) % (HID * HID + HID);
    return q < HID * HID ? (int)wt_off(l) + (int)(cm_off(128, q / HID, q % HID) / 2) : -1;
}

__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    mbar_arrive_expect_tx(bar, bytes);
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// operand bits of the instruction descriptor: A / B with the M / N dimension leading
constexpr uint32_t A_MN = 1u << 15, B_MN = 1u << 16;

// Descriptors of K-slab q (16 deep) of a buffer of R rows in the core-matrix layout: rows as
// the M/N dimension (K along the columns), or as K (M/N along the columns).
__device__ __forceinline__ uint64_t rows_mn(const void *p, int R, int q)
{
    return sdesc(reinterpret_cast<const char *>(p) + q * 2 * R * 16, R * 16, 128);
}
__device__ __forceinline__ uint64_t rows_k(const void *p, int R, int q)
{
    return sdesc(reinterpret_cast<const char *>(p) + q * 256, 128, R * 16);
}

// Row r, units 8 u8 .. 8 u8 + 7 of a 128-row operand.
__device__ __forceinline__ void put8(uint16_t *buf, int r, int u8, const float *v)
{
    *reinterpret_cast<uint4 *>(reinterpret_cast<char *>(buf) + u8 * 2048 + (r >> 3) * 128 + (r & 7) * 16) =
        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}

__global__ void __launch_bounds__(TT, 1)
k_train_tile(const float *__restrict__ params, const uint16_t *__restrict__ wt, const float *__restrict__ X,
             const float *__restrict__ T, int n, int chunk, float4 *__restrict__ Zs, float *__restrict__ part,
             double *loss, int *__restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    TrainSmem &sm = *reinterpret_cast<TrainSmem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, half = warp >> 2;
    const int r = (warp & 3) * 32 + (tid & 31);        // sample row = TMEM lane
    const int i0 = blockIdx.x * chunk, rows = min(chunk, n - i0);
    part += (int64_t)blockIdx.x * kPartStride;
    Zs += (int64_t)blockIdx.x * 4 * (HID / 4) * 128;   // [layer][column / 4][row]

    if (tid == 0) {
        mbar_init(&sm.bar, 1);
        mbar_init(&sm.wbar, 1);
    }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (half == 0) {
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (r < rows)
            for (int k = 0; k < IN; ++k) v[k] = X[3 * (int64_t)(i0 + r) + k];
        put8(sm.x, r, 0, v);
        v[0] = v[1] = v[2] = 0.f;
        put8(sm.x, r, 1, v);
    } else {
        sm.bias[0][r] = params[boff(0) + r];
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = sm.tmem;
    const uint32_t lane0 = (uint32_t)(warp & 3) << 21;  // this warp's TMEM lanes
    uint32_t phase = 0, wphase = 0;
    // products / a weight copy in flight that nothing waited for
    bool ok = true, pending = false, wpending = true;
    if (tid == 0) bulk_load(sm.w, wt, wt_bytes(0), &sm.wbar);

    // every thread: wait for the products / for the weights (bounded, one verdict per block)
    auto wait_mma = [&]() {
        ok = mbar_wait_block(&sm.bar, phase);
        if (ok) {
            phase ^= 1u;
            pending = false;
        }
        tc_fence_after();
        return ok;
    };
    auto wait_w = [&]() {
        ok = mbar_wait_block(&sm.wbar, wphase);
        if (ok) {
            wphase ^= 1u;
            wpending = false;
        }
        return ok;
    };
    auto publish = [&]() {  // shared-memory operands written, TMEM reads done
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
    };

    // ---- forward
    do {
        if (!wait_w()) break;
        if (tid == 0) {
            tc_fence_after();
            umma(tbase + ACC, rows_mn(sm.x, 128, 0), rows_mn(sm.w, 128, 0), idesc_bf16(128, 128), 0u);
            umma_commit(&sm.bar);
        }
        pending = true;
        for (int L = 1; L <= 4 && ok; ++L) {  // hidden layer L: Z_L, A_L, then the next product
            if (!wait_mma()) break;
            if (tid == 0) bulk_load(sm.w, wt + wt_off(L), wt_bytes(L), &sm.wbar);
            wpending = true;
            const float *bias = sm.bias[(L - 1) & 1];
            float4 *zrow = Zs + ((int64_t)(L - 1) * 32 + half * 16) * 128 + r;
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                uint32_t v[32];
                const int col = half * 64 + c * 32;
                tmem_ld32_nowait(tbase + ACC + lane0 + (uint32_t)col, v);
                tmem_wait_ld();
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float z[8], a[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        z[e] = __fadd_rn(__uint_as_float(v[8 * q + e]), bias[col + 8 * q + e]);
                        a[e] = silu(z[e]);
                    }
                    zrow[(c * 8 + 2 * q) * 128] = make_float4(z[0], z[1], z[2], z[3]);
                    zrow[(c * 8 + 2 * q + 1) * 128] = make_float4(z[4], z[5], z[6], z[7]);
                    put8(sm.act[L - 1], r, col / 8 + q, a);
                }
            }
            if (half == 0 && r < lout(L)) sm.bias[L & 1][r] = params[boff(L) + r];
            publish();
            if (!wait_w()) break;
            if (tid == 0) {
                tc_fence_after();
                const uint32_t id = L < 4 ? idesc_bf16(128, 128) : idesc_bf16(128, 16);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    umma(tbase + ACC, rows_mn(sm.act[L - 1], 128, q), rows_mn(sm.w, L < 4 ? 128 : 16, q), id, q > 0);
                umma_commit(&sm.bar);
            }
            pending = true;
        }
        if (!ok || !wait_mma()) break;

        // ---- output: Y, its gradient, the loss
        if (half == 0) {
            uint32_t v[8];
            tmem_ld8(tbase + ACC + lane0, v);
            float g[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            double l = 0.0;
            const float nout = (float)((int64_t)n * OUT);
            if (r < rows)
#pragma unroll
                for (int k = 0; k < OUT; ++k) {
                    const float d = __fadd_rn(__uint_as_float(v[k]), sm.bias[0][k]) - T[6 * (int64_t)(i0 + r) + k];
                    g[k] = 2.f * d / nout;
                    l += (double)d * d;
                }
            put8(sm.g5, r, 0, g);
#pragma unroll
            for (int k = 0; k < OUT; ++k) sm.stage[0][r * SLD + k] = g[k];
            g[0] = g[1] = g[2] = g[3] = g[4] = g[5] = 0.f;
            put8(sm.g5, r, 1, g);
            if (loss) {
                for (int off = 16; off > 0; off >>= 1) l += __shfl_down_sync(0xffffffffu, l, off);
                if ((tid & 31) == 0) atomicAdd(loss, l / (double)((int64_t)n * OUT));
            }
        }
        publish();
        if (tid == 0) {
            tc_fence_after();
            // dW_5^T (inputs x outputs) = A_4^T G_5, dA_4 = G_5 W_5
#pragma unroll
            for (int q = 0; q < 8; ++q)
                umma(tbase + ACCW + 128, rows_k(sm.act[3], 128, q), rows_k(sm.g5, 128, q),
                     idesc_bf16(128, 16) | A_MN | B_MN, q > 0);
            umma(tbase + ACC, rows_mn(sm.g5, 128, 0), rows_k(sm.w, 16, 0), idesc_bf16(128, 128) | B_MN, 0u);
            umma_commit(&sm.bar);
        }
        pending = true;
        if (tid < OUT) {
            float s = 0.f;
            for (int k = 0; k < rows; ++k) s = __fadd_rn(s, sm.stage[0][k * SLD + tid]);
            part[boff(4) + tid] = s;
        }

        // ---- backward through hidden layer L: G_L = dA_L silu'(Z_L)
        for (int L = 4; L >= 1 && ok; --L) {
            float4 zp[16];
            const float4 *zrow = Zs + ((int64_t)(L - 1) * 32 + half * 16) * 128 + r;
#pragma unroll
            for (int q = 0; q < 16; ++q) zp[q] = zrow[q * 128];
            if (!wait_mma()) break;  // dA_L, and dW_{L+1}: A_L's place and the weights are free
            if (tid == 0 && L > 1) bulk_load(sm.w, wt + wt_off(L - 1), wt_bytes(L - 1), &sm.wbar);
            wpending = L > 1;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t v[32];
                const int col = half * 64 + c * 32;
                tmem_ld32_nowait(tbase + ACC + lane0 + (uint32_t)col, v);
                tmem_wait_ld();
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 z0 = zp[c * 8 + 2 * q], z1 = zp[c * 8 + 2 * q + 1];
                    const float z[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
                    float g[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        g[e] = __uint_as_float(v[8 * q + e]) * silu_prime(z[e]);
                        sm.stage[half][r * SLD + 8 * q + e] = g[e];
                    }
                    put8(sm.act[L - 1], r, col / 8 + q, g);
                }
                __syncthreads();
                if ((warp & 3) == 0) {  // the bias sums of these columns, rows in order
                    const float *st = sm.stage[half] + (tid & 31);
                    float s = 0.f;
#pragma unroll 16
                    for (int k = 0; k < rows; ++k) s = __fadd_rn(s, st[k * SLD]);
                    part[boff(L - 1) + col + (tid & 31)] = s;
                }
                if (c == 0) __syncthreads();
            }
            publish();
            if (L > 1 && !wait_w()) break;
            if (tid == 0) {
                tc_fence_after();
                const uint32_t aw = tbase + ACCW + 128u * (uint32_t)(L & 1);
                if (L > 1) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)  // dW_L = G_L^T A_{L-1}
                        umma(aw, rows_k(sm.act[L - 1], 128, q), rows_k(sm.act[L - 2], 128, q),
                             idesc_bf16(128, 128) | A_MN | B_MN, q > 0);
#pragma unroll
                    for (int q = 0; q < 8; ++q)  // dA_{L-1} = G_L W_L
                        umma(tbase + ACC, rows_mn(sm.act[L - 1], 128, q), rows_k(sm.w, 128, q),
                             idesc_bf16(128, 128) | B_MN, q > 0);
                } else {
#pragma unroll
                    for (int q = 0; q < 8; ++q)  // dW_1 = G_1^T X
                        umma(aw, rows_k(sm.act[0], 128, q), rows_k(sm.x, 128, q), idesc_bf16(128, 16) | A_MN | B_MN,
                             q > 0);
                }
                umma_commit(&sm.bar);
            }
            pending = true;
            // the previous layer's weight gradient, while these products run
            const uint32_t pw = tbase + ACCW + 128u * (uint32_t)((L + 1) & 1) + lane0;
            if (L == 4) {
                if (half == 0) {
                    uint32_t v[8];
                    tmem_ld8(tbase + ACCW + 128 + lane0, v);
#pragma unroll
                    for (int o = 0; o < OUT; ++o) part[woff(4) + o * HID + r] = __uint_as_float(v[o]);
                }
            } else {
#pragma unroll 1
                for (int c = 0; c < 2; ++c) {
                    uint32_t v[32];
                    const int col = half * 64 + c * 32;
                    tmem_ld32_nowait(pw + (uint32_t)col, v);
                    tmem_wait_ld();
                    float4 *dst = reinterpret_cast<float4 *>(part + woff(L) + (int64_t)r * HID + col);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        dst[q] = make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                                             __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
                }
            }
            tc_fence_before();
        }
        if (!ok || !wait_mma()) break;
        if (half == 0) {
            uint32_t v[8];
            tmem_ld8(tbase + ACCW + 128 + lane0, v);
#pragma unroll
            for (int k = 0; k < IN; ++k) part[woff(0) + r * IN + k] = __uint_as_float(v[k]);
        }
    } while (false);
    if (!ok) {
        if (tid == 0) atomicExch(err, kErrTrainTimeout);
        if (tid == 0 && pending) mbar_wait_bounded(&sm.bar, phase);    // let late products land
        if (tid == 0 && wpending) mbar_wait_bounded(&sm.wbar, wphase);  // and a late copy
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(512u) : "memory");
}

// grad[e] = sum of the blocks' partial gradients in order; ADAM: the update instead, and the
// packed weights of the next step.  Read-bound: 128 blocks' partials are 26 MB in L2.
template <bool ADAM>
__global__ void __launch_bounds__(128)
k_train_finish(const float *__restrict__ part, int nsplit, float *__restrict__ grad, float *__restrict__ p,
               float *__restrict__ m, float *__restrict__ v, uint16_t *__restrict__ wt, float lr, float b1, float b2,
               float eps, float c1, float c2)
{
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= (int)NPARAM) return;
    float s = 0.f;
    int z = 0;
    for (; z + 16 <= nsplit; z += 16) {
        float t[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) t[k] = __ldcs(part + (int64_t)(z + k) * kPartStride + i);
#pragma unroll
        for (int k = 0; k < 16; ++k) s += t[k];
    }
    for (; z < nsplit; ++z) s += part[(int64_t)z * kPartStride + i];
    if (!ADAM) {
        grad[i] = s;
        return;
    }
    adam_update(p, s, m, v, i, lr, b1, b2, eps, c1, c2);
    const int at = packed_at(i);
    if (at >= 0) wt[at] = __bfloat16_as_ushort(__float2bfloat16(p[i]));
}

__global__ void k_train_pack(const float *__restrict__ p, uint16_t *__restrict__ wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int)NPARAM) return;
    const int at = packed_at(i);
    if (at >= 0) wt[at] = __bfloat16_as_ushort(__float2bfloat16(p[i]));
}

}  // namespace

int64_t train_weights_elems() { return WT_TOTAL; }

cudaError_t pack_train(const float *params, uint16_t *wt, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(wt, 0, sizeof(uint16_t) * WT_TOTAL, s);  // the K and N padding
    if (e != cudaSuccess) return e;
    k_train_pack<<<(unsigned)((NPARAM + 255) / 256), 256, 0, s>>>(params, wt);
    return cudaGetLastError();
}

// 16384 samples on a GB300: this launch 38.9 us, the finish 10.4, the samples 46 (a share of a
// launch for 16 steps), against 570 for the general path's launches and 240 for a step's
// samples on their own.  What is left is the chain of ten products and epilogues per block.
cudaError_t launch_train_tiles(const float *params, const uint16_t *wt, const float *X, const float *T, int n,
                               float *Zs, float *part, double *loss, int *err, cudaStream_t s)
{
    static PerDevice ready;
    cudaError_t e = ready.once([] { return allow_dynamic_smem(k_train_tile, (int)sizeof(TrainSmem)); });
    if (e != cudaSuccess) return e;
    if (loss && (e = cudaMemsetAsync(loss, 0, sizeof(double), s)) != cudaSuccess) return e;
    const int nsplit = train_splits(n), chunk = (n + nsplit - 1) / nsplit;
    k_train_tile<<<nsplit, TT, sizeof(TrainSmem), s>>>(params, wt, X, T, n, chunk, reinterpret_cast<float4 *>(Zs), part,
                                                       loss, err);
    return cudaGetLastError();
}

cudaError_t launch_train_grad(const float *part, int n, float *grad, cudaStream_t s)
{
    k_train_finish<false><<<(unsigned)((NPARAM + 127) / 128), 128, 0, s>>>(part, train_splits(n), grad, nullptr, nullptr,
                                                                           nullptr, nullptr, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f);
    return cudaGetLastError();
}

cudaError_t launch_train_adam(const float *part, int n, float *params, float *m, float *v, uint16_t *wt, float lr,
                              float b1, float b2, float eps, int step, cudaStream_t s)
{
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    k_train_finish<true><<<(unsigned)((NPARAM + 127) / 128), 128, 0, s>>>(part, train_splits(n), nullptr, params, m, v,
                                                                          wt, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

}  // namespace mlp
}  // namespace gals
