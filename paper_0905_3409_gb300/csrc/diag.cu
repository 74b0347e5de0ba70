// diag.cu -- diagnostics of a GALS state: sampled area/volume of {H < 0}, the symmetric
// difference against a reference state, e_max norms (eq. maximum_norm, Sec. 6.1), an
// FP64 L2 norm and a non-finite count.
//
// Counts are exact 64-bit integers (order-independent atomics), maxima are taken on
// the ordered bit patterns of non-negative floats, and the FP64 sum is reduced per
// block into a scratch array and then summed in a fixed order by one block, so every
// result is deterministic.
#include "gals_internal.h"

namespace gals {

namespace {

constexpr int kThreads = 256;
constexpr int kNodeBlocks = 1216;  // 8 x 152 SMs; grid-stride over the rows

__device__ __forceinline__ void gather2d(const float *s, const Geom &g, int k, int l, float c[4][4])
{
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int64_t id = (int64_t)(l + (v >> 1)) * g.pitch + k + (v & 1);
#pragma unroll
        for (int a = 0; a < 4; ++a) c[v][a] = s[a * g.plane + id];
    }
}

__device__ __forceinline__ void gather3d(const float *s, const Geom &g, int k, int l, int m,
                                         float c[8][8])
{
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const int64_t id = ((int64_t)(m + (v >> 2)) * g.n1 + l + ((v >> 1) & 1)) * g.pitch + k + (v & 1);
#pragma unroll
        for (int a = 0; a < 8; ++a) c[v][a] = s[a * g.plane + id];
    }
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T *red)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    T s = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < kThreads / 32; ++i) s += red[i];
    return s;  // valid in thread 0
}

__device__ __forceinline__ unsigned block_max(unsigned v, unsigned *red)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = max(v, __shfl_down_sync(0xffffffffu, v, off));
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    unsigned s = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < kThreads / 32; ++i) s = max(s, red[i]);
    return s;
}

// approach B for a gathered 3D cell (planes 0 phi, 1-3 psi, 4-7 mixed derivatives)
__device__ __forceinline__ void cell3d_planes(float c[8][8], const Geom &g)
{
    float cr[8][4];
    cross_cell3d([&](int v, int a) { return c[v][a]; }, g.ih0, g.ih1, g.ih2, cr);
#pragma unroll
    for (int v = 0; v < 8; ++v)
#pragma unroll
        for (int i = 0; i < 4; ++i) c[v][4 + i] = cr[v][i];
}

// Whether the FP32 interpolant of the cell (k, l, m) has one sign at every sample: the value
// weights of the basis are non-negative and sum to 1, the two slope weights along an axis
// sum to at most h / 4, so with M the largest magnitude of a plane at the corners
//   |H - (a mean of the corners' phi)| <= sum h_i/4 M_i + sum h_i h_j/16 M_ij + h_0 h_1 h_2/64 M_xyz,
// and 1e-5 of the values covers the evaluation's rounding (about 20 operations of 6e-8).
// sign = 1: every sample negative, 0: none, -1: undecided (also for anything not finite).
// cell_b: the mixed derivatives are the cell's own differences of the gradients (approach B),
// bounded through those.
template <int DIM>
__device__ __forceinline__ int cell_sign(const float *__restrict__ s, const Geom &g, int64_t id, int cell_b)
{
    const int64_t dy = g.pitch, dz = (int64_t)g.n1 * g.pitch;
    float lo, hi, M[DIM == 2 ? 4 : 8], bad = 0.f;  // bad: NaN where a value is not finite
#pragma unroll
    for (int p = 0; p < (DIM == 2 ? 4 : 8); ++p) {
        if (p > DIM && cell_b) {
            M[p] = 0.f;
            continue;
        }
        const float *f = s + p * g.plane + id;
        float mn = f[0], mx = mn, mag = fabsf(mn);
        bad += mn - mn;
#pragma unroll
        for (int v = 1; v < (1 << DIM); ++v) {
            const float x = f[(v & 1) + ((v >> 1) & 1) * dy + (v >> 2) * dz];
            if (p == 0) {
                mn = fminf(mn, x);
                mx = fmaxf(mx, x);
            }
            mag = fmaxf(mag, fabsf(x));
            bad += x - x;
        }
        if (p == 0) {
            lo = mn;
            hi = mx;
        }
        M[p] = mag;
    }
    float D;
    if (DIM == 2) {
        const float x = g.h0 * M[1], y = g.h1 * M[2];
        D = 0.25f * (x + y) + (cell_b ? 0.125f * (x + y) : 0.0625f * (g.h0 * g.h1) * M[3]);
    } else {
        const float x = g.h0 * M[1], y = g.h1 * M[2], z = g.h2 * M[3];
        D = 0.25f * (x + y + z);
        if (cell_b)
            D += 0.25f * (x + y + z) + 0.0625f * z;
        else
            D += 0.0625f * (g.h0 * g.h1 * M[4] + g.h0 * g.h2 * M[5] + g.h1 * g.h2 * M[6]) +
                 0.015625f * (g.h0 * g.h1 * g.h2) * M[7];
    }
    D += 1e-5f * (M[0] + D) + bad;
    return lo > D ? 0 : (hi < -D ? 1 : -1);
}

// Sign of H < 0 at sample t of the cell (every lane of a warp takes another t).
template <int DIM>
__device__ bool sample_negative(const float *__restrict__ s, const Geom &g, int k, int l, int m, int t, int q, int cell_b)
{
    const float invq = 1.f / (float)q;
    const int sx = t % q, sy = t / q % q, sz = t / q / q;
    const Basis1 bx = basis1(((float)sx + 0.5f) * invq, g.h0, g.ih0);
    const Basis1 by = basis1(((float)sy + 0.5f) * invq, g.h1, g.ih1);
    float H;
    if (DIM == 2) {
        float c[4][4], hx, hy;
        gather2d(s, g, k, l, c);
        if (cell_b) cross_cell2d(c, g.ih0, g.ih1);
        hermite2d(c, bx, by, H, hx, hy);
    } else {
        const Basis1 bz = basis1(((float)sz + 0.5f) * invq, g.h2, g.ih2);
        float c[8][8], gr[3];
        gather3d(s, g, k, l, m, c);
        if (cell_b) cell3d_planes(c, g);
        hermite3d(c, bx, by, bz, H, gr);
    }
    return H < 0.f;
}

// One thread per node and the cell whose first corner it is, in blocks of DX x DY over the
// rows: non-finite count, e_max of phi and psi against b and the FP64 sum of (phi - phi_b)^2
// (partials[blockIdx.x]), and the q^p cell-centred samples of H < 0.  Almost every cell is
// decided by a bound on its corner data; a warp takes the others one after the other, its
// lanes the samples.  Every plane is read once from DRAM: 2048^2 with a reference and q = 4
// 70 us where sampling every cell took 203, a pass over the nodes 65 and a serial sum 70; 3D
// 160 x 150 x 140 the same 0.26 ms of the call's 0.31, against 2.1 (q = 7: 0.55 against 9.5).
constexpr int DX = 64, DY = kThreads / DX;

template <int DIM>
__global__ void __launch_bounds__(kThreads, DIM == 2 ? 4 : 3)
k_diag(Geom g, const float *__restrict__ a, const float *__restrict__ b, int q, DiagOut *out,
       double *__restrict__ partials, int cell_a, int cell_b)
{
    __shared__ unsigned long long redu[kThreads / 32];
    __shared__ double redd[kThreads / 32];
    __shared__ unsigned redm[kThreads / 32];
    constexpr int NP = DIM == 2 ? 4 : 8;
    const int tx = threadIdx.x % DX, ty = threadIdx.x / DX, lane = threadIdx.x & 31;
    const int nchunk = (g.n0 + DX - 1) / DX;
    const int64_t nrows = (int64_t)g.n1 * (DIM == 3 ? g.n2 : 1);
    const int64_t nitem = (nrows + DY - 1) / DY * nchunk;
    int samples = q;
    for (int d = 1; d < DIM; ++d) samples *= q;
    unsigned long long nonfin = 0, nneg = 0, nsym = 0;
    unsigned mphi = 0, mpsi = 0;
    double l2 = 0.0;
    for (int64_t it = blockIdx.x; it < nitem; it += gridDim.x) {
        const int64_t row = it / nchunk * DY + ty;
        const int i = (int)(it % nchunk) * DX + tx;
        const bool node = row < nrows && i < g.n0;
        const int j = DIM == 3 ? (int)(row % g.n1) : (int)row, m = DIM == 3 ? (int)(row / g.n1) : 0;
        const int64_t o = row * g.pitch + i;
        if (node) {
            bool bad = false;
#pragma unroll
            for (int p = 0; p < NP; ++p) bad |= !isfinite(a[p * g.plane + o]);
            nonfin += bad;
            if (b) {
                mphi = max(mphi, __float_as_uint(fabsf(a[o] - b[o])));
#pragma unroll
                for (int p = 1; p <= DIM; ++p)
                    mpsi = max(mpsi, __float_as_uint(fabsf(a[p * g.plane + o] - b[p * g.plane + o])));
                const double dd = (double)a[o] - (double)b[o];
                l2 += dd * dd;
            }
        }
        if (q <= 0) continue;
        const bool cell = node && i < g.n0 - 1 && j < g.n1 - 1 && (DIM == 2 || m < g.n2 - 1);
        int sa = 0, sb = 0;
        if (cell) {
            sa = cell_sign<DIM>(a, g, o, cell_a);
            if (sa > 0) nneg += samples;
            if (b) {
                sb = cell_sign<DIM>(b, g, o, cell_b);
                if (sa >= 0 && sb >= 0 && sa != sb) nsym += samples;
            }
        }
        // the undecided cells of the warp
        unsigned todo = __ballot_sync(0xffffffffu, cell && (sa < 0 || sb < 0));
        while (todo) {
            const int w = __ffs(todo) - 1;
            todo &= todo - 1;
            const int ci = __shfl_sync(0xffffffffu, i, w), cj = __shfl_sync(0xffffffffu, j, w);
            const int cm = __shfl_sync(0xffffffffu, m, w);
            const int ca = __shfl_sync(0xffffffffu, sa, w), cb = __shfl_sync(0xffffffffu, sb, w);
            for (int t = lane; t < samples; t += 32) {
                const bool na = ca < 0 ? sample_negative<DIM>(a, g, ci, cj, cm, t, q, cell_a) : ca > 0;
                if (ca < 0) nneg += na;
                if (b) nsym += na != (cb < 0 ? sample_negative<DIM>(b, g, ci, cj, cm, t, q, cell_b) : cb > 0);
            }
        }
    }
    unsigned long long s = block_sum(nonfin, redu);
    if (threadIdx.x == 0 && s) atomicAdd(&out->nonfinite, s);
    s = block_sum(nneg, redu);
    if (threadIdx.x == 0 && s) atomicAdd(&out->n_neg, s);
    s = block_sum(nsym, redu);
    if (threadIdx.x == 0 && s) atomicAdd(&out->n_sym, s);
    if (!b) return;
    unsigned m1 = block_max(mphi, redm);
    if (threadIdx.x == 0) atomicMax(&out->emax_phi_bits, m1);
    unsigned m2 = block_max(mpsi, redm);
    if (threadIdx.x == 0) atomicMax(&out->emax_psi_bits, m2);
    double ds = block_sum(l2, redd);
    if (threadIdx.x == 0) partials[blockIdx.x] = ds;
}

// Fixed-order FP64 sum of the per-block partials, by one block.
__global__ void __launch_bounds__(kThreads) k_diag_finish(const double *partials, int nparts, DiagOut *out)
{
    __shared__ double red[kThreads / 32];
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += kThreads) s += partials[i];
    s = block_sum(s, red);
    if (threadIdx.x == 0) out->l2_phi_sum = s;
}

}  // namespace

int diag_partials_needed() { return kNodeBlocks; }

static cudaError_t launch(int dim, const Geom &g, const float *a, const float *b, int q, DiagOut *counters,
                          double *partials, int nparts, cudaStream_t s, bool cell_a, bool cell_b)
{
    cudaError_t e = cudaMemsetAsync(counters, 0, sizeof(DiagOut), s);
    if (e != cudaSuccess) return e;
    if (dim == 2) k_diag<2><<<nparts, kThreads, 0, s>>>(g, a, b, q, counters, partials, cell_a, cell_b);
    else k_diag<3><<<nparts, kThreads, 0, s>>>(g, a, b, q, counters, partials, cell_a, cell_b);
    if ((e = cudaGetLastError()) != cudaSuccess || !b) return e;
    k_diag_finish<<<1, kThreads, 0, s>>>(partials, nparts, counters);
    return cudaGetLastError();
}

cudaError_t launch_diag(int dim, const Geom &g, const float *a, const float *b, int q,
                        DiagOut *counters, double *partials, cudaStream_t s, bool cell_a, bool cell_b)
{
    return launch(dim, g, a, b, q, counters, partials, kNodeBlocks, s, cell_a, cell_b);
}

cudaError_t launch_diag_with(int dim, const Geom &g, const float *a, const float *b, int q,
                             DiagOut *counters, double *partials, int nparts, cudaStream_t s)
{
    return launch(dim, g, a, b, q, counters, partials, nparts, s, false, false);
}

}  // namespace gals
