// diag.cu -- diagnostics of a GALS state: sampled area/volume of {H < 0}, the symmetric
// difference against a reference state, e_max norms (eq. maximum_norm, Sec. 6.1), an
// FP64 L2 norm and a non-finite count.
//
// Counts are exact 64-bit integers (order-independent atomics), maxima are taken on
// the ordered bit patterns of non-negative floats, and the FP64 sum is reduced per
// block into a scratch array and then summed in a fixed order by one block, so every
// result is deterministic.
#include "gals_internal.h"
#include "tma.cuh"

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

// Whether the FP32 interpolant of a cell has one sign at every sample: the value
// weights of the basis are non-negative and sum to 1, the two slope weights along an axis
// sum to at most h / 4, so with M the largest magnitude of a plane at the corners
//   |H - (a mean of the corners' phi)| <= sum h_i/4 M_i + sum h_i h_j/16 M_ij + h_0 h_1 h_2/64 M_xyz,
// and 1e-5 of the values covers the evaluation's rounding (about 20 operations of 6e-8).
// sign = 1: every sample negative, 0: none, -1: undecided (also for anything not finite).
// value(p, v): plane p at vertex v.  cell_b: the mixed derivatives are the cell's own
// differences of the gradients (approach B), bounded through those.  Every rounding is
// written out: two kernels decide the same cells.
template <int DIM, class V>
__device__ __forceinline__ int cell_sign(const Geom &g, int cell_b, V value)
{
    float lo, hi, M[DIM == 2 ? 4 : 8], bad = 0.f;  // bad: NaN where a value is not finite
#pragma unroll
    for (int p = 0; p < (DIM == 2 ? 4 : 8); ++p) {
        if (p > DIM && cell_b) {
            M[p] = 0.f;
            continue;
        }
        float mn = value(p, 0), mx = mn, mag = fabsf(mn);
        bad += mn - mn;
#pragma unroll
        for (int v = 1; v < (1 << DIM); ++v) {
            const float x = value(p, v);
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
    const float x = __fmul_rn(g.h0, M[1]), y = __fmul_rn(g.h1, M[2]), xy = __fadd_rn(x, y);
    const float hxy = __fmul_rn(g.h0, g.h1);
    float D;
    if (DIM == 2) {
        D = cell_b ? __fmul_rn(0.375f, xy) : __fmaf_rn(__fmul_rn(0.0625f, hxy), M[3], __fmul_rn(0.25f, xy));
    } else {
        const float z = __fmul_rn(g.h2, M[3]), xyz = __fadd_rn(xy, z);
        if (cell_b) {
            D = __fmaf_rn(0.5f, xyz, __fmul_rn(0.0625f, z));
        } else {
            const float m = __fmaf_rn(hxy, M[4], __fmaf_rn(__fmul_rn(g.h0, g.h2), M[5], __fmul_rn(__fmul_rn(g.h1, g.h2), M[6])));
            D = __fmaf_rn(__fmul_rn(0.015625f, __fmul_rn(hxy, g.h2)), M[7], __fmaf_rn(0.0625f, m, __fmul_rn(0.25f, xyz)));
        }
    }
    D = __fadd_rn(__fmaf_rn(1e-5f, __fadd_rn(M[0], D), D), bad);
    return lo > D ? 0 : (hi < -D ? 1 : -1);
}

// The sign of the cell whose first corner is the node at id.
template <int DIM>
__device__ __forceinline__ int cell_sign_at(const float *__restrict__ s, const Geom &g, int64_t id, int cell_b)
{
    const int64_t dy = g.pitch, dz = (int64_t)g.n1 * g.pitch;
    return cell_sign<DIM>(g, cell_b, [&](int p, int v) {
        return s[p * g.plane + id + (v & 1) + ((v >> 1) & 1) * dy + (v >> 2) * dz];
    });
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

// The nodes and cells in items of 2^lx x (256 >> lx) nodes over the rows (narrow items on narrow
// grids), a thread per node; the lanes of warp w % 8 of item w / 8.
struct Place {
    int i, j, m;
    int64_t row, at;   // row of the grid, element of a plane
    bool node, cell;   // a node; the first corner of a cell
};

template <int DIM>
__device__ __forceinline__ Place place_of(const Geom &g, int lx, int64_t item, int tid)
{
    const int nchunk = ((g.n0 - 1) >> lx) + 1;
    Place p;
    p.row = item / nchunk * (kThreads >> lx) + (tid >> lx);
    p.i = ((int)(item % nchunk) << lx) + (tid & ((1 << lx) - 1));
    p.node = p.row < (int64_t)g.n1 * (DIM == 3 ? g.n2 : 1) && p.i < g.n0;
    p.j = DIM == 3 ? (int)(p.row % g.n1) : (int)p.row;
    p.m = DIM == 3 ? (int)(p.row / g.n1) : 0;
    p.at = p.row * g.pitch + p.i;
    p.cell = p.node && p.i < g.n0 - 1 && p.j < g.n1 - 1 && (DIM == 2 || p.m < g.n2 - 1);
    return p;
}

template <int DIM> __host__ __device__ __forceinline__ int64_t items_of(const Geom &g, int lx)
{
    const int64_t rows = (int64_t)g.n1 * (DIM == 3 ? g.n2 : 1), per = kThreads >> lx;
    return (rows + per - 1) / per * (((g.n0 - 1) >> lx) + 1);
}

// A warp samples its undecided cells together, 32 / S at a time with S lanes each (S: the samples
// rounded up to a power of two, at most 32).
__device__ __forceinline__ int lanes_per_cell(int samples) { return samples >= 32 ? 32 : 1 << (32 - __clz(samples - 1)); }

// Whether they are better sampled a lane per cell, every lane all samples of its cell from
// registers: by the evaluations on the longest lane, where the other way's gather for every
// evaluation counts as two.  Counted as two / one / none, q = 4 with a reference, us: smooth
// 150 x 110 x 150 326 / 342 / 402, 100 x 90 x 130 223 / 250 / 267, 60^3 98 / 93 / 94 (few warps
// each: there the second kernel's start shows); noise 60^3 200 / 200 / 436, 2048^2 323 / 323 / 901.
__device__ __forceinline__ bool dense_warp(int cells, int samples)
{
    const int S = lanes_per_cell(samples), rounds = (cells * S + 31) / 32 * ((samples + S - 1) / S);
    return 3 * rounds > samples + 2;
}

// How many warps may be left to k_diag_dense one by one: what its list holds, and an eighth of
// the grid's.
template <int DIM> __device__ __forceinline__ unsigned list_limit(const Geom &g, int lx)
{
    const int64_t eighth = items_of<DIM>(g, lx) * (kThreads / 32 / 8);
    return eighth < kDiagList ? (unsigned)eighth : kDiagList;
}

// One thread per node and the cell whose first corner it is: non-finite count, e_max of phi and
// psi against b and the FP64 sum of (phi - phi_b)^2 (partials[blockIdx.x]), and the q^p
// cell-centred samples of H < 0.  Almost every cell of a smooth state is decided by a bound on
// its corner data; a warp takes the others together, its lanes the samples, unless they are
// many (dense_warp): such warps are left to k_diag_dense, the first of them by a list (a smooth
// state's few, where an interface runs along a row).  Past list_limit k_diag_dense samples every
// cell of the grid, as one would without the bound, and what is found here (pre_neg, pre_sym)
// does not count: the blocks stop looking at cells.
// Every plane is read once from DRAM.  Calls, us, sampling every cell / a warp per undecided
// cell / now: 2048^2 with a reference, q = 4: smooth 365 / 113 / 112, noise 366 / 1406 / 323; q = 1:
// noise 218 / 1406 / 162; 3D 128^3, q = 2: smooth 403 / 227 / 200, noise 402 / 1909 / 387.
template <int DIM, int LX>
__global__ void __launch_bounds__(kThreads, DIM == 2 ? 4 : 3)
k_diag(Geom g, int lx_, const float *__restrict__ a, const float *__restrict__ b, int q, DiagOut *out,
       double *__restrict__ partials, unsigned *__restrict__ list, int cell_a, int cell_b)
{
    __shared__ unsigned long long redu[kThreads / 32];
    __shared__ double redd[kThreads / 32];
    __shared__ unsigned redm[kThreads / 32];
    __shared__ unsigned char order[kThreads / 32][32];
    constexpr int NP = DIM == 2 ? 4 : 8;
    const int lx = LX > 0 ? LX : lx_, lane = threadIdx.x & 31;
    const int64_t nitem = items_of<DIM>(g, lx);
    const unsigned limit = list_limit<DIM>(g, lx);
    unsigned noted = 0, turn = 0;
    pdl_release();  // k_diag_dense may be placed when the last blocks have started
    int samples = q;
    for (int d = 1; d < DIM; ++d) samples *= q;
    unsigned long long nonfin = 0, nneg = 0, nsym = 0;
    unsigned mphi = 0, mpsi = 0;
    double l2 = 0.0;
    for (int64_t it = blockIdx.x; it < nitem; it += gridDim.x) {
        const Place P = place_of<DIM>(g, lx, it, threadIdx.x);
        const int64_t o = P.at;
        const bool look = q > 0 && noted <= limit;
        // at items 2, 4, 8, 16, 24, ... and for the next one (at every item the read cost 15 of 48 us);
        // one lane's reading for the whole warp, whose lanes have to look alike (the votes below)
        if (q > 0 && ((++turn & 7) == 0 || turn == 2 || turn == 4))
            noted = __shfl_sync(0xffffffffu, *(volatile unsigned *)&out->dense, 0);
        if (P.node) {
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
        if (!look) continue;
        int sa = 0, sb = 0;
        if (P.cell) {
            sa = cell_sign_at<DIM>(a, g, o, cell_a);
            if (sa > 0) nneg += samples;
            if (b) {
                sb = cell_sign_at<DIM>(b, g, o, cell_b);
                if (sa >= 0 && sb >= 0 && sa != sb) nsym += samples;
            }
        }
        // the undecided cells of the warp
        unsigned todo = __ballot_sync(0xffffffffu, P.cell && (sa < 0 || sb < 0));
        if (!todo) continue;
        const int cells = __popc(todo), S = lanes_per_cell(samples), warp = threadIdx.x >> 5;
        if (dense_warp(cells, samples)) {
            if (lane == 0) {
                const unsigned slot = atomicAdd(&out->dense, 1u);
                if (slot < limit) list[slot] = (unsigned)(it * (kThreads / 32) + warp);
            }
            continue;
        }
        // in vain if other warps have filled the list meanwhile (a warp of a 3D grid at q = 7 may
        // take 50 us here)
        if (samples > 64 && __any_sync(0xffffffffu, *(volatile unsigned *)&out->dense > limit)) continue;
        // the undecided cells in order, for the lanes that sample them
        if (todo >> lane & 1) order[warp][__popc(todo & ((1u << lane) - 1))] = lane;
        __syncwarp();
        for (int base = 0; base < cells; base += 32 / S) {
            const int at = base + lane / S, w = order[warp][min(at, cells - 1)];
            const int ci = __shfl_sync(0xffffffffu, P.i, w), cj = __shfl_sync(0xffffffffu, P.j, w);
            const int cm = __shfl_sync(0xffffffffu, P.m, w);
            const int ca = __shfl_sync(0xffffffffu, sa, w), cb = __shfl_sync(0xffffffffu, sb, w);
            for (int t = at < cells ? lane % S : samples; t < samples; t += S) {
                const bool na = ca < 0 ? sample_negative<DIM>(a, g, ci, cj, cm, t, q, cell_a) : ca > 0;
                if (ca < 0) nneg += na;
                if (b) nsym += na != (cb < 0 ? sample_negative<DIM>(b, g, ci, cj, cm, t, q, cell_b) : cb > 0);
            }
        }
        __syncwarp();  // order is the next item's
    }
    unsigned long long s = block_sum(nonfin, redu);
    if (threadIdx.x == 0 && s) atomicAdd(&out->nonfinite, s);
    s = block_sum(nneg, redu);
    if (threadIdx.x == 0 && s) atomicAdd(&out->pre_neg, s);
    s = block_sum(nsym, redu);
    if (threadIdx.x == 0 && s) atomicAdd(&out->pre_sym, s);
    if (!b) return;
    unsigned m1 = block_max(mphi, redm);
    if (threadIdx.x == 0) atomicMax(&out->emax_phi_bits, m1);
    unsigned m2 = block_max(mpsi, redm);
    if (threadIdx.x == 0) atomicMax(&out->emax_psi_bits, m2);
    double ds = block_sum(l2, redd);
    if (threadIdx.x == 0) partials[blockIdx.x] = ds;
}

// A cell's data in registers: gathered, its mixed derivatives by approach B, H < 0 at a sample.
template <int DIM>
__device__ __forceinline__ void load_cell(const float *__restrict__ s, const Geom &g, int k, int l, int m,
                                          float (&c)[1 << DIM][1 << DIM])
{
    if constexpr (DIM == 2) gather2d(s, g, k, l, c);
    else gather3d(s, g, k, l, m, c);
}

template <int DIM>
__device__ __forceinline__ void cross_cell(const Geom &g, float (&c)[1 << DIM][1 << DIM])
{
    if constexpr (DIM == 2) cross_cell2d(c, g.ih0, g.ih1);
    else cell3d_planes(c, g);
}

template <int DIM>
__device__ __forceinline__ bool negative(const float (&c)[1 << DIM][1 << DIM], const Basis1 &bx, const Basis1 &by,
                                         const Basis1 &bz)
{
    float H, gr[3];
    if constexpr (DIM == 2) hermite2d(c, bx, by, H, gr[0], gr[1]);
    else hermite3d(c, bx, by, bz, H, gr);
    return H < 0.f;
}

// Samples of cells a lane per cell: LISTED, the undecided cells of the `count` warps of the list (the
// bound counted the others), else every cell of the grid.
template <int DIM, bool LISTED>
__device__ __forceinline__ void sample_cells(const Geom &g, int lx, const float *__restrict__ a, const float *__restrict__ b,
                                             int q, const unsigned *__restrict__ list, unsigned count, int cell_a,
                                             int cell_b, unsigned long long &nneg, unsigned long long &nsym)
{
    constexpr int W = kThreads / 32;
    const int64_t nc0 = g.n0 - 1, nc1 = g.n1 - 1, ncell = nc0 * nc1 * (DIM == 3 ? g.n2 - 1 : 1);
    // lines of samples along x; of a short list each of `parts` warps takes every parts-th line
    // (up to four rounds of the resident warps: 128^3, q = 4, smooth 285 us against 298 with one)
    const int lines = DIM == 3 ? q * q : q;
    const int parts = LISTED ? max(1, min(lines, (int)(4 * gridDim.x * W / count))) : 1;
    const int64_t total = LISTED ? (int64_t)count * parts * 32 : ncell;
    const float invq = 1.f / (float)q;
    for (int64_t c = (int64_t)blockIdx.x * kThreads + threadIdx.x; c < total; c += (int64_t)gridDim.x * kThreads) {
        int k, l, m;
        if (LISTED) {
            const unsigned w = list[(c >> 5) / parts];
            const Place P = place_of<DIM>(g, lx, w / W, (int)(w % W) * 32 + (int)(c & 31));
            if (!P.cell) continue;
            k = P.i; l = P.j; m = P.m;
        } else {
            k = (int)(c % nc0); l = (int)(c / nc0 % nc1); m = DIM == 3 ? (int)(c / (nc0 * nc1)) : 0;
        }
        float ca[1 << DIM][1 << DIM], cb[1 << DIM][1 << DIM];
        int sa = -1, sb = -1;
        load_cell<DIM>(a, g, k, l, m, ca);
        if (b) load_cell<DIM>(b, g, k, l, m, cb);
        if (LISTED) {
            sa = cell_sign<DIM>(g, cell_a, [&](int p, int v) { return ca[v][p]; });
            sb = b ? cell_sign<DIM>(g, cell_b, [&](int p, int v) { return cb[v][p]; }) : 0;
            if (sa >= 0 && sb >= 0) continue;
        }
        if (cell_a) cross_cell<DIM>(g, ca);
        if (b && cell_b) cross_cell<DIM>(g, cb);
        int neg = 0, sym = 0;
        for (int line = LISTED ? (int)((c >> 5) % parts) : 0; line < lines; line += parts) {
            const Basis1 bz = basis1(((float)(line / q) + 0.5f) * invq, g.h2, g.ih2);
            const Basis1 by = basis1(((float)(line % q) + 0.5f) * invq, g.h1, g.ih1);
            for (int sx = 0; sx < q; ++sx) {
                const Basis1 bx = basis1(((float)sx + 0.5f) * invq, g.h0, g.ih0);
                const bool na = negative<DIM>(ca, bx, by, bz);
                if (!LISTED || sa < 0) neg += na;
                if (b) {
                    const bool nb = negative<DIM>(cb, bx, by, bz);
                    sym += LISTED ? (sa < 0 ? na : sa > 0) != (sb < 0 ? nb : sb > 0) : na != nb;
                }
            }
        }
        nneg += neg;
        nsym += sym;
    }
}

// What k_diag left over (see there): the warps of its list, or the whole grid.  The first block adds
// what k_diag counted to the former and sums the partials in a fixed order.
template <int DIM>
__global__ void __launch_bounds__(kThreads)
k_diag_dense(Geom g, int lx, const float *__restrict__ a, const float *__restrict__ b, int q, DiagOut *out,
             const double *__restrict__ partials, int nparts, const unsigned *__restrict__ list, int cell_a, int cell_b)
{
    __shared__ unsigned long long redu[kThreads / 32];
    __shared__ double redd[kThreads / 32];
    pdl_wait();
    const unsigned dense = *(volatile unsigned *)&out->dense;
    const bool listed = dense <= list_limit<DIM>(g, lx);
    if (blockIdx.x == 0) {
        if (b) {
            double s = 0.0;
            for (int i = threadIdx.x; i < nparts; i += kThreads) s += partials[i];
            s = block_sum(s, redd);
            if (threadIdx.x == 0) out->l2_phi_sum = s;
        }
        if (threadIdx.x == 0 && listed) {
            atomicAdd(&out->n_neg, out->pre_neg);
            atomicAdd(&out->n_sym, out->pre_sym);
        }
    }
    if (dense == 0) return;
    unsigned long long nneg = 0, nsym = 0;
    if (listed) sample_cells<DIM, true>(g, lx, a, b, q, list, dense, cell_a, cell_b, nneg, nsym);
    else sample_cells<DIM, false>(g, lx, a, b, q, list, dense, cell_a, cell_b, nneg, nsym);
    unsigned long long s = block_sum(nneg, redu);
    if (threadIdx.x == 0 && s) atomicAdd(&out->n_neg, s);
    s = block_sum(nsym, redu);
    if (threadIdx.x == 0 && s) atomicAdd(&out->n_sym, s);
}

}  // namespace

int diag_partials_needed() { return kNodeBlocks; }

template <int DIM>
static cudaError_t launch(const Geom &g, const float *a, const float *b, int q, DiagOut *counters, double *partials,
                          int nparts, unsigned *list, cudaStream_t s, bool cell_a, bool cell_b)
{
    cudaError_t e = cudaMemsetAsync(counters, 0, sizeof(DiagOut), s);
    if (e != cudaSuccess) return e;
    // items as narrow as the grid (5 x 200000: 75 us in 64 columns, 36 in 8); a constant for all but
    // narrow grids (3D 128^3 with a reference, q = 1: 188 us against 204)
    const int lx = g.n0 > 32 ? 6 : (g.n0 > 16 ? 5 : (g.n0 > 8 ? 4 : 3));
    auto kern = lx == 6 ? k_diag<DIM, 6> : k_diag<DIM, 0>;
    kern<<<nparts, kThreads, 0, s>>>(g, lx, a, b, q, counters, partials, list, cell_a, cell_b);
    if ((e = cudaGetLastError()) != cudaSuccess || (!b && q <= 0)) return e;
    // as many blocks as are resident at once, striding over the warps: a second, part-filled
    // wave of them cost half their time again
    static PerDevice fit;
    int blocks = 1;
    e = fit.get(&blocks, [](int *n) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const cudaError_t x = cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_diag_dense<DIM>, kThreads, 0);
        *n = (*n < 1 ? 1 : *n) * (sms < 1 ? 1 : sms);
        return x;
    });
    if (e != cudaSuccess) return e;
    return launch_kernel(k_diag_dense<DIM>, dim3(q > 0 ? blocks : 1), dim3(kThreads), 0, s, true, g, lx, a, b, q,
                         counters, partials, nparts, list, (int)cell_a, (int)cell_b);
}

cudaError_t launch_diag(int dim, const Geom &g, const float *a, const float *b, int q, DiagOut *counters,
                        double *partials, int nparts, unsigned *list, cudaStream_t s, bool cell_a, bool cell_b)
{
    return dim == 2 ? launch<2>(g, a, b, q, counters, partials, nparts, list, s, cell_a, cell_b)
                    : launch<3>(g, a, b, q, counters, partials, nparts, list, s, cell_a, cell_b);
}

}  // namespace gals
