// kernels.cuh -- hot-path kernels of one PCG iteration: CSR SpMV, the colour phases of
// the multicolour Gauss-Seidel smoothers, l1-Jacobi, the transfer operators I_P / I_R
// (Eq. 10), the dense coarsest solve and the fused PCG vector updates.
//
// Rows are processed by sub-warps of TPR lanes (TPR in {4, 8, 16, 32}): the lanes of a
// sub-warp stride over the row's entries, so the column and value loads of consecutive
// lanes are coalesced, and the partial sums meet in a fixed xor-shuffle tree. Every
// reduction uses a fixed grid and a fixed summation tree, so results are bitwise
// reproducible from run to run.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace pk {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBlock = 256;
constexpr int kRedGrid = 152 * 4;  // most blocks of the reduction kernels
// Grid of an element-wise reduction over n elements: one element a thread up to kRedGrid
// blocks. On a short vector the atomics of 608 arriving blocks cost more than the sums.
inline unsigned red_grid(int64_t n) {
    return (unsigned)(n <= kBlock ? 1 : n >= (int64_t)kRedGrid * kBlock ? kRedGrid : (n + kBlock - 1) / kBlock);
}

template <typename T>
__device__ __forceinline__ T ldg(const T *p) {
    return __ldg(p);
}

// Matrix entries are read once per application and streamed: loads marked evict-first
// (ld.global.cs) keep them from pushing the gathered vector out of L2, which the colour
// phases and the SpMV read many times.
template <typename T>
__device__ __forceinline__ T ldst(const T *p) {
    return __ldcs(p);
}

// sum over the TPR lanes of a sub-warp (every lane of the warp must call this)
template <int TPR, typename A>
__device__ __forceinline__ A subwarp_sum(A v) {
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Entries per batch: a lane issues the column and value loads of kBatch entries (as
// predicated loads) before the first dependent gather of x, so the whole batch's memory
// traffic is in flight at once. Small colour phases are latency-bound and need this.
constexpr int kBatch = 8;

// sum_{e in [lo,hi)} val[e] * x[col[e]] accumulated in A by the lanes of a sub-warp,
// lane `sub` adding entries lo+sub, lo+sub+TPR, ... in that order
template <int TPR, typename A, typename VT, typename XT, int NB = kBatch>
__device__ __forceinline__ A row_dot(int64_t lo, int64_t hi, int sub, const int32_t *__restrict__ col,
                                     const VT *__restrict__ val, const XT *__restrict__ x) {
    A acc = A(0);
    for (int64_t base = lo + sub; base < hi; base += NB * TPR) {
        int c[NB];
        A v[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int64_t e = base + (int64_t)k * TPR;
            const bool ok = e < hi;
            c[k] = ok ? ldg(&col[e]) : -1;
            v[k] = ok ? (A)ldg(&val[e]) : A(0);
        }
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (c[k] >= 0) acc += v[k] * (A)ldg(&x[c[k]]);
    }
    return subwarp_sum<TPR>(acc);
}

// ---------------------------------------------------------------------------------
// Deterministic reductions. The order of every addition is fixed by the grid alone,
// never by timing.
//  - strided_sum: thread t of a block adds a[lo + t], a[lo + t + blockDim], ... below
//    hi in that order (loads issued eight at a time).
//  - block_partials: a warp shuffle tree, then the block's warps in order, into
//    partials[block].
//  - grid_reduce: the last block to arrive (fence and atomic counter) adds the block
//    partials with strided_sum and a block tree.
// The PCG's reductions run in element-wise kernels of at most kRedGrid blocks. GB300 issues one
// warp-wide FP64 instruction per 16 cycles per SM, so a shuffle tree of doubles at the
// end of every warp of a one-row-per-thread SpMV (5 adds per 32 rows) costs about as
// much as streaming the operand vectors once more: the PCG's fine SpMV writes q only,
// and the dot products read their vectors in a kernel of their own. FGMRES's residual
// and the Stokes operator (off the headline path) still reduce inside their full-grid
// kernels.
// ---------------------------------------------------------------------------------
__device__ __forceinline__ double strided_sum(const double *a, int64_t lo, int64_t hi, int stride_nv, int q) {
    constexpr int U = 8;
    const int64_t bd = blockDim.x;
    double x = 0.0;
    for (int64_t b0 = lo + threadIdx.x; b0 < hi; b0 += U * bd) {
        double t[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t b = b0 + u * bd;
            t[u] = b < hi ? __ldcg(&a[b * stride_nv + q]) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (b0 + u * bd < hi) x += t[u];
    }
    return x;
}

template <int NV>
__device__ __forceinline__ void block_partials(double (&v)[NV], double *partials) {
    __shared__ double sh[NV][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double x = v[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        if (lane == 0) sh[q][wid] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            double s = 0.0;
            for (int w = 0; w < nw; ++w) s += sh[q][w];
            partials[(int64_t)blockIdx.x * NV + q] = s;
        }
    }
}

template <int NV>
__device__ __forceinline__ bool grid_reduce(double (&v)[NV], double *partials, unsigned *counter,
                                            double (&tot)[NV]) {
    __shared__ double sh[NV][32];
    __shared__ int last;
    block_partials<NV>(v, partials);
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned prev = atomicAdd(counter, 1u);
        last = (prev == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double x = strided_sum(partials, 0, gridDim.x, NV, q);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        if (lane == 0) sh[q][wid] = x;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double s = 0.0;
        for (int w = 0; w < nw; ++w) s += sh[q][w];
        tot[q] = s;
    }
    if (threadIdx.x == 0) *counter = 0u;
    return true;
}

// ---------------------------------------------------------------------------------
// Plain CSR SpMV y = A x (transfer operators, level residual parts)
// ---------------------------------------------------------------------------------
template <int TPR, typename A, typename VT, typename XT, typename YT>
__global__ void __launch_bounds__(kBlock) k_spmv(int64_t n, const int64_t *__restrict__ ptr,
                                                 const int32_t *__restrict__ col, const VT *__restrict__ val,
                                                 const XT *__restrict__ x, YT *__restrict__ y) {
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool ok = row < n;
    int64_t lo = ok ? ptr[row] : 0, hi = ok ? ptr[row + 1] : 0;
    A s = row_dot<TPR, A>(lo, hi, sub, col, val, x);
    if (ok && sub == 0) y[row] = (YT)s;
}

// Restriction fused with the l1-Jacobi pre-smoothing step from zero of the level it
// feeds: b = R x (as k_spmv) and x_c = b / l1 (as k_jacobi0) in one pass, bitwise the two
// kernels' results.
template <int TPR, typename A, typename VT, typename XT, typename PT>
__global__ void __launch_bounds__(kBlock) k_restrict_jacobi0(int64_t n, const int64_t *__restrict__ ptr,
                                                             const int32_t *__restrict__ col,
                                                             const VT *__restrict__ val, const XT *__restrict__ x,
                                                             const PT *__restrict__ l1, PT *__restrict__ b,
                                                             PT *__restrict__ xc) {
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool ok = row < n;
    int64_t lo = ok ? ptr[row] : 0, hi = ok ? ptr[row + 1] : 0;
    A s = row_dot<TPR, A>(lo, hi, sub, col, val, x);
    if (ok && sub == 0) {
        const PT bi = (PT)s;
        b[row] = bi;
        xc[row] = bi / l1[row];
    }
}

// b = I_P^T x with I_P^T's values given by one-byte codes (value tab[code]), fused like
// k_restrict_jacobi0 with the level's first l1-Jacobi step xc = b / l1; the same lanes,
// batches and order of additions as row_dot, so the result equals k_restrict_jacobi0's
template <int TPR, typename PT, typename XT>
__global__ void __launch_bounds__(kBlock) k_restrict_code_jacobi0(int64_t n, const int64_t *__restrict__ ptr,
                                                                  const int32_t *__restrict__ col,
                                                                  const uint8_t *__restrict__ code,
                                                                  const PT *__restrict__ tab,
                                                                  const XT *__restrict__ x,
                                                                  const PT *__restrict__ l1, PT *__restrict__ b,
                                                                  PT *__restrict__ xc) {
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool ok = row < n;
    const int64_t lo = ok ? ptr[row] : 0, hi = ok ? ptr[row + 1] : 0;
    PT acc = PT(0);
    for (int64_t base = lo + sub; base < hi; base += kBatch * TPR) {
        int c[kBatch];
        PT v[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int64_t e = base + (int64_t)k * TPR;
            const bool in = e < hi;
            c[k] = in ? ldg(&col[e]) : -1;
            v[k] = in ? ldg(&tab[ldg(&code[e])]) : PT(0);
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
            if (c[k] >= 0) acc += v[k] * (PT)ldg(&x[c[k]]);
    }
    acc = subwarp_sum<TPR>(acc);
    if (ok && sub == 0) {
        b[row] = acc;
        xc[row] = acc / l1[row];
    }
}

// r = b - A x
template <int TPR, typename A, typename VT, typename T>
__global__ void __launch_bounds__(kBlock) k_residual(int64_t n, const int64_t *__restrict__ ptr,
                                                     const int32_t *__restrict__ col, const VT *__restrict__ val,
                                                     const T *__restrict__ b, const T *__restrict__ x,
                                                     T *__restrict__ r) {
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool ok = row < n;
    int64_t lo = ok ? ptr[row] : 0, hi = ok ? ptr[row + 1] : 0;
    const A bi = (ok && sub == 0) ? (A)b[row] : A(0);
    A s = row_dot<TPR, A>(lo, hi, sub, col, val, x);
    if (ok && sub == 0) r[row] = (T)(bi - s);
}

// ---------------------------------------------------------------------------------
// Multicolour Gauss-Seidel colour phases on a colour split (positions p in [pb, pe)
// hold row perm[p]; L/U hold the entries of lower/higher colour).
// forward from zero:   y_i = (r_i - sum_L a_ij y_j) / a_ii
// backward from there: y_i = y_i - (sum_U a_ij y_j) / a_ii
// backward full sweep: x_i = (b_i - sum_L a_ij x_j - sum_U a_ij x_j) / a_ii
// ---------------------------------------------------------------------------------
// Programmatic dependent launch (sm_90+): a kernel launched with programmatic stream
// serialization may start while its predecessor is still running. It lets its own
// successor launch at once, loads the data no kernel of the solve writes (the matrix),
// then waits until the predecessor has finished and its writes are visible before it
// touches any vector. Without the launch attribute both instructions are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One colour phase of the symmetric Gauss-Seidel sweep from zero (CSR colour split):
//   BACK = false: y_i = (r_i - sum_L a_ij y_j) / a_ii
//   BACK = true:  y_i = y_i - (sum_U a_ij y_j) / a_ii
// Static loads (position, bounds, diagonal, first batch of the row's entries) happen
// before the dependency wait, so they overlap the previous phase. A lane takes NB
// entries per batch (entries sub, sub + TPR, ...): NB is fitted to the colour's longest
// row part, because every FMA slot of a batch is issued whether its entry exists or not
// and GB300's FP64 pipe is narrow. Lane `sub` adds its entries in ascending order for
// every NB, so the result does not depend on NB.
template <int TPR, int NB, typename PT, typename TR, bool BACK>
__global__ void __launch_bounds__(kBlock) k_gs_phase(int64_t pb, int64_t pe, const int32_t *__restrict__ perm,
                                                     const int64_t *__restrict__ xptr, const int32_t *__restrict__ xcol,
                                                     const PT *__restrict__ xval, const PT *__restrict__ dinv,
                                                     const TR *r, PT *y) {
    pdl_trigger();
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t p = pb + gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool ok = p < pe;
    const bool lead = ok && sub == 0;
    const int32_t i = lead ? perm[p] : 0;
    const PT di = lead ? dinv[p] : PT(1);
    const int64_t lo = ok ? xptr[p] : 0, hi = ok ? xptr[p + 1] : 0;
    int c[NB];
    PT v[NB];
    const int64_t b0 = lo + sub;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const int64_t e = b0 + (int64_t)k * TPR;
        const bool in = e < hi;
        c[k] = in ? ldst(&xcol[e]) : -1;
        v[k] = in ? ldst(&xval[e]) : PT(0);
    }
    // entries of the warp's busiest lane: FMA slots past it are skipped by a warp-uniform
    // branch (an issued FP64 slot costs the same whether a lane uses it or not)
    const unsigned mine = hi > b0 ? (unsigned)((hi - b0 + TPR - 1) / TPR) : 0u;
    const int wmax = (int)__reduce_max_sync(kFull, mine);
    pdl_wait();
    PT own = PT(0);
    if (lead) own = BACK ? y[i] : (PT)r[i];
    PT acc = PT(0);
#pragma unroll
    for (int k = 0; k < NB; ++k)
        if (k < wmax && c[k] >= 0) acc += v[k] * y[c[k]];
    for (int k0 = NB; k0 < wmax; k0 += NB) {
        const int64_t base = b0 + (int64_t)k0 * TPR;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int64_t e = base + (int64_t)k * TPR;
            const bool in = e < hi;
            c[k] = in ? ldst(&xcol[e]) : -1;
            v[k] = in ? ldst(&xval[e]) : PT(0);
        }
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (k0 + k < wmax && c[k] >= 0) acc += v[k] * y[c[k]];
    }
    acc = subwarp_sum<TPR>(acc);
    if (lead) y[i] = BACK ? own - acc * di : (own - acc) * di;
}

// One colour phase over interleaved slices (slices.cu), one warp per slice: W steps of 32
// entries, T lanes per row; the sums are those of k_gs_phase with T lanes. Over whole rows
// (r = b) the BACK = false form is a phase of a full sweep, y_i = (b_i - sum a_ij y_j) / a_ii.
//
// Small phases are bound by their chain of dependent accesses and FP64 adds, large ones by
// the L2 sectors and L1 lines they touch. In the row-pointer layout a group of 4 lanes reads
// 16 unaligned bytes of columns and 32 of values per step: 0.59 lines an entry besides the
// 0.39 of the gathers (host count at P4 7^3). A slice's step is one line of columns and two
// of values: 0.1 lines an entry. FP64 S_k, us before -> after (graph replays): P4 48^3
// 2325 -> 1804, P4 24^3 597 -> 446, P3 32^3 359 -> 276, P2 33^3 129 -> 89, P2 8^3 46 -> 38;
// FP32: P4 48^3 1379 -> 1204, P3 32^3 191 -> 170, P3 9^3 68 -> 65. At P4 48^3 FP64 it reads
// about 1.0 sectors an entry at the 300 G sectors/s that random gathers reach there.
//
// NV vectors at once (r and y of vector v at r + v n, y + v n): the slice is read once.
//
// LATE: the successor may launch only once this phase's wait is over, so no more than one
// phase waits at a time (slice_late in solve.cu says when that is faster).
template <int NB, int NV, bool LATE, typename PT, typename TR, bool BACK>
__global__ void __launch_bounds__(kBlock) k_slice_phase(int64_t s0, int64_t s1, const int4 *__restrict__ meta,
                                                        const int32_t *__restrict__ rows,
                                                        const PT *__restrict__ dinv, const int32_t *__restrict__ col,
                                                        const PT *__restrict__ val, const TR *r, PT *y, int64_t n) {
    if (!LATE) pdl_trigger();
    const int64_t s = s0 + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (s >= s1) {  // a whole warp
        pdl_wait();
        return;
    }
    const int4 m = meta[s];
    const int w = m.w & 0xfffff, lt = (m.w >> 20) & 15, nr = (m.w >> 24) & 255;
    const int64_t e0 = (((int64_t)m.y << 32) | (uint32_t)m.x) + lane;
    int c[NB];
    PT v[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const bool in = k < w;
        c[k] = in ? ldst(&col[e0 + 32 * k]) : -1;
        v[k] = in ? ldst(&val[e0 + 32 * k]) : PT(0);
    }
    const int q = lane >> lt;
    const bool lead = (lane & ((1 << lt) - 1)) == 0 && q < nr;
    const int32_t i = lead ? rows[m.z + q] : 0;
    const PT di = lead ? dinv[m.z + q] : PT(1);
    pdl_wait();
    if (LATE) pdl_trigger();
    PT own[NV], acc[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) {
        own[u] = PT(0);
        if (lead) own[u] = BACK ? y[u * n + i] : (PT)r[u * n + i];
        acc[u] = PT(0);
    }
#pragma unroll
    for (int k = 0; k < NB; ++k)
        if (k < w && c[k] >= 0) {
#pragma unroll
            for (int u = 0; u < NV; ++u) acc[u] += v[k] * y[u * n + c[k]];
        }
    for (int k0 = NB; k0 < w; k0 += NB) {
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const bool in = k0 + k < w;
            c[k] = in ? ldst(&col[e0 + 32 * (int64_t)(k0 + k)]) : -1;
            v[k] = in ? ldst(&val[e0 + 32 * (int64_t)(k0 + k)]) : PT(0);
        }
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (k0 + k < w && c[k] >= 0) {
#pragma unroll
                for (int u = 0; u < NV; ++u) acc[u] += v[k] * y[u * n + c[k]];
            }
    }
    for (int o = 1 << lt >> 1; o > 0; o >>= 1) {
#pragma unroll
        for (int u = 0; u < NV; ++u) acc[u] += __shfl_xor_sync(kFull, acc[u], o);
    }
    if (lead) {
#pragma unroll
        for (int u = 0; u < NV; ++u) y[u * n + i] = BACK ? own[u] - acc[u] * di : (own[u] - acc[u]) * di;
    }
}

// The loads of a colour phase without its dependency: every position of [0, n) at
// once, out[i] = dinv_i * sum_part a_ij x_j with x read-only (a measurement of the
// smoother's memory work without the barriers between colours; not used by a solve).
template <int TPR, int NB, typename PT>
__global__ void __launch_bounds__(kBlock) k_split_pass(int64_t n, const int32_t *__restrict__ perm,
                                                       const int64_t *__restrict__ xptr,
                                                       const int32_t *__restrict__ xcol,
                                                       const PT *__restrict__ xval, const PT *__restrict__ dinv,
                                                       const PT *__restrict__ x, PT *__restrict__ out) {
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t p = gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool ok = p < n;
    const int64_t lo = ok ? xptr[p] : 0, hi = ok ? xptr[p + 1] : 0;
    PT acc = PT(0);
    for (int64_t base = lo + sub; base < hi; base += (int64_t)NB * TPR) {
        int c[NB];
        PT v[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int64_t e = base + (int64_t)k * TPR;
            const bool in = e < hi;
            c[k] = in ? ldst(&xcol[e]) : -1;
            v[k] = in ? ldst(&xval[e]) : PT(0);
        }
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (c[k] >= 0) acc += v[k] * x[c[k]];
    }
    acc = subwarp_sum<TPR>(acc);
    if (ok && sub == 0) out[perm[p]] = acc * dinv[p];
}

// The same phase over a capped grid: sub-warp g takes rows pb + g, pb + g + nsub, ...
// (nsub sub-warps in the grid) and loads the next row's position, diagonal and first
// batch of entries while the current row's gathers are in flight, with the bounds of
// the row after that one step further ahead. Each row's sum is formed exactly as in
// k_gs_phase<TPR, NB> (bitwise the same result). The grid is at most the blocks that
// are resident at once, so on phases of several waves no block waits for a slot and
// every lane group keeps a row's loads in flight behind the current one.
// The loop runs while the warp's first sub-warp has a row, so every lane of the warp
// reaches the shuffles; a sub-warp past the end takes no entries and stores nothing.
template <int TPR, int NB, typename PT>
__device__ __forceinline__ void gs_row_static(int64_t q, bool ok, bool lead, int sub, int64_t lo, int64_t hi,
                                              const int32_t *__restrict__ perm, const int32_t *__restrict__ xcol,
                                              const PT *__restrict__ xval, const PT *__restrict__ dinv,
                                              int32_t &i, PT &di, int (&c)[NB], PT (&v)[NB]) {
    i = (ok && lead) ? perm[q] : 0;
    di = (ok && lead) ? dinv[q] : PT(1);
    const int64_t b0 = lo + sub;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const int64_t e = b0 + (int64_t)k * TPR;
        const bool in = e < hi;
        c[k] = in ? ldst(&xcol[e]) : -1;
        v[k] = in ? ldst(&xval[e]) : PT(0);
    }
}

template <int TPR, int NB, typename PT, typename TR, bool BACK>
__global__ void __launch_bounds__(kBlock) k_gs_phase_gs(int64_t pb, int64_t pe, const int32_t *__restrict__ perm,
                                                        const int64_t *__restrict__ xptr,
                                                        const int32_t *__restrict__ xcol,
                                                        const PT *__restrict__ xval, const PT *__restrict__ dinv,
                                                        const TR *r, PT *y) {
    pdl_trigger();
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nsub = (int64_t)gridDim.x * blockDim.x / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool lead = sub == 0;
    int64_t p = pb + gt / TPR;
    int64_t pw = pb + (gt & ~(int64_t)31) / TPR;  // the warp's first sub-warp's row
    bool ok = p < pe;
    int64_t lo = ok ? xptr[p] : 0, hi = ok ? xptr[p + 1] : 0;
    int32_t i;
    PT di;
    int c[NB];
    PT v[NB];
    gs_row_static<TPR, NB, PT>(p, ok, lead, sub, lo, hi, perm, xcol, xval, dinv, i, di, c, v);
    int64_t pn = p + nsub;
    int64_t lon = pn < pe ? xptr[pn] : 0, hin = pn < pe ? xptr[pn + 1] : 0;
    pdl_wait();
    while (pw < pe) {
        // next row: static loads now, consumed in the next pass
        const bool okn = pn < pe;
        int32_t i_n;
        PT di_n;
        int cn[NB];
        PT vn[NB];
        gs_row_static<TPR, NB, PT>(pn, okn, lead, sub, lon, hin, perm, xcol, xval, dinv, i_n, di_n, cn, vn);
        const int64_t pnn = pn + nsub;
        const int64_t lonn = pnn < pe ? xptr[pnn] : 0, hinn = pnn < pe ? xptr[pnn + 1] : 0;
        // this row
        PT own = PT(0);
        if (ok && lead) own = BACK ? y[i] : (PT)r[i];
        PT acc = PT(0);
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (c[k] >= 0) acc += v[k] * y[c[k]];
        for (int64_t base = lo + sub + (int64_t)NB * TPR; base < hi; base += (int64_t)NB * TPR) {
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const int64_t e = base + (int64_t)k * TPR;
                const bool in = e < hi;
                c[k] = in ? ldst(&xcol[e]) : -1;
                v[k] = in ? ldst(&xval[e]) : PT(0);
            }
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (c[k] >= 0) acc += v[k] * y[c[k]];
        }
        acc = subwarp_sum<TPR>(acc);
        if (ok && lead) y[i] = BACK ? own - acc * di : (own - acc) * di;
        // advance
        p = pn;
        pw += nsub;
        ok = okn;
        i = i_n;
        di = di_n;
        lo = lon;
        hi = hin;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            c[k] = cn[k];
            v[k] = vn[k];
        }
        pn = pnn;
        lon = lonn;
        hin = hinn;
    }
}

// The same phase with two rows per sub-warp: rows p and p + half of the colour (no edge
// joins two rows of one colour, so neither reads the other's result). Both rows' loads
// are issued before either row's gathers, doubling the loads in flight per lane for
// phases that are bound by load latency. Each row's sum is formed exactly as above.
template <int TPR, int NB, typename PT, typename TR, bool BACK>
__global__ void __launch_bounds__(kBlock) k_gs_phase2(int64_t pb, int64_t pe, const int32_t *__restrict__ perm,
                                                      const int64_t *__restrict__ xptr,
                                                      const int32_t *__restrict__ xcol, const PT *__restrict__ xval,
                                                      const PT *__restrict__ dinv, const TR *r, PT *y) {
    pdl_trigger();
    const int64_t half = (pe - pb + 1) / 2;
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t p0 = pb + gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    int64_t pr[2] = {p0, p0 + half};
    bool ok[2], lead[2];
    int32_t i[2];
    PT di[2];
    int64_t lo[2], hi[2];
    int c[2][NB];
    PT v[2][NB];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        ok[q] = (q == 0 ? pr[0] < pb + half : pr[1] < pe);
        lead[q] = ok[q] && sub == 0;
        i[q] = lead[q] ? perm[pr[q]] : 0;
        di[q] = lead[q] ? dinv[pr[q]] : PT(1);
        lo[q] = ok[q] ? xptr[pr[q]] : 0;
        hi[q] = ok[q] ? xptr[pr[q] + 1] : 0;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int64_t e = lo[q] + sub + (int64_t)k * TPR;
            const bool in = e < hi[q];
            c[q][k] = in ? ldst(&xcol[e]) : -1;
            v[q][k] = in ? ldst(&xval[e]) : PT(0);
        }
    }
    pdl_wait();
    PT own[2], acc[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        own[q] = PT(0);
        if (lead[q]) own[q] = BACK ? y[i[q]] : (PT)r[i[q]];
        acc[q] = PT(0);
    }
    PT x[2][NB];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < NB; ++k) x[q][k] = c[q][k] >= 0 ? y[c[q][k]] : PT(0);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (c[q][k] >= 0) acc[q] += v[q][k] * x[q][k];
        for (int64_t base = lo[q] + sub + (int64_t)NB * TPR; base < hi[q]; base += (int64_t)NB * TPR) {
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const int64_t e = base + (int64_t)k * TPR;
                const bool in = e < hi[q];
                c[q][k] = in ? ldst(&xcol[e]) : -1;
                v[q][k] = in ? ldst(&xval[e]) : PT(0);
            }
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (c[q][k] >= 0) acc[q] += v[q][k] * y[c[q][k]];
        }
        acc[q] = subwarp_sum<TPR>(acc[q]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
        if (lead[q]) y[i[q]] = BACK ? own[q] - acc[q] * di[q] : (own[q] - acc[q]) * di[q];
}

template <int TPR, int NB, typename PT>
__global__ void __launch_bounds__(kBlock) k_gs_bwd_full(int64_t pb, int64_t pe, const int32_t *__restrict__ perm,
                                                        const int64_t *__restrict__ lptr, const int32_t *__restrict__ lcol,
                                                        const PT *__restrict__ lval, const int64_t *__restrict__ uptr,
                                                        const int32_t *__restrict__ ucol, const PT *__restrict__ uval,
                                                        const PT *__restrict__ diag, const PT *__restrict__ b,
                                                        PT *x) {
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t p = pb + gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool ok = p < pe;
    const bool lead = ok && sub == 0;
    const int32_t i = lead ? perm[p] : 0;
    const PT d = lead ? diag[p] : PT(1);
    const int64_t llo = ok ? lptr[p] : 0, lhi = ok ? lptr[p + 1] : 0;
    const int64_t ulo = ok ? uptr[p] : 0, uhi = ok ? uptr[p + 1] : 0;
    const PT bi = lead ? b[i] : PT(0);
    PT sl = row_dot<TPR, PT, PT, PT, NB>(llo, lhi, sub, lcol, lval, (const PT *)x);
    PT su = row_dot<TPR, PT, PT, PT, NB>(ulo, uhi, sub, ucol, uval, (const PT *)x);
    if (lead) x[i] = (bi - sl - su) / d;
}

// l1-Jacobi from zero: x = r / d
template <typename PT, typename TR>
__global__ void k_jacobi0(int64_t n, const PT *__restrict__ d, const TR *__restrict__ r, PT *__restrict__ x) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = (PT)r[i] / d[i];
}

// z_i = zs_i + sum_j Pi_ij w_j (I_P has at most 4 entries per row: one thread per row)
template <typename PT, typename ZT>
__global__ void k_prolong_add(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                              const PT *__restrict__ val, const PT *__restrict__ w, const PT *zs, ZT *z) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    PT s = PT(0);
    for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e) s += val[e] * w[col[e]];
    z[i] = (ZT)zs[i] + (ZT)s;
}

// x_i += sum_j P_ij xc_j
template <int TPR, typename PT>
__global__ void __launch_bounds__(kBlock) k_prolong_inplace(int64_t n, const int64_t *__restrict__ ptr,
                                                            const int32_t *__restrict__ col,
                                                            const PT *__restrict__ val, const PT *__restrict__ xc,
                                                            PT *__restrict__ x) {
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = gt / TPR;
    const int sub = threadIdx.x & (TPR - 1);
    const bool ok = row < n;
    int64_t lo = ok ? ptr[row] : 0, hi = ok ? ptr[row + 1] : 0;
    const PT xi = (ok && sub == 0) ? x[row] : PT(0);
    PT s = row_dot<TPR, PT>(lo, hi, sub, col, val, xc);
    if (ok && sub == 0) x[row] = xi + s;
}

// A sum of products in the dense products below. FP32 carries the rounding errors of its
// products and sums along (Dot2 of Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26, 2005): a row
// has up to 5120 terms where a colour phase's has tens, so plain FP32 sums are further off than
// the sweeps they replace. Against FP64, B r at P2 8^3: 6.5e-8 as sweeps, 1.2e-7 with plain sums,
// 3.4e-8 so; the V-cycle at P3 16^3: 8.6e-8, 1.3e-7, 4.6e-8. The FP32 pipe has room for it beside
// the loads: P2 8^3's product takes 12 us instead of 10, its solve 0.86 ms instead of 0.825. (Errors
// carried every two products leave P1 9^3, 512 rows, 7% further off than its sweeps.)
template <typename T>
struct DenseSum {
    T s = T(0);
    __device__ __forceinline__ void add(T a, T b) { s += a * b; }
    __device__ __forceinline__ void merge(const DenseSum &o) { s += o.s; }
    __device__ __forceinline__ DenseSum shfl_xor(int o) const {
        DenseSum t;
        t.s = __shfl_xor_sync(kFull, s, o);
        return t;
    }
    template <typename TX>
    __device__ __forceinline__ TX value() const { return (TX)s; }
};
template <>
struct DenseSum<float> {
    float s = 0.0f, c = 0.0f;
    // s + v exactly as the rounded sum and its error
    __device__ __forceinline__ void two_sum(float v, float e) {
        const float t = __fadd_rn(s, v), w = __fsub_rn(t, s);
        e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, w)), __fsub_rn(v, w)));
        s = t;
        c = __fadd_rn(c, e);
    }
    __device__ __forceinline__ void add(float a, float b) {
        const float p = __fmul_rn(a, b);
        two_sum(p, __fmaf_rn(a, b, -p));
    }
    __device__ __forceinline__ void merge(const DenseSum &o) { two_sum(o.s, o.c); }
    __device__ __forceinline__ DenseSum shfl_xor(int o) const {
        DenseSum t;
        t.s = __shfl_xor_sync(kFull, s, o);
        t.c = __shfl_xor_sync(kFull, c, o);
        return t;
    }
    template <typename TX>
    __device__ __forceinline__ TX value() const { return (TX)s + (TX)c; }
};

// x = M b for the dense tail of the V-cycle or a small problem's whole preconditioner (one warp
// per row; small blocks, so that a few hundred rows spread over the chip). Bound by reading M:
// eight loads in flight per lane and four partial sums.
template <typename PT, typename TB, typename TX>
__global__ void __launch_bounds__(128) k_dense_mv(int64_t n, const PT *__restrict__ M, const TB *__restrict__ b,
                                                  TX *__restrict__ x) {
    const int lane = threadIdx.x & 31;
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (row >= n) return;  // whole warp leaves together
    const PT *m = M + row * n;
    DenseSum<PT> acc[4];
    int64_t j = lane;
    for (; j + 7 * 32 < n; j += 8 * 32) {
        PT u[8], v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            u[k] = ldg(&m[j + 32 * k]);
            v[k] = (PT)ldg(&b[j + 32 * k]);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k & 3].add(u[k], v[k]);
    }
    PT u[8], v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const bool in = j + 32 * k < n;
        u[k] = in ? ldg(&m[j + 32 * k]) : PT(0);
        v[k] = in ? (PT)ldg(&b[j + 32 * k]) : PT(0);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (j + 32 * k - lane < n) acc[k & 3].add(u[k], v[k]);
    acc[0].merge(acc[1]);
    acc[2].merge(acc[3]);
    acc[0].merge(acc[2]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[0].merge(acc[0].shfl_xor(o));
    if (lane == 0) x[row] = acc[0].template value<TX>();
}

// ---------------------------------------------------------------------------------
// SELL-32 kernels: one thread per row; a warp is one slice, so every column and value
// load of the warp is one contiguous access. Padding entries carry column -1.
// ---------------------------------------------------------------------------------
// One colour phase of the symmetric Gauss-Seidel sweep from zero over the SELL-32 slices
// [s0, s1) of a colour-sorted split, one thread per row (no reduction across lanes):
//   BACK = false: y_i = (r_i - sum_L a_ij y_j) * dinv_i
//   BACK = true:  y_i = y_i - (sum_U a_ij y_j) * dinv_i
// Padding positions (perm < 0) only carry column -1 entries. Launched with PDL: static
// loads before the dependency wait.
template <typename PT, typename TR, bool BACK>
__global__ void __launch_bounds__(kBlock) k_sell_phase(int64_t s0, int64_t s1, const int32_t *__restrict__ perm,
                                                       const int64_t *__restrict__ sptr, const int32_t *__restrict__ sw,
                                                       const int32_t *__restrict__ col, const PT *__restrict__ val,
                                                       const PT *__restrict__ dinv, const TR *r, PT *y) {
    pdl_trigger();
    const int64_t q = s0 * 32 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= s1 * 32) return;
    const int64_t s = q >> 5;
    const int32_t i = perm[q];
    const int64_t base = sptr[s] + (q & 31);
    const int w = sw[s];
    const PT di = dinv[q];
    int c[kBatch];
    PT v[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
        const bool in = k < w;
        c[k] = in ? ldst(&col[base + 32 * (int64_t)k]) : -1;
        v[k] = in ? ldst(&val[base + 32 * (int64_t)k]) : PT(0);
    }
    pdl_wait();
    PT own = PT(0);
    if (i >= 0) own = BACK ? y[i] : (PT)r[i];
    PT acc = PT(0);
#pragma unroll
    for (int k = 0; k < kBatch; ++k)
        if (c[k] >= 0) acc += v[k] * y[c[k]];
    for (int k0 = kBatch; k0 < w; k0 += kBatch) {
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const bool in = k0 + k < w;
            c[k] = in ? ldst(&col[base + 32 * (int64_t)(k0 + k)]) : -1;
            v[k] = in ? ldst(&val[base + 32 * (int64_t)(k0 + k)]) : PT(0);
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
            if (c[k] >= 0) acc += v[k] * y[c[k]];
    }
    if (i >= 0) y[i] = BACK ? own - acc * di : (own - acc) * di;
}

}  // namespace pk
