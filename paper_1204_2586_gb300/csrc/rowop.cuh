// rowop.cuh -- the fine operator A_h as the fused Krylov kernels (PCG in solve.cu,
// FGMRES in gmres.cu) read it: the layout setup chose.
#pragma once

#include "kernels.cuh"

namespace pk {

// The fine operator A_h as the fused Krylov kernels see it: CSR rows read by sub-warps of
// TPR lanes (TPR > 0, options.spmv_threads), or interleaved slices of its rows (slices.cu)
// read one warp per slice (TPR < 0).
//
// The product is bound by HBM and the FP64 pipe together (2 flops per 12 bytes; both floors
// within 20%), so what counts is one FP64 slot per entry and no row that holds its warp
// back: one lane per row where there are rows enough, lanes doubling with the length. With
// 32 rows in their natural order per warp (SELL-32, the former layout) the vertex rows of
// P4, 370 entries, ran on one lane each. us, before -> after: P4 24^3 150 -> 120, P3 24^3
// 46 -> 37, P3 32^3 86 -> 79, P4 48^3 1015 -> 986, P2 33^3 27 -> 23, P2 21^3 10.0 -> 8.7.
struct RowOp {
    const int64_t *ptr;
    const int32_t *col;
    const double *val;
    const int4 *meta = nullptr;
    const int32_t *rows = nullptr;
    int64_t nslices = 0;
};

inline RowOp fine_op(const pkasp_problem *p) {
    if (p->spmv_tpr > 500) {
        const DSlices &S = p->fsv;
        return RowOp{nullptr, S.col, S.val, S.meta, S.rows, S.nslices};
    }
    return RowOp{p->Ah.ptr, p->Ah.col, p->Ah.val};
}

// Grid of the kernels that read A_h through for_rows (some of them reduce one value
// with grid_reduce): a warp per slice or a sub-warp (CSR) per row, as in the plain
// SpMV, up to the capacity of the partials buffer (kRedGrid * 4 * PKASP_MAX_COLS
// values). A grid of kRedGrid blocks striding over the rows left the SpMV at about 1.5x
// the plain one's time.
inline unsigned fine_grid(const pkasp_problem *p) {
    const int64_t threads = p->spmv_tpr > 500 ? p->fsv.nslices * 32 : p->nh * p->spmv_tpr;
    const int64_t g = std::max<int64_t>(1, (threads + kBlock - 1) / kBlock);
    return (unsigned)std::min<int64_t>(g, (int64_t)kRedGrid * 4 * PKASP_MAX_COLS);
}

// f(row, (A x)_row) for every row, grid-stride; every lane of a warp runs the same
// number of trips (the shuffles of the CSR form need the whole warp)
template <int TPR, class F>
__device__ __forceinline__ void for_rows(int64_t n, const RowOp &A, const double *x, F f) {
    if constexpr (TPR < 0) {
        const int lane = threadIdx.x & 31;
        const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
        for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < A.nslices; s += nwarps) {
            const int4 m = A.meta[s];
            const int w = m.w & 0xfffff, lt = (m.w >> 20) & 15, nr = (m.w >> 24) & 255, q = lane >> lt;
            const int64_t e0 = (((int64_t)m.y << 32) | (uint32_t)m.x) + lane;
            const bool lead = (lane & ((1 << lt) - 1)) == 0 && q < nr;
            const int32_t row = lead ? A.rows[m.z + q] : 0;
            double acc = 0.0;
            for (int k0 = 0; k0 < w; k0 += kBatch) {
                int c[kBatch];
                double v[kBatch];
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    const bool in = k0 + k < w;
                    c[k] = in ? ldst(&A.col[e0 + 32 * (int64_t)(k0 + k)]) : -1;
                    v[k] = in ? ldst(&A.val[e0 + 32 * (int64_t)(k0 + k)]) : 0.0;
                }
#pragma unroll
                for (int k = 0; k < kBatch; ++k)
                    if (k0 + k < w && c[k] >= 0) acc += v[k] * x[c[k]];
            }
            for (int o = 1 << lt >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
            if (lead) f((int64_t)row, acc);
        }
    } else {
        const int sub = threadIdx.x & (TPR - 1);
        const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
        const int rpw = 32 / TPR, sg = (threadIdx.x & 31) / TPR;
        for (int64_t base = warp * rpw; base < n; base += nwarps * rpw) {
            const int64_t row = base + sg;
            const bool ok = row < n;
            int64_t lo = ok ? A.ptr[row] : 0, hi = ok ? A.ptr[row + 1] : 0;
            double s = row_dot<TPR, double>(lo, hi, sub, A.col, A.val, x);
            if (ok && sub == 0) f(row, s);
        }
    }
}

// kernel template dispatch on the fine SpMV layout (500 + t = interleaved slices, t = CSR
// with t lanes)
#define PK_FMT_SWITCH(tpr, BODY)                          \
    switch ((tpr) > 500 ? -1 : (tpr)) {                   \
        case -1: { constexpr int TPR = -1; BODY; } break; \
        case 4: { constexpr int TPR = 4; BODY; } break;   \
        case 8: { constexpr int TPR = 8; BODY; } break;   \
        case 16: { constexpr int TPR = 16; BODY; } break; \
        default: { constexpr int TPR = 32; BODY; } break; \
    }

}  // namespace pk
