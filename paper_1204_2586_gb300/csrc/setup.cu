// setup.cu -- device-side construction of the auxiliary-space preconditioner:
//   * the P1 algebraic multigrid hierarchy on A_H (Step 1 of Algorithm 2.1 solved by one
//     AMG cycle, Remark 2.1): strength of connection (Sec. 6.2), PMIS coarsening and
//     extended+i interpolation (cited in Sec. 1 and 6.1), Galerkin products P^T A P
//     (the relation A_H = I_R A_h I_P of Sec. 2 applied level by level) and a dense
//     inverse of the coarsest matrix.
// Everything that decides an integer (colours, strength, C/F) is computed from the same
// FP64 values by integer-exact rules, so it is reproducible; floating-point sums run in a
// fixed order per entry (one thread or one warp per row, no atomics on values).
#include <algorithm>
#include <cstring>

#include "internal.h"
#include "pmis.cuh"

namespace pk {

void to32(const double *x, float *y, int64_t n, cudaStream_t s);

namespace {

unsigned blocks_for(int64_t n, int per) {
    int64_t b = (n + per - 1) / per;
    return (unsigned)std::max<int64_t>(1, b);
}


__global__ void k_l1norm(int64_t n, const int64_t *__restrict__ ptr, const double *__restrict__ val,
                         double *__restrict__ l1) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e) s += fabs(val[e]);
    l1[i] = s;
}

// ---------------------------------------------------------------------------------
// Strength of connection (Sec. 6.2): j strong for i iff j != i and
// -a_ij > theta * max_{k != i}(-a_ik); no strong entries if that maximum is <= 0.
// ---------------------------------------------------------------------------------
__global__ void k_strength(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                           const double *__restrict__ val, double theta, uint8_t *__restrict__ strong) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double mx = 0.0;
    bool have = false;
    for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e) {
        if (col[e] == i) continue;
        double v = -val[e];
        if (!have || v > mx) mx = v;
        have = true;
    }
    const double thr = __dmul_rn(theta, mx);
    for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e) {
        uint8_t s = 0;
        if (have && mx > 0.0 && col[e] != i) s = (-val[e] > thr) ? 1 : 0;
        strong[e] = s;
    }
}

// ---------------------------------------------------------------------------------
// PMIS (De Sterck, Yang & Heys 2006), one thread per row; the per-row rules are in
// pmis.cuh (shared with the fixed-scratch entry point).
// ---------------------------------------------------------------------------------
__global__ void k_mirror(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                         int64_t *__restrict__ mirror, int *__restrict__ bad) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) pmis_mirror_row<int64_t>(i, n, ptr, col, mirror, bad);
}

__global__ void k_pmis_init(int64_t n, const int64_t *__restrict__ ptr, const int64_t *__restrict__ mirror,
                            const uint8_t *__restrict__ strong, int64_t *__restrict__ mu,
                            int8_t *__restrict__ cf, unsigned long long *__restrict__ undecided) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && pmis_init_row<int64_t>(i, ptr, mirror, strong, mu, cf)) atomicAdd(undecided, 1ull);
}

__global__ void k_pmis_select(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                              const int64_t *__restrict__ mirror, const uint8_t *__restrict__ strong,
                              const int64_t *__restrict__ mu, uint64_t stream, const int8_t *__restrict__ cf,
                              uint8_t *__restrict__ newc) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) newc[i] = pmis_select_row<int64_t>(i, ptr, col, mirror, strong, mu, stream, cf);
}

__global__ void k_pmis_commit(int64_t n, const uint8_t *__restrict__ newc, int8_t *__restrict__ cf) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && newc[i]) cf[i] = 1;
}

__global__ void k_pmis_mark_f(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                              const uint8_t *__restrict__ strong, const uint8_t *__restrict__ newc,
                              int8_t *__restrict__ cf, unsigned long long *__restrict__ undecided) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && pmis_mark_row(i, ptr, col, strong, newc, cf)) atomicAdd(undecided, 1ull);
}

__global__ void k_flag_c(int64_t n, const int8_t *__restrict__ cf, int64_t *__restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (cf[i] == 1) ? 1 : 0;
}

// ---------------------------------------------------------------------------------
// Extended+i interpolation (De Sterck, Falgout, Nolting & Yang 2008), no truncation; a
// strong F neighbour k with zero denominator is lumped into the diagonal. With cc = 1
// (extended+i+cc, the form Sec. 1 and Sec. 6.1 name) a strong F neighbour k that shares
// a strong C point with i adds none of its own C points to the interpolatory set; the
// weights then follow from the same formula over that smaller set.
// ---------------------------------------------------------------------------------
__global__ void k_extpi_ub(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                           const uint8_t *__restrict__ strong, const int8_t *__restrict__ cf,
                           int64_t *__restrict__ ub) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (cf[i] == 1) {
        ub[i] = 1;
        return;
    }
    int64_t s = 0;
    for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e) {
        if (!strong[e]) continue;
        int32_t k = col[e];
        s += 1;
        if (cf[k] == -1) s += ptr[k + 1] - ptr[k];
    }
    ub[i] = s;
}

// ---------------------------------------------------------------------------------
// Sorted set of column indices, one block of NT threads per row: candidates go into an
// open-addressing table of CAP slots in shared memory (at most half full), the distinct
// ones are then gathered and sorted there (bitonic) and written out in ascending order.
// A row with more distinct columns than that leaves cnt[row] = -1 and is taken by the
// next larger table, at last by a heap sort in global memory (union_rows). One thread
// per row with a heap sort of all candidates took 71 ms of a 312 ms setup at P3 24^3
// (few threads, each with long chains of dependent global accesses); the table form
// takes 0.35 ms.
// ---------------------------------------------------------------------------------
template <int NT, int CAP>
struct ColSet {
    static constexpr int kMost = CAP / 2;  // the other half leaves room for NT late inserts
    static_assert(CAP / 2 >= NT, "table too small for the block");
    int32_t *tab;   // [CAP]
    int32_t *list;  // [CAP]
    int *num;       // distinct entries; > kMost: overflow

    __device__ void clear() {
        for (int q = threadIdx.x; q < CAP; q += NT) tab[q] = -1;
        if (threadIdx.x == 0) *num = 0;
        __syncthreads();
    }
    __device__ bool full() const { return *(volatile int *)num > kMost; }
    __device__ void insert(int32_t v) {
        if (full()) return;  // at most NT - 1 inserts are under way past this check
        unsigned h = ((unsigned)v * 2654435761u) & (CAP - 1);
        for (;;) {
            const int32_t old = atomicCAS(&tab[h], -1, v);
            if (old == v) return;
            if (old == -1) {
                atomicAdd(num, 1);
                return;
            }
            h = (h + 1) & (CAP - 1);
        }
    }
    // sorts the set into out[0..m); returns m, or -1 after an overflow (block-uniform)
    __device__ int sorted(int32_t *out) {
        __syncthreads();
        const int m = *num;
        if (m > kMost) return -1;
        int p2 = 1;
        while (p2 < m) p2 <<= 1;
        __syncthreads();
        if (threadIdx.x == 0) *num = 0;
        for (int q = threadIdx.x; q < p2; q += NT) list[q] = INT32_MAX;
        __syncthreads();
        for (int q = threadIdx.x; q < CAP; q += NT)
            if (tab[q] != -1) list[atomicAdd(num, 1)] = tab[q];
        __syncthreads();
        for (int k = 2; k <= p2; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int t = threadIdx.x; t < p2 / 2; t += NT) {
                    const int x = ((t & ~(j - 1)) << 1) | (t & (j - 1)), y = x | j;
                    const int32_t u = list[x], v = list[y];
                    if ((u > v) == ((x & k) == 0)) {
                        list[x] = v;
                        list[y] = u;
                    }
                }
                __syncthreads();
            }
        for (int q = threadIdx.x; q < m; q += NT) out[q] = list[q];
        return m;
    }
};

// 1 when k has a strong C point that is also a strong C point of i
__device__ bool shares_strong_c(const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                                const uint8_t *__restrict__ strong, const int8_t *__restrict__ cf, int64_t i,
                                int32_t k) {
    for (int64_t f = ptr[k]; f < ptr[k + 1]; ++f) {
        if (!strong[f] || cf[col[f]] != 1) continue;
        for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e)
            if (strong[e] && col[e] == col[f]) return true;
    }
    return false;
}

// The columns that a row of the product or of the interpolation may hold, as seen by one
// lane group: visit(i, part, nparts, f) calls f(column) for the candidates of row i that
// fall to lane `part` of `nparts`. ub is the row's number of candidates with repeats.
struct HatCands {  // interpolatory set of F row i: strong C neighbours, and those of strong F neighbours
    const int64_t *__restrict__ ptr;
    const int32_t *__restrict__ col;
    const uint8_t *__restrict__ strong;
    const int8_t *__restrict__ cf;
    int cc;
    // C rows interpolate from themselves alone
    __device__ bool single(int64_t i) const { return cf[i] == 1; }
    template <class F>
    __device__ void visit(int64_t i, int part, int nparts, F f) const {
        for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e) {
            if (!strong[e]) continue;
            const int32_t k = col[e];
            if (cf[k] == 1) {
                if (part == 0) f(k);
            } else if (!cc || !shares_strong_c(ptr, col, strong, cf, i, k)) {
                for (int64_t q = ptr[k] + part; q < ptr[k + 1]; q += nparts)
                    if (strong[q] && cf[col[q]] == 1) f(col[q]);
            }
        }
    }
};

struct GemmCands {  // columns of row i of A B
    const int64_t *__restrict__ aptr;
    const int32_t *__restrict__ acol;
    const int64_t *__restrict__ bptr;
    const int32_t *__restrict__ bcol;
    __device__ bool single(int64_t) const { return false; }
    template <class F>
    __device__ void visit(int64_t i, int part, int nparts, F f) const {
        // eight lanes per row of B (fewer than 32 entries are usual), several rows at once
        const int w = nparts < 8 ? nparts : 8;
        for (int64_t e = aptr[i] + part / w; e < aptr[i + 1]; e += nparts / w) {
            const int32_t k = acol[e];
            for (int64_t q = bptr[k] + part % w; q < bptr[k + 1]; q += w) f(bcol[q]);
        }
    }
};

// rows[0..*nrows) (or all rows 0..n-1 when rows is null): the sorted set of row i goes to
// scratch[ub_off[i]..], its size to cnt[i]; rows that overflow are listed in over[0..*nover)
template <int NT, int CAP, class C>
__global__ void __launch_bounds__(NT) k_union_rows(int64_t n, const int32_t *__restrict__ rows,
                                                   const unsigned *__restrict__ nrows, C cands,
                                                   const int64_t *__restrict__ ub_off,
                                                   int32_t *__restrict__ scratch, int64_t *__restrict__ cnt,
                                                   int32_t *__restrict__ over, unsigned *__restrict__ nover) {
    extern __shared__ int32_t smem[];  // table, list
    __shared__ int num;
    ColSet<NT, CAP> set{smem, smem + CAP, &num};
    const int64_t total = rows ? (int64_t)*nrows : n;
    for (int64_t q = blockIdx.x; q < total; q += gridDim.x) {
        const int64_t i = rows ? rows[q] : q;
        if (cands.single(i)) {
            if (threadIdx.x == 0) cnt[i] = 1;
            continue;
        }
        __syncthreads();
        set.clear();
        cands.visit(i, threadIdx.x, NT, [&](int32_t v) { set.insert(v); });
        const int m = set.sorted(scratch + ub_off[i]);
        if (threadIdx.x == 0) {
            cnt[i] = m;
            if (m < 0) over[atomicAdd(nover, 1u)] = (int32_t)i;
        }
    }
}

__device__ void heap_sort_i32(int32_t *a, int64_t m) {
    auto sift = [&](int64_t root, int64_t end) {
        while (2 * root + 1 < end) {
            int64_t c = 2 * root + 1;
            if (c + 1 < end && a[c + 1] > a[c]) ++c;
            if (a[root] >= a[c]) return;
            int32_t t = a[root];
            a[root] = a[c];
            a[c] = t;
            root = c;
        }
    };
    for (int64_t s = m / 2 - 1; s >= 0; --s) sift(s, m);
    for (int64_t end = m - 1; end > 0; --end) {
        int32_t t = a[0];
        a[0] = a[end];
        a[end] = t;
        sift(0, end);
    }
}

// the rows that no table holds (thousands of distinct columns): one thread per row
template <class C>
__global__ void k_union_heap(const int32_t *__restrict__ rows, const unsigned *__restrict__ nrows, C cands,
                             const int64_t *__restrict__ ub_off, int32_t *__restrict__ scratch,
                             int64_t *__restrict__ cnt) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < (int64_t)*nrows;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = rows[q];
        int32_t *h = scratch + ub_off[i];
        int64_t m = 0;
        cands.visit(i, 0, 1, [&](int32_t v) { h[m++] = v; });
        heap_sort_i32(h, m);
        int64_t u = 0;
        for (int64_t x = 0; x < m; ++x)
            if (x == 0 || h[x] != h[x - 1]) h[u++] = h[x];
        cnt[i] = u;
    }
}

__device__ __forceinline__ double abar(double akl, double akk) {
    if (akk > 0.0) return akl < 0.0 ? akl : 0.0;
    if (akk < 0.0) return akl > 0.0 ? akl : 0.0;
    return akl;
}

__device__ __forceinline__ int64_t find_sorted(const int32_t *h, int64_t m, int32_t v) {
    int64_t lo = 0, hi = m;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (h[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return (lo < m && h[lo] == v) ? lo : -1;
}

// adds the lanes' values v (where has) to acc in lane order, one after another: the sum
// is that of a loop over the entries, which the oracle runs too
__device__ __forceinline__ double ordered_add(double acc, bool has, double v) {
    for (unsigned m = __ballot_sync(0xffffffffu, has); m; m &= m - 1)
        acc = __dadd_rn(acc, __shfl_sync(0xffffffffu, v, __ffs(m) - 1));
    return acc;
}

// One warp per row; the lanes share the entries of the row being read, and every sum runs
// in the order of those entries (ordered_add; a weight w[q] gets its terms in the order
// of the strong F neighbours). Thread per row was bound by its chains of dependent
// accesses: 43 of 312 ms of the setup at P3 24^3, against 0.7 ms here.
__global__ void k_extpi_fill(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                             const double *__restrict__ val, const uint8_t *__restrict__ strong,
                             const int8_t *__restrict__ cf, const int64_t *__restrict__ cidx,
                             const int64_t *__restrict__ ub_off, const int32_t *__restrict__ scratch,
                             const int64_t *__restrict__ pptr, int32_t *__restrict__ pcol, double *pval) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n) return;  // a whole warp, as every branch below
    const int64_t o = pptr[i];
    if (cf[i] == 1) {
        if (lane == 0) {
            pcol[o] = (int32_t)cidx[i];
            pval[o] = 1.0;
        }
        return;
    }
    const int64_t m = pptr[i + 1] - o;
    if (m == 0) return;
    const int32_t *h = scratch + ub_off[i];
    double *w = pval + o;
    for (int64_t q = lane; q < m; q += 32) {
        w[q] = 0.0;
        pcol[o + q] = (int32_t)cidx[h[q]];
    }
    __syncwarp();
    const int64_t lo = ptr[i], hi = ptr[i + 1];
    const int64_t di = lower_bound_col(col, lo, hi, (int32_t)i);
    double diag = di < hi && col[di] == (int32_t)i ? val[di] : 0.0;
    for (int64_t e0 = lo; e0 < hi; e0 += 32) {
        const int64_t e = e0 + lane;
        const bool off = e < hi && col[e] != i;
        const double v = off ? val[e] : 0.0;
        const int64_t q = off ? find_sorted(h, m, col[e]) : -1;
        if (q >= 0) w[q] = v;
        diag = ordered_add(diag, off && q < 0 && !strong[e], v);
    }
    __syncwarp();
    for (int64_t e = lo; e < hi; ++e) {
        if (!strong[e]) continue;
        const int32_t k = col[e];
        if (cf[k] != -1) continue;
        const double aik = val[e];
        const int64_t klo = ptr[k], khi = ptr[k + 1];
        const int64_t dk = lower_bound_col(col, klo, khi, k);
        const double akk = dk < khi && col[dk] == k ? val[dk] : 0.0;
        double d = 0.0;
        for (int64_t f0 = klo; f0 < khi; f0 += 32) {
            const int64_t f = f0 + lane;
            const int32_t l = f < khi ? col[f] : k;
            const bool in = l != k && (l == i || find_sorted(h, m, l) >= 0);
            d = ordered_add(d, in, in ? abar(val[f], akk) : 0.0);
        }
        if (d == 0.0) {
            diag = __dadd_rn(diag, aik);
            continue;
        }
        for (int64_t f0 = klo; f0 < khi; f0 += 32) {
            const int64_t f = f0 + lane;
            const int32_t l = f < khi ? col[f] : k;
            const int64_t q = l != k && l != i ? find_sorted(h, m, l) : -1;
            const bool in = l != k && (l == i || q >= 0);
            const double t = in ? __ddiv_rn(__dmul_rn(aik, abar(val[f], akk)), d) : 0.0;
            if (q >= 0) w[q] = __dadd_rn(w[q], t);
            diag = ordered_add(diag, in && l == i, t);
        }
        __syncwarp();  // w is read by other lanes for the next neighbour
    }
    for (int64_t q = lane; q < m; q += 32) w[q] = __ddiv_rn(-w[q], diag);
}

// ---------------------------------------------------------------------------------
// Transpose (R = P^T): count, scan, scatter, then sort every row of R by column.
// ---------------------------------------------------------------------------------
__global__ void k_count_cols(int64_t nnz, const int32_t *__restrict__ col, unsigned long long *__restrict__ cnt) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < nnz) atomicAdd(&cnt[col[e]], 1ull);
}

__global__ void k_transpose_scatter(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                                    const double *__restrict__ val, unsigned long long *__restrict__ fill,
                                    int32_t *__restrict__ tcol, double *__restrict__ tval) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e) {
        unsigned long long q = atomicAdd(&fill[col[e]], 1ull);
        tcol[q] = (int32_t)i;
        tval[q] = val[e];
    }
}

// one warp per row: an entry's place is the number of smaller columns in its row (the
// columns of a row are distinct)
__global__ void k_sort_rows(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ icol,
                            const double *__restrict__ ival, int32_t *__restrict__ col, double *__restrict__ val) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    const int64_t lo = ptr[i], hi = ptr[i + 1];
    for (int64_t x = lo + lane; x < hi; x += 32) {
        const int32_t c = icol[x];
        int64_t at = lo;
        for (int64_t y = lo; y < hi; ++y) at += icol[y] < c;
        col[at] = c;
        val[at] = ival[x];
    }
}

// ---------------------------------------------------------------------------------
// SpGEMM C = A B: the sorted columns of every row (union_rows), then one warp per row
// adds the products in the order of A's row and then B's row (the lanes take the entries
// of one row of B, which are distinct columns): a fixed order per entry.
// ---------------------------------------------------------------------------------
__global__ void k_gemm_ub(int64_t n, const int64_t *__restrict__ aptr, const int32_t *__restrict__ acol,
                          const int64_t *__restrict__ bptr, int64_t *__restrict__ ub) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t s = 0;
    for (int64_t e = aptr[i]; e < aptr[i + 1]; ++e) s += bptr[acol[e] + 1] - bptr[acol[e]];
    ub[i] = s;
}

__global__ void k_gemm_numeric(int64_t n, const int64_t *__restrict__ aptr, const int32_t *__restrict__ acol,
                               const double *__restrict__ aval, const int64_t *__restrict__ bptr,
                               const int32_t *__restrict__ bcol, const double *__restrict__ bval,
                               const int64_t *__restrict__ ub_off, const int32_t *__restrict__ scratch,
                               const int64_t *__restrict__ cptr, int32_t *__restrict__ ccol, double *cval) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    const int64_t lo = cptr[i], m = cptr[i + 1] - lo;
    const int32_t *h = scratch + ub_off[i];
    for (int64_t q = lane; q < m; q += 32) {
        ccol[lo + q] = h[q];
        cval[lo + q] = 0.0;
    }
    __syncwarp();
    for (int64_t e = aptr[i]; e < aptr[i + 1]; ++e) {
        const int32_t k = acol[e];
        const double a = aval[e];
        for (int64_t f = bptr[k] + lane; f < bptr[k + 1]; f += 32) {
            const int64_t q = find_sorted(h, m, bcol[f]);
            if (q >= 0) cval[lo + q] = __dadd_rn(cval[lo + q], __dmul_rn(a, bval[f]));
        }
        __syncwarp();  // the next row of B may reach the same entries from other lanes
    }
}

// ---------------------------------------------------------------------------------
// Coarsest level: explicit inverse of a dense SPD matrix by in-place block Gauss-Jordan
// elimination, kGj rows at a time and without pivoting (every pivot of a positive definite
// matrix is the square of a Cholesky pivot; one that is not positive reports the matrix).
// For the pivot block K:  D = A_KK^{-1},  R = D A_K*,  A_i* -= A_iK R  for i outside K
// (columns K start from 0 there), A_K* = R with D in its columns K. The n^3 FMAs need many
// SMs (2 FP64 FMAs per clock per SM): one block's Cholesky factor and triangular solves
// took 0.61 ms for 73 rows and grew with their cube; three small launches per pivot block
// take 0.29 ms with the allocations around them (0.23 ms for 62 rows).
// ---------------------------------------------------------------------------------
constexpr int kGj = 32;

__global__ void k_csr_to_dense(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                               const double *__restrict__ val, double *__restrict__ D) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int64_t e = ptr[i]; e < ptr[i + 1]; ++e) D[i * n + col[e]] = val[e];
}

// D = inverse of the pivot block at k0 (32 x 32 threads; rows past n are the identity)
__global__ void __launch_bounds__(kGj *kGj) k_gj_pivot(int64_t n, int64_t k0, const double *__restrict__ A,
                                                       double *__restrict__ D, int *__restrict__ bad) {
    __shared__ double a[kGj][kGj + 1];
    const int i = threadIdx.y, j = threadIdx.x;
    const bool in = k0 + i < n && k0 + j < n;
    a[i][j] = in ? A[(k0 + i) * n + k0 + j] : (i == j ? 1.0 : 0.0);
    __syncthreads();
    for (int p = 0; p < kGj; ++p) {
        const double aip = a[i][p];
        __syncthreads();
        if (i == p) {  // one warp: the pivot row
            double piv = aip;
            if (!(piv > 0.0)) {
                if (j == 0) atomicExch(bad, 1);
                piv = 1.0;
            }
            const double inv = 1.0 / piv;
            a[p][j] = j == p ? inv : a[p][j] * inv;
        }
        __syncthreads();
        if (i != p) a[i][j] = (j == p ? 0.0 : a[i][j]) - aip * a[p][j];
        __syncthreads();
    }
    D[i * kGj + j] = a[i][j];
}

// R = D A_K* (its columns K hold D) and C = A_*K, one thread per column (row)
__global__ void k_gj_panels(int64_t n, int64_t k0, const double *__restrict__ A, const double *__restrict__ D,
                            double *__restrict__ R, double *__restrict__ C) {
    __shared__ double d[kGj * kGj];
    for (int q = threadIdx.x; q < kGj * kGj; q += blockDim.x) d[q] = D[q];
    __syncthreads();
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double v[kGj];
#pragma unroll
    for (int q = 0; q < kGj; ++q) v[q] = k0 + q < n ? A[(k0 + q) * n + j] : 0.0;
    const int64_t own = j - k0;
    for (int q = 0; q < kGj; ++q) {
        double t = 0.0;
#pragma unroll
        for (int u = 0; u < kGj; ++u) t += d[q * kGj + u] * v[u];
        R[(int64_t)q * n + j] = own >= 0 && own < kGj ? d[q * kGj + own] : t;
    }
    for (int q = 0; q < kGj; ++q) C[j * kGj + q] = k0 + q < n ? A[j * n + k0 + q] : 0.0;
}

__global__ void k_gj_update(int64_t n, int64_t k0, const double *__restrict__ R, const double *__restrict__ C,
                            double *__restrict__ A) {
    __shared__ double r[kGj][kGj], c[kGj][kGj + 1];
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    const int64_t j = (int64_t)blockIdx.x * kGj + tx, i0 = (int64_t)blockIdx.y * kGj;
    for (int q = ty; q < kGj; q += 8) {
        r[q][tx] = j < n ? R[(int64_t)q * n + j] : 0.0;
        c[q][tx] = i0 + q < n ? C[(i0 + q) * kGj + tx] : 0.0;
    }
    __syncthreads();
    if (j >= n) return;
    const bool jk = j >= k0 && j < k0 + kGj;
    for (int q = ty; q < kGj; q += 8) {
        const int64_t i = i0 + q;
        if (i >= n) break;
        if (i >= k0 && i < k0 + kGj) {
            A[i * n + j] = r[i - k0][tx];
            continue;
        }
        double t = jk ? 0.0 : A[i * n + j];
#pragma unroll
        for (int u = 0; u < kGj; ++u) t -= c[q][u] * r[u][tx];
        A[i * n + j] = t;
    }
}

// ---------------------------------------------------------------------------------
// host drivers
// ---------------------------------------------------------------------------------
}  // namespace

namespace {

// the sorted candidate columns of every row: a block of one warp and a 1024-slot table per
// row (28 blocks of 8 KB per SM), then 256 threads and 16384 slots for the rows that
// overflow it, then the heap sort
template <class C>
void union_rows(int64_t n, const C &cands, const int64_t *ub_off, int32_t *scratch, int64_t *cnt, DevPool &tmp,
                cudaStream_t s) {
    if (n <= 0) return;
    int32_t *over = tmp.get<int32_t>(2 * n);
    unsigned *nover = tmp.get<unsigned>(2);
    PK_CUDA(cudaMemsetAsync(nover, 0, sizeof(unsigned) * 2, s));
    constexpr int cap1 = 1024, cap2 = 16384;
    k_union_rows<32, cap1, C><<<(unsigned)std::min<int64_t>(n, 152 * 28), 32, 2 * cap1 * sizeof(int32_t), s>>>(
        n, nullptr, nullptr, cands, ub_off, scratch, cnt, over, nover);
    PK_LAUNCH();
    unsigned left[2];
    PK_CUDA(cudaMemcpyAsync(left, nover, sizeof(left), cudaMemcpyDeviceToHost, s));
    PK_CUDA(cudaStreamSynchronize(s));
    if (left[0] == 0) return;
    auto big = k_union_rows<256, cap2, C>;
    const size_t sm2 = 2 * cap2 * sizeof(int32_t);
    PK_CUDA(cudaFuncSetAttribute(big, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm2));
    big<<<(unsigned)std::min<unsigned>(left[0], 152), 256, sm2, s>>>(n, over, nover, cands, ub_off, scratch, cnt,
                                                                    over + n, nover + 1);
    PK_LAUNCH();
    k_union_heap<C><<<152, 128, 0, s>>>(over + n, nover + 1, cands, ub_off, scratch, cnt);
    PK_LAUNCH();
}

}  // namespace

double *row_l1(DevPool &pool, const DCSR &A, cudaStream_t s) {
    double *l1 = pool.get<double>(A.n > 0 ? A.n : 1);
    if (A.n > 0) {
        k_l1norm<<<blocks_for(A.n, 256), 256, 0, s>>>(A.n, A.ptr, A.val, l1);
        PK_LAUNCH();
    }
    return l1;
}

// C = A B on the device (A: n x k, B: k x m)
void spgemm(DevPool &pool, const DCSR &A, const DCSR &B, DCSR &C, cudaStream_t s) {
    const int64_t n = A.n;
    DevPool tmp;
    try {
        int64_t *ub = tmp.get<int64_t>(n + 1);
        if (n > 0) {
            k_gemm_ub<<<blocks_for(n, 256), 256, 0, s>>>(n, A.ptr, A.col, B.ptr, ub);
            PK_LAUNCH();
        }
        exclusive_scan(ub, n, s);
        int64_t tot = read_i64(ub + n, s);
        if (tot > ((int64_t)1 << 31)) fail(PKASP_ENOMEM, "Galerkin product scratch above 2^31 entries");
        int32_t *scr = tmp.get<int32_t>(tot > 0 ? tot : 1);
        int64_t *cnt = tmp.get<int64_t>(n + 1);
        union_rows(n, GemmCands{A.ptr, A.col, B.ptr, B.col}, ub, scr, cnt, tmp, s);
        exclusive_scan(cnt, n, s);
        int64_t nnz = read_i64(cnt + n, s);
        dcsr_alloc(pool, C, n, B.m, nnz);
        PK_CUDA(cudaMemcpyAsync(C.ptr, cnt, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToDevice, s));
        if (n > 0) {
            k_gemm_numeric<<<blocks_for(n * 32, 128), 128, 0, s>>>(n, A.ptr, A.col, A.val, B.ptr, B.col, B.val, ub, scr,
                                                             C.ptr, C.col, C.val);
            PK_LAUNCH();
        }
        PK_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
        cudaStreamSynchronize(s);
        tmp.free_all();
        throw;
    }
    tmp.free_all();
}

void transpose(DevPool &pool, const DCSR &A, DCSR &T, cudaStream_t s) {
    DevPool tmp;
    try {
        const int64_t m = A.m;
        unsigned long long *cnt = tmp.get<unsigned long long>(m + 1);
        PK_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * (m + 1), s));
        if (A.nnz > 0) {
            k_count_cols<<<blocks_for(A.nnz, 256), 256, 0, s>>>(A.nnz, A.col, cnt);
            PK_LAUNCH();
        }
        static_assert(sizeof(unsigned long long) == sizeof(int64_t), "scan type");
        exclusive_scan(reinterpret_cast<int64_t *>(cnt), m, s);
        dcsr_alloc(pool, T, m, A.n, A.nnz);
        int32_t *ucol = tmp.get<int32_t>(A.nnz > 0 ? A.nnz : 1);  // entries in the order of arrival
        double *uval = tmp.get<double>(A.nnz > 0 ? A.nnz : 1);
        PK_CUDA(cudaMemcpyAsync(T.ptr, cnt, sizeof(int64_t) * (m + 1), cudaMemcpyDeviceToDevice, s));
        if (A.n > 0) {
            k_transpose_scatter<<<blocks_for(A.n, 256), 256, 0, s>>>(A.n, A.ptr, A.col, A.val, cnt, ucol, uval);
            PK_LAUNCH();
        }
        if (m > 0) {
            k_sort_rows<<<blocks_for(m * 32, 128), 128, 0, s>>>(m, T.ptr, ucol, uval, T.col, T.val);
            PK_LAUNCH();
        }
        PK_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
        cudaStreamSynchronize(s);
        tmp.free_all();
        throw;
    }
    tmp.free_all();
}

// PMIS on a structurally symmetric pattern with given strength flags.
void pmis_run(int64_t n, const int64_t *ptr, const int32_t *col, const uint8_t *strong, uint64_t stream,
              int8_t *cf, cudaStream_t s) {
    DevPool tmp;
    try {
        int64_t nnz = read_i64(ptr + n, s);
        int64_t *mirror = tmp.get<int64_t>(nnz > 0 ? nnz : 1);
        int64_t *mu = tmp.get<int64_t>(n > 0 ? n : 1);
        uint8_t *newc = tmp.get<uint8_t>(n > 0 ? n : 1);
        int *bad = tmp.get<int>(1);
        unsigned long long *und = tmp.get<unsigned long long>(1);
        PK_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), s));
        PK_CUDA(cudaMemsetAsync(und, 0, sizeof(unsigned long long), s));
        if (n > 0) {
            k_mirror<<<blocks_for(n, 256), 256, 0, s>>>(n, ptr, col, mirror, bad);
            PK_LAUNCH();
            k_pmis_init<<<blocks_for(n, 256), 256, 0, s>>>(n, ptr, mirror, strong, mu, cf, und);
            PK_LAUNCH();
        }
        int hb = 0;
        unsigned long long left = 0;
        PK_CUDA(cudaMemcpyAsync(&hb, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
        PK_CUDA(cudaMemcpyAsync(&left, und, sizeof(left), cudaMemcpyDeviceToHost, s));
        PK_CUDA(cudaStreamSynchronize(s));
        if (hb == 2) fail(PKASP_EINVAL, "PMIS: a column index lies outside [0, n)");
        if (hb) fail(PKASP_EINVAL, "PMIS needs a structurally symmetric pattern with ascending columns in every row");
        int rounds = 0;
        while (left > 0) {
            PK_CUDA(cudaMemsetAsync(und, 0, sizeof(unsigned long long), s));
            k_pmis_select<<<blocks_for(n, 256), 256, 0, s>>>(n, ptr, col, mirror, strong, mu, stream, cf, newc);
            PK_LAUNCH();
            k_pmis_commit<<<blocks_for(n, 256), 256, 0, s>>>(n, newc, cf);
            PK_LAUNCH();
            k_pmis_mark_f<<<blocks_for(n, 256), 256, 0, s>>>(n, ptr, col, strong, newc, cf, und);
            PK_LAUNCH();
            PK_CUDA(cudaMemcpyAsync(&left, und, sizeof(left), cudaMemcpyDeviceToHost, s));
            PK_CUDA(cudaStreamSynchronize(s));
            if (++rounds > n + 8) fail(PKASP_ECUDA, "PMIS did not terminate");
        }
    } catch (...) {
        cudaStreamSynchronize(s);
        tmp.free_all();
        throw;
    }
    tmp.free_all();
}

void pmis_device(int64_t n, const int64_t *ptr, const int32_t *col, const uint8_t *strong, uint64_t stream_id,
                 int8_t *cf, cudaStream_t s) {
    pmis_run(n, ptr, col, strong, stream_id, cf, s);
}

// One coarsening step on level L: strength, PMIS, ext+i P, R = P^T, A_c = R (A P).
// Returns false when PMIS keeps no point or every point (the level becomes the coarsest).
// ---------------------------------------------------------------------------------
// Interpolation truncation (optional): in every row drop |w| < tf * max|w|, keep the
// pmax largest |w| of the rest (ties: the lower column), scale the kept weights to the
// row's original sum. One thread per row; kept entries stay in column order.
// ---------------------------------------------------------------------------------
__device__ __forceinline__ bool trunc_keep(const int32_t *col, const double *val, int64_t lo, int64_t hi,
                                           int64_t e, double cut, int pmax) {
    const double a = fabs(val[e]);
    if (a < cut) return false;
    if (pmax <= 0) return true;
    int rank = 0;  // candidates ahead of e: larger |w|, or equal |w| and a lower column
    for (int64_t f = lo; f < hi; ++f) {
        const double b = fabs(val[f]);
        if (b < cut || f == e) continue;
        if (b > a || (b == a && col[f] < col[e])) ++rank;
    }
    return rank < pmax;
}

__global__ void k_trunc_count(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                              const double *__restrict__ val, double tf, int pmax, int64_t *__restrict__ cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t lo = ptr[i], hi = ptr[i + 1];
    double mx = 0.0;
    for (int64_t e = lo; e < hi; ++e) mx = fmax(mx, fabs(val[e]));
    const double cut = tf > 0.0 ? tf * mx : -1.0;
    int64_t c = 0;
    for (int64_t e = lo; e < hi; ++e) c += trunc_keep(col, val, lo, hi, e, cut, pmax);
    cnt[i] = c;
}

__global__ void k_trunc_fill(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                             const double *__restrict__ val, double tf, int pmax, const int64_t *__restrict__ optr,
                             int32_t *__restrict__ ocol, double *__restrict__ oval) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t lo = ptr[i], hi = ptr[i + 1];
    double mx = 0.0, sum = 0.0;
    for (int64_t e = lo; e < hi; ++e) {
        mx = fmax(mx, fabs(val[e]));
        sum += val[e];
    }
    const double cut = tf > 0.0 ? tf * mx : -1.0;
    int64_t o = optr[i];
    double kept = 0.0;
    for (int64_t e = lo; e < hi; ++e)
        if (trunc_keep(col, val, lo, hi, e, cut, pmax)) {
            ocol[o] = col[e];
            oval[o] = val[e];
            kept += val[e];
            ++o;
        }
    if (o - optr[i] < hi - lo && kept != 0.0) {
        const double scale = sum / kept;
        for (int64_t q = optr[i]; q < o; ++q) oval[q] *= scale;
    }
}

bool coarsen(DevPool &pool, Level &L, double theta, uint64_t pmis_stream, DCSR &Ac, cudaStream_t s,
             double trunc_factor, int pmax, int cc) {
    const DCSR &A = L.A;
    const int64_t n = A.n;
    L.strong = pool.get<uint8_t>(A.nnz > 0 ? A.nnz : 1);
    L.cf = pool.get<int8_t>(n > 0 ? n : 1);
    k_strength<<<blocks_for(n, 256), 256, 0, s>>>(n, A.ptr, A.col, A.val, theta, L.strong);
    PK_LAUNCH();
    pmis_run(n, A.ptr, A.col, L.strong, pmis_stream, L.cf, s);
    DevPool tmp;
    bool ok = true;
    try {
        int64_t *cidx = tmp.get<int64_t>(n + 1);
        k_flag_c<<<blocks_for(n, 256), 256, 0, s>>>(n, L.cf, cidx);
        PK_LAUNCH();
        exclusive_scan(cidx, n, s);
        const int64_t nc = read_i64(cidx + n, s);
        if (nc == 0 || nc == n) {
            ok = false;
        } else {
            int64_t *ub = tmp.get<int64_t>(n + 1);
            k_extpi_ub<<<blocks_for(n, 256), 256, 0, s>>>(n, A.ptr, A.col, L.strong, L.cf, ub);
            PK_LAUNCH();
            exclusive_scan(ub, n, s);
            int64_t tot = read_i64(ub + n, s);
            if (tot > ((int64_t)1 << 31)) fail(PKASP_ENOMEM, "interpolation scratch above 2^31 entries");
            int32_t *scr = tmp.get<int32_t>(tot > 0 ? tot : 1);
            int64_t *cnt = tmp.get<int64_t>(n + 1);
            union_rows(n, HatCands{A.ptr, A.col, L.strong, L.cf, cc}, ub, scr, cnt, tmp, s);
            exclusive_scan(cnt, n, s);
            int64_t pnnz = read_i64(cnt + n, s);
            const bool trunc = trunc_factor > 0.0 || pmax > 0;
            DCSR full;  // ext+i before truncation (scratch when truncating)
            dcsr_alloc(trunc ? tmp : pool, full, n, nc, pnnz);
            PK_CUDA(cudaMemcpyAsync(full.ptr, cnt, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToDevice, s));
            k_extpi_fill<<<blocks_for(n * 32, 128), 128, 0, s>>>(n, A.ptr, A.col, A.val, L.strong, L.cf, cidx, ub, scr,
                                                            full.ptr, full.col, full.val);
            PK_LAUNCH();
            if (trunc) {
                int64_t *tc = tmp.get<int64_t>(n + 1);
                k_trunc_count<<<blocks_for(n, 256), 256, 0, s>>>(n, full.ptr, full.col, full.val, trunc_factor, pmax,
                                                                 tc);
                PK_LAUNCH();
                exclusive_scan(tc, n, s);
                const int64_t tnnz = read_i64(tc + n, s);
                dcsr_alloc(pool, L.P, n, nc, tnnz);
                PK_CUDA(cudaMemcpyAsync(L.P.ptr, tc, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToDevice, s));
                k_trunc_fill<<<blocks_for(n, 256), 256, 0, s>>>(n, full.ptr, full.col, full.val, trunc_factor, pmax,
                                                                L.P.ptr, L.P.col, L.P.val);
                PK_LAUNCH();
            } else {
                L.P = full;
            }
            PK_CUDA(cudaStreamSynchronize(s));
            transpose(pool, L.P, L.R, s);
            DCSR AP;
            DevPool aptmp;
            try {
                spgemm(aptmp, A, L.P, AP, s);
                spgemm(pool, L.R, AP, Ac, s);
            } catch (...) {
                cudaStreamSynchronize(s);
                aptmp.free_all();
                throw;
            }
            aptmp.free_all();
        }
        PK_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
        cudaStreamSynchronize(s);
        tmp.free_all();
        throw;
    }
    tmp.free_all();
    return ok;
}

// Dense inverse of the coarsest matrix (block Gauss-Jordan, above).
void coarse_inverse(DevPool &pool, const DCSR &A, double **inv, cudaStream_t s) {
    const int64_t n = A.n;
    if (n > 8192) fail(PKASP_ENOMEM, "coarsest level has more than 8192 rows; raise max_levels or coarse_size");
    DevPool tmp;
    try {
        double *A0 = pool.get<double>(n * n > 0 ? n * n : 1);
        double *D = tmp.get<double>(kGj * kGj), *R = tmp.get<double>(kGj * std::max<int64_t>(n, 1)),
               *C = tmp.get<double>(kGj * std::max<int64_t>(n, 1));
        int *bad = tmp.get<int>(1);
        *inv = A0;
        PK_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), s));
        PK_CUDA(cudaMemsetAsync(A0, 0, sizeof(double) * n * n, s));
        if (n > 0) {
            k_csr_to_dense<<<blocks_for(n, 128), 128, 0, s>>>(n, A.ptr, A.col, A.val, A0);
            PK_LAUNCH();
        }
        const unsigned tiles = blocks_for(n, kGj);
        for (int64_t k0 = 0; k0 < n; k0 += kGj) {
            k_gj_pivot<<<1, dim3(kGj, kGj), 0, s>>>(n, k0, A0, D, bad);
            PK_LAUNCH();
            k_gj_panels<<<blocks_for(n, 64), 64, 0, s>>>(n, k0, A0, D, R, C);
            PK_LAUNCH();
            k_gj_update<<<dim3(tiles, tiles), dim3(kGj, 8), 0, s>>>(n, k0, R, C, A0);
            PK_LAUNCH();
        }
        int hb = 0;
        PK_CUDA(cudaMemcpyAsync(&hb, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
        PK_CUDA(cudaStreamSynchronize(s));
        if (hb) fail(PKASP_EBREAKDOWN, "coarsest AMG matrix is not positive definite");
    } catch (...) {
        cudaStreamSynchronize(s);
        tmp.free_all();
        throw;
    }
    tmp.free_all();
}

}  // namespace pk
