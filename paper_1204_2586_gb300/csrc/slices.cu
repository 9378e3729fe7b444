// slices.cu -- interleaved slices: the layout in which the fine smoother's colour phases
// read A_h (kernels.cuh, k_slice_phase). A slice is the work of one warp: 32 / T rows of
// one colour with T lanes each, W steps; step k of lane l is entry base + 32 k + l, so the
// 32 columns of a step are one 128-byte line and its FP64 values two. Lane (row r, sub)
// takes the row's entries sub, sub + T, ... in that order; shorter rows are padded with
// column -1.
//
// T is T0 for rows of up to `steps` T0 entries and doubles with the length beyond (32 at
// most), so no row takes a long chain of steps on few lanes (slice_shape in solve.cu picks
// both). Within a colour the rows are ordered by T and W, largest first, in row order
// within equal T and W: the padding is then 7% at P4 and 9% at P3 with 4 lanes and 16 steps
// (host count; 23% and 29% in row order), and the longest slices start first.
#include <algorithm>

#include "internal.h"

namespace pk {
namespace {

// (T, W) classes of a colour: T = 32, 16 .. 1 by W, empty
int keys_of(int steps) { return 2 + 5 * steps; }

unsigned blocks_for(int64_t n, int per) {
    int64_t b = (n + per - 1) / per;
    return (unsigned)std::max<int64_t>(1, b);
}

// Lanes of a row part of len entries.
__host__ __device__ inline int lanes_of(int64_t len, int t0, int steps) {
    int t = t0;
    while (t < 32 && len > (int64_t)steps * t) t <<= 1;
    return t;
}

// Class of a row part: 0 for 32 lanes, then 16 lanes with steps, steps - 1, ... steps, then
// 8 lanes, ...; the last class holds the empty parts.
__host__ __device__ inline int class_of(int64_t len, int t0, int steps) {
    if (len == 0) return 1 + 5 * steps;
    const int t = lanes_of(len, t0, steps);
    if (t == 32) return 0;
    const int w = (int)((len + t - 1) / t);
    int rank = 0;
    for (int u = 16; u > t; u >>= 1) ++rank;
    return 1 + rank * steps + (steps - w);
}

// The parts that a layout is built from: the lower or upper parts of a colour split, whole
// rows without their diagonal (full: rows perm[p] of a matrix), or the rows themselves (perm
// is null).
struct Parts {
    const int64_t *ptr;
    const int32_t *col;
    const double *val;
    const int32_t *perm;
    bool full;
    __device__ int64_t lo(int64_t p) const { return ptr[full ? (int64_t)perm[p] : p]; }
    __device__ int64_t hi(int64_t p) const { return ptr[(full ? (int64_t)perm[p] : p) + 1]; }
    __device__ int64_t len(int64_t p) const { return hi(p) - lo(p) - (full ? 1 : 0); }
    __device__ int32_t row(int64_t p) const { return perm ? perm[p] : (int32_t)p; }
};

__global__ void k_slice_keys(int64_t n, Parts A, int t0, int steps, const int32_t *__restrict__ colour,
                             int32_t *__restrict__ key, int *__restrict__ maxlen) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int len = 0;
    if (p < n) {
        len = (int)A.len(p);
        key[p] = (colour ? colour[A.row(p)] * (2 + 5 * steps) : 0) + class_of(len, t0, steps);
    }
    len = __reduce_max_sync(0xffffffffu, len);
    if ((threadIdx.x & 31) == 0 && len > 0) atomicMax(maxlen, len);
}

struct Group {  // the slices of one class of one colour
    int64_t s0, p0, count;  // first slice, first ordered position, rows
    int32_t lt, pad;        // log2 of the lanes per row
};

__device__ __forceinline__ int group_of(const Group *__restrict__ g, int ng, int64_t s) {
    int lo = 0, hi = ng - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (g[mid].s0 <= s) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// steps of every slice (width[s], in entries: 32 W) and its meta without the base
__global__ void k_slice_meta(int64_t ns, const Group *__restrict__ g, int ng, Parts A,
                             const int32_t *__restrict__ order, int64_t *__restrict__ width,
                             int4 *__restrict__ meta) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const Group gr = g[group_of(g, ng, s)];
    const int t = 1 << gr.lt, rows = 32 / t;
    const int64_t first = gr.p0 + (s - gr.s0) * rows;
    const int nr = (int)min((int64_t)rows, gr.p0 + gr.count - first);
    int64_t w = 0;
    for (int r = 0; r < nr; ++r) w = max(w, (A.len(order[first + r]) + t - 1) / t);
    width[s] = 32 * w;
    meta[s] = make_int4(0, 0, (int)first, (int)w | (gr.lt << 20) | (nr << 24));
}

__global__ void k_slice_base(int64_t ns, const int64_t *__restrict__ base, int4 *__restrict__ meta) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const int64_t b = base[s];
    meta[s].x = (int)(uint32_t)(b & 0xffffffffll);
    meta[s].y = (int)(b >> 32);
}

// one warp per slice
template <typename PT>
__global__ void k_slice_fill(int64_t ns, const int4 *__restrict__ meta, Parts A, const int32_t *__restrict__ order,
                             const double *__restrict__ dinv, int32_t *__restrict__ scol, PT *__restrict__ sval,
                             int32_t *__restrict__ rows, PT *__restrict__ sdinv) {
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (s >= ns) return;
    const int4 m = meta[s];
    const int64_t base = ((int64_t)m.y << 32) | (uint32_t)m.x;
    const int w = m.w & 0xfffff, lt = (m.w >> 20) & 15, nr = (m.w >> 24) & 255, t = 1 << lt;
    const int sub = lane & (t - 1), r = lane >> lt;
    const bool ok = r < nr;
    const int64_t p = ok ? order[m.z + r] : 0;
    const int32_t i = ok ? A.row(p) : -1;
    const int64_t lo = ok ? A.lo(p) : 0, len = ok ? A.len(p) : 0;
    // whole rows skip their diagonal: entries from there on move down by one
    int64_t skip = len;
    if (A.full && ok) {
        int64_t a = 0, b = len + 1;
        while (a < b) {
            const int64_t mid = (a + b) >> 1;
            if (A.col[lo + mid] < i) a = mid + 1;
            else b = mid;
        }
        skip = a;
    }
    for (int k = 0; k < w; ++k) {
        const int64_t q = (int64_t)k * t + sub;
        const bool real = q < len;
        const int64_t e = lo + q + (q >= skip && A.full ? 1 : 0);
        scol[base + 32 * (int64_t)k + lane] = real ? A.col[e] : -1;
        sval[base + 32 * (int64_t)k + lane] = real ? (PT)A.val[e] : PT(0);
    }
    if (ok && sub == 0) {
        rows[m.z + r] = i;
        if (dinv) sdinv[m.z + r] = (PT)dinv[p];
    }
}

}  // namespace

// part: 0 lower, 1 upper, 2 whole rows of A without the diagonal, 3 the rows of A themselves
// (no colours: one list of slices). Rows whose upper part is empty are left out (their phase
// would change nothing).
void build_slices(DevPool &pool, const DCSR &A, const DSplit &sp, int part, int t0, int steps, bool fp32, DSlices &S,
                  cudaStream_t s) {
    S = DSlices{};
    S.t0 = t0;
    S.steps = steps;
    const int64_t n = A.n;
    const bool plain = part == 3;
    const int ncol = plain ? 1 : sp.ncol, keys = keys_of(steps);
    const Parts P = plain ? Parts{A.ptr, A.col, A.val, nullptr, false}
                    : part == 2 ? Parts{A.ptr, A.col, A.val, sp.perm, true}
                    : part == 1 ? Parts{sp.uptr, sp.ucol, sp.uval, sp.perm, false}
                                : Parts{sp.lptr, sp.lcol, sp.lval, sp.perm, false};
    S.off.assign(ncol + 1, 0);
    if (n == 0) return;
    DevPool tmp;
    try {
        int32_t *key = tmp.get<int32_t>(n), *order = tmp.get<int32_t>(n);
        int *maxlen = tmp.get<int>(1);
        PK_CUDA(cudaMemsetAsync(maxlen, 0, sizeof(int), s));
        k_slice_keys<<<blocks_for(n, 256), 256, 0, s>>>(n, P, t0, steps, plain ? nullptr : sp.colour, key, maxlen);
        PK_LAUNCH();
        std::vector<int64_t> koff;
        key_sort(n, key, (int64_t)ncol * keys, order, koff, s);
        int longest = 0;
        PK_CUDA(cudaMemcpyAsync(&longest, maxlen, sizeof(int), cudaMemcpyDeviceToHost, s));
        PK_CUDA(cudaStreamSynchronize(s));
        if (longest >= (32 << 20)) fail(PKASP_ENOMEM, "a row of A_h has more than 2^25 entries");
        std::vector<Group> groups;
        int64_t ns = 0;
        for (int c = 0; c < ncol; ++c) {
            for (int q = 0; q < keys; ++q) {
                const int64_t p0 = koff[(int64_t)c * keys + q], m = koff[(int64_t)c * keys + q + 1] - p0;
                if (m == 0 || (part == 1 && q == keys - 1)) continue;
                int lt = 5;  // class 0: 32 lanes; empty parts: one lane
                if (q == keys - 1) lt = 0;
                else if (q > 0) lt = 4 - (q - 1) / steps;
                groups.push_back(Group{ns, p0, m, lt, 0});
                const int rows = 32 >> lt;
                ns += (m + rows - 1) / rows;
            }
            S.off[c + 1] = ns;
        }
        S.nslices = ns;
        S.meta = pool.get<int4>(std::max<int64_t>(ns, 1));
        S.rows = pool.get<int32_t>(n);
        if (!plain && fp32) S.dinv32 = pool.get<float>(n);
        if (!plain && !fp32) S.dinv = pool.get<double>(n);
        Group *dg = tmp.get<Group>(std::max<size_t>(groups.size(), 1));
        int64_t *width = tmp.get<int64_t>(ns + 1);
        if (ns > 0) {
            PK_CUDA(cudaMemcpyAsync(dg, groups.data(), sizeof(Group) * groups.size(), cudaMemcpyHostToDevice, s));
            k_slice_meta<<<blocks_for(ns, 128), 128, 0, s>>>(ns, dg, (int)groups.size(), P, order, width, S.meta);
            PK_LAUNCH();
            exclusive_scan(width, ns, s);
            k_slice_base<<<blocks_for(ns, 256), 256, 0, s>>>(ns, width, S.meta);
            PK_LAUNCH();
            S.entries = read_i64(width + ns, s);
        }
        S.col = pool.get<int32_t>(std::max<int64_t>(S.entries, 1));
        if (fp32) S.val32 = pool.get<float>(std::max<int64_t>(S.entries, 1));
        else S.val = pool.get<double>(std::max<int64_t>(S.entries, 1));
        if (ns > 0) {
            if (fp32)
                k_slice_fill<float><<<blocks_for(ns * 32, 256), 256, 0, s>>>(ns, S.meta, P, order, plain ? nullptr : sp.dinv, S.col,
                                                                            S.val32, S.rows, S.dinv32);
            else
                k_slice_fill<double><<<blocks_for(ns * 32, 256), 256, 0, s>>>(ns, S.meta, P, order, plain ? nullptr : sp.dinv, S.col,
                                                                             S.val, S.rows, S.dinv);
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

}  // namespace pk
