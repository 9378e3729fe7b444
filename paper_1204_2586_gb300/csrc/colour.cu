// colour.cu -- Jones-Plassmann colouring of a matrix graph and the colour split used by
// the multicolour Gauss-Seidel smoothers (the paper's hybrid GS of Sec. 6.1 replaced by a
// GS that parallelises over colours), built on the device. The host reads back only the
// colour count, the colour offsets and four row lengths per colour.
#include <algorithm>

#include "internal.h"
#include "pmis.cuh"

namespace pk {
namespace {

unsigned blocks_for(int64_t n, int per) {
    int64_t b = (n + per - 1) / per;
    return (unsigned)std::max<int64_t>(1, b);
}

// ---------------------------------------------------------------------------------
// Jones-Plassmann colouring, priority (degree, hash, -index), largest first: a row takes
// the smallest colour unused by its neighbours of higher priority, once all of those are
// coloured. The result is the sequential greedy colouring in priority order, whatever the
// schedule. The schedule here does each row's work once: every row counts its uncoloured
// neighbours of higher priority; a row whose count is zero stands in the current round's
// list, takes its colour, and takes one off the count of each uncoloured neighbour, which
// joins the next round's list when its count reaches zero. (Rescanning every uncoloured
// row each round, with each neighbour's degree counted from its row, took 116 ms of a
// 312 ms setup at P3 24^3; now the whole split of A_h, colours included, takes 2.6 ms.)
//
// kJpLanes lanes share a row: rows have 15 (P1) to 75 (P4) entries on average, so eight
// lanes read them in a few coalesced steps and leave enough rows in flight.
// ---------------------------------------------------------------------------------
constexpr int kJpLanes = 8;

// off-diagonal entries of each row (columns ascend, so the diagonal is found by bisection)
__global__ void k_jp_degree(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                            int32_t *__restrict__ deg) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t lo = ptr[i], hi = ptr[i + 1];
    const int64_t d = lower_bound_col(col, lo, hi, (int32_t)i);
    deg[i] = (int32_t)(hi - lo - (d < hi && col[d] == (int32_t)i));
}

__global__ void k_jp_count(int64_t n, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
                           const int32_t *__restrict__ deg, uint64_t stream, int32_t *__restrict__ cnt,
                           int32_t *__restrict__ list, unsigned *__restrict__ ctr) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kJpLanes;
    const int sub = threadIdx.x & (kJpLanes - 1);
    if (i >= n) return;  // a whole lane group
    const unsigned gm = ((1u << kJpLanes) - 1u) << (threadIdx.x & 31 & ~(kJpLanes - 1));
    const int32_t di = deg[i];
    const uint64_t hi = splitmix64(stream, (uint64_t)i);
    int c = 0;
    for (int64_t e = ptr[i] + sub; e < ptr[i + 1]; e += kJpLanes) {
        const int32_t j = col[e];
        if (j == i) continue;
        const int32_t dj = deg[j];
        bool first;  // j before i
        if (dj != di) first = dj > di;
        else {
            const uint64_t hj = splitmix64(stream, (uint64_t)j);
            first = hj != hi ? hj > hi : j < i;
        }
        c += first;
    }
#pragma unroll
    for (int o = kJpLanes / 2; o > 0; o >>= 1) c += __shfl_xor_sync(gm, c, o);
    if (sub == 0) {
        cnt[i] = c;
        if (c == 0) list[atomicAdd(&ctr[0], 1u)] = (int32_t)i;
    }
}

// Round r: the rows of list `in` (ctr[r % 3] of them) take their colours; rows made ready
// go to `out` (counted in ctr[(r + 1) % 3]); the counter of the round after is cleared.
// No two rows of a list are neighbours, and a coloured neighbour of row i always comes
// before i, so the colours read here are final.
__global__ void k_jp_round(const int64_t *__restrict__ ptr, const int32_t *__restrict__ col, int32_t *colour,
                           int32_t *cnt, const int32_t *__restrict__ in, int32_t *__restrict__ out, unsigned *ctr,
                           int r, int *maxcol) {
    const unsigned nf = ctr[r % 3];
    if (blockIdx.x == 0 && threadIdx.x == 0) ctr[(r + 2) % 3] = 0u;
    const unsigned ngrp = gridDim.x * (blockDim.x / kJpLanes);
    const int sub = threadIdx.x & (kJpLanes - 1);
    const unsigned gm = ((1u << kJpLanes) - 1u) << (threadIdx.x & 31 & ~(kJpLanes - 1));
    int most = 0;
    for (unsigned q = (blockIdx.x * blockDim.x + threadIdx.x) / kJpLanes; q < nf; q += ngrp) {
        const int32_t i = in[q];
        const int64_t lo = ptr[i], hi = ptr[i + 1];
        int base = 0, c = -1;
        while (c < 0) {
            unsigned long long used = 0ull;
            for (int64_t e = lo + sub; e < hi; e += kJpLanes) {
                const int32_t j = col[e];
                if (j == i) continue;
                const int cj = colour[j] - base;
                if (cj >= 0 && cj < 64) used |= 1ull << cj;
            }
#pragma unroll
            for (int o = kJpLanes / 2; o > 0; o >>= 1) used |= __shfl_xor_sync(gm, used, o);
            if (~used != 0ull) c = base + __ffsll((long long)~used) - 1;
            else base += 64;
        }
        for (int64_t e = lo + sub; e < hi; e += kJpLanes) {
            const int32_t j = col[e];
            if (j == i || colour[j] >= 0) continue;
            if (atomicSub(&cnt[j], 1) == 1) out[atomicAdd(&ctr[(r + 1) % 3], 1u)] = j;
        }
        if (sub == 0) colour[i] = c;
        most = max(most, c + 1);
    }
    if (most > 0 && sub == 0) atomicMax(maxcol, most);
}

// The same rounds in one block, with colours, counts and lists in shared memory, one warp per
// row. A coarse level is nearly dense, so its rounds are many (592 rows with 124 entries each:
// hundreds) and hold a row or two: a launch each took 3.2 ms of a 17 ms setup for those rows
// at P3 24^3. Up to kJpSmall rows; with more a block is the smaller part of the chip.
constexpr int kJpSmall = 4096;

__global__ void __launch_bounds__(1024) k_jp_small(int n, const int64_t *__restrict__ ptr,
                                                   const int32_t *__restrict__ col, const int32_t *__restrict__ cnt0,
                                                   const int32_t *__restrict__ list0, const unsigned *__restrict__ nlist,
                                                   int32_t *__restrict__ colour, int *__restrict__ maxcol) {
    extern __shared__ int32_t jp_smem[];
    int32_t *clr = jp_smem, *cnt = clr + n, *in = cnt + n, *out = in + n;
    __shared__ int num[2];
    __shared__ int most;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        num[0] = (int)*nlist;
        num[1] = 0;
        most = 0;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        clr[q] = -1;
        cnt[q] = cnt0[q];
        if (q < num[0]) in[q] = list0[q];
    }
    __syncthreads();
    // every row enters a list once, so the rounds end
    for (int cur = 0; num[cur] > 0; cur ^= 1) {
        const int nf = num[cur];
        for (int q = warp; q < nf; q += 32) {
            const int32_t i = in[q];
            const int64_t lo = ptr[i], hi = ptr[i + 1];
            int base = 0, c = -1;
            while (c < 0) {
                unsigned long long used = 0ull;
                for (int64_t e = lo + lane; e < hi; e += 32) {
                    const int32_t j = col[e];
                    const int cj = j == i ? -1 : clr[j] - base;
                    if (cj >= 0 && cj < 64) used |= 1ull << cj;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) used |= __shfl_xor_sync(0xffffffffu, used, o);
                if (~used != 0ull) c = base + __ffsll((long long)~used) - 1;
                else base += 64;
            }
            for (int64_t e = lo + lane; e < hi; e += 32) {
                const int32_t j = col[e];
                if (j == i || clr[j] >= 0) continue;
                if (atomicSub(&cnt[j], 1) == 1) out[atomicAdd(&num[cur ^ 1], 1)] = j;
            }
            if (lane == 0) {
                clr[i] = c;
                atomicMax(&most, c + 1);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) num[cur] = 0;
        int32_t *t = in;
        in = out;
        out = t;
        __syncthreads();
    }
    for (int q = threadIdx.x; q < n; q += blockDim.x) colour[q] = clr[q];
    if (threadIdx.x == 0) *maxcol = most;
}

int jp_colour(int64_t n, const int64_t *ptr, const int32_t *col, uint64_t stream, int32_t *colour, DevPool &tmp,
              cudaStream_t s) {
    int32_t *deg = tmp.get<int32_t>(n), *cnt = tmp.get<int32_t>(n);
    int32_t *list[2] = {tmp.get<int32_t>(n), tmp.get<int32_t>(n)};
    unsigned *ctr = tmp.get<unsigned>(4);  // three rotating list lengths; then the colour count
    int *maxc = reinterpret_cast<int *>(ctr + 3);
    PK_CUDA(cudaMemsetAsync(colour, 0xff, sizeof(int32_t) * n, s));
    PK_CUDA(cudaMemsetAsync(ctr, 0, sizeof(unsigned) * 4, s));
    k_jp_degree<<<blocks_for(n, 256), 256, 0, s>>>(n, ptr, col, deg);
    PK_LAUNCH();
    k_jp_count<<<blocks_for(n * kJpLanes, 256), 256, 0, s>>>(n, ptr, col, deg, stream, cnt, list[0], ctr);
    PK_LAUNCH();
    if (n <= kJpSmall) {
        const size_t smem = sizeof(int32_t) * 4 * (size_t)n;
        PK_CUDA(cudaFuncSetAttribute(k_jp_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(sizeof(int32_t) * 4 * kJpSmall)));
        k_jp_small<<<1, 1024, smem, s>>>((int)n, ptr, col, cnt, list[0], ctr, colour, maxc);
        PK_LAUNCH();
        int h = 0;
        PK_CUDA(cudaMemcpyAsync(&h, maxc, sizeof(int), cudaMemcpyDeviceToHost, s));
        PK_CUDA(cudaStreamSynchronize(s));
        return h;
    }
    // a round's list is rarely longer than a few percent of the rows; rounds run in
    // batches of 32 between two looks at the list length (an empty round costs a launch)
    const unsigned grid = (unsigned)std::min<int64_t>(152 * 4, blocks_for(n * kJpLanes, 256));
    for (int64_t r = 0;; r += 32) {
        for (int q = 0; q < 32; ++q) {
            const int rr = (int)((r + q) % 6);  // lists alternate, counters rotate
            k_jp_round<<<grid, 256, 0, s>>>(ptr, col, colour, cnt, list[rr & 1], list[(rr & 1) ^ 1], ctr, rr % 3,
                                           maxc);
            PK_LAUNCH();
        }
        unsigned h[4];
        PK_CUDA(cudaMemcpyAsync(h, ctr, sizeof(h), cudaMemcpyDeviceToHost, s));
        PK_CUDA(cudaStreamSynchronize(s));
        if (h[(r + 32) % 3] == 0u) return (int)h[3];
        if (r > n + 64) fail(PKASP_ECUDA, "colouring did not terminate");
    }
}

// ---------------------------------------------------------------------------------
// Stable counting sort by a small key. One warp walks kSortChunk consecutive rows and
// counts them per key (rows of equal key within 32 found with a match, their leader adds
// the count: no atomics); the counts, key-major, are scanned; the warp walks its rows
// again and places them. (The host did this on a copy of the colours. At P4 48^3 the whole
// split of A_h, 7 million rows, takes 24 ms.)
// ---------------------------------------------------------------------------------
constexpr int kSortChunk = 1024;

template <bool PLACE>
__global__ void k_key_sort(int64_t n, const int32_t *__restrict__ key, int64_t nchunks, int64_t *cnt,
                           int32_t *__restrict__ perm) {
    const int64_t chunk = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (chunk >= nchunks) return;  // a whole warp
    for (int64_t b = chunk * kSortChunk; b < (chunk + 1) * kSortChunk && b < n; b += 32) {
        const int64_t i = b + lane;
        const bool in = i < n;
        const int32_t k = in ? key[i] : -1;
        const unsigned m = __match_any_sync(0xffffffffu, k);
        const int leader = __ffs(m) - 1;
        int64_t *slot = &cnt[(int64_t)max(k, 0) * nchunks + chunk];
        int64_t at = 0;
        if (in && lane == leader) {
            at = *slot;
            *slot = at + __popc(m);
        }
        if (PLACE) {
            at = __shfl_sync(0xffffffffu, at, leader);
            if (in) perm[at + __popc(m & ((1u << lane) - 1u))] = (int32_t)i;
        }
        __syncwarp();
    }
}

// longest and 90th-percentile lower and upper part of each colour (lengths above 511
// count as 511: they only choose lanes and batch sizes, which are the same from 256 on)
constexpr int kLenCap = 512;
__global__ void k_colour_lengths(const int64_t *__restrict__ off, const int64_t *__restrict__ lptr,
                                 const int64_t *__restrict__ uptr, int4 *__restrict__ out) {
    __shared__ int hl[kLenCap], hu[kLenCap];
    for (int q = threadIdx.x; q < kLenCap; q += blockDim.x) hl[q] = hu[q] = 0;
    __syncthreads();
    const int64_t pb = off[blockIdx.x], pe = off[blockIdx.x + 1];
    for (int64_t p = pb + threadIdx.x; p < pe; p += blockDim.x) {
        atomicAdd(&hl[min((int64_t)kLenCap - 1, lptr[p + 1] - lptr[p])], 1);
        atomicAdd(&hu[min((int64_t)kLenCap - 1, uptr[p + 1] - uptr[p])], 1);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    int v[4] = {0, 0, 0, 0};  // lmax, umax, l90, u90
    const int64_t at = ((pe - pb) * 9) / 10;
    int64_t sl = 0, su = 0;
    for (int q = 0; q < kLenCap; ++q) {
        if (hl[q]) v[0] = q;
        if (hu[q]) v[1] = q;
        if (sl <= at) v[2] = hl[q] ? q : v[2];
        if (su <= at) v[3] = hu[q] ? q : v[3];
        sl += hl[q];
        su += hu[q];
    }
    out[blockIdx.x] = make_int4(v[0], v[1], v[2], v[3]);
}

// ---------------------------------------------------------------------------------
// Colour split
// ---------------------------------------------------------------------------------
__global__ void k_split_count(int64_t n, const int32_t *__restrict__ perm, const int64_t *__restrict__ ptr,
                              const int32_t *__restrict__ col, const int32_t *__restrict__ colour,
                              int64_t *__restrict__ lcnt, int64_t *__restrict__ ucnt) {
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kJpLanes;
    const int sub = threadIdx.x & (kJpLanes - 1);
    if (p >= n) return;
    const unsigned gm = ((1u << kJpLanes) - 1u) << (threadIdx.x & 31 & ~(kJpLanes - 1));
    const int32_t i = perm[p];
    const int ci = colour[i];
    int l = 0, u = 0;
    for (int64_t e = ptr[i] + sub; e < ptr[i + 1]; e += kJpLanes) {
        const int32_t j = col[e];
        if (j == i) continue;
        if (colour[j] < ci) ++l;
        else ++u;  // a proper colouring leaves no equal colours off the diagonal
    }
#pragma unroll
    for (int o = kJpLanes / 2; o > 0; o >>= 1) {
        l += __shfl_xor_sync(gm, l, o);
        u += __shfl_xor_sync(gm, u, o);
    }
    if (sub == 0) {
        lcnt[p] = l;
        ucnt[p] = u;
    }
}

// A lane group takes eight entries of its row at a time; ballots give each entry its
// place, so both parts keep the row's ascending column order.
__global__ void k_split_fill(int64_t n, const int32_t *__restrict__ perm, const int64_t *__restrict__ ptr,
                             const int32_t *__restrict__ col, const double *__restrict__ val,
                             const int32_t *__restrict__ colour, const int64_t *__restrict__ lptr,
                             const int64_t *__restrict__ uptr, int32_t *__restrict__ lcol,
                             double *__restrict__ lval, int32_t *__restrict__ ucol, double *__restrict__ uval,
                             double *__restrict__ diag, double *__restrict__ dinv, int *__restrict__ bad) {
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kJpLanes;
    const int sub = threadIdx.x & (kJpLanes - 1);
    if (p >= n) return;
    const int shift = threadIdx.x & 31 & ~(kJpLanes - 1);
    const unsigned gm = ((1u << kJpLanes) - 1u) << shift;
    const int32_t i = perm[p];
    const int ci = colour[i];
    int64_t lo = lptr[p], uo = uptr[p];
    double d = 0.0;
    const int64_t hi = ptr[i + 1];
    for (int64_t e0 = ptr[i]; e0 < hi; e0 += kJpLanes) {
        const int64_t e = e0 + sub;
        const bool in = e < hi;
        const int32_t j = in ? col[e] : -1;
        const double v = in ? val[e] : 0.0;
        const bool own = in && j == i;
        const int cj = in ? colour[j] : 0;
        const bool low = in && !own && cj < ci, up = in && !own && cj >= ci;
        if (up && cj == ci) atomicExch(bad, 2);
        if (own) d = v;
        const unsigned ml = (__ballot_sync(gm, low) & gm) >> shift, mu = (__ballot_sync(gm, up) & gm) >> shift;
        const unsigned below = (1u << sub) - 1u;
        if (low) {
            const int64_t q = lo + __popc(ml & below);
            lcol[q] = j;
            lval[q] = v;
        }
        if (up) {
            const int64_t q = uo + __popc(mu & below);
            ucol[q] = j;
            uval[q] = v;
        }
        lo += __popc(ml);
        uo += __popc(mu);
    }
    // one lane of the group holds the diagonal, the others 0
#pragma unroll
    for (int o = kJpLanes / 2; o > 0; o >>= 1) {
        const double t = __shfl_xor_sync(gm, d, o);
        if (d == 0.0) d = t;
    }
    if (sub == 0) {
        if (d == 0.0) atomicExch(bad, 1);
        diag[p] = d;
        dinv[p] = d != 0.0 ? 1.0 / d : 0.0;
    }
}

}  // namespace

void key_sort(int64_t n, const int32_t *key, int64_t nkeys, int32_t *perm, std::vector<int64_t> &off,
              cudaStream_t s) {
    off.assign(nkeys + 1, 0);
    off[nkeys] = n;
    if (n <= 0) return;
    const int64_t nchunks = (n + kSortChunk - 1) / kSortChunk;
    DevPool tmp;
    try {
        int64_t *cnt = tmp.get<int64_t>(nkeys * nchunks + 1);
        PK_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int64_t) * nkeys * nchunks, s));
        k_key_sort<false><<<blocks_for(nchunks * 32, 128), 128, 0, s>>>(n, key, nchunks, cnt, nullptr);
        PK_LAUNCH();
        exclusive_scan(cnt, nkeys * nchunks, s);
        PK_CUDA(cudaMemcpy2DAsync(off.data(), sizeof(int64_t), cnt, sizeof(int64_t) * nchunks, sizeof(int64_t),
                                  nkeys, cudaMemcpyDeviceToHost, s));
        k_key_sort<true><<<blocks_for(nchunks * 32, 128), 128, 0, s>>>(n, key, nchunks, cnt, perm);
        PK_LAUNCH();
        PK_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
        cudaStreamSynchronize(s);
        tmp.free_all();
        throw;
    }
    tmp.free_all();
}

// Colour split of A for the multicolour Gauss-Seidel sweeps.
void build_split(DevPool &pool, const DCSR &A, uint64_t stream, bool want32, DSplit &sp, cudaStream_t s) {
    DevPool tmp;
    try {
        const int64_t n = A.n;
        sp.colour = pool.get<int32_t>(n > 0 ? n : 1);
        sp.ncol = n > 0 ? jp_colour(n, A.ptr, A.col, stream, sp.colour, tmp, s) : 0;
        // rows by colour, in row order within a colour
        sp.perm = pool.get<int32_t>(n > 0 ? n : 1);
        key_sort(n, sp.colour, sp.ncol, sp.perm, sp.off, s);
        sp.lptr = pool.get<int64_t>(n + 1);
        sp.uptr = pool.get<int64_t>(n + 1);
        if (n > 0) {
            k_split_count<<<blocks_for(n * kJpLanes, 256), 256, 0, s>>>(n, sp.perm, A.ptr, A.col, sp.colour, sp.lptr,
                                                                        sp.uptr);
            PK_LAUNCH();
        }
        exclusive_scan(sp.lptr, n, s);
        exclusive_scan(sp.uptr, n, s);
        sp.nnz_l = read_i64(sp.lptr + n, s);
        sp.nnz_u = read_i64(sp.uptr + n, s);
        sp.lmax.assign(sp.ncol, 0);
        sp.umax.assign(sp.ncol, 0);
        sp.l90.assign(sp.ncol, 0);
        sp.u90.assign(sp.ncol, 0);
        if (sp.ncol > 0) {
            // longest and 90th-percentile lower/upper part of each colour: they fix the lanes
            // per row and the entries per batch of that colour's phase
            int64_t *doff = tmp.get<int64_t>(sp.ncol + 1);
            int4 *dlen = tmp.get<int4>(sp.ncol);
            std::vector<int4> len(sp.ncol);
            PK_CUDA(cudaMemcpyAsync(doff, sp.off.data(), sizeof(int64_t) * (sp.ncol + 1), cudaMemcpyHostToDevice, s));
            k_colour_lengths<<<(unsigned)sp.ncol, 512, 0, s>>>(doff, sp.lptr, sp.uptr, dlen);
            PK_LAUNCH();
            PK_CUDA(cudaMemcpyAsync(len.data(), dlen, sizeof(int4) * sp.ncol, cudaMemcpyDeviceToHost, s));
            PK_CUDA(cudaStreamSynchronize(s));
            for (int c = 0; c < sp.ncol; ++c) {
                sp.lmax[c] = len[c].x;
                sp.umax[c] = len[c].y;
                sp.l90[c] = len[c].z;
                sp.u90[c] = len[c].w;
            }
        }
        sp.lcol = pool.get<int32_t>(sp.nnz_l > 0 ? sp.nnz_l : 1);
        sp.lval = pool.get<double>(sp.nnz_l > 0 ? sp.nnz_l : 1);
        sp.ucol = pool.get<int32_t>(sp.nnz_u > 0 ? sp.nnz_u : 1);
        sp.uval = pool.get<double>(sp.nnz_u > 0 ? sp.nnz_u : 1);
        sp.diag = pool.get<double>(n > 0 ? n : 1);
        sp.dinv = pool.get<double>(n > 0 ? n : 1);
        int *bad = tmp.get<int>(1);
        PK_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), s));
        if (n > 0) {
            k_split_fill<<<blocks_for(n * kJpLanes, 256), 256, 0, s>>>(n, sp.perm, A.ptr, A.col, A.val, sp.colour,
                                                                       sp.lptr, sp.uptr, sp.lcol, sp.lval, sp.ucol,
                                                                       sp.uval, sp.diag, sp.dinv, bad);
            PK_LAUNCH();
        }
        int hb = 0;
        PK_CUDA(cudaMemcpyAsync(&hb, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
        PK_CUDA(cudaStreamSynchronize(s));
        if (hb == 1) fail(PKASP_EBREAKDOWN, "zero diagonal entry in a smoothed matrix");
        if (hb == 2) fail(PKASP_ECUDA, "colouring left two neighbours with the same colour");
        if (want32) {
            sp.lval32 = pool.get<float>(sp.nnz_l > 0 ? sp.nnz_l : 1);
            sp.uval32 = pool.get<float>(sp.nnz_u > 0 ? sp.nnz_u : 1);
            sp.diag32 = pool.get<float>(n > 0 ? n : 1);
            sp.dinv32 = pool.get<float>(n > 0 ? n : 1);
            to32(sp.lval, sp.lval32, sp.nnz_l, s);
            to32(sp.uval, sp.uval32, sp.nnz_u, s);
            to32(sp.diag, sp.diag32, n, s);
            to32(sp.dinv, sp.dinv32, n, s);
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
