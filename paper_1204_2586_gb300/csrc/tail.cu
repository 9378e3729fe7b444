// tail.cu -- the dense tail of the V-cycle. On a small level the cycle from there down is a
// chain of launches that each move a few kilobytes: with Gauss-Seidel levels one per colour
// and sweep (402 rows still have 53 colours), each 2-4 us. But V is a fixed linear operator
// of b, so setup applies it to the identity (all columns at once, from the coarsest level
// up) and the solve multiplies by that n x n matrix, as it always did with the coarsest
// inverse: one launch that reads n^2 entries. The matrix is formed in FP64.
//
// One column block of a level is kCols threads wide; a thread carries one column through the
// row sums, so reads of the dense operand are coalesced and the matrix entry is a broadcast.
#include <algorithm>
#include <cmath>

#include "internal.h"

namespace pk {
namespace {

constexpr int kCols = 128;  // columns of a block

unsigned tiles(int64_t n) { return (unsigned)((n + kCols - 1) / kCols); }

// Y_r = c0 * I_r + Y_r * keep + scale_r * (sum_e a_e X_e) with rows r = rows[p] (or p)
//   rows/ptr per position p; one block per position and column block
__global__ void __launch_bounds__(kCols) k_tail_rows(int64_t n, int64_t p0, const int32_t *__restrict__ rows,
                                                     const int64_t *__restrict__ ptr,
                                                     const int32_t *__restrict__ col, const double *__restrict__ val,
                                                     const double *X, double *Y, double ident, double keep,
                                                     double sign) {
    const int64_t p = p0 + blockIdx.x, c = (int64_t)blockIdx.y * kCols + threadIdx.x;
    if (c >= n) return;
    const int64_t r = rows ? rows[p] : p;
    double acc = 0.0;
    const int64_t hi = ptr[p + 1];
    for (int64_t e = ptr[p]; e < hi; ++e) acc += val[e] * X[(int64_t)col[e] * n + c];
    const double own = keep != 0.0 ? keep * Y[r * n + c] : 0.0;
    Y[r * n + c] = (r == c ? ident : 0.0) + own + sign * acc;
}

// one Gauss-Seidel colour: X_r = (I_r - sum_lower a X - [full] sum_upper a X) * dinv; or
// (back) the second half of the symmetric sweep, X_r -= (sum_upper a X) * dinv
__global__ void __launch_bounds__(kCols) k_tail_gs(int64_t n, int64_t p0, const int32_t *__restrict__ rows,
                                                   const int64_t *__restrict__ lptr,
                                                   const int32_t *__restrict__ lcol,
                                                   const double *__restrict__ lval, const int64_t *__restrict__ uptr,
                                                   const int32_t *__restrict__ ucol,
                                                   const double *__restrict__ uval, const double *__restrict__ dinv,
                                                   int full, int back, double *X) {
    const int64_t p = p0 + blockIdx.x, c = (int64_t)blockIdx.y * kCols + threadIdx.x;
    if (c >= n) return;
    const int64_t r = rows[p];
    double acc = 0.0;
    if (!back)
        for (int64_t e = lptr[p]; e < lptr[p + 1]; ++e) acc += lval[e] * X[(int64_t)lcol[e] * n + c];
    if (full || back)
        for (int64_t e = uptr[p]; e < uptr[p + 1]; ++e) acc += uval[e] * X[(int64_t)ucol[e] * n + c];
    X[r * n + c] = back ? X[r * n + c] - acc * dinv[p] : ((r == c ? 1.0 : 0.0) - acc) * dinv[p];
}

// X = D^{-1} (the l1-Jacobi step from zero on the identity); X += D^{-1} R
__global__ void k_tail_jacobi0(int64_t n, const double *__restrict__ d, double *__restrict__ X) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n * n) return;
    const int64_t r = q / n;
    X[q] = r == q % n ? 1.0 / d[r] : 0.0;
}
__global__ void k_tail_jacobi(int64_t n, const double *__restrict__ d, const double *__restrict__ R,
                              double *__restrict__ X) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < n * n) X[q] += R[q] / d[q / n];
}

// C[m][n] = A[m][k] B[k][n]: 32 x 32 tiles, four rows per thread
__global__ void __launch_bounds__(256) k_tail_gemm(int64_t m, int64_t n, int64_t k, const double *__restrict__ A,
                                                   const double *__restrict__ B, double *__restrict__ C) {
    __shared__ double a[32][33], b[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
    const int64_t i0 = (int64_t)blockIdx.y * 32, j = (int64_t)blockIdx.x * 32 + tx;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t k0 = 0; k0 < k; k0 += 32) {
        for (int q = ty; q < 32; q += 8) {
            a[q][tx] = i0 + q < m && k0 + tx < k ? A[(i0 + q) * k + k0 + tx] : 0.0;
            b[q][tx] = k0 + q < k && j < n ? B[(k0 + q) * n + j] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int u = 0; u < 32; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] += a[ty + 8 * q][u] * b[u][tx];
        __syncthreads();
    }
    if (j >= n) return;
    for (int q = 0; q < 4; ++q)
        if (i0 + ty + 8 * q < m) C[(i0 + ty + 8 * q) * n + j] = acc[q];
}

// X += I_P M I_P^T (rows of I_P have at most four entries)
__global__ void __launch_bounds__(kCols) k_tail_coarse(int64_t n, int64_t nc, const int64_t *__restrict__ ptr,
                                                       const int32_t *__restrict__ col,
                                                       const double *__restrict__ val, const double *__restrict__ M,
                                                       double *__restrict__ X) {
    const int64_t r = blockIdx.x, c = (int64_t)blockIdx.y * kCols + threadIdx.x;
    if (c >= n) return;
    double acc = 0.0;
    for (int64_t e = ptr[r]; e < ptr[r + 1]; ++e) {
        double t = 0.0;
        for (int64_t f = ptr[c]; f < ptr[c + 1]; ++f) t += M[(int64_t)col[e] * nc + col[f]] * val[f];
        acc += val[e] * t;
    }
    X[r * n + c] += acc;
}

// Modelled time (us) of one cycle from level l down, as launches. Gauss-Seidel: a launch
// per colour and sweep, 3.4 us each in the row layout (P2 21^3 FP64, 202 phases of three
// levels: 709 us) and 1.6 to 2.4 in slices, which picks the same levels on the hierarchies of
// P1 problems from 17^3 to 64^3;
// l1-Jacobi: five launches of 2 us each besides the next level (P2 8^3: 18 us over two
// levels).
double launches_us(const Level &L, bool jacobi) { return jacobi ? 11.0 : 10.0 + 2 * 3.4 * L.sp.ncol; }
// and of the dense product: a launch, then n^2 FMAs at the FP64 pipe's 0.55 10^6 a us (the
// reads of 8 n^2 bytes at 5 10^6 a us hide behind them), or 4 n^2 bytes at that rate in FP32
double dense_us(double n, bool fp32) { return 2.5 + n * n / (fp32 ? 1.2e6 : 0.55e6); }

}  // namespace

// Level at which the cycle becomes one dense product: the highest where that is modelled
// faster than the launches below it, within 5120 rows and n nnz <= 4 10^9 (the FMAs of one of the
// level's own passes over the identity; the coarse product adds n_c^2 n of them: a setup of P1 17^3,
// 4096 rows over 1241, takes 19 ms).
int tail_level(const pkasp_problem *p) {
    const bool jacobi = p->opt.level_smoother == PKASP_SMOOTHER_L1JACOBI;
    const bool fp32 = p->opt.precond_precision == PKASP_PREC_FP32;
    const int last = (int)p->lev.size() - 1;
    int best = last;
    double below = dense_us((double)p->lev[last].A.n, fp32);
    for (int l = last - 1; l >= 0; --l) {
        const Level &L = p->lev[l];
        const double n = (double)L.A.n;
        below += launches_us(L, jacobi);
        if (L.A.n > 5120 || n * (double)L.A.nnz > 4e9) break;
        if (dense_us(n, fp32) < below) {
            best = l;
            below = dense_us(n, fp32);
        }
    }
    return best;
}

// The same for the cycle of a block of NC columns, which takes the dense matrix of p->tail or,
// where that takes longer, the launches down to the coarsest inverse. In the additive form both
// run beside the fine sweeps (S): launches wait most of their time and hide behind them, the
// product wants the FP64 pipe and the L1 as they do and adds to them. So the times (us) compared
// are  max(S, D) + share min(S, D)  for the product and  max(S, L)  for the launches; with no
// sweep beside them D and L. w is NC / 64, `row` a level's mean row in units of 50 entries:
//   D  chain n W / 32 for a group's entries one after another, or the n^2 NC FMAs (a warp a row,
//      so whole rounds of eight rows on each of 152 SMs) at `rate` a us
//   L  Gauss-Seidel: level + a phase a colour and sweep of c0 + c1 w + row (c2 + c3 w);
//      l1-Jacobi: level + row (c2 + c3 w); and the product of the coarsest level
// Fitted to graph solves with and without the product, P1 7^3 to 42^3, P2 9^3 to 32^3, P3 9^3
// to 21^3, P4 8^3 to 16^3, constant and lognormal coefficients, widths 4 to 64, as is the estimate
// of S: the constants stand for the choice they make, not for a kernel alone. Of 864 pairs ten
// come out more than 3% above the faster side (13% at most), none more than 2% above the launches.
// Taking the product always had made wide blocks up to twice as slow:
// an iteration of P2 17^3, 64 columns, FP64, Gauss-Seidel levels 1724 us as launches and 3321 with
// 4096 rows dense; with l1-Jacobi levels and n^2 NC <= 10^7, P1 9^3, 32 columns 162 and 210.
struct BlockCycle {
    double chain, rate, share, level, c0, c1, c2, c3;
};
constexpr BlockCycle kBlockCycle[2][2] = {  // [FP32][l1-Jacobi]
    {{0.078, 0.33e6, 1.1, 30, 3.3, 7.1, 2.3, 9.4}, {0.87, 0.67e6, 0.62, 24, 0, 0, 160, 19}},
    {{0.018, 1.3e6, 0.45, 410, 0.73, 0, 6.8, 0}, {0.17, 0.90e6, 0.076, 33, 0, 0, 55, 0.54}}};

int block_tail_level(const pkasp_problem *p, int NC) {
    const bool jacobi = p->opt.level_smoother == PKASP_SMOOTHER_L1JACOBI;
    const bool fp32 = p->opt.precond_precision == PKASP_PREC_FP32;
    const BlockCycle &c = kBlockCycle[fp32][jacobi];
    const int last = (int)p->lev.size() - 1, W = NC % 32 == 0 ? 32 : NC % 16 == 0 ? 16 : NC % 8 == 0 ? 8 : 4;
    const double w = NC / 64.0;
    auto product = [&](int l) {
        const double n = (double)p->lev[l].A.n;
        return 3.0 + std::max(c.chain * n * W / 32, std::ceil(n / 1216) * 1216 * n * NC / c.rate);
    };
    double launches = product(last);
    for (int l = p->tail; l < last; ++l) {
        const Level &L = p->lev[l];
        const double row = (double)L.A.nnz / (double)L.A.n / 50, each = c.c0 + c.c1 * w + row * (c.c2 + c.c3 * w);
        launches += c.level + (jacobi ? 1 : 2 * L.sp.ncol) * each;
    }
    double sweeps = 0;
    if (p->opt.mode == PKASP_MODE_ADDITIVE && p->opt.smoother == PKASP_SMOOTHER_SGS) {
        const double row = (double)p->Ah.nnz / (double)p->nh / 50, ph = 2.0 * p->fine.ncol, m = 1e-6 * (double)p->Ah.nnz;
        sweeps = fp32 ? ph * (1.5 + row * (1.5 + 3.2 * w)) + m * (0.42 * NC + 9.7)
                      : ph * (1.3 + row * (2.4 + 6.1 * w)) + m * (2.4 * NC + 17.0);
    }
    const double d = product(p->tail);
    return std::max(sweeps, d) + c.share * std::min(sweeps, d) < std::max(sweeps, launches) ? p->tail : last;
}

// Whether the whole additive preconditioner B = S_k + I_P V I_P^T of a small problem is
// applied as one dense product: its sweeps cost 1.5 us a phase, whatever their size. An iteration
// (us, Gauss-Seidel levels, kappa = 1; product, sweeps):
//   3375 rows  P2 8^3 FP64 60.6, 70.7, FP32 44.4, 65.5; P1 16^3 62, 76 and 47, 61; P4 4^3 60, 148
//              and 43, 129
//   4096 rows  P1 17^3 80, 92 and 49, 63
//   4913 rows  P2 9^3 94, 75 and 53, 69; P3 6^3 91, 102 and 54, 92
// The order changes between 3400 and 4900 rows for FP64 and few colours. The bound of 3400 rows is
// that line (92 MB of matrix in FP64), taken for all degrees and both precisions, and the one of
// 6 10^8 entries times rows keeps the setup's work at 1 ms: FP32, P3 and P4 would gain beyond them
// (P4 4^3 has 6.3 10^8; its setup takes 3.5 ms with the product and 1.4 without). An explicit
// layout of the smoother keeps its sweeps.
bool dense_prec(const pkasp_problem *p) {
    const pkasp_options &o = p->opt;
    if (o.mode != PKASP_MODE_ADDITIVE || o.smoother != PKASP_SMOOTHER_SGS || o.smoother_layout != 0 ||
        o.spmv_threads != 0 || p->tail != 0)
        return false;
    const double n = (double)p->nh;
    return p->nh <= 3400 && n * (double)p->Ah.nnz <= 6e8 &&
           dense_us(n, o.precond_precision == PKASP_PREC_FP32) < 3.0 * p->fine.ncol;
}

// B from M = V on level 0 (n_H x n_H, FP64)
void build_dense_prec(pkasp_problem *p, const double *M, DevPool &tmp, cudaStream_t s) {
    const bool fp32 = p->opt.precond_precision == PKASP_PREC_FP32;
    const int64_t n = p->nh;
    double *X = (fp32 ? tmp : p->setup_pool).get<double>(n * n);
    const DSplit &sp = p->fine;
    for (int q = 0; q < 2 * sp.ncol; ++q) {
        const int back = q >= sp.ncol, c = back ? 2 * sp.ncol - 1 - q : q;
        const int64_t pb = sp.off[c], m = sp.off[c + 1] - pb;
        if (m == 0) continue;
        k_tail_gs<<<dim3((unsigned)m, tiles(n)), kCols, 0, s>>>(n, pb, sp.perm, sp.lptr, sp.lcol, sp.lval, sp.uptr,
                                                                sp.ucol, sp.uval, sp.dinv, 0, back, X);
        PK_LAUNCH();
    }
    k_tail_coarse<<<dim3((unsigned)n, tiles(n)), kCols, 0, s>>>(n, p->nH, p->Pi.ptr, p->Pi.col, p->Pi.val, M, X);
    PK_LAUNCH();
    if (fp32) {
        p->d_dense32 = p->setup_pool.get<float>(n * n);
        to32(X, p->d_dense32, n * n, s);
    } else {
        p->d_dense = X;
    }
}

// M = V on level p->tail, from the coarsest inverse up; into d_tail (or d_tail32); then the
// whole preconditioner of a small problem
void build_tail(pkasp_problem *p, cudaStream_t s) {
    const int last = (int)p->lev.size() - 1;
    p->tail = tail_level(p);
    p->d_tail = p->d_cinv;
    p->d_tail32 = p->d_cinv32;
    const bool dense = dense_prec(p);
    if (p->tail == last && !dense) return;
    const bool jacobi = p->opt.level_smoother == PKASP_SMOOTHER_L1JACOBI;
    const bool fp32 = p->opt.precond_precision == PKASP_PREC_FP32;
    DevPool tmp;
    try {
        const double *Mc = p->d_cinv;
        for (int l = last - 1; l >= p->tail; --l) {
            Level &L = p->lev[l];
            const int64_t n = L.A.n, nc = L.R.n;
            // the matrix of the tail itself outlives setup when it is the one in use
            double *X = (l == p->tail && !fp32 ? p->setup_pool : tmp).get<double>(n * n);
            double *R = tmp.get<double>(n * n), *B = tmp.get<double>(nc * n), *W = tmp.get<double>(nc * n);
            const unsigned ct = tiles(n), flat = (unsigned)((n * n + 255) / 256);
            const DSplit &sp = L.sp;
            auto gs = [&](int c, int full) {
                const int64_t pb = sp.off[c], m = sp.off[c + 1] - pb;
                if (m == 0) return;
                k_tail_gs<<<dim3((unsigned)m, ct), kCols, 0, s>>>(n, pb, sp.perm, sp.lptr, sp.lcol, sp.lval, sp.uptr,
                                                                  sp.ucol, sp.uval, sp.dinv, full, 0, X);
                PK_LAUNCH();
            };
            auto residual = [&] {  // R = I - A X
                k_tail_rows<<<dim3((unsigned)n, ct), kCols, 0, s>>>(n, 0, nullptr, L.A.ptr, L.A.col, L.A.val, X, R,
                                                                    1.0, 0.0, -1.0);
                PK_LAUNCH();
            };
            if (jacobi) {
                k_tail_jacobi0<<<flat, 256, 0, s>>>(n, L.l1, X);
                PK_LAUNCH();
            } else {
                for (int c = 0; c < sp.ncol; ++c) gs(c, 0);
            }
            residual();
            k_tail_rows<<<dim3((unsigned)nc, ct), kCols, 0, s>>>(n, 0, nullptr, L.R.ptr, L.R.col, L.R.val, R, B, 0.0,
                                                                 0.0, 1.0);
            PK_LAUNCH();
            k_tail_gemm<<<dim3((unsigned)((n + 31) / 32), (unsigned)((nc + 31) / 32)), 256, 0, s>>>(nc, n, nc, Mc, B,
                                                                                                   W);
            PK_LAUNCH();
            k_tail_rows<<<dim3((unsigned)n, ct), kCols, 0, s>>>(n, 0, nullptr, L.P.ptr, L.P.col, L.P.val, W, X, 0.0,
                                                                1.0, 1.0);
            PK_LAUNCH();
            if (jacobi) {
                residual();
                k_tail_jacobi<<<flat, 256, 0, s>>>(n, L.l1, R, X);
                PK_LAUNCH();
            } else {
                for (int c = sp.ncol - 1; c >= 0; --c) gs(c, 1);
            }
            Mc = X;
        }
        if (dense) build_dense_prec(p, Mc, tmp, s);
        const int64_t n = p->lev[p->tail].A.n;
        if (p->tail == last) {
            // the coarsest inverse itself
        } else if (fp32) {
            p->d_tail32 = p->setup_pool.get<float>(n * n);
            to32(Mc, p->d_tail32, n * n, s);
            p->d_tail = nullptr;
        } else {
            p->d_tail = const_cast<double *>(Mc);
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
