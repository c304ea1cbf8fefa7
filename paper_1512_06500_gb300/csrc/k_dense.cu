// FP64 dense building blocks of the Krylov solver: tall-skinny products with a deterministic
// split-K reduction, small products, Cholesky with inverse, and seeded Gaussian blocks.
#include "eda_internal.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

namespace eda {

namespace {

constexpr int TN_KB = 32;       // rows of A/B staged per pass
constexpr int TN_TM = 32;       // output tile rows
constexpr int TN_THREADS = 256;

// Tile (bx, by) with bx >= by of the lower triangle of a T x T tile grid from its index
// q = bx (bx + 1) / 2 + by (row by row).
__device__ __forceinline__ void tri_tile(int q, int& bx, int& by) {
    // single precision, corrected below: an FP64 square root takes the FP64 pipe for longer than some callers' products
    int x = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
    while ((x + 1) * (x + 2) / 2 <= q) ++x;
    while (x * (x + 1) / 2 > q) --x;
    bx = x;
    by = q - x * (x + 1) / 2;
}

// partial[s][j][i] = sum over rows r of split s of A[r, i0+i] * B[r, j0+j]. SYM (A = B, m = p, TP = TN_TM):
// only the tiles with i0 >= j0 are launched (blockIdx.x runs over the lower triangle of the tile grid);
// a diagonal tile computes entries (i, j) and (j, i) from the same products in the same order, so it is
// exactly symmetric.
template <int TP, class T, bool SYM = false>
__global__ void __launch_bounds__(TN_THREADS) k_gemm_tn_partial(int64_t d, int m, int p, const T* __restrict__ A,
                                                                int64_t lda, const T* __restrict__ B, int64_t ldb,
                                                                int64_t rows_per_split, T* __restrict__ partial) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(B); PDL_ARG(partial);
    __shared__ T As[TN_KB][TN_TM + 1];
    __shared__ T Bs[TN_KB][TP + 1];
    int bx = blockIdx.x, by = blockIdx.y;
    if (SYM) tri_tile(blockIdx.x, bx, by);
    const int i0 = bx * TN_TM;
    const int j0 = by * TP;
    const int s = blockIdx.z;
    const int64_t r_begin = (int64_t)s * rows_per_split;
    const int64_t r_end = min(d, r_begin + rows_per_split);
    // thread -> outputs: TM*TP outputs over 256 threads
    constexpr int OUT = TN_TM * TP / TN_THREADS;      // 1 (TP=8), 2 (TP=16), 4 (TP=32)
    constexpr int TPT = (TP >= 16) ? 2 : 1;           // columns per thread
    constexpr int TMT = OUT / TPT;                    // rows per thread
    const int tx = threadIdx.x % (TN_TM / TMT);       // row group
    const int ty = threadIdx.x / (TN_TM / TMT);       // column group
    T acc[TMT][TPT];
#pragma unroll
    for (int a = 0; a < TMT; ++a)
#pragma unroll
        for (int b = 0; b < TPT; ++b) acc[a][b] = T(0);

    // the next chunk of rows is read into registers while the current one is multiplied, so the
    // global-memory latency overlaps the FP64 work (the products and their order are unchanged)
    constexpr int PA = TN_KB * TN_TM / TN_THREADS;                  // A elements per thread and chunk
    constexpr int PB = (TN_KB * TP + TN_THREADS - 1) / TN_THREADS;  // B elements per thread and chunk
    T ra[PA], rb[PB];
    auto fetch = [&](int64_t r0) {
#pragma unroll
        for (int q = 0; q < PA; ++q) {
            const int e = threadIdx.x + q * TN_THREADS;
            const int rr = e % TN_KB, cc = e / TN_KB;
            const int64_t r = r0 + rr;
            const int c = i0 + cc;
            ra[q] = (r < r_end && c < m) ? A[(int64_t)c * lda + r] : T(0);
        }
#pragma unroll
        for (int q = 0; q < PB; ++q) {
            const int e = threadIdx.x + q * TN_THREADS;
            const int rr = e % TN_KB, cc = e / TN_KB;
            const int64_t r = r0 + rr;
            const int c = j0 + cc;
            rb[q] = (e < TN_KB * TP && r < r_end && c < p) ? B[(int64_t)c * ldb + r] : T(0);
        }
    };
    if (r_begin < r_end) fetch(r_begin);
    for (int64_t r0 = r_begin; r0 < r_end; r0 += TN_KB) {
        // stage A rows r0..r0+KB of columns i0..i0+TM and the matching rows of B
#pragma unroll
        for (int q = 0; q < PA; ++q) {
            const int e = threadIdx.x + q * TN_THREADS;
            As[e % TN_KB][e / TN_KB] = ra[q];
        }
#pragma unroll
        for (int q = 0; q < PB; ++q) {
            const int e = threadIdx.x + q * TN_THREADS;
            if (e < TN_KB * TP) Bs[e % TN_KB][e / TN_KB] = rb[q];
        }
        __syncthreads();
        if (r0 + TN_KB < r_end) fetch(r0 + TN_KB);
#pragma unroll 8
        for (int rr = 0; rr < TN_KB; ++rr) {
            T av[TMT], bv[TPT];
#pragma unroll
            for (int a = 0; a < TMT; ++a) av[a] = As[rr][tx + a * (TN_TM / TMT)];
#pragma unroll
            for (int b = 0; b < TPT; ++b) bv[b] = Bs[rr][ty + b * (TP / TPT)];
#pragma unroll
            for (int a = 0; a < TMT; ++a)
#pragma unroll
                for (int b = 0; b < TPT; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
        }
        __syncthreads();
    }
    PDL_NEXT();
    T* out = partial + (int64_t)s * m * p;
#pragma unroll
    for (int a = 0; a < TMT; ++a)
#pragma unroll
        for (int b = 0; b < TPT; ++b) {
            const int i = i0 + tx + a * (TN_TM / TMT);
            const int j = j0 + ty + b * (TP / TPT);
            if (i < m && j < p) out[(int64_t)j * m + i] = acc[a][b];
        }
}

// The symmetric product A^T A of a narrow block (m <= 32 columns: the CholQR Grams), partial sums by CTA in the layout of
// k_gemm_tn_partial. The FP64 pipe bounds it, so only the m (m + 1) / 2 entries of the lower triangle are computed: the
// items (row phase r < R, entry e of the triangle) are dealt to the lanes of each warp, ACC or fewer accumulators a lane, and
// a step of a warp takes R rows of the block, so that almost every lane of every FP64 instruction works (m = 8: 9 instructions
// for 8 rows; the 32 x 32 tiles of the general kernel take 32 a row). Rows come through shared memory, the next chunk
// read into registers meanwhile; the warps' sums are added in order at the end.
// GB300: d = 16384, m = 16 59 -> 17.8 us; d = 65536, m = 32 111 -> 90 us (69 us at the FP64 rate); d = 256, m = 1 .. 7
// 19 -> 8 us. Two CTAs per SM (a few accumulators spill at m > 16: 104 us with one).
constexpr int SN_THREADS = 256;
constexpr int SN_MAXM = 32;
template <int ACC, int CH, int MC, class T>
__global__ void __launch_bounds__(SN_THREADS, 2) k_syrk_narrow(int64_t d, int m, const T* __restrict__ A, int64_t lda,
                                                            int64_t rows_per_split, int R, T* __restrict__ partial) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(partial);
    constexpr int LD = MC | 1;   // odd: the columns of a row and the rows of a column fall into different banks
    __shared__ T As[CH][LD];
    __shared__ T tot[32 * ACC];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int tri = m * (m + 1) / 2, items = R * tri;
    const int64_t r_begin = (int64_t)blockIdx.x * rows_per_split, r_end = min(d, r_begin + rows_per_split);
    // this lane's items: offsets of the two factors within a step's rows
    int off[ACC];
    T acc[ACC];
#pragma unroll
    for (int k = 0; k < ACC; ++k) {
        const int it = lane + 32 * k;
        const int r = it < items ? it / tri : 0, e = it < items ? it % tri : 0;
        int i, j;
        tri_tile(e, i, j);
        off[k] = (r * LD + i) << 16 | (r * LD + j);
        acc[k] = T(0);
    }
    constexpr int PA = CH * MC / SN_THREADS;
    T ra[PA];
    auto fetch = [&](int64_t r0) {
#pragma unroll
        for (int q = 0; q < PA; ++q) {
            const int e = tid + q * SN_THREADS;
            const int64_t r = r0 + e % CH;
            const int c = e / CH;
            ra[q] = (r < r_end && c < m) ? A[(int64_t)c * lda + r] : T(0);
        }
    };
    if (r_begin < r_end) fetch(r_begin);
    for (int64_t r0 = r_begin; r0 < r_end; r0 += CH) {
#pragma unroll
        for (int q = 0; q < PA; ++q) {
            const int e = tid + q * SN_THREADS;
            As[e % CH][e / CH] = ra[q];
        }
        __syncthreads();
        if (r0 + CH < r_end) fetch(r0 + CH);
        // the warp's steps of R rows (rows at or beyond r_end are zero; R divides CH)
        const int live = (int)min((int64_t)CH, r_end - r0);
        for (int rr = w * R; rr < live; rr += (SN_THREADS / 32) * R) {
            const T* base = &As[rr][0];
            // groups of four: their eight loads are in flight together (lanes beyond the items repeat item 0)
#pragma unroll
            for (int k0 = 0; k0 < ACC; k0 += 4) {
                if (32 * k0 >= items) break;
                T x[4], y[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (k0 + u < ACC) {
                        x[u] = base[off[k0 + u] >> 16];
                        y[u] = base[off[k0 + u] & 0xffff];
                    }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (k0 + u < ACC) acc[k0 + u] = fma(x[u], y[u], acc[k0 + u]);
            }
        }
        __syncthreads();
    }
    PDL_NEXT();
    for (int v = 0; v < SN_THREADS / 32; ++v) {
        if (w == v) {
#pragma unroll
            for (int k = 0; k < ACC; ++k) tot[lane + 32 * k] = v == 0 ? acc[k] : tot[lane + 32 * k] + acc[k];
        }
        __syncthreads();
    }
    T* out = partial + (int64_t)blockIdx.x * m * m;
    for (int e = tid; e < tri; e += SN_THREADS) {
        int i, j;
        tri_tile(e, i, j);
        T v = tot[e];
        for (int r = 1; r < R; ++r) v += tot[r * tri + e];
        out[(int64_t)j * m + i] = v;
    }
}

// C[i, j] = alpha * sum_s partial[s][j][i] + beta * C[i, j]. Small split counts: one thread per
// output, splits summed in order. Large split counts: one warp per output, lane l sums splits
// l, l + 32, ... in order, then a fixed butterfly across lanes (deterministic either way).
// SYM: only entries with i >= j are summed; each is written to (i, j) and mirrored to (j, i).
__device__ __forceinline__ void tn_store(double* C, int ldc, int i, int j, double acc, double alpha, double beta,
                                         bool sym) {
    double v = alpha * acc;
    if (beta != 0.0) v = fma(beta, C[(int64_t)j * ldc + i], v);
    C[(int64_t)j * ldc + i] = v;
    if (sym && i != j) {
        double w = alpha * acc;
        if (beta != 0.0) w = fma(beta, C[(int64_t)i * ldc + j], w);
        C[(int64_t)i * ldc + j] = w;
    }
}

template <class T>
__global__ void k_gemm_tn_reduce(int m, int p, int splits, const T* __restrict__ partial, double alpha,
                                 double beta, double* __restrict__ C, int ldc, bool sym) {
    PDL_ENTER();
    PDL_ARG(partial); PDL_ARG(C);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)m * p) return;
    const int i = (int)(e % m), j = (int)(e / m);
    if (sym && i < j) return;
    double acc = 0.0;
    for (int s = 0; s < splits; ++s) acc += (double)partial[(int64_t)s * m * p + e];
    tn_store(C, ldc, i, j, acc, alpha, beta, sym);
}

template <class T>
__global__ void k_gemm_tn_reduce_warp(int m, int p, int splits, const T* __restrict__ partial, double alpha,
                                      double beta, double* __restrict__ C, int ldc, bool sym) {
    PDL_ENTER();
    PDL_ARG(partial); PDL_ARG(C);
    const int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (e >= (int64_t)m * p) return;
    const int i = (int)(e % m), j = (int)(e / m);
    if (sym && i < j) return;
    const int64_t mp = (int64_t)m * p;
    double a0 = 0.0, a1 = 0.0;
    int s = lane;
    for (; s + 32 < splits; s += 64) {
        a0 += (double)partial[(int64_t)s * mp + e];
        a1 += (double)partial[(int64_t)(s + 32) * mp + e];
    }
    if (s < splits) a0 += (double)partial[(int64_t)s * mp + e];
    double acc = a0 + a1;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) tn_store(C, ldc, i, j, acc, alpha, beta, sym);
}

// C[r, c] = beta * C0[r, c] + alpha * sum_l A[r, l] B[l, c] for tall A (d x m) and small B
// (m x p). A CTA owns 32 rows and NC columns; its eight warps (two per SM sub-partition, so that
// one issues FP64 work while the other waits on a load) split the inner dimension into eighths,
// each thread keeps NC independent accumulators, the slice of B sits in shared memory, and the
// partial sums of the eighths are added in a fixed pairwise order at the end, a column per warp (one
// warp adding all of them took as long as the products of m = 64). For an upper
// triangular B (ub) each warp stops at row c0 + NC of B, below which the CTA's columns are zero: the
// partition of the inner dimension is unchanged and only exact zero terms are left out.
// KS = 1 (few inner rows and warps enough for every sub-partition): a warp takes 32 rows of its own over the whole inner
// dimension; nothing is added across warps, a quarter of the FP64 instructions at m = 32. GB300, 65536 rows,
// m = p = 32, upper triangular: 114 -> 86 us (FP64 bound 84); 4096 rows, 8 columns, m = 240, KS = 8: 23 -> 19.6 us.
constexpr int kNnWholeM = 64;
template <int NC, class T, int KS = 8>
__global__ void __launch_bounds__(256) k_gemm_nn(int64_t d, int m, int p, double alpha, const T* __restrict__ A,
                                                 int64_t lda, const double* __restrict__ B, int ldb, double beta,
                                                 const T* C0, int64_t ldc0, T* C, int64_t ldc, int ub) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(B); PDL_ARG(C0); PDL_ARG(C);
    constexpr int LCH = 256;                 // rows of B staged per pass
    __shared__ T Bs[LCH][NC];
    __shared__ T red[KS == 1 ? 1 : 8][NC][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t r = (KS == 1 ? (int64_t)blockIdx.x * 8 + w : (int64_t)blockIdx.x) * 32 + lane;
    const int c0 = blockIdx.y * NC;
    const int nc = min(NC, p - c0);
    const int lim = ub ? min(m, c0 + NC) : m;   // rows of B that can be nonzero in these columns
    T acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = T(0);
    const bool live = r < d;
    const T* Ar = A + (live ? r : 0);
    for (int l0 = 0; l0 < m; l0 += LCH) {
        const int lc = min(LCH, m - l0);
        __syncthreads();
        for (int e = threadIdx.x; e < lc * NC; e += blockDim.x) {
            const int l = e / NC, c = e % NC;
            Bs[l][c] = (c < nc) ? (T)B[(int64_t)(c0 + c) * ldb + l0 + l] : T(0);
        }
        __syncthreads();
        const int q = (lc + KS - 1) / KS;
        const int lb = KS == 1 ? 0 : w * q, le = min(min(lc, lb + q), lim - l0);
        int l = lb;
        // groups of four rows of A, the next group read while the current one is multiplied
        T a[4];
        if (l + 3 < le) {
#pragma unroll
            for (int u = 0; u < 4; ++u) a[u] = live ? Ar[(int64_t)(l0 + l + u) * lda] : T(0);
        }
        for (; l + 3 < le; l += 4) {
            T an[4];
            const bool more = l + 7 < le;
            if (more) {
#pragma unroll
                for (int u = 0; u < 4; ++u) an[u] = live ? Ar[(int64_t)(l0 + l + 4 + u) * lda] : T(0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int c = 0; c < NC; ++c) acc[c] = fma(a[u], Bs[l + u][c], acc[c]);
            if (more) {
#pragma unroll
                for (int u = 0; u < 4; ++u) a[u] = an[u];
            }
        }
        for (; l < le; ++l) {
            const T a0 = live ? Ar[(int64_t)(l0 + l) * lda] : T(0);
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] = fma(a0, Bs[l][c], acc[c]);
        }
    }
    PDL_NEXT();
    auto put = [&](int c, T sum) {
        T v = (T)alpha * sum;
        if (beta != 0.0) v = fma((T)beta, C0[(int64_t)(c0 + c) * ldc0 + r], v);
        C[(int64_t)(c0 + c) * ldc + r] = v;
    };
    if (KS == 1) {
        if (!live) return;
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (c < nc) put(c, acc[c]);
        return;
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) red[w][c][lane] = acc[c];
    __syncthreads();
    if (w >= nc || !live) return;
    T x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = red[KS == 1 ? 0 : u][w][lane];
    put(w, ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7])));
}

// Small C (m x p) = alpha A B + beta C (both operands untransposed) with a long inner dimension:
// CTA = 8 warps for one (32-row block, column); warp w sums its eighth of the inner dimension with
// eight independent chains (eight loads of A in flight per lane: at these sizes the product is bound
// by load latency, then by the FP64 pipe), and the eighths are added in a fixed order through shared
// memory.
// SYM (m = p, a symmetric product and C): entries i >= j only, each written to (i, j) and (j, i); the grid's x runs over
// the CTAs that hold such entries, column after column.
constexpr int kSplitkWarps = 8;
template <bool SYM>
__global__ void __launch_bounds__(32 * kSplitkWarps) k_gemm_small_nn_splitk(int m, int p, int kk, double alpha,
                                                                           const double* __restrict__ A, int lda,
                                                                           const double* __restrict__ B, int ldb,
                                                                           double beta, double* __restrict__ C,
                                                                           int ldc) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(B); PDL_ARG(C);
    __shared__ double part[kSplitkWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int ib = blockIdx.x, j = blockIdx.y;
    if (SYM) {
        // blocks of 32 columns from the right: column block c has nb - c row blocks a column
        const int nb = (m + 31) / 32;
        int c = 0, e = blockIdx.x;
        while (e >= 32 * (nb - c)) e -= 32 * (nb - c), ++c;
        ib = c + e % (nb - c);
        j = 32 * c + e / (nb - c);
        if (j >= m) return;   // uniform over the CTA
    }
    const int i = ib * 32 + lane;
    const int q = (kk + kSplitkWarps - 1) / kSplitkWarps;
    const int lb = w * q, le = min(kk, lb + q);
    double a[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) a[u] = 0.0;
    if (i < m) {
        const double* Bj = B + (int64_t)j * ldb;
        int l = lb;
        for (; l + 7 < le; l += 8) {
#pragma unroll
            for (int u = 0; u < 8; ++u) a[u] = fma(A[(int64_t)(l + u) * lda + i], Bj[l + u], a[u]);
        }
        for (; l < le; ++l) a[0] = fma(A[(int64_t)l * lda + i], Bj[l], a[0]);
    }
    PDL_NEXT();
    part[w][lane] = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
    __syncthreads();
    if (w == 0 && i < m) {
        const double acc = ((part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane])) +
                           ((part[4][lane] + part[5][lane]) + (part[6][lane] + part[7][lane]));
        if (SYM && i < j) return;
        double v = alpha * acc;
        if (beta != 0.0) v = fma(beta, C[(int64_t)j * ldc + i], v);
        C[(int64_t)j * ldc + i] = v;
        if (SYM) C[(int64_t)i * ldc + j] = v;
    }
}

__global__ void k_gemm_small(bool ta, bool tb, int m, int p, int kk, double alpha, const double* __restrict__ A,
                             int lda, const double* __restrict__ B, int ldb, double beta, double* __restrict__ C,
                             int ldc) {
    PDL_ENTER();
    PDL_ARG(A); PDL_ARG(B); PDL_ARG(C);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= m || j >= p) return;
    double acc0 = 0.0, acc1 = 0.0, acc2 = 0.0, acc3 = 0.0;
    int l = 0;
    for (; l + 3 < kk; l += 4) {
        if (ta) {
            acc0 = fma(A[(int64_t)i * lda + l], tb ? B[(int64_t)l * ldb + j] : B[(int64_t)j * ldb + l], acc0);
            acc1 = fma(A[(int64_t)i * lda + l + 1], tb ? B[(int64_t)(l + 1) * ldb + j] : B[(int64_t)j * ldb + l + 1], acc1);
            acc2 = fma(A[(int64_t)i * lda + l + 2], tb ? B[(int64_t)(l + 2) * ldb + j] : B[(int64_t)j * ldb + l + 2], acc2);
            acc3 = fma(A[(int64_t)i * lda + l + 3], tb ? B[(int64_t)(l + 3) * ldb + j] : B[(int64_t)j * ldb + l + 3], acc3);
        } else {
            acc0 = fma(A[(int64_t)l * lda + i], tb ? B[(int64_t)l * ldb + j] : B[(int64_t)j * ldb + l], acc0);
            acc1 = fma(A[(int64_t)(l + 1) * lda + i], tb ? B[(int64_t)(l + 1) * ldb + j] : B[(int64_t)j * ldb + l + 1], acc1);
            acc2 = fma(A[(int64_t)(l + 2) * lda + i], tb ? B[(int64_t)(l + 2) * ldb + j] : B[(int64_t)j * ldb + l + 2], acc2);
            acc3 = fma(A[(int64_t)(l + 3) * lda + i], tb ? B[(int64_t)(l + 3) * ldb + j] : B[(int64_t)j * ldb + l + 3], acc3);
        }
    }
    for (; l < kk; ++l) {
        const double a = ta ? A[(int64_t)i * lda + l] : A[(int64_t)l * lda + i];
        const double b = tb ? B[(int64_t)l * ldb + j] : B[(int64_t)j * ldb + l];
        acc0 = fma(a, b, acc0);
    }
    double v = alpha * ((acc0 + acc1) + (acc2 + acc3));
    if (beta != 0.0) v = fma(beta, C[(int64_t)j * ldc + i], v);
    C[(int64_t)j * ldc + i] = v;
}

// 1 / x for a positive normal x: the hardware's 20-bit approximation (PTX rcp.approx.ftz.f64) and two
// Newton-Raphson steps r <- r + r (1 - x r), each doubling the correct bits. The IEEE division is used where
// x or 1 / x leaves the approximation's range.
__device__ __forceinline__ double newton_rcp(double x) {
    const int ex = (__double2hiint(x) >> 20) & 0x7ff;
    if (ex < 24 || ex > 2022) return 1.0 / x;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// Upper Cholesky G = R^T R with rank detection and X = R^{-1}, one CTA of eight warps, b <= 32 NC; the pivot
// order, threshold, lost list and status bits are those of k_chol_inv. The kernel is a chain of b pivots on an
// FP64 pipe that holds a warp instruction for about 64 cycles, so the work is arranged to keep FP64
// instructions off that chain:
//  - G and the inverse are eliminated together as [G | I] -> [R | R^{-T}]: row i keeps G's entries c >= i and the
//    inverse's entries c < i (its unit diagonal is implicit), one b x b square in registers, warp w owning rows
//    w, w + 8, ... and lane l columns l, l + 32, ... There is no back substitution after the factorisation.
//  - rows stay unscaled (G[i, :] -= (u_i / g_j) u for the pivot row u): one reciprocal per pivot, no square root;
//    the square roots and the scaling follow at the end, for all rows at once.
//  - the owner of row j + 1 updates that row first, publishes it and its reciprocal, and updates its other rows
//    while the other warps update theirs: one barrier per pivot, the pivot row double-buffered.
// A kept pivot far below its column's own squared norm (kCholWeak) is counted in lost[b + 1]: that column of X = A R^{-1}
// is A's rounding errors magnified, and no longer orthogonal to what A's columns were orthogonal to.
// GB300, one launch: b = 16 12 us and b = 32 22 us (30 and 76 us by one warp with a back substitution), b = 64 88 us
// (220 us with three barriers, a division and a square root per pivot).
constexpr double kCholWeak = 1e-10;
template <int NC>
__global__ void __launch_bounds__(256) k_chol_inv_pair(int b, double* G, int ldg, double* Rinv, double rank_tol,
                                                       double piv_min2, int* status, int* lost, const NoteRef note) {
    PDL_ENTER();
    PDL_ARG(G); PDL_ARG(Rinv); PDL_ARG(status); PDL_ARG(lost);
    constexpr int NR = 4 * NC;               // rows per warp
    __shared__ double urow[2][32 * NC];      // the pivot row: G's part c >= j, the inverse's part c < j
    __shared__ double ginv[2];               // 1 / pivot, 0 where the pivot is lost
    __shared__ double gpiv[32 * NC];         // pivots (0 where lost)
    __shared__ double rdiag[32 * NC];        // 1 / sqrt(pivot)
    __shared__ double diag0[32 * NC];        // the squared column norms (G's diagonal)
    __shared__ double s_thr;
    __shared__ int s_nlost, s_nweak;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double a[NR][NC];
#pragma unroll
    for (int q = 0; q < NR; ++q) {
        const int i = w + 8 * q;
#pragma unroll
        for (int h = 0; h < NC; ++h) {
            const int c = lane + 32 * h;
            a[q][h] = (i < b && c < b && c >= i) ? G[(int64_t)c * ldg + i] : 0.0;
        }
    }
    if (w == 0) {
        double mx = 0.0;
        bool bad = false;
#pragma unroll
        for (int h = 0; h < NC; ++h) {
            const int c = lane + 32 * h;
            const double g = c < b ? G[(int64_t)c * ldg + c] : 0.0;
            diag0[c] = g;
            bad |= !isfinite(g);
            mx = fmax(mx, fabs(g));
        }
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, ST_NONFINITE);
        // a zero diagonal loses every pivot
        if (lane == 0) {
            s_thr = mx == 0.0 ? INFINITY : fmax(rank_tol * mx, piv_min2);
            s_nlost = 0;
            s_nweak = 0;
        }
    }
    __syncthreads();
    const double thr = s_thr;
    // row i (register row v, owned by this warp) becomes pivot row i: publish it with its reciprocal
    auto publish = [&](int i, const double (&v)[NC]) {
        double g = v[0];
#pragma unroll
        for (int h = 1; h < NC; ++h)
            if (h == (i >> 5)) g = v[h];
        g = __shfl_sync(0xffffffffu, g, i & 31);
        const bool lost_i = !(g > thr);
#pragma unroll
        for (int h = 0; h < NC; ++h) urow[i & 1][lane + 32 * h] = v[h];
        if (lane == 0) {
            ginv[i & 1] = lost_i ? 0.0 : newton_rcp(g);
            gpiv[i] = lost_i ? 0.0 : g;
            if (lost_i) {
                if (lost) lost[s_nlost] = i;
                ++s_nlost;
                atomicOr(status, ST_RANKLOSS);
            }
        }
    };
    if (w == 0) publish(0, a[0]);
    __syncthreads();
    for (int j = 0; j + 1 < b; ++j) {
        const double gi = ginv[j & 1];
        const double* u = urow[j & 1];
        double uc[NC], f[NC];
#pragma unroll
        for (int h = 0; h < NC; ++h) {
            const int c = lane + 32 * h;
            uc[h] = c == j ? 1.0 : u[c];     // column j of the inverse's part: its unit diagonal
            f[h] = u[c] * gi;                // u_i / g_j for row i = c
        }
        // rows i > j: columns c <= j (inverse) and c >= i (G)
        auto update = [&](int i, double (&v)[NC]) {
            double fi = f[0];
#pragma unroll
            for (int h = 1; h < NC; ++h)
                if (h == (i >> 5)) fi = f[h];
            fi = __shfl_sync(0xffffffffu, fi, i & 31);
#pragma unroll
            for (int h = 0; h < NC; ++h) {
                // a 32-column slice strictly between the two parts holds nothing (uniform over the warp)
                if (32 * h > j && 32 * h + 31 < i) continue;
                const int c = lane + 32 * h;
                const double x = fma(-fi, uc[h], v[h]);
                if (c <= j || c >= i) v[h] = x;
            }
        };
        const int nx = j + 1;
        if ((nx & 7) == w) {
#pragma unroll
            for (int q = 0; q < NR; ++q)
                if (w + 8 * q == nx) {
                    update(nx, a[q]);
                    publish(nx, a[q]);
                }
        }
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            const int i = w + 8 * q;
            if (i > nx && i < b) update(i, a[q]);
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < b; i += blockDim.x) {
        const double g = gpiv[i];
        rdiag[i] = g > 0.0 ? 1.0 / sqrt(g) : 0.0;
        if (g > 0.0 && g < kCholWeak * diag0[i]) atomicAdd(&s_nweak, 1);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NR; ++q) {
        const int i = w + 8 * q;
        if (i >= b) break;
        const double sc = rdiag[i];
#pragma unroll
        for (int h = 0; h < NC; ++h) {
            const int c = lane + 32 * h;
            if (c >= b) continue;
            const double v = sc > 0.0 ? a[q][h] * sc : 0.0;   // a lost row of R, and of R^{-T}, is zero
            G[(int64_t)c * ldg + i] = c >= i ? v : 0.0;
            Rinv[(int64_t)i * b + c] = c < i ? v : (c == i ? sc : 0.0);
        }
    }
    if (threadIdx.x == 0 && lost) {
        lost[b] = s_nlost;
        lost[b + 1] = s_nweak;
        note_write(note, s_nlost, s_nweak);
    }
}

// The same by one CTA in global memory, for any b: two divisions a column and a back substitution.
__global__ void k_chol_inv(int b, double* G, int ldg, double* Rinv, double rank_tol, double piv_min2, int* status,
                           int* lost, const NoteRef note) {
    PDL_WAIT();
    PDL_ARG(G); PDL_ARG(Rinv); PDL_ARG(status); PDL_ARG(lost);
    __shared__ double maxdiag;
    __shared__ int nlost;
    __shared__ double piv;
    if (threadIdx.x == 0) {
        double mx = 0.0;
        bool bad = false;
        for (int j = 0; j < b; ++j) {
            const double g = G[(int64_t)j * ldg + j];
            if (!isfinite(g)) bad = true;
            mx = fmax(mx, fabs(g));
        }
        maxdiag = mx;
        nlost = 0;
        if (bad) atomicOr(status, ST_NONFINITE);
    }
    __syncthreads();
    const double thr = fmax(rank_tol * maxdiag, piv_min2);
    for (int j = 0; j < b; ++j) {
        if (threadIdx.x == 0) {
            const double g = G[(int64_t)j * ldg + j];
            if (!(g > thr) || maxdiag == 0.0) {
                piv = 0.0;
                if (lost) lost[nlost] = j;
                nlost++;
                atomicOr(status, ST_RANKLOSS);
            } else {
                piv = sqrt(g);
            }
            G[(int64_t)j * ldg + j] = piv;
        }
        __syncthreads();
        const double rjj = piv;
        // row j of R: G[j, c] / r_jj for c > j (upper triangle, column-major: G[c*ldg + j])
        for (int c = j + 1 + threadIdx.x; c < b; c += blockDim.x) {
            const double v = (rjj > 0.0) ? G[(int64_t)c * ldg + j] / rjj : 0.0;
            G[(int64_t)c * ldg + j] = v;
        }
        __syncthreads();
        // trailing update of the upper triangle: G[c1, c2] -= R[j, c1] R[j, c2], j < c1 <= c2
        const int rem = b - j - 1;
        for (int e = threadIdx.x; e < rem * rem; e += blockDim.x) {
            const int c1 = j + 1 + e % rem, c2 = j + 1 + e / rem;
            if (c1 <= c2) G[(int64_t)c2 * ldg + c1] -= G[(int64_t)c1 * ldg + j] * G[(int64_t)c2 * ldg + j];
        }
        __syncthreads();
    }
    // zero the strict lower triangle
    for (int e = threadIdx.x; e < b * b; e += blockDim.x) {
        const int r = e % b, c = e / b;
        if (r > c) G[(int64_t)c * ldg + r] = 0.0;
    }
    __syncthreads();
    // Rinv by back substitution, one column per thread
    for (int c = threadIdx.x; c < b; c += blockDim.x) {
        for (int i = b - 1; i >= 0; --i) {
            double v = (i == c) ? 1.0 : 0.0;
            if (i > c) v = 0.0;
            else {
                for (int l = i + 1; l <= c; ++l) v -= G[(int64_t)l * ldg + i] * Rinv[(int64_t)c * b + l];
                const double rii = G[(int64_t)i * ldg + i];
                v = (rii > 0.0) ? v / rii : 0.0;
            }
            Rinv[(int64_t)c * b + i] = v;
        }
    }
    if (!lost) return;
    if (threadIdx.x == 0) lost[b] = nlost;
    __shared__ int nweak;
    if (threadIdx.x == 0) nweak = 0;
    __syncthreads();
    for (int c = threadIdx.x; c < b; c += blockDim.x) {
        double sum = 0.0;   // the column's squared norm, from its column of R
        for (int r = 0; r <= c; ++r) sum = fma(G[(int64_t)c * ldg + r], G[(int64_t)c * ldg + r], sum);
        const double p = G[(int64_t)c * ldg + c];
        if (p > 0.0 && p * p < kCholWeak * sum) atomicAdd(&nweak, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        lost[b + 1] = nweak;
        note_write(note, nlost, nweak);
    }
}

// the register-resident factorisation up to this size (three 32-column slices a lane)
constexpr int kCholPairMax = 96;

template <class Ti, class To>
__global__ void k_copy(int64_t rows, int cols, const Ti* __restrict__ A, int64_t lda, To* __restrict__ B,
                       int64_t ldb) {
    PDL_ENTER();
    PDL_ARG(A); PDL_ARG(B);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= rows * cols) return;
    const int64_t r = e % rows, c = e / rows;
    B[c * ldb + r] = (To)A[c * lda + r];
}

__global__ void k_symmetrize(int m, double* A, int lda) {
    PDL_ENTER();
    PDL_ARG(A);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)m * m) return;
    const int r = (int)(e % m), c = (int)(e / m);
    if (r < c) {
        const double v = 0.5 * (A[(int64_t)c * lda + r] + A[(int64_t)r * lda + c]);
        A[(int64_t)c * lda + r] = v;
        A[(int64_t)r * lda + c] = v;
    }
}

// splitmix64 finaliser (Steele, Lea and Flood, 2014) as a counter-based generator.
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

template <class T>
__global__ void k_fill_gaussian(int64_t rows, int cols, T* A, int64_t lda, uint64_t seed, uint64_t sid) {
    PDL_ENTER();
    PDL_ARG(A);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= rows * cols) return;
    const int64_t r = e % rows, c = e / rows;
    const uint64_t h1 = mix64(seed ^ mix64(sid * 0x100000001B3ull + (uint64_t)e));
    const uint64_t h2 = mix64(h1 + 0x632BE59BD9B4E019ull);
    const double u1 = ((h1 >> 11) + 1) * (1.0 / 9007199254740993.0);   // (0, 1]
    const double u2 = (h2 >> 11) * (1.0 / 9007199254740992.0);         // [0, 1)
    A[c * lda + r] = (T)(sqrt(-2.0 * log(u1)) * cospi(2.0 * u2));       // Box-Muller
}

template <class T>
__global__ void k_col_norms(int64_t rows, const T* __restrict__ A, int64_t lda, double* out) {
    PDL_ENTER();
    PDL_ARG(A); PDL_ARG(out);
    const int c = blockIdx.x;
    double acc = 0.0;
    for (int64_t r = threadIdx.x; r < rows; r += blockDim.x) {
        const double v = (double)A[(int64_t)c * lda + r];
        acc = fma(v, v, acc);
    }
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        out[c] = sqrt(s);
    }
}

}  // namespace

namespace {

int g_sm_count = 0;   // streaming multiprocessors of the device the split counts are sized for

template <class T>
int gemm_tn_impl(int64_t d, int m, int p, double alpha, const T* A, int64_t lda, const T* B, int64_t ldb,
                 double beta, double* C, int ldc, void* partial_buf, size_t partial_cap, bool sym, cudaStream_t s) {
    if (m <= 0 || p <= 0) return EDA_OK;
    T* partial = static_cast<T*>(partial_buf);
    const int TP = sym ? TN_TM : (p <= 8 ? 8 : (p <= 16 ? 16 : 32));
    const int tm = ceil_div(m, TN_TM);
    const int tiles = sym ? tm * (tm + 1) / 2 : tm * ceil_div(p, TP);
    const int nsm = sm_count();
    // algorithmic work of this product, by the definition (one triangle for the symmetric case):
    // flops 2 d m p (SYRK: d m (m + 1)), bytes: A and B read once, C written once, in the storage type
    const double flops = sym ? (double)d * m * (m + 1.0) : 2.0 * (double)d * m * p;
    const double bytes = (double)sizeof(T) * (double)d * (sym ? m : (double)m + p) + 8.0 * m * p;
    ProfScope prof(std::is_same<T, double>::value ? "tn_f64" : "tn_f32", s, flops, bytes);
    if (sym && m <= SN_MAXM && d > 0) {
        // narrow blocks: one triangle of entries dealt to the lanes. Rows evenly over up to two CTAs per SM (a CTA with a
        // chunk more than the others would set the time), at least 64 a CTA
        int64_t G = std::max<int64_t>(1, std::min<int64_t>(2 * nsm, d / 64));
        while (G > 1 && (size_t)G * m * m > partial_cap) --G;
        if ((size_t)G * m * m > partial_cap) return EDA_ERR_INVALID_ARG;
        const int64_t rw = (d + G - 1) / G;
        G = (d + rw - 1) / rw;
        const int tri = m * (m + 1) / 2;
        const int cap = 32 * (m <= 8 ? 9 : (m <= 16 ? 17 : 33));
        int R = 32;
        while (R * tri > cap) R >>= 1;
        if (m <= 8) EDA_CUDA_TRY((launch_spread(k_syrk_narrow<9, 256, 8, T>, dim3((unsigned)G), dim3(SN_THREADS), 0, s,
            d, m, A, lda, rw, R, partial)));
        else if (m <= 16) EDA_CUDA_TRY((launch_spread(k_syrk_narrow<17, 128, 16, T>, dim3((unsigned)G), dim3(SN_THREADS),
            0, s, d, m, A, lda, rw, R, partial)));
        else EDA_CUDA_TRY((launch_spread(k_syrk_narrow<33, 64, 32, T>, dim3((unsigned)G), dim3(SN_THREADS), 0, s, d, m,
            A, lda, rw, R, partial)));
        const int64_t out = (int64_t)m * m;
        if (G >= 16)
            EDA_CUDA_TRY((launch_chained(k_gemm_tn_reduce_warp<T>, dim3(ceil_div(out * 32, 256)), dim3(256), 0, s, m, m,
                (int)G, partial, alpha, beta, C, ldc,
            true)));
        else
            EDA_CUDA_TRY((launch_chained(k_gemm_tn_reduce<T>, dim3(ceil_div(out, 256)), dim3(256), 0, s, m, m, (int)G,
                partial, alpha, beta, C, ldc, true)));
        return EDA_OK;
    }
    // Split count: the kernel is FP64- or bandwidth-bound per SM, so an SM holding one CTA more than
    // the others sets the time. Among counts giving 1.8 to 4 CTAs per SM (after rounding the split
    // rows to TN_KB), take the one that fills the SMs most evenly, tiles * splits over
    // nsm * ceil(tiles * splits / nsm), preferring fewer splits unless another fills 2 % better.
    int splits = 1;
    {
        const int smax = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(4 * nsm, tiles), (d + 63) / 64));
        const int smin = std::min(smax, std::max(1, (int)std::ceil(1.8 * nsm / tiles)));
        double best = -1.0;
        for (int s0 = smin; s0 <= smax; ++s0) {
            int64_t rw = (d + s0 - 1) / s0;
            rw = (rw + TN_KB - 1) / TN_KB * TN_KB;
            const int sc = (int)std::max<int64_t>(1, (d + rw - 1) / rw);
            const int64_t ctas = (int64_t)tiles * sc;
            const double fill = (double)ctas / ((double)nsm * (double)((ctas + nsm - 1) / nsm));
            if (fill > best + 0.02) {
                best = fill;
                splits = sc;
            }
        }
    }
    while (splits > 1 && (size_t)splits * m * p > partial_cap) --splits;
    if ((size_t)splits * m * p > partial_cap) return EDA_ERR_INVALID_ARG;
    int64_t rows = (d + splits - 1) / splits;
    rows = (rows + TN_KB - 1) / TN_KB * TN_KB;
    splits = (int)std::max<int64_t>(1, (d + rows - 1) / rows);
    if (d > 0) {
        if (sym) {
            dim3 grid(tiles, 1, splits);
            EDA_CUDA_TRY((launch_spread(k_gemm_tn_partial<32, T, true>, grid, dim3(TN_THREADS), 0, s, d, m, p, A, lda, B,
                ldb, rows, partial)));
        } else {
            dim3 grid(tm, ceil_div(p, TP), splits);
            if (TP == 8) EDA_CUDA_TRY((launch_spread(k_gemm_tn_partial<8, T>, grid, dim3(TN_THREADS), 0, s, d, m, p, A,
                lda, B, ldb, rows, partial)));
            else if (TP == 16) EDA_CUDA_TRY((launch_spread(k_gemm_tn_partial<16, T>, grid, dim3(TN_THREADS), 0, s, d, m,
                p, A, lda, B, ldb, rows, partial)));
            else EDA_CUDA_TRY((launch_spread(k_gemm_tn_partial<32, T>, grid, dim3(TN_THREADS), 0, s, d, m, p, A, lda, B,
                ldb, rows, partial)));
        }
    } else {
        splits = 0;
    }
    const int64_t tot = (int64_t)m * p;
    if (splits >= 16 && tot <= 65536)
        EDA_CUDA_TRY((launch_chained(k_gemm_tn_reduce_warp<T>, dim3(ceil_div(tot * 32, 256)), dim3(256), 0, s, m, p,
            splits, partial, alpha, beta, C, ldc,
            sym)));
    else
        EDA_CUDA_TRY((launch_chained(k_gemm_tn_reduce<T>, dim3(ceil_div(tot, 256)), dim3(256), 0, s, m, p, splits,
            partial, alpha, beta, C, ldc, sym)));
    return EDA_OK;
}

}  // namespace

int sm_count() {
    // queried once per process for the current device (every handle of a process uses one GPU type)
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0)
            g_sm_count = n;
        else
            g_sm_count = 148;
        cudaGetLastError();
    });
    return g_sm_count;
}

template <class T>
int gemm_tn(int64_t d, int m, int p, double alpha, const T* A, int64_t lda, const T* B, int64_t ldb, double beta,
            double* C, int ldc, void* partial_buf, size_t partial_cap, cudaStream_t s) {
    return gemm_tn_impl<T>(d, m, p, alpha, A, lda, B, ldb, beta, C, ldc, partial_buf, partial_cap, false, s);
}

template <class T>
int syrk_tn(int64_t d, int m, double alpha, const T* A, int64_t lda, double beta, double* C, int ldc,
            void* partial_buf, size_t partial_cap, cudaStream_t s) {
    return gemm_tn_impl<T>(d, m, m, alpha, A, lda, A, lda, beta, C, ldc, partial_buf, partial_cap, true, s);
}

template <class T>
int gemm_nn(int64_t d, int m, int p, double alpha, const T* A, int64_t lda, const double* B, int ldb, double beta,
            const T* C0, int64_t ldc0, T* C, int64_t ldc, cudaStream_t s, bool b_upper) {
    if (d <= 0 || p <= 0) return EDA_OK;
    // algorithmic work: 2 d m p flops (2 d sum_c min(m, c + 1) for an upper triangular B); A read once,
    // C0 read (beta != 0) and C written once
    double terms = (double)m * p;
    if (b_upper) {
        terms = 0.0;
        for (int c = 0; c < p; ++c) terms += std::min(m, c + 1);
    }
    ProfScope prof(std::is_same<T, double>::value ? "nn_f64" : "nn_f32", s, 2.0 * (double)d * terms,
                   (double)sizeof(T) * (double)d * (m + (beta != 0.0 ? 2.0 : 1.0) * p) + 8.0 * m * p);
    const int ub = b_upper ? 1 : 0;
    const int rowblocks = ceil_div(d, 32);
    // columns per thread: as many as possible while at least ~one CTA per SM stays busy
    if (p >= 6 && m <= kNnWholeM && (int64_t)rowblocks * ceil_div(p, 8) >= 4 * sm_count()) {
        EDA_CUDA_TRY((launch_spread(k_gemm_nn<8, T, 1>, dim3(ceil_div(rowblocks, 8), ceil_div(p, 8)), dim3(256), 0, s, d, m, p,
            alpha, A, lda, B, ldb, beta, C0, ldc0, C, ldc, ub)));
    } else if (p >= 6 && (int64_t)rowblocks * ceil_div(p, 8) >= 120) {
        EDA_CUDA_TRY((launch_spread(k_gemm_nn<8, T>, dim3(rowblocks, ceil_div(p, 8)), dim3(256), 0, s, d, m, p, alpha, A,
            lda, B, ldb, beta, C0, ldc0, C, ldc, ub)));
    } else if (p >= 3 && (int64_t)rowblocks * ceil_div(p, 4) >= 120) {
        EDA_CUDA_TRY((launch_spread(k_gemm_nn<4, T>, dim3(rowblocks, ceil_div(p, 4)), dim3(256), 0, s, d, m, p, alpha, A,
            lda, B, ldb, beta, C0, ldc0, C, ldc, ub)));
    } else if (p >= 2) {
        EDA_CUDA_TRY((launch_spread(k_gemm_nn<2, T>, dim3(rowblocks, ceil_div(p, 2)), dim3(256), 0, s, d, m, p, alpha, A,
            lda, B, ldb, beta, C0, ldc0, C, ldc, ub)));
    } else {
        EDA_CUDA_TRY((launch_spread(k_gemm_nn<1, T>, dim3(rowblocks, p), dim3(256), 0, s, d, m, p, alpha, A, lda, B, ldb,
            beta, C0, ldc0, C, ldc, ub)));
    }
    return EDA_OK;
}

template <class Ti, class To>
int copy_mat(int64_t rows, int cols, const Ti* A, int64_t lda, To* B, int64_t ldb, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_copy<Ti, To>, dim3(ceil_div(rows * cols, 256)), dim3(256), 0, s, rows, cols, A, lda,
        B, ldb)));
    return EDA_OK;
}

template <class T>
int fill_gaussian(int64_t rows, int cols, T* A, int64_t lda, uint64_t seed, uint64_t stream_id, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_fill_gaussian<T>, dim3(ceil_div(rows * cols, 256)), dim3(256), 0, s, rows, cols, A,
        lda, seed, stream_id)));
    return EDA_OK;
}

template <class T>
int col_norms(int64_t rows, int cols, const T* A, int64_t lda, double* out, cudaStream_t s) {
    if (cols <= 0) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_col_norms<T>, dim3(cols), dim3(256), 0, s, rows, A, lda, out)));
    return EDA_OK;
}

template int gemm_tn<double>(int64_t, int, int, double, const double*, int64_t, const double*, int64_t, double,
                             double*, int, void*, size_t, cudaStream_t);
template int gemm_tn<float>(int64_t, int, int, double, const float*, int64_t, const float*, int64_t, double,
                            double*, int, void*, size_t, cudaStream_t);
template int syrk_tn<double>(int64_t, int, double, const double*, int64_t, double, double*, int, void*, size_t,
                             cudaStream_t);
template int syrk_tn<float>(int64_t, int, double, const float*, int64_t, double, double*, int, void*, size_t,
                            cudaStream_t);
template int gemm_nn<double>(int64_t, int, int, double, const double*, int64_t, const double*, int, double,
                             const double*, int64_t, double*, int64_t, cudaStream_t, bool);
template int gemm_nn<float>(int64_t, int, int, double, const float*, int64_t, const double*, int, double,
                            const float*, int64_t, float*, int64_t, cudaStream_t, bool);
template int copy_mat<double, double>(int64_t, int, const double*, int64_t, double*, int64_t, cudaStream_t);
template int copy_mat<float, float>(int64_t, int, const float*, int64_t, float*, int64_t, cudaStream_t);
template int copy_mat<double, float>(int64_t, int, const double*, int64_t, float*, int64_t, cudaStream_t);
template int copy_mat<float, double>(int64_t, int, const float*, int64_t, double*, int64_t, cudaStream_t);
template int fill_gaussian<double>(int64_t, int, double*, int64_t, uint64_t, uint64_t, cudaStream_t);
template int fill_gaussian<float>(int64_t, int, float*, int64_t, uint64_t, uint64_t, cudaStream_t);
template int col_norms<double>(int64_t, int, const double*, int64_t, double*, cudaStream_t);
template int col_norms<float>(int64_t, int, const float*, int64_t, double*, cudaStream_t);

int gemm_tn_f64(int64_t d, int m, int p, double alpha, const double* A, int64_t lda, const double* B, int64_t ldb,
                double beta, double* C, int ldc, double* partial, size_t partial_cap, cudaStream_t s) {
    return gemm_tn<double>(d, m, p, alpha, A, lda, B, ldb, beta, C, ldc, partial, partial_cap, s);
}

int syrk_f64(int64_t d, int m, double alpha, const double* A, int64_t lda, double beta, double* C, int ldc,
             double* partial, size_t partial_cap, cudaStream_t s) {
    return syrk_tn<double>(d, m, alpha, A, lda, beta, C, ldc, partial, partial_cap, s);
}

int gemm_nn_f64(int64_t d, int m, int p, double alpha, const double* A, int64_t lda, const double* B, int ldb,
                double beta, const double* C0, int64_t ldc0, double* C, int64_t ldc, cudaStream_t s) {
    return gemm_nn<double>(d, m, p, alpha, A, lda, B, ldb, beta, C0, ldc0, C, ldc, s);
}

int gemm_small_f64(bool ta, bool tb, int m, int p, int kk, double alpha, const double* A, int lda, const double* B,
                   int ldb, double beta, double* C, int ldc, cudaStream_t s) {
    if (m <= 0 || p <= 0) return EDA_OK;
    if (!ta && !tb && kk >= 64) {
        EDA_CUDA_TRY((launch_chained(k_gemm_small_nn_splitk<false>, dim3(ceil_div(m, 32), p), dim3(32 * kSplitkWarps), 0,
            s, m, p, kk, alpha, A, lda, B, ldb,
            beta, C, ldc)));
        return EDA_OK;
    }
    // one warp per CTA (32 rows of one column): FP64 work spreads over all SMs
    dim3 blk(32, 1), grid(ceil_div(m, 32), p);
    EDA_CUDA_TRY((launch_spread(k_gemm_small, grid, blk, 0, s, ta, tb, m, p, kk, alpha, A, lda, B, ldb, beta, C, ldc)));
    return EDA_OK;
}

int gemm_small_sym_f64(int m, double alpha, const double* A, int lda, const double* B, int ldb, double beta, double* C,
                       int ldc, cudaStream_t s) {
    if (m < 64) return gemm_small_f64(false, false, m, m, m, alpha, A, lda, B, ldb, beta, C, ldc, s);
    const int nb = ceil_div(m, 32);
    EDA_CUDA_TRY((launch_spread(k_gemm_small_nn_splitk<true>, dim3(32 * (nb * (nb + 1) / 2)), dim3(32 * kSplitkWarps), 0,
        s, m, m, m, alpha, A, lda, B, ldb,
            beta, C, ldc)));
    return EDA_OK;
}

int chol_inv_small(int b, double* G, int ldg, double* Rinv, double rank_tol, double piv_min2, int* status, int* lost,
                   cudaStream_t s, const NoteRef& note) {
    if (b <= 32)
        EDA_CUDA_TRY((launch_chained(k_chol_inv_pair<1>, dim3(1), dim3(256), 0, s, b, G, ldg, Rinv, rank_tol, piv_min2,
            status, lost, note)));
    else if (b <= 64)
        EDA_CUDA_TRY((launch_chained(k_chol_inv_pair<2>, dim3(1), dim3(256), 0, s, b, G, ldg, Rinv, rank_tol, piv_min2,
            status, lost, note)));
    else if (b <= kCholPairMax)
        EDA_CUDA_TRY((launch_chained(k_chol_inv_pair<3>, dim3(1), dim3(256), 0, s, b, G, ldg, Rinv, rank_tol, piv_min2,
            status, lost, note)));
    else
        EDA_CUDA_TRY((launch_chained(k_chol_inv, dim3(1), dim3(256), 0, s, b, G, ldg, Rinv, rank_tol, piv_min2, status,
            lost, note)));
    return EDA_OK;
}

namespace {
// B (rows x cols, ldb) = 0 below the diagonal (strict lower triangle of a square or tall block)
__global__ void k_zero_lower(int m, double* A, int lda) {
    PDL_ENTER();
    PDL_ARG(A);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)m * m) return;
    const int r = (int)(e % m), c = (int)(e / m);
    if (r > c) A[(int64_t)c * lda + r] = 0.0;
}
__global__ void k_zero_all(int m, double* A, int lda) {
    PDL_ENTER();
    PDL_ARG(A);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)m * m) return;
    A[(int64_t)(e / m) * lda + e % m] = 0.0;
}
}  // namespace

size_t chol_inv_blocked_doubles(int m) { return (size_t)kCholBlock * m + (size_t)kCholBlock * kCholBlock; }

// Right-looking blocked Cholesky G = R^T R (R upper, in place, strict lower triangle zeroed) and R^{-1}, in
// blocks of kCholBlock: the diagonal block by the one-CTA factorisation (with its rank detection), the row
// panel R12 = R11^{-T} G12 and the trailing update G22 -= R12^T R12 as multi-CTA products; then R^{-1} block
// column by block column, X[:j, j] = -X[:j, :j] R[:j, j] R_jj^{-1}. work: chol_inv_blocked_doubles(m);
// partial: split-K partials of at least m * m doubles.
int chol_inv_blocked(int m, double* G, int ldg, double* Rinv, int ldr, double rank_tol, int* status, double* work,
                     double* partial, size_t pcap, cudaStream_t s) {
    constexpr int NB = kCholBlock;
    double* T = work;                          // NB x m
    double* Dinv = work + (size_t)NB * m;      // NB x NB
    // R^{-1} starts as zero: its blocks below the block diagonal are never written and are read as zeros
    EDA_CUDA_TRY((launch_chained(k_zero_all, dim3(ceil_div((int64_t)m * m, 256)), dim3(256), 0, s, m, Rinv, ldr)));
    for (int j0 = 0; j0 < m; j0 += NB) {
        const int nb = std::min(NB, m - j0);
        double* G11 = G + (int64_t)j0 * ldg + j0;
        EDA_TRY(chol_inv_small(nb, G11, ldg, Dinv, rank_tol, 0.0, status, nullptr, s));
        // R^{-1} diagonal block
        EDA_TRY(copy_mat_f64(nb, nb, Dinv, nb, Rinv + (int64_t)j0 * ldr + j0, ldr, s));
        const int r = m - j0 - nb;
        if (r > 0) {
            double* G12 = G + (int64_t)(j0 + nb) * ldg + j0;
            double* G22 = G + (int64_t)(j0 + nb) * ldg + j0 + nb;
            // R12 = R11^{-T} G12
            EDA_TRY(gemm_small_f64(true, false, nb, r, nb, 1.0, Dinv, nb, G12, ldg, 0.0, T, nb, s));
            EDA_TRY(copy_mat_f64(nb, r, T, nb, G12, ldg, s));
            // G22 -= R12^T R12 (a product reduced over the nb rows of R12)
            EDA_TRY(gemm_tn_f64(nb, r, r, -1.0, G12, ldg, G12, ldg, 1.0, G22, ldg, partial, pcap, s));
        }
    }
    EDA_CUDA_TRY((launch_chained(k_zero_lower, dim3(ceil_div((int64_t)m * m, 256)), dim3(256), 0, s, m, G, ldg)));
    // off-diagonal blocks of R^{-1}: X[:j0, j-block] = -X[:j0, :j0] (R[:j0, j-block] R_jj^{-1})
    for (int j0 = NB; j0 < m; j0 += NB) {
        const int nb = std::min(NB, m - j0);
        const double* Rj = G + (int64_t)j0 * ldg;                       // R[:j0, j-block]
        const double* Xjj = Rinv + (int64_t)j0 * ldr + j0;              // R_jj^{-1}
        EDA_TRY(gemm_small_f64(false, false, j0, nb, nb, 1.0, Rj, ldg, Xjj, ldr, 0.0, T, j0, s));
        EDA_TRY(gemm_small_f64(false, false, j0, nb, j0, -1.0, Rinv, ldr, T, j0, 0.0, Rinv + (int64_t)j0 * ldr, ldr,
                               s));
    }
    return EDA_OK;
}

int chol_inv_auto(int b, double* G, int ldg, double* Rinv, double rank_tol, int* status, double* work, double* partial,
                  size_t pcap, cudaStream_t s) {
    if (b <= kCholPairMax) return chol_inv_small(b, G, ldg, Rinv, rank_tol, 0.0, status, nullptr, s);
    return chol_inv_blocked(b, G, ldg, Rinv, b, rank_tol, status, work, partial, pcap, s);
}

int copy_mat_f64(int64_t rows, int cols, const double* A, int64_t lda, double* B, int64_t ldb, cudaStream_t s) {
    return copy_mat<double, double>(rows, cols, A, lda, B, ldb, s);
}

int symmetrize_f64(int m, double* A, int lda, cudaStream_t s) {
    if (m <= 1) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_symmetrize, dim3(ceil_div((int64_t)m * m, 256)), dim3(256), 0, s, m, A, lda)));
    return EDA_OK;
}

int fill_gaussian_f64(int64_t rows, int cols, double* A, int64_t lda, uint64_t seed, uint64_t stream_id,
                      cudaStream_t s) {
    return fill_gaussian<double>(rows, cols, A, lda, seed, stream_id, s);
}

int col_norms_f64(int64_t rows, int cols, const double* A, int64_t lda, double* out, cudaStream_t s) {
    return col_norms<double>(rows, cols, A, lda, out, s);
}

}  // namespace eda
