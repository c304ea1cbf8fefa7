// FP64 symmetric eigensolver for the small matrices of the method: the Gram matrices
// G = H^T H (the spectra D = Sigma^2 of Eqs. (3.4)-(3.6)) and the block-tridiagonal Lanczos
// matrix T of the Rayleigh-Ritz step.
//
// Route: Householder reduction to tridiagonal form (from n = 288 a cooperative grid with the columns
// resident in its CTAs' shared memory; below that, or when the GPU is shared, one thread-block cluster;
// beyond what shared memory holds, a cooperative grid streaming the matrix through L2; all with bounded
// waits) -> eigenvalues by 33-way
// multisection on Sturm counts (one warp per eigenvalue) -> eigenvectors of the tridiagonal
// by inverse iteration with partial pivoting (one thread per eigenvector) -> modified
// Gram-Schmidt inside tight clusters (one warp per cluster) -> back-transformation with the
// stored reflectors. Callers add a Newton-Schulz step for orthogonality across near clusters.
#include "eda_internal.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <cfloat>
#include <cmath>

namespace eda {

namespace {

constexpr int TRI_THREADS = 256;

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Bounded grid-wide barrier for a cooperative launch. On timeout it records ST_TIMEOUT and
// returns; the kernel then runs to completion with stale data and the host reports the error.
__device__ void grid_sync(GridBarrier bar, int* status) {
    if (gridDim.x == 1) {
        __syncthreads();
        return;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned g = ld_acquire_u32(bar.gen);
        __threadfence();
        const unsigned ticket = atomicAdd(bar.count, 1u);
        if (ticket == gridDim.x - 1) {
            atomicExch(bar.count, 0u);
            __threadfence();
            atomicAdd(bar.gen, 1u);
        } else {
            long long it = 0;
            while (ld_acquire_u32(bar.gen) == g) {
                if (++it > bar.spin_limit) {
                    atomicOr(status, ST_TIMEOUT);
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    __syncthreads();
}

__device__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    // pairwise tree over the warps: the same fixed order in every thread and every CTA
    const int nw = blockDim.x >> 5;
    if (nw == 4) return (red[0] + red[1]) + (red[2] + red[3]);
    if (nw == 8) return ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
    double sacc = 0.0;
    for (int i = 0; i < nw; ++i) sacc += red[i];
    return sacc;
}

// Householder tridiagonalisation of the full symmetric n x n matrix A (ld n), in place.
// HV[j * n + i] receives reflector j (u_j[j+1] = 1, zero above), tau[j] its scalar.
// vbuf: 2n doubles (p vector and a copy of the current column).
__global__ void __launch_bounds__(TRI_THREADS) k_tridiag(int n, double* A, double* HV, double* dgl, double* eoff,
                                                         double* tau, double* pglob, GridBarrier bar, int* status) {
    extern __shared__ double sm[];
    double* v = sm;          // n
    double* w = sm + n;      // n
    __shared__ double red[32];
    const int C = gridDim.x, cta = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;

    for (int j = 0; j + 2 < n; ++j) {
        const int i0 = j + 1;                // trailing block starts here
        // ---- Householder vector of column j (computed redundantly by every CTA) ----
        double ss = 0.0;
        for (int i = i0 + 1 + threadIdx.x; i < n; i += blockDim.x) {
            const double x = A[(int64_t)j * n + i];
            ss = fma(x, x, ss);
        }
        ss = block_sum(ss, red);
        const double alpha = A[(int64_t)j * n + i0];
        double beta, tj, scal;
        if (ss == 0.0) {
            beta = alpha;
            tj = 0.0;
            scal = 0.0;
        } else {
            beta = -copysign(sqrt(fma(alpha, alpha, ss)), alpha);
            tj = (beta - alpha) / beta;
            scal = 1.0 / (alpha - beta);
        }
        for (int i = i0 + threadIdx.x; i < n; i += blockDim.x)
            v[i] = (i == i0) ? 1.0 : A[(int64_t)j * n + i] * scal;
        __syncthreads();
        if (cta == 0) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) HV[(int64_t)j * n + i] = (i >= i0) ? v[i] : 0.0;
            if (threadIdx.x == 0) {
                eoff[j] = beta;
                tau[j] = tj;
            }
        }
        if (tj == 0.0) {
            grid_sync(bar, status);   // keep every CTA on the same barrier count
            grid_sync(bar, status);
            continue;
        }
        // ---- p[r] = tau * sum_c A[c, r] v[c] for owned rows r (column r is contiguous) ----
        for (int r = i0 + cta + C * warp; r < n; r += C * nwarps) {
            double acc = 0.0;
            const double* col = A + (int64_t)r * n;
            for (int c = i0 + lane; c < n; c += 32) acc = fma(col[c], v[c], acc);
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
            if (lane == 0) pglob[r] = tj * acc;
        }
        grid_sync(bar, status);
        // ---- w = p - (tau/2)(p^T v) v, then A22 -= v w^T + w v^T on owned columns ----
        double pv = 0.0;
        for (int i = i0 + threadIdx.x; i < n; i += blockDim.x) {
            const double pi = pglob[i];
            w[i] = pi;
            pv = fma(pi, v[i], pv);
        }
        pv = block_sum(pv, red);
        const double kk = 0.5 * tj * pv;
        for (int i = i0 + threadIdx.x; i < n; i += blockDim.x) w[i] = fma(-kk, v[i], w[i]);
        __syncthreads();
        for (int r = i0 + cta + C * warp; r < n; r += C * nwarps) {
            double* col = A + (int64_t)r * n;
            const double vr = v[r], wr = w[r];
            for (int c = i0 + lane; c < n; c += 32) col[c] -= fma(v[c], wr, w[c] * vr);
        }
        grid_sync(bar, status);
    }
    if (cta == 0) {
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            dgl[i] = A[(int64_t)i * n + i];
            if (i + 2 >= n) {
                if (i + 1 < n) eoff[i] = A[(int64_t)i * n + i + 1];
                tau[i] = 0.0;
                for (int r = 0; r < n; ++r) HV[(int64_t)i * n + r] = 0.0;
            }
        }
        if (threadIdx.x == 0) eoff[n - 1] = 0.0;
    }
}

// Householder tridiagonalisation with one exchange between CTAs per column, on a cooperative grid (CL = false) or
// in one thread-block cluster (CL = true). Column r of the symmetric matrix is owned by CTA r % G and stays in its
// shared memory (in a cluster, for large n, in a global slab of that CTA).
//
// Every CTA holds the current column x = A[c.., c] and forms its reflector itself: v = x - beta e_{c+1} (rows
// c + 1.., unscaled), H = I - tau v v^T with tau = 1 / (beta (beta - alpha)). What the CTAs exchange for column c is
// p = tau A v, each entry from the owner of its row, and the next column A[.., c + 1] before its update, from its owner.
// From these every CTA forms, with the same operations in the same order,
//     K = (tau / 2) v^T p,  w = p - K v,  x' = A[.., c + 1] - v w_{c+1} - w v_{c+1},  ||x'||
// and then updates its own columns (A <- A - v w^T - w v^T) and multiplies them by x' in the same pass; the reflector's
// scalars beta', tau' are formed by one warp beside that pass and applied afterwards, A v' = A x' - beta' A e_{c+2}.
//
// What bounds it: per column one exchange and a chain of FP64 instructions (each holds a sub-partition's pipe for about
// 64 cycles whatever the number of lanes), so the design spends CTA-wide redundant work to have one exchange instead of
// two, keeps square root and reciprocal beside the pass, and reduces with one warp per sub-partition.
//   Grid: the exchanged values are written once to their own place (row c of two n x n buffers, filled before the launch
// with a bit pattern that no result has) and polled there by the reader: no barrier, flag or fence is on the path, each
// value vouches for itself. The polls are bounded (ST_TIMEOUT); a thread that gave up once does not wait again.
//   Cluster: entries in the owners' shared memory, read through distributed shared memory after one cluster barrier;
// p is double-buffered, and a column is never written again once it is next.
// GB300, against two barriers (or cluster barriers) per column and the reflector formed by its owner alone: grid n = 700
// 7.66 -> 4.62 ms, n = 668 7.13 -> 4.30 ms; cluster n = 144 0.95 -> 0.51 ms, n = 100 0.55 -> 0.33 ms.
constexpr int TD_WARPS = 8;                             // warps that share the owned columns; one more forms the scalars
constexpr int TD_THREADS = 32 * TD_WARPS + 32;
constexpr int TD_RED = 128;                             // threads (one warp per sub-partition) of the vector work

// Warps per owned column in the pass over the columns: enough tasks to even out the sub-partitions.
__host__ __device__ inline int td_split(int ncl) { return ncl >= TD_WARPS ? 1 : (ncl > 4 ? 4 : 2); }
__host__ __device__ inline int td_dots(int ncl) { return ncl * 32 * td_split(ncl); }
constexpr unsigned long long TD_EMPTY = ~0ull;          // "not written yet": a NaN with this payload is never stored

__device__ __forceinline__ unsigned long long td_ld(const double* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void td_st(double* p, double x) {
    unsigned long long v = (unsigned long long)__double_as_longlong(x);
    if (v == TD_EMPTY) v = 0x7FF8000000000000ull;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// 1 / x for a positive normal x: PTX rcp.approx.ftz.f64 (20 bits) and two Newton-Raphson steps; the IEEE division where x
// or 1 / x leaves the approximation's range.
__device__ __forceinline__ double td_rcp(double x) {
    const int ex = (__double2hiint(x) >> 20) & 0x7ff;
    if (ex < 24 || ex > 2022) return 1.0 / x;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}

// sqrt(x), x >= 0: PTX rsqrt.approx.ftz.f64 and two Goldschmidt steps on g ~ sqrt(x), h ~ 1 / (2 sqrt(x))
// (r = 1/2 - g h, g <- g + g r, h <- h + h r); the library's square root outside the approximation's range.
__device__ __forceinline__ double td_sqrt(double x) {
    const int ex = (__double2hiint(x) >> 20) & 0x7ff;
    if (ex < 24 || ex > 2022) return sqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double g = x * y, h = 0.5 * y;
    double r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    h = fma(h, r, h);
    r = fma(-g, h, 0.5);
    return fma(g, r, g);
}

template <bool CL>
__global__ void __launch_bounds__(TD_THREADS) k_tridiag_x(int n, const double* __restrict__ Ain, int lda, double* Aglob,
                                                          int in_smem, double* pbuf, double* cbuf, double* HV, double* dgl,
                                                          double* eoff, double* tau, long long spin, int* status) {
    namespace cg = cooperative_groups;
    extern __shared__ double sm[];
    __shared__ double red[2][TD_RED / 32];   // partial sums of v^T p and of ||x'||^2
    __shared__ double s_pc, s_alpha;         // p_c; x'_{c+1}
    __shared__ double s_beta, s_tau, s_htau, s_v1;   // the current reflector: beta, tau, tau / 2, v_{c+1}
    const int G = gridDim.x, cta = blockIdx.x;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int NW = TD_WARPS;
    const int ncl = (n + G - 1) / G;
    double* vs = sm;                     // n: reflector of the previous column (entries below its first)
    double* xs = sm + n;                 // n: the current column
    double* ws = sm + 2 * n;             // n: p, then w
    const int split = td_split(ncl);
    double* sdot = sm + 3 * n;             // ncl x (32 split): the lanes' partial sums of A x
    double* pin = sdot + td_dots(ncl);     // cluster: 2 x n, p of this column and of the next (written by all CTAs)
    double* Aloc = CL ? (in_smem ? pin + 2 * n : Aglob + (size_t)cta * ncl * n) : pin;

    for (int q = 0; q < ncl; ++q) {
        const int r = q * G + cta;
        if (r >= n) break;
        for (int i = tid; i < n; i += TD_THREADS)
            Aloc[(size_t)q * n + i] = 0.5 * (Ain[(int64_t)r * lda + i] + Ain[(int64_t)i * lda + r]);
    }
    for (int i = tid; i < n; i += TD_THREADS) {
        vs[i] = 0.0;
        ws[i] = 0.0;
        xs[i] = 0.5 * (Ain[i] + Ain[(int64_t)i * lda]);
    }
    if (tid == 0) s_tau = s_htau = s_v1 = 0.0;
    __syncthreads();

    for (int c = 0; c + 1 < n; ++c) {
        double ss = 0.0;
        if (c > 0) {
            // ---- p (warps 0-3) and the raw column c (warps 4-7) into ws and xs; v^T p ----
            const bool first = tid < TD_RED;   // the last warp (the scalars') takes no part
            double acc = 0.0;
            double* dst = first ? ws : xs;
            const double vc = s_v1;
            auto take = [&](int i, double x) {
                dst[i] = x;
                if (first) {
                    acc = fma(i == c ? vc : vs[i], x, acc);
                    if (i == c) s_pc = x;
                }
            };
            if (CL) {
                cg::cluster_group cluster = cg::this_cluster();
                const int oc = c & (G - 1);   // a cluster's size is a power of two
                const double* own = in_smem ? cluster.map_shared_rank(Aloc, oc) : Aglob + (size_t)oc * ncl * n;
                const double* col = own + (size_t)(c / G) * n;
                const double* src = first ? pin + ((c - 1) & 1) * n : col;
                if (warp < NW)
                    for (int i = c + (tid & (TD_RED - 1)); i < n; i += TD_RED) take(i, src[i]);
            } else if (warp < NW) {
                const double* src = (first ? pbuf : cbuf) + (size_t)(c - 1) * n;
                // one lane waits for its value before the warp reads all of them: the polls of every lane of every CTA
                // would slow down the writes that they wait for
                if (lane == 0 && c + tid % TD_RED < n) {
                    long long polls = 0;
                    while (td_ld(src + c + tid % TD_RED) == TD_EMPTY && spin >= 0 && ++polls <= spin) {
                    }
                }
                __syncwarp();
                for (int i0 = c + (tid & (TD_RED - 1)); i0 < n; i0 += 4 * TD_RED) {
                    unsigned long long u[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) u[k] = i0 + k * TD_RED < n ? td_ld(src + i0 + k * TD_RED) : 0ull;
                    long long polls = 0;
                    while (u[0] == TD_EMPTY || u[1] == TD_EMPTY || u[2] == TD_EMPTY || u[3] == TD_EMPTY) {
                        if (++polls > spin) {
                            if (spin >= 0) atomicOr(status, ST_TIMEOUT);
                            spin = -1;   // this thread does not wait again
                            break;
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (u[k] == TD_EMPTY) u[k] = td_ld(src + i0 + k * TD_RED);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (i0 + k * TD_RED < n) take(i0 + k * TD_RED, __longlong_as_double((long long)u[k]));
                }
            }
            if (first) {
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0) red[0][warp] = acc;
            }
            __syncthreads();
            // ---- w and the finished column x' ----
            if (first) {
                const double K = s_htau * ((red[0][0] + red[0][1]) + (red[0][2] + red[0][3]));
                const double wc = fma(-K, vc, s_pc);
                for (int i = c + tid; i < n; i += TD_RED) {
                    const double vi = i == c ? vc : vs[i];
                    const double wi = fma(-K, vi, ws[i]);
                    const double xi = fma(-wi, vc, fma(-vi, wc, xs[i]));
                    ws[i] = wi;
                    xs[i] = xi;
                    if (i >= c + 2) ss = fma(xi, xi, ss);
                    if (i == c + 1) s_alpha = xi;
                    if (i == c && cta == 0) dgl[c] = xi;
                }
            } else if (warp < NW && cta == (c - 1) % G) {
                // the previous reflector, for the back-transformation
                for (int i = tid - TD_RED; i < n; i += TD_RED)
                    HV[(int64_t)(c - 1) * n + i] = i < c ? 0.0 : (i == c ? vc : vs[i]);
            }
        } else if (tid < TD_RED) {
            for (int i = tid; i < n; i += TD_RED) {
                const double xi = xs[i];
                if (i >= 2) ss = fma(xi, xi, ss);
                if (i == 1) s_alpha = xi;
                if (i == 0 && cta == 0) dgl[0] = xi;
            }
        }
        if (tid < TD_RED) {
            for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (lane == 0) red[1][warp] = ss;
        }
        __syncthreads();
        if (c + 2 == n) break;
        // ---- the reflector's scalars (one warp) beside the update of the owned columns and their products with x' ----
        if (warp == NW) {
            const double alpha = s_alpha;
            const double sig = (red[1][0] + red[1][1]) + (red[1][2] + red[1][3]);
            double beta = alpha, t = 0.0, v1 = 0.0;
            // Tests on the bits: a comparison would take the FP64 pipe. A column below 2^-450 ends the coupling (graded matrices
            // come down to 1e-160 where their eigenvectors have converged): its tau, the square's reciprocal, times the
            // matrix would leave the exponent range.
            const double nn = fma(alpha, alpha, sig);
            if (__double_as_longlong(sig) != 0 && __double2hiint(nn) >= (1023 - 900) << 20) {
                const double ab = td_sqrt(nn);
                const double av = fabs(alpha) + ab;   // |alpha - beta|: beta has the other sign
                t = td_rcp(ab * av);
                const int sg = __double2hiint(alpha) & 0x80000000;
                beta = __hiloint2double(__double2hiint(ab) | (sg ^ 0x80000000), __double2loint(ab));
                v1 = __hiloint2double(__double2hiint(av) | sg, __double2loint(av));
            }
            if (lane == 0) {
                s_beta = beta;
                s_tau = t;
                s_htau = 0.5 * t;
                s_v1 = v1;
                if (cta == 0) {
                    eoff[c] = beta;
                    tau[c] = t;
                }
            }
        }
        const int i0 = c + 1;
        const int q0 = (i0 - cta + G - 1) / G;   // first owned slot with a column >= i0
        // few tasks: none on the scalar warp's sub-partition (warps 0 and 4)
        const int ntask = (ncl - q0) * split;
        const bool apart = ntask <= 2 * (NW - 2);
        const int tw = apart ? ((warp & 3) == 0 ? ntask : (warp < 4 ? warp - 1 : warp - 2)) : warp;
        for (int task = tw; warp < NW && task < ntask; task += apart ? NW - 2 : NW) {
            const int q = q0 + task / split, part = task % split;
            const int r = q * G + cta;
            if (r >= n) break;
            double* col = Aloc + (size_t)q * n;
            const double vr = vs[r], wr = ws[r];
            double* pub = (!CL && r == i0) ? cbuf + (size_t)c * n : nullptr;   // the next column: publish it on the way
            double acc0 = 0.0, acc1 = 0.0;
            int i = i0 + 32 * part + lane;
            const int st = 32 * split;
            for (; i + st < n; i += 2 * st) {
                const double a0 = fma(-ws[i], vr, fma(-vs[i], wr, col[i]));
                const double a1 = fma(-ws[i + st], vr, fma(-vs[i + st], wr, col[i + st]));
                col[i] = a0;
                col[i + st] = a1;
                if (pub) {
                    td_st(pub + i, a0);
                    td_st(pub + i + st, a1);
                }
                acc0 = fma(a0, xs[i], acc0);
                acc1 = fma(a1, xs[i + st], acc1);
            }
            if (i < n) {
                const double a0 = fma(-ws[i], vr, fma(-vs[i], wr, col[i]));
                col[i] = a0;
                if (pub) td_st(pub + i, a0);
                acc0 = fma(a0, xs[i], acc0);
            }
            sdot[(q * split + part) * 32 + lane] = acc0 + acc1;
        }
        // ---- p = tau (A x' - beta A e_{c+1}) of the owned rows: the lanes' sums by 8 threads a column, or by a warp,
        //      while the scalar warp still works (a barrier of the other warps alone), then the scalars ----
        const int tpc = split == 1 ? 8 : 32;           // threads per column
        const int g = tid & (tpc - 1), cps = (32 * NW) / tpc;
        constexpr int MAXP = 16;                       // rounds held in registers: up to 512 columns a CTA (n = 1024, two CTAs)
        double ax[MAXP], a0[MAXP];
        if (warp < NW) {
            asm volatile("bar.sync 1, %0;" ::"n"(32 * NW) : "memory");
#pragma unroll
            for (int u = 0; u < MAXP; ++u) {
                ax[u] = a0[u] = 0.0;
                const int q = q0 + u * cps + tid / tpc;
                if (q0 + u * cps + (32 * warp) / tpc >= ncl) break;   // none of this warp's columns (uniform)
                if (q < ncl) {
                    const double* d = sdot + (size_t)q * split * 32 + g;
                    if (split == 1) ax[u] = (d[0] + d[8]) + (d[16] + d[24]);
                    else if (split == 2) ax[u] = d[0] + d[32];
                    else ax[u] = (d[0] + d[32]) + (d[64] + d[96]);
                    a0[u] = Aloc[(size_t)q * n + i0];
                }
                for (int o = tpc >> 1; o > 0; o >>= 1) ax[u] += __shfl_xor_sync(0xffffffffu, ax[u], o);
            }
        }
        __syncthreads();
        if (warp < NW) {
            const double tj = s_tau, bj = s_beta;
#pragma unroll
            for (int u = 0; u < MAXP; ++u) {
                const int q = q0 + u * cps + tid / tpc;
                if (q0 + u * cps + (32 * warp) / tpc >= ncl) break;
                const int r = q * G + cta;
                if (q >= ncl || r >= n) continue;
                const double p = tj * fma(-bj, a0[u], ax[u]);
                if (CL) {
                    double* mine = pin + (c & 1) * n + r;
                    for (int k = g; k < G; k += tpc) *cg::this_cluster().map_shared_rank(mine, k) = p;
                } else if (g == 0) {
                    td_st(pbuf + (size_t)c * n + r, p);
                }
            }
        }
        double* sw = vs;   // x' becomes the reflector (its first entry is s_v1)
        vs = xs;
        xs = sw;
        if (CL) cg::this_cluster().sync();
    }
    if (n >= 2) {
        // column n - 2 is x'; the last diagonal entry is the owner's, updated by the last reflector
        if (cta == 0 && tid == 0) eoff[n - 2] = xs[n - 1];
        if (cta == (n - 1) % G && tid == 0) {
            const double a = Aloc[(size_t)((n - 1) / G) * n + n - 1];
            dgl[n - 1] = fma(-2.0 * vs[n - 1], ws[n - 1], a);
        }
    } else if (cta == 0 && tid == 0) {
        dgl[0] = xs[0];
    }
    if (cta == 0) {
        for (int jj = (n >= 2 ? n - 2 : 0); jj < n; ++jj) {
            if (tid == 0) tau[jj] = 0.0;
            for (int i = tid; i < n; i += TD_THREADS) HV[(int64_t)jj * n + i] = 0.0;
        }
        if (tid == 0) eoff[n - 1] = 0.0;
    }
    if (CL) cg::this_cluster().sync();   // no CTA leaves while another may still read its shared memory
}

__device__ __forceinline__ bool abs_less(double a, double b) {   // |a| < |b|
    return (__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFll) < (__double_as_longlong(b) & 0x7FFFFFFFFFFFFFFFll);
}
__device__ __forceinline__ bool is_zero(double a) { return (__double_as_longlong(a) << 1) == 0; }
// 1 / x for any sign: td_rcp on |x| with the sign put back
__device__ __forceinline__ double signed_rcp(double x) {
    const double r = td_rcp(fabs(x));
    return __hiloint2double(__double2hiint(r) | (__double2hiint(x) & 0x80000000), __double2loint(r));
}

// Number of eigenvalues below x of the tridiagonal with diagonal d and squared off-diagonal e2, in
// single precision (ratio form q_i = (d_i - x) - e2_{i-1} / q_{i-1}, small pivots replaced).
__device__ __forceinline__ int sturm_count_f32(int n, const float* d, const float* e2, float x, float pivmin) {
    int cnt = 0;
    float q = d[0] - x;
    if (fabsf(q) < pivmin) q = -pivmin;
    cnt += (q < 0.f);
    for (int i = 1; i < n; ++i) {
        q = (d[i] - x) - __fdividef(e2[i - 1], q);
        if (fabsf(q) < pivmin) q = -pivmin;
        cnt += (q < 0.f);
    }
    return cnt;
}

// The same count in double precision without divisions: the leading principal minors
// p_i = det(T_i - x I) obey
// p_i = (d_{i-1} - x) p_{i-1} - e2_{i-2} p_{i-2}, and the number of sign changes along
// p_0 = 1, p_1, ..., p_n is the number of eigenvalues below x (Sturm). Sign tests use the sign
// bit (integer pipe); an exact zero takes the sign opposite to its predecessor (a sign change,
// as a zero pivot does in the ratio form); every fourth step the pair (p_{i-1}, p_i) is rescaled
// by a power of two when its exponent drifts, which keeps every sign and ratio exact.
__device__ __forceinline__ double fix_zero(double p, double prev) {
    const int hi = __double2hiint(p), lo = __double2loint(p);
    if (((hi & 0x7fffffff) | lo) != 0) return p;
    return __hiloint2double((~__double2hiint(prev) & 0x80000000) | 0x00100000, 0);   // -sign(prev) * DBL_MIN
}

__device__ __forceinline__ void rescale_pair(double& pc, double& pm, int& shift) {
    const int ex = (__double2hiint(pc) >> 20) & 0x7ff;
    if (ex > 1023 + 480 || ex < 1023 - 480) {
        const double sc = __hiloint2double((2046 - ex) << 20, 0);   // 2^(1023 - ex)
        pc *= sc;
        pm *= sc;
        shift += ex - 1023;
    }
}

// The number of eigenvalues below x0 by that recurrence (one shift per thread), and the value of the characteristic
// polynomial there as val 2^shift.
__device__ __forceinline__ int sturm_count1_f64(int n, const double* d, const double* e2, double x0, double* val = nullptr,
                                                int* shift = nullptr) {
    double pm0 = 1.0;
    double pc0 = fix_zero(d[0] - x0, 1.0);
    int c0 = (int)((unsigned)__double2hiint(pc0) >> 31);
    int sh = 0;
    for (int i = 1; i < n; ++i) {
        const double di = d[i], ei = e2[i - 1];
        const double pn0 = fix_zero(fma(di - x0, pc0, -ei * pm0), pc0);
        c0 += (int)(((unsigned)__double2hiint(pn0) ^ (unsigned)__double2hiint(pc0)) >> 31);
        pm0 = pc0;
        pc0 = pn0;
        if ((i & 3) == 0) rescale_pair(pc0, pm0, sh);
    }
    if (val) {
        *val = pc0;
        *shift = sh;
    }
    return c0;
}

// The root in [0, 1] of the cubic through f(-1), f(0), f(1), f(2), f(0) and f(1) of opposite signs: Newton's iteration on
// the interpolation polynomial in Newton's form from the chord's root (which is returned when the iteration leaves [0, 1]).
__device__ __forceinline__ double cubic_root01(double fm, double f0, double f1, double f2) {
    const double d01 = f1 - f0, d1m = 0.5 * (f1 - fm);
    const double d2 = d01 - d1m;
    const double d3 = 0.5 * (fma(f2 - fm, 1.0 / 3.0, -d1m) - d2);
    const double s0 = fabs(f0) * td_rcp(fabs(f0) + fabs(f1));
    double s = s0;
    for (int it = 0; it < 3; ++it) {
        const double q = fma(s + 1.0, d3, d2);
        const double r = fma(s - 1.0, q, d01);
        const double dp = fma(s, fma(s - 1.0, d3, q), r);
        s = fma(-fma(s, r, f0), signed_rcp(dp), s);
    }
    return s >= 0.0 && s <= 1.0 ? s : s0;
}

// One CTA of two warps per wanted eigenvalue (ascending index il + blockIdx.x). The tridiagonal is
// scaled by 1 / ||T||; 33-way multisection first on single-precision counts (fast; both warps run it
// alike) until the interval is 1e-5 wide, then, after widening it by that margin (far above the
// single-precision backward error of the count, about 1e-6), 65-way multisection on double-precision
// counts down to ~eps: lane l of warp 0 counts at the shift 2 l + 1 of the 65-way split and lane l of
// warp 1 at 2 l + 2, so each warp's FP64 chain carries one shift (the FP64 pipe of a sub-partition
// holds a warp instruction for ~64 cycles, so two warps on two sub-partitions halve the time).
//
// A double-precision round gains 6 bits and costs n dependent steps, so the first one also gives the polynomial's values:
// when the four shifts around the bracket hold this eigenvalue alone, the cubic through them puts it within about
// (h / gap)^3 of the bracket's width h (3e-7), and the second round counts at x* +- h 2^-i, i = 0 .. 31: whatever
// the quality of x*, the counts make the new bracket, about as wide as x* was wrong. Two or three rounds then do the work
// of six. GB300: n = 698 and 100, all eigenvalues, 1.70 -> 1.13 ms; n = 668, 92 of them 0.73 -> 0.56; n = 144, 99 of them
// 0.165 -> 0.085.
__global__ void __launch_bounds__(64) k_bisect(int n, const double* __restrict__ dgl, const double* __restrict__ eoff,
                                                int il, int nw, double* w) {
    PDL_WAIT();
    PDL_ARG(dgl); PDL_ARG(eoff); PDL_ARG(w);
    extern __shared__ double smb[];
    double* d64 = smb;                                     // n
    double* e264 = smb + n;                                // n
    float* d32 = reinterpret_cast<float*>(smb + 2 * n);    // n
    float* e232 = d32 + n;                                 // n
    __shared__ double s_tnorm;
    __shared__ unsigned s_ball[2];
    __shared__ double s_f[64];
    __shared__ int s_fs[64], s_cnt[64];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    // ||T||_inf by warp 0
    if (threadIdx.x < 32) {
        double m = 0.0;
        for (int i = lane; i < n; i += 32) {
            const double r = fabs(dgl[i]) + ((i > 0) ? fabs(eoff[i - 1]) : 0.0) + ((i + 1 < n) ? fabs(eoff[i]) : 0.0);
            m = fmax(m, r);
        }
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) s_tnorm = (m > 0.0) ? m : 1.0;
    }
    __syncthreads();
    const double tn = s_tnorm, itn = 1.0 / tn;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double di = dgl[i] * itn;
        const double ei = (i + 1 < n) ? eoff[i] * itn : 0.0;
        d64[i] = di;
        e264[i] = ei * ei;
        d32[i] = (float)di;
        e232[i] = (float)(ei * ei);
    }
    __syncthreads();
    const int gw = blockIdx.x;
    if (gw >= nw) return;                                   // uniform over the CTA
    const int idx = il + gw;
    // scaled Gershgorin interval is inside [-1, 1]
    float lo = -1.0f - 1e-6f, hi = 1.0f + 1e-6f;
    const float piv32 = 1e-30f;
    for (int round = 0; round < 8 && hi - lo > 1e-5f; ++round) {
        const float step = (hi - lo) / 33.f;
        const float x = lo + (lane + 1) * step;
        const int cnt = sturm_count_f32(n, d32, e232, x, piv32);
        const unsigned above = __ballot_sync(0xffffffffu, cnt > idx);
        if (above == 0u) {
            lo = __shfl_sync(0xffffffffu, x, 31);
        } else {
            const int l = __ffs(above) - 1;
            const float xl = __shfl_sync(0xffffffffu, x, l);
            const float xp = __shfl_sync(0xffffffffu, x, l > 0 ? l - 1 : 0);
            if (l > 0) lo = xp;
            hi = xl;
        }
    }
    double dlo = (double)lo - 1e-5, dhi = (double)hi + 1e-5;
    // first double-precision round: 64 shifts from dlo to dhi, both included (lane l of warp 0 at shift 2 l, of warp 1 at
    // 2 l + 1), so that it confirms the bracket and divides it; the full interval when the bracket fails
    {
        const double step = (dhi - dlo) * (1.0 / 63.0);
        const int me = 2 * lane + wp;
        double f;
        int fs;
        const int c = sturm_count1_f64(n, d64, e264, me == 63 ? dhi : fma((double)me, step, dlo), &f, &fs);
        s_f[me] = f;
        s_fs[me] = fs;
        s_cnt[me] = c;
        __syncthreads();
        if (s_cnt[0] > idx || s_cnt[63] <= idx) {
            dlo = -1.0 - 1e-12;
            dhi = 1.0 + 1e-12;
        } else {
            // the first shift with more than idx eigenvalues below it
            int k = 1;
            {
                const unsigned b0 = __ballot_sync(0xffffffffu, s_cnt[lane] > idx);
                const unsigned b1 = __ballot_sync(0xffffffffu, s_cnt[32 + lane] > idx);
                k = b0 ? __ffs(b0) - 1 : 31 + __ffs(b1);
            }
            const double x0 = fma((double)(k - 1), step, dlo), x1 = k == 63 ? dhi : fma((double)k, step, dlo);
            const bool alone = k >= 2 && k <= 62 && s_cnt[k - 2] == idx && s_cnt[k + 1] == idx + 1;
            dlo = x0;
            dhi = x1;
            if (alone) {
                // values at the four shifts on one scale (powers of two; far smaller ones vanish)
                double v[4];
                int top = s_fs[k - 2];
#pragma unroll
                for (int u = 1; u < 4; ++u) top = max(top, s_fs[k - 2 + u]);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int sh = s_fs[k - 2 + u] - top;
                    v[u] = sh < -500 ? 0.0 : s_f[k - 2 + u] * __hiloint2double((1023 + sh) << 20, 0);
                }
                const double xs = fma(cubic_root01(v[0], v[1], v[2], v[3]), step, x0);
                // second round: x* -+ step 2^-i, ascending with the index
                auto at = [&](int m) {
                    return m < 32 ? fma(-step, __hiloint2double((1023 - m) << 20, 0), xs)
                                  : fma(step, __hiloint2double((1023 - (63 - m)) << 20, 0), xs);
                };
                const int c2 = sturm_count1_f64(n, d64, e264, at(me));
                __syncthreads();   // the first round's counts have been read
                s_cnt[me] = c2;
                __syncthreads();
                const unsigned b0 = __ballot_sync(0xffffffffu, s_cnt[lane] > idx);
                const unsigned b1 = __ballot_sync(0xffffffffu, s_cnt[32 + lane] > idx);
                const int m = b0 ? __ffs(b0) - 1 : (b1 ? 31 + __ffs(b1) : 64);
                if (m > 0) dlo = fmax(dlo, at(m - 1));
                if (m < 64) dhi = fmin(dhi, at(m));
            }
        }
        __syncthreads();
    }
    for (int round = 0; round < 24; ++round) {
        const double width = dhi - dlo;
        if (width <= 2.0 * DBL_EPSILON * fmax(fabs(dlo), fabs(dhi)) || width <= 0.5 * DBL_EPSILON) break;
        const double step = width / 65.0;
        const double x = dlo + (2 * lane + 1 + wp) * step;   // warp 0: shifts 2 l + 1, warp 1: 2 l + 2
        const int c = sturm_count1_f64(n, d64, e264, x);
        const unsigned b = __ballot_sync(0xffffffffu, c > idx);
        if (lane == 0) s_ball[wp] = b;
        __syncthreads();
        const unsigned b0 = s_ball[0], b1 = s_ball[1];
        __syncthreads();
        const unsigned above = b0 | b1;
        if (above == 0u) {
            dlo = dlo + (2 * 31 + 2) * step;
        } else {
            const int l = __ffs(above) - 1;
            const bool first = (b0 >> l) & 1u;
            const double a0 = dlo + (2 * l + 1) * step;
            const double a1 = dlo + (2 * l + 2) * step;
            const double pl = dlo + (2 * (l > 0 ? l - 1 : 0) + 2) * step;
            if (first) {
                if (l > 0) dlo = pl;
                dhi = a0;
            } else {
                dlo = a0;
                dhi = a1;
            }
        }
    }
    if (threadIdx.x == 0) w[gw] = 0.5 * (dlo + dhi) * tn;
}

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Inverse iteration, one thread per eigenvector; factor arrays laid out [array][i][q] so that
// the threads of a warp touch consecutive addresses. Gaussian elimination with partial pivoting
// of T - lambda I, two triangular solves a pass, two passes from a counter-based random start.
//
// What bounds it is the chain of FP64 instructions of a thread (each about 64 cycles, whatever the number of warps), so a
// row takes as few as it can: 8 in the elimination (one Newton reciprocal per pivot), 1 or 2 in the forward and 3 in the
// backward solve, 2 for the norm; comparisons, maxima and the start vector use the bits, the scale between the passes is
// a power of two, the normalisation is left to the transposition. The rows of a pass are read IV_U at a time, the next
// group while the current one is used; the interchanges are one bit a row. GB300: n = 288, nv = 199 450 -> 225 us;
// n = nv = 698 and 100 together 1.77 -> 0.97 ms; n = 144, nv = 99 305 -> 175 us.
constexpr int IV_U = 8;

__global__ void __launch_bounds__(32) k_invit(int n, int nv, const double* __restrict__ dgl,
                                              const double* __restrict__ eoff, const double* __restrict__ lam, double* lu,
                                              double* Zt, uint64_t seed) {
    PDL_WAIT();
    PDL_ARG(dgl); PDL_ARG(eoff); PDL_ARG(lam); PDL_ARG(lu); PDL_ARG(Zt);
    const int lane = threadIdx.x;
    // ||T||_inf, by the whole warp
    double tn = 0.0;
    for (int i = lane; i < n; i += 32) {
        const double r = fabs(dgl[i]) + ((i > 0) ? fabs(eoff[i - 1]) : 0.0) + ((i + 1 < n) ? fabs(eoff[i]) : 0.0);
        tn = fmax(tn, r);
    }
    for (int o = 16; o > 0; o >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
    const int q = blockIdx.x * blockDim.x + lane;
    if (q >= nv) return;
    const int64_t S = nv;
    double* DL = lu;                           // multipliers
    double* RD = lu + (int64_t)n * S;          // reciprocal pivots
    double* DU = lu + 2 * (int64_t)n * S;      // first superdiagonal of U
    double* DU2 = lu + 3 * (int64_t)n * S;     // second superdiagonal of U
    unsigned* PIV = reinterpret_cast<unsigned*>(lu + 4 * (int64_t)n * S);   // bit i % 32 of word i / 32: rows i, i + 1 swapped
    double* x = Zt;
    const double l = lam[q];
    const double tiny = fmax(DBL_EPSILON * tn, DBL_MIN);
    double dcur = dgl[0] - l;
    double ucur = (n > 1) ? eoff[0] : 0.0;
    unsigned bits = 0;
    for (int i = 0; i + 1 < n; ++i) {
        const double sub = eoff[i];                    // T[i+1, i]
        const double dnext = dgl[i + 1] - l;
        const double unext = (i + 2 < n) ? eoff[i + 1] : 0.0;
        const bool swap = abs_less(dcur, sub);
        const double piv = swap ? sub : (is_zero(dcur) ? tiny : dcur);
        const double r = signed_rcp(piv);
        const double f = (swap ? dcur : sub) * r;
        RD[i * S + q] = r;
        DL[i * S + q] = f;
        DU[i * S + q] = swap ? dnext : ucur;
        DU2[i * S + q] = swap ? unext : 0.0;
        if (swap) bits |= 1u << (i & 31);
        if ((i & 31) == 31 || i + 2 == n) {
            PIV[(i >> 5) * S + q] = bits;
            bits = 0;
        }
        const double hi = swap ? ucur : dnext, lo = swap ? dnext : ucur;
        dcur = fma(-f, lo, hi);
        ucur = swap ? -f * unext : unext;
    }
    RD[(int64_t)(n - 1) * S + q] = signed_rcp(is_zero(dcur) ? tiny : dcur);
    // start vector, uniform in [-1, 1): 52 bits of the hash as the fraction of a number in [1, 2)
    auto start = [&](int i) {
        const uint64_t h = mix64(seed ^ mix64(((uint64_t)q << 32) + (uint64_t)i + 0x5851F42D4C957F2Dull));
        return fma(2.0, __longlong_as_double((long long)((h >> 12) | 0x3FF0000000000000ull)), -3.0);
    };
    double sc = 1.0;   // power-of-two scale of the previous pass, applied to x as it is read
    for (int it = 0; it < 2; ++it) {
        // forward: L^{-1} P b, the running entry carried in a register
        auto in = [&](int i) { return it == 0 ? start(i) : x[(int64_t)i * S + q]; };
        double carry = in(0);
        if (it > 0) carry *= sc;
        double f[IV_U], nx[IV_U];
        auto load = [&](int i0, double (&ff)[IV_U], double (&xx)[IV_U]) {
#pragma unroll
            for (int u = 0; u < IV_U; ++u) {
                const int i = i0 + u;
                if (i + 1 < n) {
                    ff[u] = DL[(int64_t)i * S + q];
                    xx[u] = in(i + 1);
                }
            }
        };
        load(0, f, nx);
        unsigned pv = 0;
        for (int i0 = 0; i0 + 1 < n; i0 += IV_U) {
            double fn[IV_U], xn[IV_U];
            if ((i0 & 31) == 0) pv = PIV[(i0 >> 5) * S + q];
            if (i0 + IV_U + 1 < n) load(i0 + IV_U, fn, xn);
#pragma unroll
            for (int u = 0; u < IV_U; ++u) {
                const int i = i0 + u;
                if (i + 1 < n) {
                    const double b = it > 0 ? nx[u] * sc : nx[u];
                    const bool swap = (pv >> (i & 31)) & 1u;
                    const double keep = swap ? b : carry;      // this row of the permuted right-hand side
                    const double other = swap ? carry : b;
                    x[(int64_t)i * S + q] = keep;
                    carry = fma(-f[u], keep, other);
                }
            }
#pragma unroll
            for (int u = 0; u < IV_U; ++u) {
                f[u] = fn[u];
                nx[u] = xn[u];
            }
        }
        x[(int64_t)(n - 1) * S + q] = carry;
        // back: U^{-1}, carrying the two previous solution entries
        double v1 = 0.0, v2 = 0.0;
        int mx = 0;   // largest biased exponent
        double xv[IV_U], du[IV_U], du2[IV_U], rd[IV_U];
        auto loadb = [&](int i0, double (&a)[IV_U], double (&b)[IV_U], double (&c)[IV_U], double (&d)[IV_U]) {
#pragma unroll
            for (int u = 0; u < IV_U; ++u) {
                const int i = i0 - u;
                if (i >= 0) {
                    a[u] = x[(int64_t)i * S + q];
                    b[u] = (i + 1 < n) ? DU[(int64_t)i * S + q] : 0.0;
                    c[u] = (i + 2 < n) ? DU2[(int64_t)i * S + q] : 0.0;
                    d[u] = RD[(int64_t)i * S + q];
                }
            }
        };
        loadb(n - 1, xv, du, du2, rd);
        for (int i0 = n - 1; i0 >= 0; i0 -= IV_U) {
            double xn[IV_U], dn[IV_U], d2n[IV_U], rn[IV_U];
            if (i0 - IV_U >= 0) loadb(i0 - IV_U, xn, dn, d2n, rn);
#pragma unroll
            for (int u = 0; u < IV_U; ++u) {
                const int i = i0 - u;
                if (i >= 0) {
                    const double v = fma(-du2[u], v2, fma(-du[u], v1, xv[u])) * rd[u];
                    x[(int64_t)i * S + q] = v;
                    mx = max(mx, (__double2hiint(v) >> 20) & 0x7ff);
                    v2 = v1;
                    v1 = v;
                }
            }
#pragma unroll
            for (int u = 0; u < IV_U; ++u) {
                xv[u] = xn[u];
                du[u] = dn[u];
                du2[u] = d2n[u];
                rd[u] = rn[u];
            }
        }
        // 2^-(exponent of the largest entry); a zero or non-finite vector comes out zero
        sc = (mx > 0 && mx < 0x7ff) ? __hiloint2double(max(1, min(0x7fe, 2046 - mx)) << 20, 0) : 0.0;
    }
    // norm of the scaled vector; the normalisation factor goes where the pivots were
    double nrm = 0.0;
    for (int i0 = 0; i0 < n; i0 += 2 * IV_U) {
        double xv[2 * IV_U];
#pragma unroll
        for (int u = 0; u < 2 * IV_U; ++u) xv[u] = i0 + u < n ? x[(int64_t)(i0 + u) * S + q] : 0.0;
#pragma unroll
        for (int u = 0; u < 2 * IV_U; ++u) {
            const double t = xv[u] * sc;
            nrm = fma(t, t, nrm);
        }
    }
    RD[q] = (nrm > 0.0) ? sc / sqrt(nrm) : 0.0;
}

// Zt (row-major n x nv) times its column factors -> Z (column-major, ldz), by 32 x 32 tiles through shared memory
__global__ void __launch_bounds__(256) k_transpose_out(int n, int nv, const double* __restrict__ Zt,
                                                       const double* __restrict__ fac, double* __restrict__ Z, int ldz) {
    PDL_ENTER();
    PDL_ARG(Zt); PDL_ARG(fac); PDL_ARG(Z);
    __shared__ double t[32][33];
    const int q0 = blockIdx.y * 32, i0 = blockIdx.x * 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double f = q0 + lane < nv ? fac[q0 + lane] : 0.0;
    for (int r = w; r < 32; r += 8)
        if (i0 + r < n && q0 + lane < nv) t[r][lane] = Zt[(int64_t)(i0 + r) * nv + q0 + lane] * f;
    __syncthreads();
    for (int c = w; c < 32; c += 8)
        if (q0 + c < nv && i0 + lane < n) Z[(int64_t)(q0 + c) * ldz + i0 + lane] = t[lane][c];
}

// Z <- H_0 H_1 ... H_{n-3} Z in blocks of WY_B reflectors, last block first. A block is I - V U^{-1} V^T with V its
// reflectors (n x 32) and U upper triangular, U_ii = 1 / tau_i and U_ik = v_i^T v_k above the diagonal (the inverse of the
// compact WY factor; Joffrain, Low, Quintana-Orti, van de Geijn and Van Zee, "Accumulating Householder transformations,
// revisited", ACM TOMS 32, 2006). Applied one by one, each reflector of each column costs a reduction over all warps,
// as many FP64 instructions as the products themselves at n = 700; here a CTA keeps NC columns of Z in shared memory, takes
// the 32 NC products of a block with packed reductions, solves with U by one warp per column and updates the rows with no
// reduction at all. The FP64 pipe bounds it (n^2 FMAs a column, each CTA on its own SM): n = nv = 698 2.58 -> 0.80 ms,
// n = 668, nv = 92 1.13 -> 0.39, n = 288, nv = 199 0.40 -> 0.25, n = 144, nv = 99 0.12 -> 0.07.
constexpr int WY_B = 32;

// Upper triangles of V^T V of every block: G[kb][i][k], i < k. grid (blocks, 8): four rows i each; a warp per product.
__global__ void __launch_bounds__(256) k_wy_gram(int n, const double* __restrict__ HV, double* __restrict__ G) {
    PDL_WAIT();
    PDL_ARG(HV); PDL_ARG(G);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int j0 = blockIdx.x * WY_B, m = min(WY_B, n - 2 - j0);
    double* g = G + (size_t)blockIdx.x * WY_B * WY_B;
    for (int ii = 0; ii < 4; ++ii) {
        const int i = 4 * blockIdx.y + ii;
        const double* vi = HV + (int64_t)(j0 + i) * n;
        for (int k = i + 1 + w; k < m; k += 8) {
            const double* vk = HV + (int64_t)(j0 + k) * n;   // zero above row j0 + k + 1
            double a0 = 0.0, a1 = 0.0;
            int r = j0 + k + 1 + lane;
            for (; r + 32 < n; r += 64) {
                a0 = fma(vi[r], vk[r], a0);
                a1 = fma(vi[r + 32], vk[r + 32], a1);
            }
            if (r < n) a0 = fma(vi[r], vk[r], a0);
            a0 += a1;
            for (int o = 16; o > 0; o >>= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
            if (lane == 0) g[i * WY_B + k] = a0;
        }
    }
}

// Sums over the lanes of N values (N a power of two up to 8): value v's sum ends in the lanes whose upper log2(N) bits,
// read from lane bit 4 down, spell v. Half of the values change sides at each of the first steps, so that 8 values take 9
// FP64 additions and not 40.
template <int N>
__device__ __forceinline__ double warp_sum_packed(double (&a)[N], int lane) {
#pragma unroll
    for (int h = N / 2, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int v = 0; v < N / 2; ++v)
            if (v < h) {
                const double keep = up ? a[v + h] : a[v], send = up ? a[v] : a[v + h];
                a[v] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    double x = a[0];
#pragma unroll
    for (int o = 16 / N; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

template <int NC>
__global__ void __launch_bounds__(256) k_wy_apply(int n, int nv, const double* __restrict__ HV,
                                                  const double* __restrict__ tau, const double* __restrict__ G, double* Z,
                                                  int ldz) {
    PDL_WAIT();
    PDL_ARG(HV); PDL_ARG(tau); PDL_ARG(G); PDL_ARG(Z);
    constexpr int NP = NC <= 1 ? 1 : (NC <= 2 ? 2 : (NC <= 4 ? 4 : 8));
    extern __shared__ double sz[];               // NC x n: this CTA's columns
    __shared__ double xs[WY_B][NC];              // V^T Z of the block, then U^{-1} V^T Z
    __shared__ double gs[WY_B][WY_B + 1];
    __shared__ double ts[WY_B];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int q0 = blockIdx.x * NC, nc = min(NC, nv - q0);
    for (int c = 0; c < NC; ++c)
        for (int i = tid; i < n; i += 256) sz[c * n + i] = c < nc ? Z[(int64_t)(q0 + c) * ldz + i] : 0.0;
    const int nr = n - 2, nb = (nr + WY_B - 1) / WY_B;
    for (int kb = nb - 1; kb >= 0; --kb) {
        const int j0 = kb * WY_B, m = min(WY_B, nr - j0);
        for (int e = tid; e < WY_B * WY_B; e += 256) {
            const int i = e / WY_B, k = e % WY_B;
            gs[i][k] = (i < k && k < m) ? G[(size_t)kb * WY_B * WY_B + e] : 0.0;
        }
        if (tid < WY_B) ts[tid] = tid < m ? tau[j0 + tid] : 0.0;
        __syncthreads();   // also: the columns are up to date
        // products of the block's reflectors with the columns, one warp per reflector
        for (int r = w; r < m; r += 8) {
            const double* v = HV + (int64_t)(j0 + r) * n;
            double a[NP];
#pragma unroll
            for (int c = 0; c < NP; ++c) a[c] = 0.0;
            for (int i = ((j0 + r + 1) & ~31) + lane; i < n; i += 32) {
                const double vi = v[i];
#pragma unroll
                for (int c = 0; c < NC; ++c) a[c] = fma(vi, sz[c * n + i], a[c]);
            }
            const double x = warp_sum_packed<NP>(a, lane);
            // the value this lane holds: lane bits 4, 3, 2 (for NP = 8), and so on
            const int val = NP == 1 ? 0 : lane / (32 / NP);
            if (lane % (32 / NP) == 0 && val < NC) xs[r][val] = x;
        }
        __syncthreads();
        // U x = V^T Z by back substitution, one warp per column, lane i holding row i
        for (int c = w; c < NC; c += 8) {
            double wi = lane < m ? xs[lane][c] : 0.0, mine = 0.0;
            for (int k = m - 1; k >= 0; --k) {
                const double xk = ts[k] * __shfl_sync(0xffffffffu, wi, k);
                if (lane == k) mine = xk;
                wi = fma(-gs[lane][k], xk, wi);   // zero at and below the diagonal
            }
            if (lane < m) xs[lane][c] = mine;
        }
        __syncthreads();
        // Z -= V x
        for (int i = j0 + 1 + tid; i < n; i += 256) {
            double z[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) z[c] = sz[c * n + i];
            const double* v = HV + (int64_t)j0 * n + i;
            for (int r = 0; r < m; r += 4) {
                double vr[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) vr[u] = r + u < m ? v[(int64_t)(r + u) * n] : 0.0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (r + u < m) {
#pragma unroll
                        for (int c = 0; c < NC; ++c) z[c] = fma(-vr[u], xs[r + u][c], z[c]);
                    }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) sz[c * n + i] = z[c];
        }
        __syncthreads();
    }
    PDL_NEXT();
    for (int c = 0; c < nc; ++c)
        for (int i = tid; i < n; i += 256) Z[(int64_t)(q0 + c) * ldz + i] = sz[c * n + i];
}

// Z <- H_0 H_1 ... H_{n-3} Z for few or short columns: one column per CTA, held in the registers of four warps
// (n <= 128 NPL), one warp per SM sub-partition: carried by a single warp, the chain of reflectors is bound by the FP64 issue rate of one
// sub-partition. Rows are dealt in 32-row stripes, row 32 (4 k + w) + lane in register k of warp w; a
// warp skips the stripes that lie wholly at or above reflector j's first nonzero row j + 1 (exact zero
// terms), the four partial dot products are added in a fixed order through shared memory (one barrier
// per reflector, the partials double-buffered), and reflector j - 1 and its scalar are read while
// reflector j is applied.
template <int NPL>
__global__ void __launch_bounds__(128) k_backtransform_w4(int n, int nv, const double* __restrict__ HV,
                                                          const double* __restrict__ tau, double* Z, int ldz) {
    PDL_WAIT();
    PDL_ARG(HV); PDL_ARG(tau); PDL_ARG(Z);
    __shared__ double red[2][4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int col = blockIdx.x;
    if (col >= nv) return;   // uniform over the CTA
    double* zc = Z + (int64_t)col * ldz;
    double z[NPL];
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
        const int i = 32 * (4 * k + w) + lane;
        z[k] = (i < n) ? zc[i] : 0.0;
    }
    // stripe k of this warp holds a row below j exactly when its last row 32 (4 k + w) + 31 exceeds j
    double un[NPL];
    double tn = 0.0;
    if (n >= 3) {
        const int j = n - 3;
        const double* u = HV + (int64_t)j * n;
        tn = __ldg(tau + j);
#pragma unroll
        for (int k = 0; k < NPL; ++k) {
            const int i = 32 * (4 * k + w) + lane;
            un[k] = (i < n && 32 * (4 * k + w) + 31 > j) ? __ldg(u + i) : 0.0;
        }
    }
    int par = 0;
    for (int j = n - 3; j >= 0; --j) {
        double uu[NPL];
#pragma unroll
        for (int k = 0; k < NPL; ++k) uu[k] = un[k];
        const double tj = tn;
        if (j > 0) {
            const double* u = HV + (int64_t)(j - 1) * n;
            tn = __ldg(tau + j - 1);
#pragma unroll
            for (int k = 0; k < NPL; ++k) {
                const int i = 32 * (4 * k + w) + lane;
                un[k] = (i < n && 32 * (4 * k + w) + 31 > j - 1) ? __ldg(u + i) : 0.0;
            }
        }
        if (tj == 0.0) continue;   // uniform over the CTA
        double d0 = 0.0, d1 = 0.0;
#pragma unroll
        for (int k = 0; k < NPL; ++k) {
            if (32 * (4 * k + w) + 31 > j) {
                if (k & 1) d1 = fma(uu[k], z[k], d1);
                else d0 = fma(uu[k], z[k], d0);
            }
        }
        double dot = d0 + d1;
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        if (lane == 0) red[par][w] = dot;
        __syncthreads();
        const double tot = (red[par][0] + red[par][1]) + (red[par][2] + red[par][3]);
        par ^= 1;
        const double f = tj * tot;
#pragma unroll
        for (int k = 0; k < NPL; ++k)
            if (32 * (4 * k + w) + 31 > j) z[k] = fma(-f, uu[k], z[k]);
    }
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
        const int i = 32 * (4 * k + w) + lane;
        if (i < n) zc[i] = z[k];
    }
}

// Largest eigenvalue of a symmetric positive semidefinite n x n matrix A (n <= 16 C) by the plain
// symmetric Lanczos recurrence u = A v_j - beta_{j-1} v_{j-1}, alpha_j = v_j^T u,
// u <- u - alpha_j v_j, beta_j = ||u||, v_{j+1} = u / beta_j, run for m steps in one thread-block
// cluster of C CTAs. The extreme Ritz values of the tridiagonal T_m converge to the extreme
// eigenvalues of A without reorthogonalisation (loss of orthogonality only adds copies of converged
// Ritz values), so the recurrence alone is kept. CTA r owns rows [r nb, r nb + nb) of A (nb <= 16)
// in its shared memory and every CTA keeps the whole current vector v; the two inner products of a
// step are summed over the CTAs in a fixed order, so every CTA holds bitwise the same alpha_j and
// beta_j. Output: T_m as dgl[0..m-1] (alpha) and eoff[0..m-1] (beta, eoff[m-1] = beta_m, the norm of
// the residual after the last step). On breakdown (beta_j at rounding level) the recurrence stops
// and the rest of T_m is zero: a diagonal block of zeros, which leaves the largest eigenvalue of the
// nonnegative spectrum unchanged. Start vector: uniform in [-1, 1] from a counter-based hash of
// (seed, index).
constexpr int LZ_THREADS = 128;
constexpr int LZ_ROWS = 16;
constexpr int LZ_GROUPS = LZ_THREADS / LZ_ROWS;

__global__ void __launch_bounds__(LZ_THREADS) k_lanczos(int n, const double* __restrict__ A, int lda, int m,
                                                        uint64_t seed, double* dgl, double* eoff) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int nb = (n + C - 1) / C;
    const int r0 = rank * nb;
    const int nr = max(0, min(n, r0 + nb) - r0);
    extern __shared__ double smz[];
    double* Aloc = smz;                    // Aloc[c * LZ_ROWS + i] = A[r0 + i, c]
    double* v = smz + (size_t)LZ_ROWS * n; // the current Lanczos vector, all n entries
    __shared__ double part[LZ_GROUPS][LZ_ROWS];
    __shared__ double vnew[LZ_ROWS];       // this CTA's rows of v_{j+1} (read by the other CTAs)
    __shared__ double red[2];              // this CTA's partial sums of the step (read by the other CTAs)
    __shared__ double s_ab[2];
    __shared__ double s_red[32];
    __shared__ int s_stop;
    const int tid = threadIdx.x, lane = tid & 31;
    const int row = tid % LZ_ROWS, grp = tid / LZ_ROWS;
    for (int e = tid; e < LZ_ROWS * n; e += LZ_THREADS) {
        const int c = e / LZ_ROWS, i = e % LZ_ROWS;
        Aloc[e] = (i < nr) ? A[(int64_t)c * lda + r0 + i] : 0.0;
    }
    // start vector: every CTA forms all n entries and their norm in the same order
    double ss = 0.0;
    for (int c = tid; c < n; c += LZ_THREADS) {
        const uint64_t h = mix64(seed ^ mix64((uint64_t)c + 0x2545F4914F6CDD1Dull));
        const double x = 2.0 * ((h >> 11) * (1.0 / 9007199254740992.0)) - 1.0;
        v[c] = x;
        ss = fma(x, x, ss);
    }
    ss = block_sum(ss, s_red);
    const double inv0 = (ss > 0.0) ? 1.0 / sqrt(ss) : 0.0;
    __syncthreads();
    for (int c = tid; c < n; c += LZ_THREADS) v[c] *= inv0;
    double vp = 0.0;                       // v_{j-1} at this thread's row (warp 0, lanes < nr)
    double beta = 0.0, anorm = 0.0;
    if (tid == 0) s_stop = 0;
    __syncthreads();
    int j = 0;
    for (; j < m; ++j) {
        // u = A v over this CTA's rows: thread (row, grp) sums the columns c = grp mod LZ_GROUPS
        double acc = 0.0;
        for (int c = grp; c < n; c += LZ_GROUPS) acc = fma(Aloc[c * LZ_ROWS + row], v[c], acc);
        part[grp][row] = acc;
        __syncthreads();
        double u = 0.0, vi = 0.0;
        if (tid < 32) {
            if (lane < nr) {
                double t = part[0][lane];
#pragma unroll
                for (int g = 1; g < LZ_GROUPS; ++g) t += part[g][lane];
                vi = v[r0 + lane];
                u = fma(-beta, vp, t);
            }
            double a = vi * u;
            for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);   // lanes < 16 hold the rows
            if (lane == 0) red[0] = a;
        }
        cluster.sync();                                    // partial alpha of every CTA published
        if (tid < 32) {
            double a = (lane < C) ? *cluster.map_shared_rank(&red[0], lane) : 0.0;
            for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);     // C <= 16
            u = (lane < nr) ? fma(-a, vi, u) : 0.0;
            double b2 = u * u;
            for (int o = 8; o > 0; o >>= 1) b2 += __shfl_xor_sync(0xffffffffu, b2, o);
            if (lane == 0) {
                s_ab[0] = a;
                red[1] = b2;
            }
        }
        cluster.sync();                                    // partial ||u||^2 of every CTA published
        if (tid < 32) {
            double b2 = (lane < C) ? *cluster.map_shared_rank(&red[1], lane) : 0.0;
            for (int o = 8; o > 0; o >>= 1) b2 += __shfl_xor_sync(0xffffffffu, b2, o);
            const double a = s_ab[0];
            // beta and 1 / beta from one reciprocal square root (each within a few ulps)
            const double rb = (b2 > 0.0) ? rsqrt(b2) : 0.0;
            const double b = b2 * rb;
            anorm = fmax(anorm, fabs(a) + b + beta);
            const bool stop = !(b > 16.0 * DBL_EPSILON * anorm);
            if (rank == 0 && lane == 0) {
                dgl[j] = a;
                eoff[j] = stop ? 0.0 : b;
            }
            if (lane < nr) {
                vp = vi;
                vnew[lane] = stop ? 0.0 : u * rb;
            }
            beta = b;
            if (lane == 0) s_stop = stop ? 1 : 0;
        }
        cluster.sync();                                    // v_{j+1} published
        if (s_stop) break;                                 // the same decision in every CTA
        for (int c = tid; c < n; c += LZ_THREADS) v[c] = cluster.map_shared_rank(vnew, c / nb)[c % nb];
        __syncthreads();
    }
    if (rank == 0)
        for (int jj = j + 1 + tid; jj < m; jj += LZ_THREADS) {
            dgl[jj] = 0.0;
            eoff[jj] = 0.0;
        }
    cluster.sync();   // no CTA leaves while another may still read its shared memory
}

// The same recurrence for a Gram too large for one cluster's shared memory (n > kLanczosMaxN), two
// launches per step with the matrix read from global memory (L2-resident at these sizes):
// k_lz_matvec forms u = A v_j (one warp per row; A is symmetric, so row r is read as its contiguous
// column r), k_lz_update the rest of the step in one CTA. The vectors rotate through three buffers
// chosen by the host; st[0] = beta_{j-1}, st[1] = the running norm estimate, st[2] = the stop flag.
// eight warps: with 32 the FP64 sums over the warps (each instruction about 64 cycles of a sub-partition's pipe) took most
// of the step (n = 2000: 30 us against 8)
constexpr int LZG_THREADS = 256;
__global__ void k_lz_start(int n, uint64_t seed, double* __restrict__ v, double* __restrict__ vprev,
                           double* __restrict__ st) {
    PDL_ENTER();
    PDL_ARG(v); PDL_ARG(vprev); PDL_ARG(st);
    __shared__ double red[32];
    double ss = 0.0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        const uint64_t h = mix64(seed ^ mix64((uint64_t)c + 0x2545F4914F6CDD1Dull));
        const double x = 2.0 * ((h >> 11) * (1.0 / 9007199254740992.0)) - 1.0;
        v[c] = x;
        vprev[c] = 0.0;
        ss = fma(x, x, ss);
    }
    ss = block_sum(ss, red);
    const double inv0 = (ss > 0.0) ? 1.0 / sqrt(ss) : 0.0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) v[c] *= inv0;
    if (threadIdx.x == 0) {
        st[0] = 0.0;
        st[1] = 0.0;
        st[2] = 0.0;
    }
}

__global__ void k_lz_matvec(int n, const double* __restrict__ A, int lda, const double* __restrict__ v,
                            double* __restrict__ u, const double* __restrict__ st) {
    PDL_ENTER();
    PDL_ARG(A); PDL_ARG(v); PDL_ARG(u); PDL_ARG(st);
    if (st[2] != 0.0) return;
    const int row = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (row >= n) return;
    const double* col = A + (int64_t)row * lda;
    double acc = 0.0;
    for (int c = lane; c < n; c += 32) acc = fma(col[c], v[c], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) u[row] = acc;
}

// u <- u - beta_{j-1} v_{j-1}; alpha_j = v_j^T u; u <- u - alpha_j v_j; beta_j = ||u||;
// v_{j+1} = u / beta_j, written over v_{j-1}. On breakdown (or after it) T's entries are zero.
__global__ void __launch_bounds__(LZG_THREADS) k_lz_update(int n, int j, double* __restrict__ u,
                                                           const double* __restrict__ v, double* __restrict__ vprev,
                                                           double* __restrict__ st, double* dgl, double* eoff) {
    PDL_ENTER();
    PDL_ARG(u); PDL_ARG(v); PDL_ARG(vprev); PDL_ARG(st); PDL_ARG(dgl); PDL_ARG(eoff);
    __shared__ double red[32];
    if (st[2] != 0.0) {
        if (threadIdx.x == 0) {
            dgl[j] = 0.0;
            eoff[j] = 0.0;
        }
        return;
    }
    const double beta = st[0];
    double a = 0.0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        const double x = fma(-beta, vprev[c], u[c]);
        u[c] = x;
        a = fma(v[c], x, a);
    }
    a = block_sum(a, red);
    double b2 = 0.0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        const double x = fma(-a, v[c], u[c]);
        u[c] = x;
        b2 = fma(x, x, b2);
    }
    b2 = block_sum(b2, red);
    const double rb = (b2 > 0.0) ? rsqrt(b2) : 0.0;
    const double b = b2 * rb;
    const double anorm = fmax(st[1], fabs(a) + b + beta);
    const bool stop = !(b > 16.0 * DBL_EPSILON * anorm);
    for (int c = threadIdx.x; c < n; c += blockDim.x) vprev[c] = stop ? 0.0 : u[c] * rb;
    __syncthreads();   // every thread has read st before thread 0 updates it
    if (threadIdx.x == 0) {
        dgl[j] = a;
        eoff[j] = stop ? 0.0 : b;
        st[0] = b;
        st[1] = anorm;
        st[2] = stop ? 1.0 : 0.0;
    }
}

// (theta_1, theta_2, |z_m|, beta_m) of the Lanczos tridiagonal: its two largest eigenvalues, the last
// entry of the unit eigenvector of theta_1, and the residual norm after the last step.
// (z: the inverse-iteration vector before its normalisation by *fac).
__global__ void k_lanczos_pack(int m, const double* w, const double* z, const double* fac, const double* eoff,
                               double* out) {
    PDL_ENTER();
    PDL_ARG(w); PDL_ARG(z); PDL_ARG(fac); PDL_ARG(eoff); PDL_ARG(out);
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    out[0] = w[m >= 2 ? 1 : 0];
    out[1] = (m >= 2) ? w[0] : -DBL_MAX;
    out[2] = fabs(z[m - 1] * fac[0]);
    out[3] = eoff[m - 1];
}

__global__ void k_copy_sq(int n, const double* A, int lda, double* B) {
    PDL_ENTER();
    PDL_ARG(A); PDL_ARG(B);
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)n * n) return;
    const int r = (int)(e % n), c = (int)(e / n);
    // symmetrise on the way in
    B[(int64_t)c * n + r] = 0.5 * (A[(int64_t)c * lda + r] + A[(int64_t)r * lda + c]);
}

}  // namespace

constexpr int kBlockClusterMin = 48;   // clusters of this many columns or more: block Gram-Schmidt
int symeig_orth_clusters(int n, int nv, const double* w, double* Z, int ldz, SymEigWork* ws, double cluster_rel,
                         int maxc, cudaStream_t s);
int symeig_backtransform(int n, int nv, double* Z, int ldz, SymEigWork* ws, cudaStream_t s);

// the cooperative grid from here when its columns fit: at n = 288 a column step takes about 5 us on either path, beyond it
// the columns of 16 CTAs grow with n while those of the grid's up to 152 stay few
constexpr int kResMinN = 288;
constexpr int kWyMinN = 64;   // back-transformation in blocks of reflectors from here; below it one launch serves

size_t symeig_work_bytes(int n, int nv) {
    const size_t nn = (size_t)n * n;
    size_t b = 0;
    auto add = [&](size_t cnt) { b += ((cnt * sizeof(double) + 255) / 256) * 256; };
    add(nn + 16 * (size_t)n);   // A (the cluster path keeps up to n + 16 columns of n; the grid path its exchange of p)
    add(n >= kResMinN ? nn : 0);   // X (the grid path's exchange of columns)
    add(nn);            // HV
    add(n);             // d
    add(n);             // e
    add(n);             // tau
    add(4 * (size_t)n); // vbuf
    add(5 * (size_t)n * std::max(nv, 1) + (size_t)n * std::max(nv, 1));  // lu + Zt
    return b + 4096;
}

int symeig_work_carve(Arena& a, int n, int nv, GridBarrier bar, SymEigWork* w) {
    const size_t nn = (size_t)n * n;
    w->A = a.take<double>(nn + 16 * (size_t)n);
    w->X = a.take<double>(n >= kResMinN ? nn : 0);
    w->partial = a.take<double>(nn);      // HV
    w->dgl = a.take<double>(n);
    w->eoff = a.take<double>(n);
    w->tau = a.take<double>(n);
    w->vbuf = a.take<double>(4 * (size_t)n);
    w->lu = a.take<double>(6 * (size_t)n * std::max(nv, 1));
    w->bar = bar;
    w->max_ctas = 0;
    if (!w->A || !w->partial || !w->dgl || !w->eoff || !w->tau || !w->vbuf || !w->lu || !w->X) return EDA_ERR_OOM;
    w->xn = n >= kResMinN ? n : 0;
    return EDA_OK;
}

constexpr int kClusterMaxN = 512;        // the cluster path up to here; a cooperative grid beyond
constexpr int kClusterMaxNShared = 1024; // limit of the cluster path when the GPU is shared (see below)

// Host threads that run many problems side by side (the batched solver) set this: a cooperative
// grid with a software grid barrier needs all its CTAs resident at once, which concurrent kernels
// of other problems can delay beyond the barrier's limit, while a thread-block cluster is scheduled
// as one unit by the hardware. Such threads take the cluster path (matrix in a global slab) up to
// kClusterMaxNShared.
thread_local bool tl_shared_gpu = false;

// Launch k_tridiag_x on one cluster of C CTAs (a power of two, 16 only when the device accepts that non-portable
// cluster size with the needed shared memory).
int launch_tridiag_cluster(int C, int n, const double* A, int lda, SymEigWork* ws, int* status, cudaStream_t s,
                           bool probe_only, bool* fits) {
    auto kern = k_tridiag_x<true>;
    static std::mutex mu;                 // the function attributes below are shared by all threads
    static size_t smem_set = 0;
    static bool attrs = false;
    const int ncl = (n + C - 1) / C;
    const size_t vec_bytes = (5 * (size_t)n + td_dots(ncl)) * sizeof(double);
    const size_t a_bytes = (size_t)ncl * n * sizeof(double);
    const int in_smem = (vec_bytes + a_bytes <= 220 * 1024) ? 1 : 0;
    const size_t smem = vec_bytes + (in_smem ? a_bytes : 0);
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!attrs) {
            attrs = true;
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            cudaGetLastError();
        }
        if (smem > smem_set) {
            EDA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)std::max<size_t>(smem, 48 * 1024)));
            smem_set = std::max<size_t>(smem, 48 * 1024);
        }
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(TD_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (probe_only) {
        int nclusters = 0;
        *fits = cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess && nclusters >= 1;
        cudaGetLastError();
        return EDA_OK;
    }
    ProfScope prof("tridiag", s, 4.0 / 3.0 * (double)n * n * n);
    EDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, n, A, lda, ws->A, in_smem, (double*)nullptr, (double*)nullptr, ws->partial,
                                    ws->dgl, ws->eoff, ws->tau, 0LL, status));
    launch_counter()++;
    return EDA_OK;
}

int tridiag_cluster(int n, const double* A, int lda, SymEigWork* ws, int* status, cudaStream_t s) {
    static int chosen_C[kClusterMaxNShared + 1] = {};   // cluster size that passed the occupancy check, per n
    static std::mutex mu;
    std::unique_lock<std::mutex> lk(mu);
    if (!chosen_C[n]) {
        // eight columns or more per CTA, one for each warp of the pass (4, 6 and 12 measured within 3 %, n = 48 .. 200)
        int want = 1;
        while (want < 16 && want * 2 * 8 <= n) want *= 2;
        int C = std::max(2, want);
        for (; C > 2; C /= 2) {
            bool fits = false;
            EDA_TRY(launch_tridiag_cluster(C, n, A, lda, ws, status, s, true, &fits));
            if (fits) break;
        }
        chosen_C[n] = C;
    }
    const int C = chosen_C[n];
    lk.unlock();
    return launch_tridiag_cluster(C, n, A, lda, ws, status, s, false, nullptr);
}

// k_tridiag_x on a cooperative grid: about four columns per CTA, at most one CTA per SM, when the owned columns and
// three work vectors fit in 220 KB of shared memory. INVALID_ARG: does not apply.
int tridiag_res(int n, const double* A, int lda, double* HV, SymEigWork* ws, int* status, int sms, cudaStream_t s) {
    const int G = std::max(1, std::min(sms, (n + 3) / 4));
    const int ncl = (n + G - 1) / G;
    const size_t smem = ((size_t)(ncl + 3) * n + td_dots(ncl)) * sizeof(double);
    if (smem > 220 * 1024 || ws->xn < n) return EDA_ERR_INVALID_ARG;
    auto kern = k_tridiag_x<false>;
    {
        static std::mutex mu;
        static size_t set = 0;
        std::lock_guard<std::mutex> lk(mu);
        if (smem > set && smem > 40 * 1024) {
            EDA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)std::max<size_t>(smem, 48 * 1024)));
            set = std::max<size_t>(smem, 48 * 1024);
        }
    }
    int per_sm = 0;
    EDA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TD_THREADS, smem));
    if (per_sm < 1 || G > per_sm * sms) return EDA_ERR_INVALID_ARG;
    // both exchange buffers to the "not written yet" pattern
    EDA_CUDA_TRY(cudaMemsetAsync(ws->A, 0xFF, (size_t)n * n * sizeof(double), s));
    EDA_CUDA_TRY(cudaMemsetAsync(ws->X, 0xFF, (size_t)n * n * sizeof(double), s));
    ProfScope prof("tridiag", s, 4.0 / 3.0 * (double)n * n * n);
    int nn = n, ld = lda, insm = 1;
    const double* a0 = A;
    double* ag = nullptr;
    double* pb = ws->A;
    double* cb = ws->X;
    double* a1 = HV;
    double* a2 = ws->dgl;
    double* a3 = ws->eoff;
    double* a4 = ws->tau;
    long long spin = ws->bar.spin_limit;
    int* st = status;
    void* args[] = {&nn, &a0, &ld, &ag, &insm, &pb, &cb, &a1, &a2, &a3, &a4, &spin, &st};
    EDA_CUDA_TRY(cudaLaunchCooperativeKernel((void*)kern, dim3(G), dim3(TD_THREADS), args, smem, s));
    launch_counter()++;
    return EDA_OK;
}

int symeig_values(int n, const double* A, int lda, int il, int iu, double* w, SymEigWork* ws, int* status,
                  cudaStream_t s) {
    if (n <= 0 || il < 0 || iu >= n || il > iu) return EDA_ERR_INVALID_ARG;
    EDA_CUDA_TRY(cudaPeekAtLastError());   // surface an error left by an earlier call at its own site
    const int nv = iu - il + 1;
    double* HV = ws->partial;
    // ---- tridiagonal reduction: resident-column grid, cluster, or L2-streaming grid (see the file header) ----
    int dev = 0;
    EDA_CUDA_TRY(cudaGetDevice(&dev));
    int sms = 0;
    EDA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // dynamic shared memory near 48 KB needs the opt-in too: the kernels also hold static shared
    // variables, and the default limit covers static + dynamic
    const size_t smem = 2 * (size_t)n * sizeof(double);
    if (smem > 40 * 1024) {
        // raise-only, under a lock: concurrent solves of different sizes share the attribute
        static std::mutex mu;
        static size_t set = 0;
        std::lock_guard<std::mutex> lk(mu);
        if (smem > set) {
            EDA_CUDA_TRY(cudaFuncSetAttribute(k_tridiag, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            set = smem;
        }
    }
    int res = EDA_ERR_INVALID_ARG;   // the resident-column grid when it applies and fits
    if (!tl_shared_gpu && n >= kResMinN) res = tridiag_res(n, A, lda, HV, ws, status, sms, s);
    if (res == EDA_OK) {
    } else if (res != EDA_ERR_INVALID_ARG) {
        return res;
    } else if (n <= (tl_shared_gpu ? kClusterMaxNShared : kClusterMaxN)) {
        EDA_TRY(tridiag_cluster(n, A, lda, ws, status, s));
    } else {
    int per_sm = 0;
    EDA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tridiag, TRI_THREADS, smem));
    // about 8 rows per CTA: more CTAs shorten each column step's FP64 chains (16 rows per CTA measured
    // 10 % slower at the Rayleigh-Ritz sizes 576-704; fewer than 8 rows gained nothing)
    int ctas = std::max(1, std::min(n / 8, sms));
    ctas = std::min(ctas, std::max(1, per_sm * sms));
    double* pglob = ws->vbuf;
    EDA_CUDA_TRY(cudaMemsetAsync(ws->bar.count, 0, sizeof(unsigned), s));
    EDA_CUDA_TRY((launch_chained(k_copy_sq, dim3(ceil_div((int64_t)n * n, 256)), dim3(256), 0, s, n, A, lda, ws->A)));
    {
        ProfScope prof("tridiag", s, 4.0 / 3.0 * (double)n * n * n);
        int nn = n;
        double* a0 = ws->A;
        double* a1 = HV;
        double* a2 = ws->dgl;
        double* a3 = ws->eoff;
        double* a4 = ws->tau;
        double* a5 = pglob;
        GridBarrier b = ws->bar;
        int* st = status;
        void* args[] = {&nn, &a0, &a1, &a2, &a3, &a4, &a5, &b, &st};
        EDA_CUDA_TRY(cudaLaunchCooperativeKernel((void*)k_tridiag, dim3(ctas), dim3(TRI_THREADS), args, smem, s));
        launch_counter()++;
    }
    }
    // ---- eigenvalues ----
    EDA_CUDA_TRY(cudaPeekAtLastError());
    const size_t bsm = 3 * (size_t)n * sizeof(double);
    if (bsm > 40 * 1024) {
        static std::mutex mu;
        static size_t set = 0;
        std::lock_guard<std::mutex> lk(mu);
        if (bsm > set) {
            EDA_CUDA_TRY(cudaFuncSetAttribute(k_bisect, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bsm));
            set = bsm;
        }
    }
    {
        ProfScope prof("bisect", s);
        // one warp per CTA: the FP64 pipe of one SM is narrow, so the warps are spread over SMs
        EDA_CUDA_TRY((launch_chained(k_bisect, dim3(nv), dim3(64), bsm, s, n, ws->dgl, ws->eoff, il, nv, w)));
    }
    return EDA_OK;
}

namespace {
// Inverse iteration for the nv eigenvalues w of the tridiagonal in ws, vectors into Z (n x nv, ldz).
int invit_vectors(int n, int nv, const double* w, double* Z, int ldz, SymEigWork* ws, uint64_t seed, cudaStream_t s) {
    double* lu = ws->lu;
    double* Zt = ws->lu + 5 * (size_t)n * nv;
    {
        ProfScope prof("invit", s);
        EDA_CUDA_TRY((launch_chained(k_invit, dim3(ceil_div(nv, 32)), dim3(32), 0, s, n, nv, ws->dgl, ws->eoff, w, lu,
            Zt, seed)));
    }
    // the normalisation factors: row 0 of the reciprocal pivots
    EDA_CUDA_TRY((launch_chained(k_transpose_out, dim3(ceil_div(n, 32), ceil_div(nv, 32)), dim3(256), 0, s, n, nv, Zt,
        lu + (size_t)n * nv, Z, ldz)));
    return EDA_OK;
}
}  // namespace

int symeig_vectors(int n, int nv, const double* w, double* Z, int ldz, SymEigWork* ws, uint64_t seed,
                   double cluster_rel, cudaStream_t s) {
    if (nv <= 0) return EDA_OK;
    EDA_TRY(invit_vectors(n, nv, w, Z, ldz, ws, seed, s));
    EDA_TRY(symeig_orth_clusters(n, nv, w, Z, ldz, ws, cluster_rel, kBlockClusterMin, s));
    return symeig_backtransform(n, nv, Z, ldz, ws, s);
}

int symeig_f64(int n, const double* A, int lda, int il, int iu, double* w, double* Z, int ldz, SymEigWork* ws,
               int* status, uint64_t seed, double cluster_rel, cudaStream_t s) {
    ProfScope prof("symeig", s);
    EDA_TRY(symeig_values(n, A, lda, il, iu, w, ws, status, s));
    if (!Z) return EDA_OK;
    return symeig_vectors(n, iu - il + 1, w, Z, ldz, ws, seed, cluster_rel, s);
}

// Cluster MGS with a tolerance relative to max |lambda|, computed on the device.
namespace {
__global__ void k_cluster_scale(int nv, const double* lam, double rel, double* out) {
    PDL_ENTER();
    PDL_ARG(lam); PDL_ARG(out);
    double m = 0.0;
    for (int i = threadIdx.x; i < nv; i += 32) m = fmax(m, fabs(lam[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) out[0] = rel * m;
}
// Columns Z[:, 0 .. bs) (bs <= 16), already orthogonal to every earlier column of their cluster: each column
// against the earlier ones of the block by classical Gram-Schmidt applied twice (the dot products of a pass
// on one warp each, the update on all threads), then normalised. Computed from the vectors themselves (not
// their Gram matrix), like the column-by-column loop it replaces, so nearly dependent inverse-iteration
// vectors of a tight cluster keep their content above the rounding level.
constexpr int kClusterBlock = 16;
__global__ void __launch_bounds__(512) k_cluster_block_cgs2(int n, double* Z, int ldz, int bs) {
    PDL_WAIT();
    PDL_ARG(Z);
    __shared__ double dots[kClusterBlock];
    __shared__ double red[16];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int c = 0; c < bs; ++c) {
        double* zc = Z + (int64_t)c * ldz;
        for (int pass = 0; pass < 2 && c > 0; ++pass) {
            if (warp < c) {
                const double* zw = Z + (int64_t)warp * ldz;
                double dot = 0.0;
                for (int i = lane; i < n; i += 32) dot = fma(zw[i], zc[i], dot);
                for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                if (lane == 0) dots[warp] = dot;
            }
            __syncthreads();
            for (int i = tid; i < n; i += blockDim.x) {
                double acc = 0.0;
                for (int w = 0; w < c; ++w) acc = fma(dots[w], Z[(int64_t)w * ldz + i], acc);
                zc[i] -= acc;
            }
            __syncthreads();
        }
        double nrm = 0.0;
        for (int i = tid; i < n; i += blockDim.x) nrm = fma(zc[i], zc[i], nrm);
        for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
        if (lane == 0) red[warp] = nrm;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
            red[0] = t > 0.0 ? 1.0 / sqrt(t) : 0.0;
        }
        __syncthreads();
        const double sc = red[0];
        for (int i = tid; i < n; i += blockDim.x) zc[i] *= sc;
        __syncthreads();
    }
}

// Modified Gram-Schmidt (two passes) inside each run of eigenvalues whose consecutive gaps are <= ctol,
// one warp per run; runs of maxc or more columns are left to the block path.
__global__ void k_cluster_mgs_dev(int n, int nv, const double* lam, const double* ctol_dev, double* Z, int ldz,
                                  int maxc) {
    PDL_ENTER();
    PDL_ARG(lam); PDL_ARG(ctol_dev); PDL_ARG(Z);
    const double ctol = ctol_dev[0];
    const int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= nv) return;
    if (q > 0 && lam[q] - lam[q - 1] <= ctol) return;
    int end = q + 1;
    while (end < nv && lam[end] - lam[end - 1] <= ctol) ++end;
    if (end - q < 2 || end - q >= maxc) return;
    for (int c = q + 1; c < end; ++c) {
        double* zc = Z + (int64_t)c * ldz;
        for (int pass = 0; pass < 2; ++pass) {
            for (int pcol = q; pcol < c; ++pcol) {
                const double* zp = Z + (int64_t)pcol * ldz;
                double dot = 0.0;
                for (int i = lane; i < n; i += 32) dot = fma(zp[i], zc[i], dot);
                for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                for (int i = lane; i < n; i += 32) zc[i] = fma(-dot, zp[i], zc[i]);
            }
        }
        double nrm = 0.0;
        for (int i = lane; i < n; i += 32) nrm = fma(zc[i], zc[i], nrm);
        for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
        const double sc = nrm > 0.0 ? 1.0 / sqrt(nrm) : 0.0;
        for (int i = lane; i < n; i += 32) zc[i] *= sc;
    }
}
}  // namespace

// Orthogonalisation of the inverse-iteration vectors inside eigenvalue clusters (runs whose consecutive
// gaps are <= cluster_rel * max |w|), in the tridiagonal basis. Runs shorter than maxc columns: modified
// Gram-Schmidt (two passes) by one warp each (k_cluster_mgs_dev). Longer runs (when eigenvalues span many
// orders of magnitude, every value near the bottom of the spectrum falls within one such run): blocks of
// kClusterBlock columns in order, each first made orthogonal to the earlier blocks of its run by block
// classical Gram-Schmidt applied twice with the multi-CTA products, then orthonormalised column by column
// (k_cluster_block_cgs2). In exact arithmetic this is the same Gram-Schmidt basis as the column loop, and
// like it every step works on the vectors, never on their Gram matrix. The cluster bounds are found on the
// host with the device's criterion and operations.
int symeig_orth_clusters(int n, int nv, const double* w, double* Z, int ldz, SymEigWork* ws, double cluster_rel,
                         int maxc, cudaStream_t s) {
    double* ctol = ws->vbuf + 2 * n;
    EDA_CUDA_TRY((launch_chained(k_cluster_scale, dim3(1), dim3(32), 0, s, nv, w, cluster_rel, ctol)));
    EDA_CUDA_TRY((launch_chained(k_cluster_mgs_dev, dim3(ceil_div((int64_t)nv * 32, 256)), dim3(256), 0, s, n, nv, w,
        ctol, Z, ldz, maxc)));
    if (maxc == INT_MAX || nv < maxc) return EDA_OK;
    std::vector<double> wh(nv);
    EDA_TRY(read_back(wh.data(), w, nv * sizeof(double), s));
    double mx = 0.0;
    for (int i = 0; i < nv; ++i) mx = std::fmax(mx, std::fabs(wh[i]));
    const double tol = cluster_rel * mx;
    std::vector<std::pair<int, int>> big;
    for (int q = 0; q < nv;) {
        int end = q + 1;
        while (end < nv && wh[end] - wh[end - 1] <= tol) ++end;
        if (end - q >= maxc) big.emplace_back(q, end);
        q = end;
    }
    if (big.empty()) return EDA_OK;
    ProfScope prof("cluster_orth", s);
    // scratch in the inverse-iteration factors (free once the vectors are in Z)
    constexpr int BS = kClusterBlock;
    double* C = ws->lu;                                   // nv x BS
    double* part = C + (size_t)nv * BS;
    const size_t cap = 6 * (size_t)n * nv;
    if ((size_t)nv * BS * 2 > cap) return EDA_ERR_INVALID_ARG;
    const size_t pcap = cap - (size_t)nv * BS;
    for (const auto& cl : big) {
        const int q = cl.first, end = cl.second;
        double* Zq = Z + (size_t)q * ldz;
        for (int j0 = q; j0 < end; j0 += BS) {
            const int bs = std::min(BS, end - j0);
            double* Zj = Z + (size_t)j0 * ldz;
            const int prev = j0 - q;
            for (int pass = 0; pass < 2 && prev > 0; ++pass) {
                EDA_TRY(gemm_tn_f64(n, prev, bs, 1.0, Zq, ldz, Zj, ldz, 0.0, C, prev, part, pcap, s));
                EDA_TRY(gemm_nn_f64(n, prev, bs, -1.0, Zq, ldz, C, prev, 1.0, Zj, ldz, Zj, ldz, s));
            }
            EDA_CUDA_TRY((launch_chained(k_cluster_block_cgs2, dim3(1), dim3(512), 0, s, n, Zj, ldz, bs)));
        }
    }
    return EDA_OK;
}

// Householder back-transformation of the tridiagonal eigenvectors Z (reflectors still in ws).
namespace {
template <int NC>
int wy_apply(int n, int nv, double* Z, int ldz, SymEigWork* ws, cudaStream_t s) {
    const size_t smem = (size_t)NC * n * sizeof(double);
    {
        // raise-only, under a lock: concurrent solves of different sizes share the attribute
        static std::mutex mu;
        static size_t set = 0;
        std::lock_guard<std::mutex> lk(mu);
        if (smem > set && smem > 32 * 1024) {
            EDA_CUDA_TRY(cudaFuncSetAttribute(k_wy_apply<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            set = smem;
        }
    }
    EDA_CUDA_TRY((launch_spread(k_wy_apply<NC>, dim3(ceil_div(nv, NC)), dim3(256), smem, s, n, nv, ws->partial, ws->tau,
        ws->A, Z, ldz)));
    return EDA_OK;
}
}  // namespace

int symeig_backtransform(int n, int nv, double* Z, int ldz, SymEigWork* ws, cudaStream_t s) {
    if (n < 3) return EDA_OK;
    ProfScope prof("backtransform", s);
    if (n < kWyMinN) {
        EDA_CUDA_TRY((launch_spread(k_backtransform_w4<2>, dim3(nv), dim3(128), 0, s, n, nv, ws->partial, ws->tau, Z, ldz)));
        return EDA_OK;
    }
    // the blocks' triangles go into the matrix copy, which the reduction has done with (n^2 + 16 n doubles hold them)
    EDA_CUDA_TRY((launch_spread(k_wy_gram, dim3(ceil_div(n - 2, WY_B), 8), dim3(256), 0, s, n, ws->partial, ws->A)));
    // columns per CTA: one wave of CTAs, at most eight, as many as fit in 200 KB
    const int fit = (int)std::max<size_t>(1, 200 * 1024 / ((size_t)n * sizeof(double)));
    const int nc = std::min(std::min(8, ceil_div(nv, sm_count())), fit);
    switch (nc) {
        case 1: return wy_apply<1>(n, nv, Z, ldz, ws, s);
        case 2: return wy_apply<2>(n, nv, Z, ldz, ws, s);
        case 3: return wy_apply<3>(n, nv, Z, ldz, ws, s);
        case 4: return wy_apply<4>(n, nv, Z, ldz, ws, s);
        case 5: return wy_apply<5>(n, nv, Z, ldz, ws, s);
        case 6: return wy_apply<6>(n, nv, Z, ldz, ws, s);
        case 7: return wy_apply<7>(n, nv, Z, ldz, ws, s);
        default: return wy_apply<8>(n, nv, Z, ldz, ws, s);
    }
}

int newton_schulz_f64(int n, int nv, double* Z, int ldz, int steps, double* tmp, double* partial, size_t partial_cap,
                      cudaStream_t s) {
    double* G = tmp;                       // nv x nv
    double* Zn = tmp + (size_t)nv * nv;    // n x nv
    for (int it = 0; it < steps; ++it) {
        EDA_TRY(syrk_f64(n, nv, 1.0, Z, ldz, 0.0, G, nv, partial, partial_cap, s));
        // Zn = 1.5 Z - 0.5 Z G
        EDA_TRY(gemm_nn_f64(n, nv, nv, -0.5, Z, ldz, G, nv, 1.5, Z, ldz, Zn, n, s));
        EDA_TRY(copy_mat_f64(n, nv, Zn, n, Z, ldz, s));
    }
    return EDA_OK;
}

int lanczos_top(int n, const double* A, int lda, int m, uint64_t seed, SymEigWork* ws, double* out,
                cudaStream_t s) {
    if (n < 1 || m < 1 || m > n) return EDA_ERR_INVALID_ARG;
    if (n > kLanczosMaxN) {
        // three n-vectors in vbuf (4 n doubles), the state after them in lu
        double* buf[3] = {ws->vbuf, ws->vbuf + n, ws->vbuf + 2 * (size_t)n};
        double* st = ws->lu;
        {
            ProfScope prof("lanczos", s);
            EDA_CUDA_TRY((launch_chained(k_lz_start, dim3(1), dim3(LZG_THREADS), 0, s, n, seed, buf[0], buf[1], st)));
            // v_j in buf[j % 2], v_{j-1} (then v_{j+1}) in buf[(j + 1) % 2], u in buf[2]
            for (int j = 0; j < m; ++j) {
                double* v = buf[j & 1];
                double* vp = buf[(j + 1) & 1];
                EDA_CUDA_TRY((launch_chained(k_lz_matvec, dim3(ceil_div((int64_t)n * 32, 256)), dim3(256), 0, s, n, A,
                    lda, v, buf[2], st)));
                EDA_CUDA_TRY((launch_chained(k_lz_update, dim3(1), dim3(LZG_THREADS), 0, s, n, j, buf[2], v, vp, st,
                    ws->dgl, ws->eoff)));
            }
        }
        const int nv = m >= 2 ? 2 : 1;
        double* w = ws->vbuf + 3 * (size_t)n;       // nv values (vbuf holds 4 n doubles)
        double* zt = ws->lu + 5 * (size_t)m;        // the eigenvector after the 5 m factor entries
        EDA_CUDA_TRY((launch_chained(k_bisect, dim3(nv), dim3(64), 3 * (size_t)m * sizeof(double), s, m, ws->dgl,
            ws->eoff, m - nv, nv, w)));
        EDA_CUDA_TRY((launch_chained(k_invit, dim3(1), dim3(32), 0, s, m, 1, ws->dgl, ws->eoff, w + nv - 1, ws->lu, zt, seed)));   // st is dead here
        EDA_CUDA_TRY((launch_chained(k_lanczos_pack, dim3(1), dim3(32), 0, s, m, w, zt, ws->lu + m, ws->eoff, out)));
        return EDA_OK;
    }
    const int C = (n + LZ_ROWS - 1) / LZ_ROWS;
    {
        static std::once_flag once;
        std::call_once(once, [] {
            cudaFuncSetAttribute(k_lanczos, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            cudaGetLastError();
        });
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(LZ_THREADS);
    cfg.dynamicSmemBytes = (size_t)(LZ_ROWS + 1) * n * sizeof(double);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    {
        ProfScope prof("lanczos", s);
        EDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_lanczos, n, A, lda, m, seed, ws->dgl, ws->eoff));
        launch_counter()++;
    }
    // the two largest eigenvalues of T_m and the eigenvector of the largest
    const int nv = m >= 2 ? 2 : 1;
    double* w = ws->vbuf;                       // nv values
    double* zt = ws->lu + 5 * (size_t)m;        // the eigenvector (m entries) after the 5 m factor entries
    EDA_CUDA_TRY((launch_chained(k_bisect, dim3(nv), dim3(64), 3 * (size_t)m * sizeof(double), s, m, ws->dgl, ws->eoff,
        m - nv, nv, w)));
    EDA_CUDA_TRY((launch_chained(k_invit, dim3(1), dim3(32), 0, s, m, 1, ws->dgl, ws->eoff, w + nv - 1, ws->lu, zt, seed)));
    EDA_CUDA_TRY((launch_chained(k_lanczos_pack, dim3(1), dim3(32), 0, s, m, w, zt, ws->lu + m, ws->eoff, out)));
    return EDA_OK;
}

bool symeig_set_shared_gpu(bool on) {
    const bool prev = tl_shared_gpu;
    tl_shared_gpu = on;
    return prev;
}

}  // namespace eda
