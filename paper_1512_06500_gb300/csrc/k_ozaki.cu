// FP64-accurate tall-skinny products on the bf16 tensor cores by error-free splitting of the operands
// into integer digit planes (Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its applications", Numerical
// Algorithms 59, 2012), arranged for tcgen05.
//
// Splitting. Each row i of an operand (the rows of the MMA's M or N side; the reduction index k runs
// along it) gets a power-of-two scale 2^{e_i} with |a_ik| < 2^{e_i}. Then
//     a_ik = 2^{e_i - 7} (s_0 + 2^-8 s_1 + ... + 2^-48 s_6) + tail,   |tail| <= 2^{e_i - 56},
// with integer digits s_q in [-128, 128]: the balanced base-256 digits of the integer nearest to
// a 2^{55 - e}, extracted with integer operations from the bits of a. A digit is exact in bf16 (8
// significant bits).
//
// Products. For D = A B^T over the reduction index (A: M x K, B: N x K, both split),
//     D_ij = 2^{e_i + f_j - 14} sum_q 2^{-8q} L_q,    L_q = sum_{a + b = q} sum_k s^A_{a,ik} s^B_{b,jk},
// truncated at q <= 6 (28 digit-plane products; the dropped terms and both tails are below 2^-53 of
// max_k |a_ik| sum_k |b_jk|). A level L_q summed over a chunk of 128 values of k is an integer below
// (q + 1) 128 2^14 < 2^24, so the tensor cores' FP32 accumulation of a chunk is exact. Each chunk's
// seven levels are read out of tensor memory, converted to integers and folded into two 64-bit
// integer sums per output (G_0 = L_0 2^16 + L_1 2^8 + L_2 and G_1 = L_3 2^24 + L_4 2^16 + L_5 2^8 + L_6),
// so the reduction over k is exact as well; the only roundings are the final conversion to FP64 and the
// 2^-56 truncation of the digits.
//
// Kernel. A CTA works on a run of K stages of one or several 128-row bands of M, 256 threads: thread 0 issues the bulk copies of
// the pre-tiled digit planes of A (one contiguous 16 KB swizzled tile per K stage of 64 and plane) and
// the TMA boxes of the seven planes of B; thread 32 issues tcgen05.mma (M = 128, K = 16, N = 32 (7 - a) for
// digit plane a of A against planes 0 .. 6 - a of B at once) into one of two accumulator sets of seven
// levels in tensor memory (7 x 32 columns each), switching sets every chunk of two K stages; warps 4-7
// drain a finished set (tcgen05.ld, integer fold) while the tensor cores fill the other. Every wait is
// bounded (ST_TIMEOUT on give-up).
#include "tc_ptx.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

namespace eda {

using namespace tc;

namespace {

constexpr int OZ_S = kOzSlices;       // digit planes
constexpr int OZ_N = 32;              // N of every MMA: the narrow operand's columns per launch
constexpr int OZ_AST = 8;             // A ring slots (one 16 KB tile of one plane each)
constexpr int OZ_BST = 2;             // B ring slots (the seven 32 x 64 planes of one K stage)
constexpr int OZ_THREADS = 256;
constexpr int kOzJoinStages = 3;      // what k_oz_join costs, in K stages of a CTA
constexpr int OZ_SET_COLS = 256;      // tensor-memory columns of one accumulator set (7 levels x 32)

struct OzRing {
    __nv_bfloat16 A[OZ_AST][TC_M * TC_KS];            // 8 x 16 KB
    __nv_bfloat16 B[OZ_BST][OZ_S][OZ_N * TC_KS];      // 2 x 7 x 4 KB
    uint64_t fullA[OZ_AST], emptyA[OZ_AST];
    uint64_t fullB[OZ_BST], emptyB[OZ_BST];
    uint64_t accFull[2], accEmpty[2];
    uint32_t tbase;
    int fail;
};
constexpr size_t oz_smem_bytes() { return sizeof(OzRing) + 1024; }

__device__ __forceinline__ OzRing& oz_ring(unsigned char* raw) {
    const uint32_t mis = smem_u32(raw) & 1023u;
    return *reinterpret_cast<OzRing*>(raw + ((1024u - mis) & 1023u));
}

// B from a pre-tiled split operand (BT mode): its planes at tiles + q * slice, kbs tiles along K per band; the
// product's 32-column block x (blockIdx.x mod nblk) is the quarter x % 4 of B's 128-row band x / 4, one contiguous
// 4 KB image per plane and stage, and the band of A is blockIdx.x / nblk: the CTAs that run together share few bands of A,
// whose tiles they then find in L2. upper: skip the blocks wholly below the diagonal (x 32 + 32 <= band 128).
struct OzBTiles {
    const __nv_bfloat16* tiles = nullptr;
    int64_t slice = 0;
    int kbs = 0;
    int nblk = 1;   // 32-column blocks
    int upper = 0;
};

// A narrow product with more bands than SMs (RUNS): the K stages of all bands, band after band, are dealt to the CTAs of
// one wave in contiguous runs, one per CTA. The roles run through the bands of their run without a pause: the copies of a
// band's first stages are in flight, and its MMAs run, while the previous band is still being folded and written. A band that
// lies in one run is written to D; of a band that several runs share, each writes the sum over its stages to its own 128 x N
// slot of partial (a run has at most two such pieces, its first, slot 2 c, and its last, slot 2 c + 1), and k_oz_join adds them
// in the order of k. One CTA a band took four rounds of 152 for 3.4 rounds of work, each with its own start and end
// (65536 x 2200 times 32 columns: 408 -> 340 us). With fewer bands than SMs the split of K stays the same for all bands: the
// CTAs of one split read the same stages of B at the same time (2200 x 65536 times 32 columns 315 us, in runs 363).
// unit: a run starts at a multiple of this many stages: 1, or the stages of a band (whole bands, nothing to join).
struct OzRuns {
    int kst;        // stages per band
    int unit;
    int64_t units;  // bands * kst / unit
    __host__ __device__ int64_t begin(int c, int ctas) const { return units * c / ctas * unit; }
    // the CTA whose run holds stage t
    __host__ __device__ int of(int64_t t, int ctas) const {
        return (int)(((t / unit + 1) * ctas + units - 1) / units) - 1;
    }
};

// round((g0 2^32 + g1) 2^{e - 62}), to nearest even, by integer operations. The two conversions and two ldexp of the plain form
// are some ten FP64 instructions, and a warp instruction of that pipe takes 64 cycles: 10 us for a warp's 32 x 32 results,
// against 1.5 here (one rounding instead of three).
__device__ __forceinline__ double oz_value(long long g0, long long g1, int e) {
    unsigned long long lo = ((unsigned long long)g0 << 32) + (unsigned long long)g1;
    long long hi = (g0 >> 32) + (g1 >> 63) + (lo < (unsigned long long)g1 ? 1 : 0);
    const bool neg = hi < 0;
    if (neg) {
        lo = 0ull - lo;
        hi = ~hi + (lo == 0 ? 1 : 0);
    }
    if (hi == 0) {   // g0 2^32 + g1 below 2^64
        if (lo == 0) return 0.0;
        hi = (long long)lo;
        lo = 0;
        e -= 64;
    }
    const int lz = __clzll(hi);
    const unsigned long long m = ((unsigned long long)hi << lz) | ((lo >> 1) >> (63 - lz)), rest = lo << lz;
    unsigned long long q = m >> 11;   // 53 bits, 2^{e + 13 - lz} times q
    const unsigned rem = (unsigned)(m & 0x7ff);
    q += (rem > 0x400u || (rem == 0x400u && (rest != 0 || (q & 1)))) ? 1 : 0;
    const int ex = e + 65 - lz + 1023;   // biased exponent
    const unsigned long long sign = neg ? 1ull << 63 : 0ull;
    if (ex >= 1 && ex <= 2045) return __longlong_as_double((long long)(((unsigned long long)(ex - 1) << 52) + q | sign));
    return ldexp(__longlong_as_double((long long)((1022ull << 52) + q | sign)), ex - 1023);   // q up to 2^53: one binade more
}

// D[i, j] (i < M, j < N) = alpha * sum_k A_ik B_jk + beta * C0[i, j]; D, C0 column-major (ld ldd, ldc0),
// the split-th slice of D at D + split * split_stride. A: digit planes at At + q * aslice, pre-tiled
// (128-row bands, kbs tiles of 64 along K per band), row scales expA. B: digit planes read through tmB
// (inner = K, outer = 7 x 32 rows: plane q is rows 32 q .. 32 q + 31), or in BT mode from bt (N rows, the
// CTA's 32 of them chosen by blockIdx.x mod nblk), row scales expB. Without RUNS: one band a CTA, K stages
// [split * kps, min(kst, (split + 1) * kps)), split = blockIdx.y.
template <bool BT, bool RUNS>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_gemm(const __nv_bfloat16* __restrict__ At, int64_t aslice, int kbs, const __grid_constant__ CUtensorMap tmB,
              const OzBTiles bt, const int* __restrict__ expA, const int* __restrict__ expB, int M, int N,
              const OzRuns runs, int kps, double alpha, double beta, const double* C0, int64_t ldc0, double* D, int64_t ldd,
              int64_t split_stride, double* partial, int* status) {
    PDL_WAIT();
    PDL_ARG(At); PDL_ARG(expA); PDL_ARG(expB); PDL_ARG(C0); PDL_ARG(D); PDL_ARG(partial); PDL_ARG(status);
    extern __shared__ unsigned char smraw[];
    OzRing& sm = oz_ring(smraw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kst = runs.kst;
    const int blk = BT ? (int)blockIdx.x % bt.nblk : 0;
    // this CTA's stages: n of them from stage k0 of band0 on, going on with stage 0 of the next band
    int band0, k0, n;
    if (!RUNS) {
        band0 = BT ? (int)blockIdx.x / bt.nblk : (int)blockIdx.x;
        k0 = blockIdx.y * kps;
        n = max(0, min(kst, k0 + kps) - k0);
        D += blockIdx.y * split_stride;
    } else {
        const int64_t t0 = runs.begin(blockIdx.x, gridDim.x), t1 = runs.begin(blockIdx.x + 1, gridDim.x);
        band0 = (int)(t0 / kst);
        k0 = (int)(t0 % kst);
        n = (int)(t1 - t0);
    }
    if (BT) {
        if (bt.upper && blk * OZ_N + OZ_N <= band0 * TC_M) return;   // the whole CTA: a uniform exit
        expB += blk * OZ_N;
        N -= blk * OZ_N;
        D += (int64_t)blk * OZ_N * ldd;
        if (C0) C0 += (int64_t)blk * OZ_N * ldc0;
    }
    if (warp == 0) {
        tmem_alloc(&sm.tbase, 2 * OZ_SET_COLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < OZ_AST; ++i) {
            mbar_init(&sm.fullA[i], 1);
            mbar_init(&sm.emptyA[i], 1);
        }
        for (int i = 0; i < OZ_BST; ++i) {
            mbar_init(&sm.fullB[i], 1);
            mbar_init(&sm.emptyB[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.accFull[i], 1);
            mbar_init(&sm.accEmpty[i], 128);
        }
        fence_mbar_init();
        sm.fail = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tbase;

    int issuedA = 0, issuedB = 0;   // producer: copies requested (for the drain after a give-up)
    bool ok = true;
    if (tid == 0) {
        // ---- producer ----
        constexpr uint32_t abytes = TC_M * TC_KS * 2;
        constexpr uint32_t bbytes = OZ_S * OZ_N * TC_KS * 2;
        int band = band0, kstage = k0;
        for (int s = 0; s < n && ok; ++s) {
            const int bslot = s % OZ_BST;
            if (s >= OZ_BST && !(ok = mbar_wait(&sm.emptyB[bslot], ((s / OZ_BST) - 1) & 1, status))) break;
            mbar_expect_tx(&sm.fullB[bslot], bbytes);
            if (BT) {
                const __nv_bfloat16* src =
                    bt.tiles + ((((int64_t)(blk >> 2)) * bt.kbs + kstage) << 13) + (int64_t)(blk & 3) * (OZ_N * TC_KS);
#pragma unroll
                for (int q = 0; q < OZ_S; ++q)
                    bulk_load(sm.B[bslot][q], src + q * bt.slice, OZ_N * TC_KS * 2, &sm.fullB[bslot]);
            } else {
#pragma unroll
                for (int q = 0; q < OZ_S; ++q)
                    tma_load_2d(sm.B[bslot][q], &tmB, kstage * TC_KS, q * OZ_N, &sm.fullB[bslot]);
            }
            issuedB = s + 1;
            for (int a = 0; a < OZ_S; ++a) {
                const int idx = s * OZ_S + a;
                const int slot = idx % OZ_AST;
                if (idx >= OZ_AST && !(ok = mbar_wait(&sm.emptyA[slot], ((idx / OZ_AST) - 1) & 1, status))) break;
                mbar_expect_tx(&sm.fullA[slot], abytes);
                bulk_load(sm.A[slot], At + a * aslice + ((int64_t)((int64_t)band * kbs + kstage) << 13), abytes,
                          &sm.fullA[slot]);
                issuedA = idx + 1;
            }
            ++kstage;
            if (RUNS && kstage == kst) {
                kstage = 0;
                ++band;
            }
        }
    } else if (tid == 32) {
        // ---- MMA issuer ----
        int kstage = k0, chunk = 0;   // chunks of two stages, cut at the end of a band
        bool first = true;
        for (int s = 0; s < n && ok; ++s) {
            const int set = chunk & 1;
            if (first && chunk >= 2 && !(ok = mbar_wait(&sm.accEmpty[set], ((chunk >> 1) - 1) & 1, status))) break;
            const int bslot = s % OZ_BST;
            if (!(ok = mbar_wait(&sm.fullB[bslot], (s / OZ_BST) & 1, status))) break;
            // descriptors differ only in their start-address field (address / 16): a K step of 16 elements
            // is +2; computed once per stage and tile
            const uint64_t bdesc = smem_desc_sw128(smem_u32(sm.B[bslot][0]));
            const uint32_t dset = tmem + (uint32_t)(set * OZ_SET_COLS);
#pragma unroll
            for (int a = 0; a < OZ_S; ++a) {
                const int idx = s * OZ_S + a;
                const int slot = idx % OZ_AST;
                if (!(ok = mbar_wait(&sm.fullA[slot], (idx / OZ_AST) & 1, status))) break;
                tc_fence_after();
                const uint64_t adesc = smem_desc_sw128(smem_u32(sm.A[slot]));
                // A plane a against B planes 0 .. 6 - a in one MMA per K step: those planes are consecutive
                // in shared memory, one operand of N = 32 (7 - a) rows, and the product with plane b lands
                // 32 b columns into the accumulator, so starting it at level column 32 a puts it in level
                // a + b. A is read from shared memory once per K step instead of once per B plane.
                const uint32_t idesc = idesc_bf16(TC_M, OZ_N * (OZ_S - a));
                const uint32_t dcol = dset + (uint32_t)(a * OZ_N);
#pragma unroll
                for (int kk = 0; kk < TC_KS / 16; ++kk) {
                    // the chunk's first MMA (a = 0, first K step) covers all seven levels and overwrites
                    const uint32_t acc = (a == 0 && kk == 0 && first) ? 0u : 1u;
                    mma_bf16(dcol, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, acc);
                }
                mma_commit(&sm.emptyA[slot]);
            }
            if (!ok) break;
            mma_commit(&sm.emptyB[bslot]);
            const bool band_end = RUNS && ++kstage == kst;
            if (band_end) kstage = 0;
            first = !first || band_end || s == n - 1;   // the chunk ends here
            if (first) {
                mma_commit(&sm.accFull[set]);
                ++chunk;
            }
        }
    }
    // ---- epilogue: warps 4-7 fold each finished chunk into exact 64-bit integer sums and write a band out at its end ----
    if (warp >= 4) {
        const int ew = warp - 4;
        const uint32_t lanebase = tmem + ((uint32_t)(32 * ew) << 16);
        bool eok = true;   // a give-up: this band and the rest of the run become NaN
        int chunk = 0, left = n, band = band0, kfrom = k0;
        do {
            const int nks = RUNS ? min(left, kst - kfrom) : n;
            long long g0[OZ_N], g1[OZ_N];
#pragma unroll
            for (int c = 0; c < OZ_N; ++c) g0[c] = g1[c] = 0;
            for (int ch = (nks + 1) >> 1; ch > 0; --ch, ++chunk) {
                const int set = chunk & 1;
                if (!(eok = eok && mbar_wait(&sm.accFull[set], (chunk >> 1) & 1, status))) break;
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < OZ_N; c0 += 8) {
                    uint32_t r[OZ_S][8];
#pragma unroll
                    for (int q = 0; q < OZ_S; ++q) tmem_ld8(lanebase + set * OZ_SET_COLS + q * OZ_N + c0, r[q]);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        long long L[OZ_S];
#pragma unroll
                        for (int q = 0; q < OZ_S; ++q) L[q] = (long long)__float2int_rn(__uint_as_float(r[q][c]));
                        g0[c0 + c] += L[0] * 65536LL + L[1] * 256LL + L[2];
                        g1[c0 + c] += ((L[3] * 256LL + L[4]) * 256LL + L[5]) * 256LL + L[6];
                    }
                }
                tc_fence_before();
                mbar_arrive(&sm.accEmpty[set]);
            }
            left -= nks;
            if (!RUNS || left == 0) PDL_NEXT();
            const int row = 32 * ew + lane, i = band * TC_M + row;
            if (i < M) {
                const int ea = expA[i];
                const bool whole = !RUNS || nks == kst;
                double* out = whole ? D + i : partial + ((int64_t)(2 * blockIdx.x + (left + nks < n ? 1 : 0)) * N) * TC_M + row;
                const int64_t ldo = whole ? ldd : TC_M;
#pragma unroll
                for (int c0 = 0; c0 < OZ_N; c0 += 8) {
                    if (c0 >= N) break;
                    // the eight loads of C0 go out together: D may be C0, so none could pass a store
                    double add[8];
                    if (whole && beta != 0.0) {
#pragma unroll
                        for (int u = 0; u < 8; ++u) add[u] = c0 + u < N ? C0[(int64_t)(c0 + u) * ldc0 + i] : 0.0;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int c = c0 + u;
                        if (c >= N) break;
                        double v = eok ? oz_value(g0[c], g1[c], ea + expB[c]) : nan("");
                        if (whole) {
                            if (alpha != 1.0) v = alpha * v;
                            if (beta != 0.0) v = fma(beta, add[u], v);
                        }
                        out[c * ldo] = v;
                    }
                }
            }
            kfrom = 0;
            ++band;
        } while (RUNS && left > 0);
        if (!eok) sm.fail = 1;
    }
    if ((tid == 0 || tid == 32) && !ok) sm.fail = 1;
    __syncthreads();
    if (tid == 0 && sm.fail) {
        // after a give-up, wait (bounded again) for this CTA's copies that may still be in flight, so
        // that none lands after the CTA's shared memory is released
        for (int i = max(0, issuedA - OZ_AST); i < issuedA; ++i)
            mbar_wait(&sm.fullA[i % OZ_AST], (i / OZ_AST) & 1, status);
        for (int i = max(0, issuedB - OZ_BST); i < issuedB; ++i)
            mbar_wait(&sm.fullB[i % OZ_BST], (i / OZ_BST) & 1, status);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 2 * OZ_SET_COLS);
}

// frexp exponent of |v| (|v| = f 2^e, f in [0.5, 1)) read from the bits of v; kOzExpZero for v = 0.
// Inf and NaN give 1025.
constexpr int kOzExpZero = -1061109568;   // every byte 0xC0: the fill of a scale array before its maxima
__device__ __forceinline__ int oz_frexp_exp(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
    if (b == 0) return kOzExpZero;
    const int ef = (int)(b >> 52);
    return ef ? ef - 1022 : -1010 - __clzll((long long)b);   // subnormal: b is the mantissa
}

// Digits of x_0 = v 2^{7 - e} (|v| < 2^e). N = v 2^{55 - e} rounded to an integer (|N| <= 2^55, the
// rounding error at most half a unit of 2^{e - 55}), written in balanced base 256: s_6 .. s_1 are its
// low bytes taken as residues in [-128, 127] from the low end, s_0 what remains (|s_0| <= 128, since
// the low digits sum to less than 2^47 in magnitude). Then x_0 = sum_q 2^{-8q} s_q up to 2^{-49}, the
// same precision as the rounding recurrence x_{q+1} = 256 (x_q - rint(x_q)).
//
// Integer operations only (the mantissa and exponent come from the bits of v): with 128 added at each of the six low bytes
// the carries of all digits are done by one addition, and the bytes are the digits plus 128. A byte becomes a number by
// its place in the mantissa of 2^23 (one byte permutation and one single-precision subtraction, both at full rate; an
// integer-to-float conversion and a rounding to bf16 run at a quarter), and its bf16 is the upper half, exactly. The
// conversions bound the column splits: 40 of them in a d = 65536, n = 2000 pipeline 1.57 -> 1.22 ms, 81 narrow ones
// 0.49 -> 0.41 ms.
//
// w[q]: digit q as single precision. Returns false for Inf or NaN (digits zero).
__device__ __forceinline__ bool oz_digits(double v, int e, uint32_t (&w)[OZ_S]) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const int ef = (int)((bits >> 52) & 0x7FF);
    unsigned long long m = bits & 0xFFFFFFFFFFFFFull;
    long long N = 0;
    if (ef != 0x7FF) {
        int ex = -1074;                       // |v| = m 2^ex
        if (ef) {
            m |= 1ull << 52;
            ex = ef - 1075;
        }
        const int sh = ex + 55 - e;           // <= 2 whenever |v| < 2^e
        if (m != 0) {
            if (sh >= 0)
                N = (long long)(m << sh);
            else if (sh > -56)
                N = (long long)((m + (1ull << (-sh - 1))) >> (-sh));
        }
        if (bits >> 63) N = -N;
    }
    const long long B = N + 0x0000808080808080ll;
    const uint32_t lo = (uint32_t)B, hi = (uint32_t)((unsigned long long)B >> 32);
    const float off = 8388608.0f + 128.0f;
    auto digit = [&](uint32_t word, uint32_t sel) {   // byte sel of word, minus 128
        return __float_as_uint(__uint_as_float(__byte_perm(word, 0x4B000000u, 0x7440u | sel)) - off);
    };
    w[6] = digit(lo, 0);
    w[5] = digit(lo, 1);
    w[4] = digit(lo, 2);
    w[3] = digit(lo, 3);
    w[2] = digit(hi, 0);
    w[1] = digit(hi, 1);
    // the top digit, signed: 1.5 x 2^23 + s_0
    w[0] = __float_as_uint(__uint_as_float(0x4B400000u + (uint32_t)((int)hi >> 16)) - 12582912.0f);
    return ef != 0x7FF;
}

// The bf16 digit planes of eight values as one 16-byte chunk a plane.
__device__ __forceinline__ bool oz_digits8(const double (&v)[8], int e, uint4 (&dg)[OZ_S]) {
    bool fin = true;
    uint32_t pk[OZ_S][4];
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
        uint32_t a[OZ_S], b[OZ_S];
        fin &= oz_digits(v[u], e, a);
        fin &= oz_digits(v[u + 1], e, b);
#pragma unroll
        for (int q = 0; q < OZ_S; ++q) pk[q][u / 2] = __byte_perm(a[q], b[q], 0x7632);   // the upper halves
    }
#pragma unroll
    for (int q = 0; q < OZ_S; ++q) dg[q] = make_uint4(pk[q][0], pk[q][1], pk[q][2], pk[q][3]);
    return fin;
}

// Column scales: e[c] = max over rows r of the frexp exponent of A[r, c] (d x ncols, lda), kOzExpZero for
// a zero column. One CTA per (column, chunk of kOzExpChunk rows); each thread issues its eight loads
// before it reduces them (the scan is bound by the number of loads in flight), and the CTA's maximum is
// merged by one atomicMax into e, which the host fills with kOzExpZero first.
constexpr int kOzExpThreads = 256;
constexpr int kOzExpPer = 8;
constexpr int kOzExpChunk = kOzExpThreads * kOzExpPer;
__global__ void __launch_bounds__(kOzExpThreads) k_oz_exp_cols(int64_t rows, const double* __restrict__ A,
                                                              int64_t lda, int* __restrict__ e) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(e);
    __shared__ int wmax[kOzExpThreads / 32];
    const int c = blockIdx.x;
    const double* col = A + (int64_t)c * lda;
    const int64_t r0 = (int64_t)blockIdx.y * kOzExpChunk + threadIdx.x;
    double v[kOzExpPer];
#pragma unroll
    for (int u = 0; u < kOzExpPer; ++u) {
        const int64_t r = r0 + (int64_t)u * kOzExpThreads;
        v[u] = r < rows ? col[r] : 0.0;
    }
    int mx = kOzExpZero;
#pragma unroll
    for (int u = 0; u < kOzExpPer; ++u) mx = max(mx, oz_frexp_exp(v[u]));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kOzExpThreads / 32; ++w) mx = max(mx, wmax[w]);
        if (mx != kOzExpZero) atomicMax(&e[c], mx);
    }
}

// Row scales of a split operand whose M rows are the ROWS of A (d x m, lda): one CTA per (256 rows, chunk of kOzRowChunk
// columns), thread per row, eight loads in flight; merged by one atomicMax a row into e, which the host fills with
// kOzExpZero first. Bound by HBM; one thread for a whole row had too few loads in
// flight (65536 x 2200 and two 65536 x 199: 0.80 -> 0.28 ms).
constexpr int kOzRowChunk = 64;
__global__ void __launch_bounds__(256) k_oz_exp_rows(int64_t rows, int cols, const double* __restrict__ A, int64_t lda,
                                                    int* __restrict__ e) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(e);
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    const int c0 = blockIdx.y * kOzRowChunk, c1 = min(cols, c0 + kOzRowChunk);
    int mx = kOzExpZero;
    for (int c = c0; c < c1; c += 8) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = c + u < c1 ? A[(int64_t)(c + u) * lda + r] : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = max(mx, oz_frexp_exp(v[u]));
    }
    if (mx != kOzExpZero) atomicMax(&e[r], mx);
}

// A chained launch where a memset would break the chain: the gap before it and after it came to 4 to 9 us, of which 2 are left.
__global__ void k_oz_fill(int* __restrict__ p, int64_t n, int v) {
    PDL_ENTER();
    PDL_ARG(p);
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) p[t] = v;
}

// A narrow operand B (K x p, ldb; its columns are the N rows of the product): column scales and the seven digit planes, in
// one launch. planes [7][32][ld] (plane q, row j at (32 q + j) ld), zero for j >= p or k >= K; e[j] the scales (0 for
// j >= p). One cluster per column: each CTA takes the maximum over its share of the column, the CTAs exchange theirs
// through distributed shared memory, and each splits its share (read again, from L2), eight consecutive k per thread: one
// 64-byte read and one 16-byte store per plane. Launch overhead bounds it at the usual sizes: a fill, a scale and a split
// launch and their gaps took about 15 us at K = 65536 and 11 us at K = 700, this one 9 and 5 us.
constexpr int OZ_NARROW_CL = 8;
__global__ void __cluster_dims__(OZ_NARROW_CL, 1, 1) __launch_bounds__(256)
    k_oz_narrow(int64_t K, int p, const double* __restrict__ B, int64_t ldb, int* __restrict__ e, int64_t ld,
                __nv_bfloat16* __restrict__ out, int* __restrict__ status) {
    PDL_ENTER();
    PDL_ARG(B); PDL_ARG(e); PDL_ARG(out); PDL_ARG(status);
    namespace cg = cooperative_groups;
    __shared__ int wmax[8];
    __shared__ int cmax;
    cg::cluster_group cluster = cg::this_cluster();
    const int j = blockIdx.y, rank = blockIdx.x;
    const int64_t groups = ld / 8;
    const double* col = B + (int64_t)j * ldb;
    int ex = 0;
    if (j < p) {   // uniform over the cluster
        int mx = kOzExpZero;
        for (int64_t g = (int64_t)rank * 256 + threadIdx.x; g < groups; g += OZ_NARROW_CL * 256) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = 8 * g + u < K ? col[8 * g + u] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) mx = max(mx, oz_frexp_exp(v[u]));
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) mx = max(mx, wmax[w]);
            cmax = mx;
        }
        cluster.sync();
        ex = kOzExpZero;
        for (int r = 0; r < OZ_NARROW_CL; ++r) ex = max(ex, *cluster.map_shared_rank(&cmax, r));
        cluster.sync();   // no CTA leaves while another reads its maximum
    }
    if (rank == 0 && threadIdx.x == 0) e[j] = ex;
    bool fin = true;
    for (int64_t g = (int64_t)rank * 256 + threadIdx.x; g < groups; g += OZ_NARROW_CL * 256) {
        const int64_t k0 = 8 * g;
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = (j < p && k0 + u < K) ? col[k0 + u] : 0.0;
        uint4 dg[OZ_S];
        fin &= oz_digits8(v, ex, dg);
#pragma unroll
        for (int q = 0; q < OZ_S; ++q) *reinterpret_cast<uint4*>(out + ((int64_t)q * OZ_N + j) * ld + k0) = dg[q];
    }
    if (!fin) atomicOr(status, ST_NONFINITE);
}

// Digit planes of the columns i0 .. i1 of A (d x m, lda) as M rows of a split operand whose K index runs down
// the columns (rows_are_cols layout), 8 consecutive k per thread: one 64-byte read of A and one 16-byte
// store per plane. e: the scales of those columns (e[i - i0]). Rows at or beyond Mvalid (the padding of
// the last 128-row band) are written as zeros.
__global__ void k_oz_split_cols8(const double* __restrict__ A, int64_t lda, int i0, int i1, int Mvalid, int64_t K,
                                 const int* __restrict__ e, int kbs, int64_t ld, __nv_bfloat16* __restrict__ out,
                                 int64_t slice, int* __restrict__ status) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(e); PDL_ARG(out); PDL_ARG(status);
    const int64_t groups = ld / 8;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)(i1 - i0) * groups) return;
    const int i = i0 + (int)(t / groups);
    const int64_t k0 = (t % groups) * 8;
    const bool row = i < Mvalid;
    const int ex = row ? e[i - i0] : 0;
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        v[u] = (row && k0 + u < K) ? A[(int64_t)i * lda + k0 + u] : 0.0;
    }
    uint4 dg[OZ_S];
    const bool fin = oz_digits8(v, ex, dg);
    if (!fin) atomicOr(status, ST_NONFINITE);
    const int64_t off = tile_off(i, k0, kbs);
#pragma unroll
    for (int q = 0; q < OZ_S; ++q)
        *reinterpret_cast<uint4*>(out + q * slice + off) = dg[q];
}

// Digit planes of the rows of A (M x K, lda; M rows = rows of A, K along its columns). One CTA per 32 rows of a tile and
// its 64 k: warp w reads k 8 w .. 8 w + 7 (each coalesced across the lanes' rows) and puts its chunks into the tile's image
// in shared memory, from where each plane's 32 rows leave as 4 contiguous KB. Written straight from the registers every
// 16-byte chunk is a store of its own to half a sector: 65536 x 2200 and two 65536 x 199 took 2.15 ms (also with 16 k a
// thread), now 0.60 ms (3.8 GB: 0.56 ms at the copy rate). Columns at or beyond K, and rows at or beyond M, are zero; the scale
// kOzExpZero of a zero row stands for any.
__global__ void __launch_bounds__(256) k_oz_split_rows(const double* __restrict__ A, int64_t lda, int64_t M, int64_t K,
                                                      const int* __restrict__ e, int kbs, int kst,
                                                      __nv_bfloat16* __restrict__ out, int64_t slice,
                                                      int* __restrict__ status) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(e); PDL_ARG(out); PDL_ARG(status);
    __shared__ __align__(16) uint4 img[OZ_S][32 * 8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)(blockIdx.x / kst) * 32, i = i0 + lane;
    const int kb = blockIdx.x % kst;
    const int ex = i < M ? e[i] : 0;
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int64_t k = (int64_t)kb * TC_KS + 8 * w + u;
        v[u] = (i < M && k < K) ? A[k * lda + i] : 0.0;
    }
    uint4 dg[OZ_S];
    if (!oz_digits8(v, ex, dg)) atomicOr(status, ST_NONFINITE);
#pragma unroll
    for (int q = 0; q < OZ_S; ++q) img[q][lane * 8 + (w ^ (lane & 7))] = dg[q];
    __syncthreads();
    const int64_t off = tile_off(i0, (int64_t)kb * TC_KS, kbs) & ~(int64_t)63;   // row i0's 64 elements, chunk 0
#pragma unroll
    for (int q = 0; q < OZ_S; ++q)
        reinterpret_cast<uint4*>(out + q * slice + off)[threadIdx.x] = img[q][threadIdx.x];
}

// Growing a row-scaled operand (the Krylov basis, M = d rows, K = the columns so far) from k0 to k1 columns:
// thread per row. A row whose scale is unchanged by the new columns gets the digits of its new 8-groups
// [k0 rounded down to 8, k1) (the part of a group below k0 rewritten with identical digits) and zeros to the end of the
// last 64-wide tile; a row whose
// scale grows records the new scale and joins list (count in list[0]) for a full re-split by
// k_oz_resplit_listed. Zero rows keep the scale kOzExpZero.
__global__ void k_oz_grow_rows(const double* __restrict__ A, int64_t lda, int64_t M, int64_t k0, int64_t k1,
                               int* __restrict__ e, int kbs, __nv_bfloat16* __restrict__ out, int64_t slice,
                               int* __restrict__ list, int* __restrict__ status) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(e); PDL_ARG(out); PDL_ARG(list); PDL_ARG(status);
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    int mnew = kOzExpZero;
    for (int64_t k = k0; k < k1; ++k) mnew = max(mnew, oz_frexp_exp(A[k * lda + i]));
    int eold = k0 == 0 ? mnew : e[i];
    if (k0 == 0) {
        e[i] = mnew;   // the first columns: their digits below, with their own scale
    } else if (mnew > eold) {
        e[i] = mnew;
        list[1 + atomicAdd(&list[0], 1)] = (int)i;
        return;
    }
    bool fin = true;
    for (int64_t kg = k0 & ~(int64_t)7; kg < ((k1 + TC_KS - 1) & ~(int64_t)(TC_KS - 1)); kg += 8) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t k = kg + u;
            v[u] = k < k1 ? A[k * lda + i] : 0.0;
        }
        uint4 dg[OZ_S];
        fin &= oz_digits8(v, eold, dg);
        const int64_t off = tile_off(i, kg, kbs);
#pragma unroll
        for (int q = 0; q < OZ_S; ++q)
            *reinterpret_cast<uint4*>(out + q * slice + off) = dg[q];
    }
    if (!fin) atomicOr(status, ST_NONFINITE);
}

// Full re-split, columns 0 .. K, of the rows in list (count list[0]), one (row, 8-group) per thread step.
__global__ void k_oz_resplit_listed(const double* __restrict__ A, int64_t lda, int64_t K, const int* __restrict__ e,
                                    int kbs, __nv_bfloat16* __restrict__ out, int64_t slice,
                                    const int* __restrict__ list, int* __restrict__ status) {
    PDL_WAIT();
    PDL_ARG(A); PDL_ARG(e); PDL_ARG(out); PDL_ARG(list); PDL_ARG(status);
    const int64_t groups = (K + TC_KS - 1) / TC_KS * (TC_KS / 8);   // whole tiles: zeros beyond K
    const int64_t total = (int64_t)list[0] * groups;
    bool fin = true;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = list[1 + t % list[0]];
        const int64_t kg = (t / list[0]) * 8;
        const int ex = e[i];
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t k = kg + u;
            v[u] = k < K ? A[k * lda + i] : 0.0;
        }
        uint4 dg[OZ_S];
        fin &= oz_digits8(v, ex, dg);
        const int64_t off = tile_off(i, kg, kbs);
#pragma unroll
        for (int q = 0; q < OZ_S; ++q)
            *reinterpret_cast<uint4*>(out + q * slice + off) = dg[q];
    }
    if (!fin) atomicOr(status, ST_NONFINITE);
}

// D[i, j] = alpha * sum_s P[s][j][i] + beta * D[i, j], splits added in order (deterministic).
__global__ void k_oz_reduce(int M, int N, int splits, const double* __restrict__ P, int64_t sstride, double alpha,
                            double beta, const double* C0, int64_t ldc0, double* D, int64_t ldd) {
    PDL_ENTER();
    PDL_ARG(P); PDL_ARG(C0); PDL_ARG(D);
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)M * N) return;
    const int i = (int)(t % M), j = (int)(t / M);
    double acc = 0.0;
    for (int s = 0; s < splits; ++s) acc += P[(int64_t)s * sstride + (int64_t)j * M + i];
    double v = alpha * acc;
    if (beta != 0.0) v = fma(beta, C0[(int64_t)j * ldc0 + i], v);
    D[(int64_t)j * ldd + i] = v;
}

// The bands that several runs share: D = alpha * (the sum of their slots, in the order of k) + beta * C0. Block row c > 0 takes
// the band in which run c begins, if it is the first run to begin inside that band; 256 of the band's 128 x N entries a CTA.
__global__ void __launch_bounds__(256) k_oz_join(const OzRuns runs, int ctas, int M, int N, const double* __restrict__ P,
                                                 double alpha, double beta, const double* C0, int64_t ldc0, double* D,
                                                 int64_t ldd) {
    PDL_ENTER();
    PDL_ARG(P); PDL_ARG(C0); PDL_ARG(D);
    const int c = blockIdx.y + 1;
    const int64_t t = runs.begin(c, ctas);
    const int band = (int)(t / runs.kst);
    const int64_t b0 = (int64_t)band * runs.kst;
    if (t == b0 || runs.begin(c - 1, ctas) > b0) return;
    const int e = blockIdx.x * 256 + threadIdx.x, row = e % TC_M, j = e / TC_M, i = band * TC_M + row;
    if (j >= N || i >= M) return;
    const int last = runs.of(b0 + runs.kst - 1, ctas);
    // run c - 1 holds the band's first stages: as its first piece if it begins with the band, else as its last
    const double* src = P + (int64_t)j * TC_M + row;
    const int64_t slot = (int64_t)N * TC_M;
    double acc = src[(2 * (c - 1) + (runs.begin(c - 1, ctas) == b0 ? 0 : 1)) * slot];
    for (int q = c; q <= last; ++q) acc += src[2 * q * slot];
    double v = alpha * acc;
    if (beta != 0.0) v = fma(beta, C0[(int64_t)j * ldc0 + i], v);
    D[(int64_t)j * ldd + i] = v;
}

int oz_attr() {
    static std::once_flag once;
    static cudaError_t rc = cudaSuccess;
    std::call_once(once, [] {
        rc = cudaFuncSetAttribute(k_oz_gemm<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)oz_smem_bytes());
        if (rc == cudaSuccess)
            rc = cudaFuncSetAttribute(k_oz_gemm<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)oz_smem_bytes());
        if (rc == cudaSuccess)
            rc = cudaFuncSetAttribute(k_oz_gemm<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)oz_smem_bytes());

    });
    EDA_CUDA_TRY(rc);
    return EDA_OK;
}

}  // namespace

size_t oz_operand_bytes(int64_t M, int64_t K) {
    const int64_t mt = (M + TC_M - 1) / TC_M, kb = (K + TC_KS - 1) / TC_KS;
    const size_t plane = (size_t)mt * kb * TC_M * TC_KS * 2;
    return OZ_S * ((plane + 255) / 256 * 256) + ((size_t)M * 4 + 255) / 256 * 256;
}

// Column scales of columns 0 .. ncols of A (K x ncols, lda) into e.
static int oz_col_exps(int64_t K, const double* A, int64_t lda, int ncols, int* e, cudaStream_t s) {
    if (ncols <= 0) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_oz_fill, dim3(ceil_div(ncols, 256)), dim3(256), 0, s, e, ncols, kOzExpZero)));
    const dim3 grid((unsigned)ncols, (unsigned)ceil_div(std::max<int64_t>(K, 1), kOzExpChunk));
    EDA_CUDA_TRY((launch_chained(k_oz_exp_cols, grid, dim3(kOzExpThreads), 0, s, K, A, lda, e)));
    return EDA_OK;
}

// Row scales of A (M x K, lda) into e.
static int oz_row_exps(int64_t M, int64_t K, const double* A, int64_t lda, int* e, cudaStream_t s) {
    if (M <= 0) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_oz_fill, dim3(ceil_div(M, 256)), dim3(256), 0, s, e, M, kOzExpZero)));
    if (K <= 0) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_oz_exp_rows, dim3((unsigned)ceil_div(M, 256), (unsigned)ceil_div(K, kOzRowChunk)),
        dim3(256), 0, s, M, (int)K, A, lda, e)));
    return EDA_OK;
}

int oz_operand_make(const double* A, int64_t lda, int64_t M, int64_t K, bool rows_are_cols, void* mem,
                    OzOperand* op, int* status, cudaStream_t s) {
    const int64_t mt = (M + TC_M - 1) / TC_M, kb = (K + TC_KS - 1) / TC_KS;
    const int64_t plane = mt * kb * TC_M * TC_KS;
    const int64_t slice = ((plane * 2 + 255) / 256 * 256) / 2;
    op->tiles = static_cast<__nv_bfloat16*>(mem);
    op->slice = slice;
    op->exps = reinterpret_cast<int*>(static_cast<char*>(mem) + OZ_S * slice * 2);
    op->M = M;
    op->K = K;
    op->kbs = (int)kb;
    op->mtiles = (int)mt;
    const int64_t ld = kb * TC_KS, mpad = mt * TC_M;
    if (rows_are_cols) {
        EDA_TRY(oz_col_exps(K, A, lda, (int)M, op->exps, s));
        EDA_CUDA_TRY((launch_chained(k_oz_split_cols8, dim3(ceil_div(mpad * (ld / 8), 256)), dim3(256), 0, s, A, lda, 0,
            (int)mpad, (int)M, K, op->exps,
            (int)kb, ld, op->tiles, slice, status)));
    } else {
        EDA_TRY(oz_row_exps(M, K, A, lda, op->exps, s));
        EDA_CUDA_TRY((launch_chained(k_oz_split_rows, dim3((unsigned)(mpad / 32 * kb)), dim3(256), 0, s, A, lda, M, K,
            op->exps, (int)kb, (int)kb, op->tiles,
            slice, status)));
    }
    return EDA_OK;
}

// A split operand with room for Mcap rows (columns of a d x Mcap matrix, K = d) or for Kcap values of K
// (rows_are_cols = false: M = d rows, K up to Kcap columns), no row filled yet. The planes are not cleared (4 GB at
// d = 65536, m = 2232): rows beyond those present only reach results that are not stored, and every write fills its 64-wide
// tile along K up to the end with zeros.
int oz_operand_init(int64_t Mcap, int64_t Kcap, void* mem, OzOperand* op, cudaStream_t s) {
    const int64_t mt = (Mcap + TC_M - 1) / TC_M, kb = (Kcap + TC_KS - 1) / TC_KS;
    const int64_t plane = mt * kb * TC_M * TC_KS;
    const int64_t slice = ((plane * 2 + 255) / 256 * 256) / 2;
    op->tiles = static_cast<__nv_bfloat16*>(mem);
    op->slice = slice;
    op->exps = reinterpret_cast<int*>(static_cast<char*>(mem) + OZ_S * slice * 2);
    op->M = 0;
    op->K = 0;
    op->kbs = (int)kb;
    op->mtiles = 0;
    (void)s;
    return EDA_OK;
}

int oz_append_cols(const double* A, int64_t lda, int i0, int i1, int64_t K, OzOperand* op, int* status,
                   cudaStream_t s) {
    if (i1 <= i0) return EDA_OK;
    EDA_TRY(oz_col_exps(K, A + (int64_t)i0 * lda, lda, i1 - i0, op->exps + i0, s));
    const int64_t ld = (int64_t)op->kbs * TC_KS;
    EDA_CUDA_TRY((launch_chained(k_oz_split_cols8, dim3(ceil_div((int64_t)(i1 - i0) * (ld / 8), 256)), dim3(256), 0, s,
        A, lda, i0, i1, i1, K, op->exps + i0, op->kbs, ld, op->tiles, op->slice, status)));
    op->M = i1;
    op->K = K;
    op->mtiles = ceil_div(i1, TC_M);
    return EDA_OK;
}

int oz_grow_rows(const double* A, int64_t lda, int64_t M, int64_t k0, int64_t k1, OzOperand* op, int* list,
                 int* status, cudaStream_t s) {
    if (k1 <= k0) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_oz_fill, dim3(1), dim3(32), 0, s, list, 1, 0)));
    EDA_CUDA_TRY((launch_chained(k_oz_grow_rows, dim3(ceil_div(M, 256)), dim3(256), 0, s, A, lda, M, k0, k1, op->exps,
        op->kbs, op->tiles, op->slice, list,
            status)));
    EDA_CUDA_TRY((launch_chained(k_oz_resplit_listed, dim3(2 * sm_count()), dim3(256), 0, s, A, lda, k1, op->exps,
        op->kbs, op->tiles, op->slice, list,
            status)));
    op->M = M;
    op->K = k1;
    op->mtiles = ceil_div(M, TC_M);
    return EDA_OK;
}

// doubles of the partial buffer: max_splits copies of a result, and two 128-row slots for each run of a narrow product
static size_t oz_partial_cap(int max_splits, int64_t Mmax) {
    return (size_t)max_splits * OZ_N * (size_t)std::max<int64_t>(Mmax, 2 * TC_M);
}

size_t oz_narrow_bytes(int64_t Kmax, int max_splits, int64_t Mmax) {
    const int64_t ld = (Kmax + TC_KS - 1) / TC_KS * TC_KS;
    return ((size_t)OZ_S * OZ_N * ld * 2 + 255) / 256 * 256 + 256 + (oz_partial_cap(max_splits, Mmax) * 8 + 255) / 256 * 256;
}

int oz_narrow_make(int64_t Kmax, int max_splits, int64_t Mmax, void* mem, OzNarrow* nb) {
    const int64_t ld = (Kmax + TC_KS - 1) / TC_KS * TC_KS;
    char* p = static_cast<char*>(mem);
    nb->planes = reinterpret_cast<__nv_bfloat16*>(p);
    p += ((size_t)OZ_S * OZ_N * ld * 2 + 255) / 256 * 256;
    nb->exps = reinterpret_cast<int*>(p);
    p += 256;
    nb->partial = reinterpret_cast<double*>(p);
    nb->pcap = oz_partial_cap(max_splits, Mmax);
    nb->ldmax = ld;
    nb->map_ld = 0;
    return EDA_OK;
}

int oz_gemm(const OzOperand& A, OzNarrow& nb, int p, const double* B, int64_t ldb, double alpha, double beta,
            const double* C0, int64_t ldc0, double* D, int64_t ldd, int* status, cudaStream_t s) {
    if (p < 1 || p > OZ_N) return EDA_ERR_INVALID_ARG;
    const int64_t ld = (A.K + TC_KS - 1) / TC_KS * TC_KS;
    if (ld > nb.ldmax) return EDA_ERR_INVALID_ARG;
    EDA_TRY(oz_attr());
    if (nb.map_ld != ld) {
        EDA_TRY(make_map(&nb.map, nb.planes, (uint64_t)ld, (uint64_t)OZ_S * OZ_N, (uint64_t)ld, OZ_N));
        nb.map_ld = ld;
    }
    // algorithmic work, as for the FP64 product it replaces: 2 M K p flops; A read once (seven bf16
    // digit planes), B read and D written once in FP64
    ProfScope prof("oz_gemm", s, 2.0 * (double)A.M * A.K * p,
                   2.0 * OZ_S * (double)A.M * A.K + 8.0 * (double)A.K * p + 8.0 * (double)A.M * p);
    EDA_CUDA_TRY((launch_chained(k_oz_narrow, dim3(OZ_NARROW_CL, OZ_N), dim3(256), 0, s, A.K, p, B, ldb, nb.exps, ld,
        nb.planes, status)));
    const int kst = (int)(ld / TC_KS);
    // One CTA an SM at most (the kernel holds all of an SM's tensor memory). Up to one band an SM: K splits that fill the SMs.
    // More: runs; of whole bands, which need no join, unless even ones are shorter by more than the join costs.
    const int nsm = sm_count();
    OzRuns runs{kst, kst, A.mtiles};
    int ctas = std::min(nsm, A.mtiles), splits = 1, kps = 0;
    if (A.mtiles <= nsm) {
        splits = std::max(1, std::min(kst / 2, nsm / std::max(1, A.mtiles)));
        while (splits > 1 && (size_t)splits * p * A.M > nb.pcap) --splits;
        kps = ceil_div(kst, splits);
        splits = ceil_div(kst, kps);
    } else if ((size_t)2 * TC_M * p * nsm <= nb.pcap &&
               (int64_t)ceil_div(A.mtiles, nsm) * kst > (int64_t)A.mtiles * kst / nsm + kOzJoinStages) {
        runs.unit = 1;
        runs.units = (int64_t)A.mtiles * kst;
    }
    const bool add = splits > 1;   // the splits' sums go to partial
    const bool join = kps == 0 && runs.unit == 1;
    {
        // the tensor-core kernel alone: it must read the seven digit planes of A and of B once and write D
        // tensor work: the 28 digit-plane products of 2 M K p flops each
        ProfScope kprof("oz_kernel", s, 56.0 * (double)A.M * A.K * p,
                        2.0 * OZ_S * ((double)A.M * A.K + (double)A.K * p) + 8.0 * (double)A.M * p);
        const OzBTiles none{};
        EDA_CUDA_TRY((launch_chained(kps ? k_oz_gemm<false, false> : k_oz_gemm<false, true>, dim3((unsigned)ctas, (unsigned)splits), dim3(OZ_THREADS), oz_smem_bytes(),
            s, A.tiles, A.slice, A.kbs, nb.map, none, A.exps, nb.exps, (int)A.M, p, runs, kps, add ? 1.0 : alpha,
            add ? 0.0 : beta, C0, ldc0, add ? nb.partial : D, add ? A.M : ldd, add ? (int64_t)p * A.M : 0, nb.partial, status)));
    }
    if (add)
        EDA_CUDA_TRY((launch_chained(k_oz_reduce, dim3(ceil_div((int64_t)A.M * p, 256)), dim3(256), 0, s, (int)A.M, p, splits,
            nb.partial, (int64_t)p * A.M, alpha, beta, C0, ldc0, D, ldd)));
    if (!join) return EDA_OK;
    EDA_CUDA_TRY((launch_chained(k_oz_join, dim3(ceil_div(TC_M * p, 256), (unsigned)(ctas - 1)), dim3(256), 0, s, runs, ctas,
        (int)A.M, p, nb.partial, alpha, beta, C0, ldc0, D, ldd)));
    return EDA_OK;
}

// D[i, j] = alpha sum_k A_ik B_jk + beta C0[i, j] for two split operands with the same K (i < A.M, j < B.M):
// one launch over (A band, B 32-row block); upper: only the blocks meeting the upper triangle i <= j, the
// rest filled by the mirror image (for products that are symmetric; blocks on the diagonal are computed whole).
__global__ void k_oz_mirror_lower(int n, double* D, int64_t ldd) {
    PDL_ENTER();
    PDL_ARG(D);
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * n) return;
    const int i = (int)(t % n), j = (int)(t / n);
    if (i > j && (j + OZ_N) / OZ_N * OZ_N <= (i / TC_M) * TC_M) D[(int64_t)j * ldd + i] = D[(int64_t)i * ldd + j];
}

int oz_gemm_tiled(const OzOperand& A, const OzOperand& B, double alpha, double beta, const double* C0, int64_t ldc0,
                  double* D, int64_t ldd, bool upper, int* status, cudaStream_t s, double* part, size_t pcap) {
    if (A.K != B.K || A.M < 1 || B.M < 1) return EDA_ERR_INVALID_ARG;
    if (upper && A.M != B.M) return EDA_ERR_INVALID_ARG;
    EDA_TRY(oz_attr());
    const int kst = ceil_div(A.K, TC_KS);   // an operand with room for more (a growing basis) has more tiles a band
    const int nblk = ceil_div(B.M, OZ_N);
    // K splits (when a partial buffer is given): the count of 1 .. 8, or up to one wave of CTAs, that fills the SMs best at one
    // CTA each; a larger count only for 4 % more (each adds a pass over the result)
    int splits = 1;
    if (part && !upper) {
        const int nsm = sm_count(), tiles = std::max(1, A.mtiles * nblk);
        double best = 0.0;
        for (int c = 1; c <= std::min(kst / 8, std::max(8, nsm / tiles)); ++c) {
            if ((size_t)c * A.M * B.M > pcap) break;
            const double fill = (double)tiles * c / ((double)nsm * ((tiles * c + nsm - 1) / nsm));
            if (fill > best + 0.04) {
                best = fill;
                splits = c;
            }
        }
    }
    const int kps = ceil_div(kst, splits);
    splits = ceil_div(kst, kps);
    const dim3 grid((unsigned)nblk * (unsigned)A.mtiles, (unsigned)splits);
    OzBTiles bt;
    bt.kbs = B.kbs;
    bt.nblk = nblk;
    bt.tiles = B.tiles;
    bt.slice = B.slice;
    bt.upper = upper ? 1 : 0;
    // tensor work of the computed blocks: 28 digit-plane products of 2 x 128 x 32 x K flops per (band, block)
    double blocks = 0.0;
    for (int b = 0; b < A.mtiles; ++b)
        for (int z = 0; z < nblk; ++z) blocks += (upper && z * OZ_N + OZ_N <= b * TC_M) ? 0.0 : 1.0;
    {
        ProfScope kprof("oz_tiled", s, 56.0 * TC_M * OZ_N * (double)kst * TC_KS * blocks,
                        2.0 * OZ_S * ((double)A.M * A.K + (double)A.K * B.M) + 8.0 * (double)A.M * B.M);
        // tmB is not read in this mode; the operand's planes are passed in bt
        static const CUtensorMap unused{};
        const OzRuns runs{kst, kst, A.mtiles};
        if (splits == 1)
            EDA_CUDA_TRY((launch_chained(k_oz_gemm<true, false>, grid, dim3(OZ_THREADS), oz_smem_bytes(), s, A.tiles, A.slice,
                A.kbs, unused, bt, A.exps,
            B.exps, (int)A.M, (int)B.M, runs, kps, alpha, beta,
            C0, ldc0, D, ldd, 0, nullptr, status)));
        else
            EDA_CUDA_TRY((launch_chained(k_oz_gemm<true, false>, grid, dim3(OZ_THREADS), oz_smem_bytes(), s, A.tiles, A.slice,
                A.kbs, unused, bt, A.exps,
            B.exps, (int)A.M, (int)B.M, runs, kps, 1.0, 0.0,
            nullptr, 0, part, A.M, (int64_t)A.M * B.M, nullptr, status)));
    }
    if (splits > 1) {
        EDA_CUDA_TRY((launch_chained(k_oz_reduce, dim3(ceil_div((int64_t)A.M * B.M, 256)), dim3(256), 0, s, (int)A.M,
            (int)B.M, splits, part,
            (int64_t)A.M * B.M, alpha, beta, C0, ldc0, D, ldd)));
    }
    if (upper) {
        EDA_CUDA_TRY((launch_chained(k_oz_mirror_lower, dim3(ceil_div((int64_t)A.M * A.M, 256)), dim3(256), 0, s,
            (int)A.M, D, ldd)));
    }
    return EDA_OK;
}

int oz_gemm_wide(const OzOperand& A, OzNarrow& nb, OzScratch& sc, int p, const double* B, int64_t ldb, double alpha,
                 double beta, const double* C0, int64_t ldc0, double* D, int64_t ldd, int* status, cudaStream_t s) {
    if (p <= OZ_N) return oz_gemm(A, nb, p, B, ldb, alpha, beta, C0, ldc0, D, ldd, status, s);
    EDA_TRY(sc.ensure(oz_operand_bytes(p, A.K)));
    OzOperand op;
    EDA_TRY(oz_operand_make(B, ldb, p, A.K, true, sc.mem, &op, status, s));
    return oz_gemm_tiled(A, op, alpha, beta, C0, ldc0, D, ldd, false, status, s, nb.partial, nb.pcap);
}

int OzScratch::ensure(size_t need) {
    if (bytes >= need) return EDA_OK;
    void* old = mem;
    mem = nullptr;
    bytes = 0;
    EDA_TRY(dev_free_idle(old));   // earlier products may still read it
    EDA_TRY(dev_alloc(&mem, need));
    bytes = need;
    return EDA_OK;
}

}  // namespace eda
