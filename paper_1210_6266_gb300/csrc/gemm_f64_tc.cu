// FP64 fronts on the tensor cores: every product of the blocked partial Cholesky (the
// updates C -= X X^T, the panel solve X = A L_kk^-T) or LU (C -= X Y) split into exact FP16 products
// (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix multiplication by
// using fast routines of matrix multiplication", 2012).
//
// The FP64 pipe retires 1.65 FMAs per clock and SM, the tensor cores about 4096 FP16 ones,
// so 36 exact FP16 products per FP64 product are over fifty times cheaper.
//
// Digits.  Row i of an operand has an exponent e_i with |entry| < 2^e_i, taken from its
// entries in the columns of the product (128 for a panel solve, up to 512 for an update).
// An entry is rounded to a multiple of 2^(e_i - FB) and written as eight balanced digits of DB
// bits, x = 2^(e_i - FB) sum_k d_k 2^(DB (7 - k)), stored as FP16 integers of magnitude at
// most 1024.  Products: C = the sum over digit pairs with i + j = d <= 7 of
// 2^(DB (14 - d)) (D_i D_j^T); a sum over pairs and K columns that stays below 2^24 is exact in FP32,
// whatever its order:
//   updates, K <= 512: DB = 7, FB = 59 (|d_k| <= 64), and e_i such that a row's sum of
//     (x 2^-e_i)^2 is at most 8: the vector of its d_0 is then no longer than 2^11.5, that of a d_k than
//     2^10.5, and by Cauchy-Schwarz a sum is at most 2 x 2^22 + (d - 1) 2^21 <= 2^24 for
//     d <= 5 (2^23 for d = 0); d = 6 and 7 could pass it by a quarter, where a lost unit
//     is 2^-62 of the product;
//   panel solve, K <= 128: DB = 8, FB = 62 (|d_0| <= 64, |d_k| <= 128): at most 2^24.
// The eight sums (one per d) are combined in 64-bit integers, rounded to FP64 once, and C is
// updated with one FP64 subtraction.  The pairs left out (d = 8 and beyond) are of
// either sign but for the squares of digit 4 on C's diagonal (X X^T): those are summed per
// row and added (without them every pivot is biased one way).
// Error of 57^3 log-normal diffusion solves (three loads) against the assembled system's
// solution, refined with extended-precision residuals: 9.0, 5.0 and 5.3e-16 this way, 37.6, 18.5
// and 16.0e-16 with FMAs on the FP64 pipe (of 37^3 convection-diffusion, LU: 4.9, 4.3, 5.9 against
// 6.7, 6.2, 7.0).  A plain FP64 CG on the unassembled operator is itself 46, 25 and 18e-16 from
// that solution and lies nearer to the FMA form's answers (17, 14, 12 against 53, 26, 18): a
// comparison with one says more about the two roundings' likeness than about either error.
// (With exponents fixed by sqrt(K_ii), most entries of a row being far smaller, 1e-11.)  A Schur
// complement that cancels to 1e-7 of its terms is off by half a unit of those terms (rms), by 2 to 5
// units with FMAs.
//
// Scale.  One exponent a row is safe for Cholesky: with K = D K0 D the entries of row i of
// [L; X] all scale with D_i, and |l_ik| <= sqrt(K_ii).  LU is not like that: with K = Dr K0 Dc
// an entry of [L; X] scales with Dr_i / Dr_k and one of [U^T; Y^T] with Dr_k Dc_j, so along
// the columns k of a panel the operands' scales run opposite ways, and what an entry 2^-59
// below its row's largest loses is not small beside the product.  So column k of [L; X] is
// split times 2^t_k and column k of [U^T; Y^T] times 2^-t_k (exact, and nothing to undo in
// the product), t_k the exponent of Dr_k as the pivot u_kk = Dr_k Dc_k gives it: half of its
// exponent (rows and columns scaled alike, the Galerkin case), all of it (scaled equations) or
// none of it (scaled unknowns), whichever of the three fits the entries of K best beside its
// diagonal (lu_scaling).  The operands of the panel solves are scaled to match.
// No power of two fits every Dr and Dc, so each split row is held against the scale that the
// same choice gives its diagonal entry of K: rows up to 2^SPREAD_MAX above it keep the
// error of a product below 2^(2 SPREAD_MAX - 59) Dr_i Dc_j (Cholesky's bound has 0 there); one
// further up raises ERR_SPREAD, and the setup factors the hierarchy again on the FP64 pipe.
// Fronts of 300 diagonally dominant unknowns with rows, or rows and columns, scaled over
// 2^-40 .. 2^40: entries of L wrong by 4e-3 with t_k = 0, now as the unscaled fronts'.  37^3
// convection-diffusion, setup + solve: 16.45 -> 16.65 ms with the scales and the subnormals below
// (57^3 FP64, for those: 61.6 -> 62.1).
//
// Kernel.  A 128 x 64 tile keeps its eight sums in TMEM (8 x 64 columns, all 512).  Digit
// rows of B are stacked in shared memory, so one MMA of N = 256 multiplies digit i of A by
// four digits of B and adds into four adjacent sums.  For 64 columns of K the eight digit
// blocks of B (64 KB, one copy) stay while the eight of A (16 KB each) stream past them:
// 192 KB loaded per 36 products, less than half the bytes per product of a plain GEMM of
// 128 x 256 tiles.  K = 512 updates of many tiles run at 40 TFLOP/s of FP64 products (1.46
// PFLOP/s of FP16 ones, the tensor pipe's rate; 1.12 on the FP64 pipe), K = 128 ones at 21
// (the epilogue's pace).  Digit blocks are stored in the swizzled shared-memory layout (64 rows
// x 128 B), so a load is one contiguous bulk copy and needs no tensor map.  The epilogue
// reads the sums into integers and releases TMEM; the rounding and the update of C (one
// row and 16 columns per thread, 16 warps: eight left it latency-bound) overlap the next
// tile's MMAs.
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>
#include <vector>

#include "rsd_internal.cuh"
#include "tcgen05.cuh"

namespace rsd {
namespace {

constexpr int ND = 8;                        // digits per entry
constexpr int TN = 64;                       // tile columns (and rows per digit block)
constexpr int TN_FEW = 16;                   // tile columns of a launch with few tiles
constexpr int KB = 64;                       // K columns per digit block
constexpr int WP = 512;                      // panel width: the longest K with exact sums
constexpr int BLK = 64 * 128;                // bytes of a digit block (64 rows x 64 FP16)
constexpr int GROUP = ND * BLK;              // a row tile's eight digits for one K block
constexpr int A_BYTES = 2 * BLK;
constexpr int UPD_DB = 7, UPD_FB = 59;       // digits of the updates
constexpr float UPD_NORM2 = 7.9f;            // a row's largest sum of (x 2^-e)^2
constexpr int SLV_DB = 8, SLV_FB = 62;       // digits of the panel solve
constexpr int EPI_WARPS = 16;                // four per TMEM lane quadrant, 16 columns each
constexpr int F64_THREADS = 64 + 32 * EPI_WARPS;
template <int W> struct F64Smem {            // W: tile columns
    static constexpr int B_BYTES = ND * W * 128;                 // a K block of B, all digits
    static constexpr int A_ST = W == TN ? 5 : 10;                // ring stages of A (two digit blocks each)
    static constexpr int TOTAL = 2 * B_BYTES + A_ST * A_BYTES + 1024 + 384;
};

// One front's operands and target of one launch.  Row tiles are 64 rows counted from the
// front's row 0; A's and B's buffers hold [K block][row tile][digit][64 x 128 B].
struct F64Task {
    const char *A, *B;
    const int *ea, *eb;                      // exponents by row of A and of B
    const int* sq;                           // per row: sum of digit 4 squared (C -= X X^T; else null)
    double *P, *U;                           // C: columns below s in P, the rest in U
    int a_nrt, b_nrt;                        // row tiles per K block
    int ldp, ldu, s;
    int r_lo, r_hi, c_lo, c_hi;              // rows and columns of C to write
    int tm0, tn0, ntm, ntn;                  // 128-row and W-column tiles
    int b_c0;                                // B's row for column c is c - b_c0 (a multiple of 64)
    int nkb, lower;
    int tile_begin;
};

// Workspace of one front's panel [L; X] (of [U^T; Y^T] too, for a nonsymmetric front)
struct F64Front {
    char *XS, *AS, *DS;                      // digits: the panel's X, the block column's A, Dinv_k
    int *ex, *aex, *dex;                     // row exponents of X, A and Dinv_k
    int* sq;                                 // per row of X: sum of digit 4 squared
    float* n2;                               // per row of X: sum of (x 2^-ex)^2
    int* tk;                                 // nonsymmetric: t_k of the panel's columns
    int nrt;
};

// ---- entry <-> digits --------------------------------------------------------------------

constexpr int E_NONE = -4000;                // exponent of a row of zeros (below any scaled entry's)

// exponent e of a finite x: |x| < 2^e (E_NONE for zero); *ok = 0 otherwise
__device__ __forceinline__ int exp_above(double x, int* ok) {
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    if (ex == 0x7ff) *ok = 0;
    return b << 1 ? ex - 1022 : E_NONE;                          // (2^-1022 for all subnormals: 59 bits hold every one)
}

// (x 2^-e)^2 for finite |x| < 2^e, to FP32 (below 2^-200: 0; a subnormal as 2^-1022 at least)
__device__ __forceinline__ float square_scaled(double x, int e) {
    const long long b = __double_as_longlong(x);
    const int f = max((int)((b >> 52) & 0x7ff), 1), ex = f - 1023 - e + 127;     // biased FP32 exponent of x 2^-e
    if (!(b << 1) || ex <= 0) return 0.f;
    const float v = __int_as_float((ex << 23) | (int)((b >> 29) & 0x7fffff));
    return v * v;
}

// round(x 2^(FB - e)) for finite |x| < 2^e
template <int FB>
__device__ __forceinline__ long long to_fixed(double x, int e) {
    const long long b = __double_as_longlong(x);
    const int eb = (int)((b >> 52) & 0x7ff), ex = max(eb, 1), sh = ex - 1075 + FB - e;     // |x| = m 2^(ex - 1075)
    if (eb == 0x7ff || sh < -54) return 0;
    const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (eb ? 0x10000000000000ull : 0ull);
    const unsigned long long f = sh >= 0 ? m << min(sh, 63) : (m + (1ull << (-sh - 1))) >> -sh;
    return b < 0 ? -(long long)f : (long long)f;
}

// balanced digits of DB bits, most significant first
template <int DB>
__device__ __forceinline__ void to_digits(long long f, int (&d)[ND]) {
    if constexpr (DB == 8) {
        uint32_t t = (uint32_t)f, u = (uint32_t)(f >> 32), carry;
#pragma unroll
        for (int k = ND - 1; k >= 4; --k) {
            d[k] = (int)(signed char)(t & 255u);
            carry = (t >> 7) & 1u;
            t = (t >> 8) + carry;
        }
        u += t;
#pragma unroll
        for (int k = 3; k >= 1; --k) {
            d[k] = (int)(signed char)(u & 255u);
            u = (uint32_t)((int)(u - (uint32_t)d[k]) >> 8);
        }
        d[0] = (int)u;
    } else {
        int t = (int)(f & 0xfffffff);
#pragma unroll
        for (int k = ND - 1; k >= 4; --k) { d[k] = ((t + 64) & 127) - 64; t = (t - d[k]) >> 7; }
        const long long h = (f >> 28) + t;                       // up to 2^31
        d[3] = (((int)h + 64) & 127) - 64;
        int u = (int)((h - d[3]) >> 7);
#pragma unroll
        for (int k = 2; k >= 1; --k) { d[k] = ((u + 64) & 127) - 64; u = (u - d[k]) >> 7; }
        d[0] = u;
    }
}

// two integers of magnitude at most 2048 as FP16
__device__ __forceinline__ uint32_t pack_top_digits(int lo, int hi) {
    const __half2 h = __floats2half2_rn((float)lo, (float)hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// two small integers as FP16 (1024 + 512 + n is exact in FP16 for |n| < 512)
__device__ __forceinline__ uint32_t pack_digits(int lo, int hi) {
    const uint32_t p = 0x66006600u + (uint32_t)((hi << 16) + lo);
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&p), __half2half2(__ushort_as_half(0x6600)));
    return *reinterpret_cast<const uint32_t*>(&h);
}

// (a1 2^S + a0) 2^e rounded to FP64 (halves away from zero), 0 <= a0 < 2^S, |a1| < 2^60
template <int S>
__device__ __forceinline__ double from_fixed(long long a1, uint32_t a0, int e) {
    const long long sign = a1 & 0x8000000000000000ll;
    if (a1 < 0) { a1 = ~a1 + (a0 == 0); a0 = S == 32 ? 0u - a0 : (0u - a0) & ((1u << (S & 31)) - 1u); }
    unsigned long long m;
    int l;
    if (a1) {
        l = __clzll(a1);
        m = ((unsigned long long)a1 << l) | (l >= S ? (unsigned long long)a0 << (l - S) : (unsigned long long)a0 >> (S - l));
    } else {
        if (!a0) return 0.0;
        m = (unsigned long long)a0 << (64 - S);
        const int z = __clzll((long long)m);
        m <<= z;
        l = 64 + z;
    }
    const int be = 11 + S - l + e + 52 + 1022;                   // biased exponent - 1
    if (be < 0) {                                                // subnormal: fewer bits
        const int sh = min(11 - be, 65);
        m = sh > 64 ? 0 : sh == 64 ? m >> 63 : (m >> sh) + ((m >> (sh - 1)) & 1);
        return __longlong_as_double(sign | (long long)m);
    }
    m = (m >> 11) + ((m >> 10) & 1);                              // 53 bits, 2^52 <= m <= 2^53
    if (be > 2045) return __longlong_as_double(sign | 0x7ff0000000000000ll);
    return __longlong_as_double(sign | (long long)(((unsigned long long)be << 52) + m));
}

// byte offset of 16-byte chunk c of row r inside a digit block (128-byte swizzle)
__device__ __forceinline__ int blk_off(int r, int c) { return r * 128 + ((c ^ (r & 7)) << 4); }

// a value that is not finite: reported like a pivot that is not positive
__device__ __forceinline__ void mark_bad(int node, int* err, int* bad_front) {
    atomicExch(&err[ERR_NOT_SPD], 1);
    atomicMin(&err[ERR_NOT_SPD_NODE], node);
    bad_front[node] = 1;
}

// ---- scale of nonsymmetric fronts ----------------------------------------------------------

constexpr int SPREAD_MAX = 4;                // see above: 2^-51 Dr_i Dc_j in the worst case

// Which power of the diagonal goes to the equations: 0 half of its exponent, 1 all, -1 none.
// w[q]: how far the largest entry of K lies above its place under q = 0, 1, -1 (in bits).
__device__ __forceinline__ int lu_scaling(const int* __restrict__ w) {
    const int w1 = w[1], w2 = w[2];
    return w[0] > min(w1, w2) + 1 ? (w1 <= w2 ? 1 : -1) : 0;
}
// exponents of Dr and Dc for a diagonal entry (or pivot) of exponent e
__device__ __forceinline__ int lu_row_exp(int q, int e) { return ((1 + q) * e) >> 1; }
__device__ __forceinline__ int lu_col_exp(int q, int e) { return ((1 - q) * e) >> 1; }

__global__ void k_lu_diag_exp(int n, const int64_t* __restrict__ rowptr, const int* __restrict__ col, const double* __restrict__ val,
                              int* __restrict__ de) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t a = rowptr[i], e = rowptr[i + 1];
    const int64_t end = e;
    while (a < e) {
        const int64_t mid = (a + e) >> 1;
        if (col[mid] < i) a = mid + 1; else e = mid;
    }
    int ok = 1;
    de[i] = a < end && col[a] == i ? exp_above(val[a], &ok) : E_NONE;
}

// largest exponent of an entry of K above Dr_i Dc_j, for the three choices; a warp a row
__global__ void __launch_bounds__(256) k_lu_spread(int n, const int64_t* __restrict__ rowptr, const int* __restrict__ col,
                                                  const double* __restrict__ val, const int* __restrict__ de, int* __restrict__ w) {
    __shared__ int s_w[3];
    if (threadIdx.x < 3) s_w[threadIdx.x] = INT_MIN;
    __syncthreads();
    const int lane = threadIdx.x & 31, warps = (int)(gridDim.x * (blockDim.x >> 5));
    int m[3] = {INT_MIN, INT_MIN, INT_MIN};
    for (int i = (int)(blockIdx.x * (blockDim.x >> 5)) + (threadIdx.x >> 5); i < n; i += warps) {
        const int di = de[i];
        if (di == E_NONE) continue;
        for (int64_t k = rowptr[i] + lane; k < rowptr[i + 1]; k += 32) {
            int ok = 1;
            const int e = exp_above(val[k], &ok), dj = de[col[k]];
            if (e == E_NONE || !ok || dj == E_NONE) continue;
#pragma unroll
            for (int h = 0; h < 3; ++h) {
                const int q = h == 2 ? -1 : h;
                m[h] = max(m[h], e - lu_row_exp(q, di) - lu_col_exp(q, dj));
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 3; ++h) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m[h] = max(m[h], __shfl_xor_sync(0xffffffffu, m[h], o));
        if (lane == 0) atomicMax(&s_w[h], m[h]);
    }
    __syncthreads();
    if (threadIdx.x < 3) atomicMax(&w[threadIdx.x], s_w[threadIdx.x]);
}

// ---- splitting -----------------------------------------------------------------------------
// Half a warp takes a row and 128 columns, eight adjacent columns (one 16-byte chunk per
// digit) to a lane.  HBM-bound: 8 bytes read and 16 written per entry.

__device__ __forceinline__ int half_warp_max(int v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ int half_warp_sum(int v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// digits of x[0..8) (scaled by 2^-e[.]) into chunk `ch` (0..15) of row r of the row tile at
// dst; the second 64 columns lie kb_stride bytes further.  Returns the sum of digit 4 squared.
template <int DB, int FB>
__device__ __forceinline__ int store_digits(const double (&x)[8], const int (&e)[8], char* dst, int64_t kb_stride, int r, int ch) {
    uint32_t o[ND][4];
    int sq = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int d[2][ND];
        to_digits<DB>(to_fixed<FB>(x[2 * q], e[2 * q]), d[0]);
        to_digits<DB>(to_fixed<FB>(x[2 * q + 1], e[2 * q + 1]), d[1]);
        sq += d[0][4] * d[0][4] + d[1][4] * d[1][4];
#pragma unroll
        for (int t = 1; t < ND; ++t) o[t][q] = pack_digits(d[0][t], d[1][t]);
        o[0][q] = pack_top_digits(d[0][0], d[1][0]);
    }
    dst += (ch >> 3) * kb_stride + blk_off(r, ch & 7);
#pragma unroll
    for (int t = 0; t < ND; ++t) *reinterpret_cast<uint4*>(dst + t * BLK) = make_uint4(o[t][0], o[t][1], o[t][2], o[t][3]);
    return sq;
}

// scale of row r of [L; X] (Dr) or of [U^T; Y^T] (Dc), from its diagonal entry of K
__device__ __forceinline__ int row_scale(const FrontDesc& f, int r, bool upper, int sc, const int* __restrict__ de) {
    const int d = de[r < f.s ? f.I[r] : f.Bd[r - f.s]];
    return upper ? lu_col_exp(sc, d) : lu_row_exp(sc, d);
}

// Operands of the panel solve at block column k: A_ij 2^-s_j (rows below the diagonal
// block) and Dinv_cj 2^s_j, s_j the exponent of L_jj (a row's entries then compare across
// columns of different scale).  blockIdx.x < na: nr rows of A, else of Dinv.
// Nonsymmetric fronts, blockIdx.z = 0: P against (U_kk^T)^-1, s_j the exponent of Dc_j; 1: PU
// against L_kk^-1, s_j that of Dr_j, which is the column's t_k too (de, the exponents of K's
// diagonal, and sw as launch_lu_scale left them; null for symmetric fronts).
__global__ void __launch_bounds__(256) k_split_a(const FrontDesc* __restrict__ fronts, const F64Front* __restrict__ wk, int k,
                                                int K0, int na, int nr, const int* __restrict__ de, const int* __restrict__ sw,
                                                int* __restrict__ err, int* __restrict__ bad_front) {
    __shared__ int sj[NB];
    const FrontDesc f = fronts[blockIdx.y];
    if (f.s <= k) return;
    const int w = min(NB, f.s - k), ch = threadIdx.x & 15, j0 = ch * 8;
    const bool isA = (int)blockIdx.x < na;
    const int r0 = isA ? k + w + (int)blockIdx.x * nr : ((int)blockIdx.x - na) * nr;
    if (isA && r0 >= f.N) return;
    const F64Front wf = wk[gridDim.z * blockIdx.y + blockIdx.z];
    const bool lu = gridDim.z == 2, upper = blockIdx.z == 1;
    const double* P = (const double*)(upper ? f.PU : f.P);
    const double* diag = (const double*)(lu ? f.PU : f.P);       // u_jj or l_jj
    const double* Dk = (const double*)(lu && !upper ? f.DinvU : f.Dinv) + (int64_t)(k / NB) * NB * NB;
    const int sc = lu ? lu_scaling(sw) : 0;
    int ok = 1, spread = 0;
    if (threadIdx.x < NB) {
        int e = (int)threadIdx.x < w ? exp_above(diag[(int64_t)(k + threadIdx.x) * f.ldp + k + threadIdx.x], &ok) : 0;
        if (lu) e = upper ? lu_row_exp(sc, e) : lu_col_exp(sc, e);
        sj[threadIdx.x] = e;
        if (lu && upper && blockIdx.x == 0) wf.tk[k - K0 + threadIdx.x] = e;
    }
    __syncthreads();
#pragma unroll 1
    for (int r = r0 + (threadIdx.x >> 4); r < r0 + nr; r += 16) {
        const bool in = isA ? r < f.N : r < w;
        const double* src = (isA ? P + (int64_t)r * f.ldp + k : Dk + r * NB) + j0;
        int top = E_NONE, e[8];
        double x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            x[q] = in && j0 + q < w ? src[q] : 0.0;
            e[q] = isA ? sj[j0 + q] : -sj[j0 + q];
            const int ex = exp_above(x[q], &ok);
            if (ex != E_NONE) top = max(top, ex - e[q]);
        }
        top = half_warp_max(top);
#pragma unroll
        for (int q = 0; q < 8; ++q) e[q] += top;
        if (in || !isA) {
            char* dst = (isA ? wf.AS : wf.DS) + (int64_t)(r >> 6) * GROUP;
            store_digits<SLV_DB, SLV_FB>(x, e, dst, (int64_t)(isA ? wf.nrt : 2) * GROUP, r & 63, ch);
            if (ch == 0) (isA ? wf.aex : wf.dex)[r] = top;
        }
        if (lu && isA && in) spread |= top > row_scale(f, r, upper, sc, de) + SPREAD_MAX;
    }
    if (!ok) mark_bad(f.node, err, bad_front);
    else if (spread) err[ERR_SPREAD] = 1;
}

// Digits of the solved rows X of block column k for the updates that follow, the panel's
// columns K0 .. k + w of a row on one exponent (from the largest entry and the norm):
// where the new block raises it, the row's earlier blocks are split again.  Nonsymmetric fronts:
// column c times 2^t_c on side 0, 2^-t_c on side 1.
__global__ void __launch_bounds__(256) k_split_x(const FrontDesc* __restrict__ fronts, const F64Front* __restrict__ wk, int k,
                                                int K0, const int* __restrict__ de, const int* __restrict__ sw,
                                                int* __restrict__ err, int* __restrict__ bad_front) {
    const FrontDesc f = fronts[blockIdx.y];
    if (f.s <= k) return;
    const F64Front wf = wk[gridDim.z * blockIdx.y + blockIdx.z];
    const int w = min(NB, f.s - k), ch = threadIdx.x & 15, j0 = ch * 8;
    if (k + w + (int)blockIdx.x * 16 >= f.N) return;
    const int r = k + w + (int)blockIdx.x * 16 + (threadIdx.x >> 4);
    const bool in = r < f.N;
    const double* src = (const double*)(blockIdx.z ? f.PU : f.P) + (int64_t)r * f.ldp + j0;
    const bool lu = gridDim.z == 2;
    const int sign = blockIdx.z ? -1 : 1;
    int ok = 1, top = E_NONE, t[8];
    double x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        x[q] = in && j0 + q < w ? src[k + q] : 0.0;
        t[q] = lu ? sign * wf.tk[k - K0 + j0 + q] : 0;
        const int ex = exp_above(x[q], &ok);
        if (ex != E_NONE) top = max(top, ex + t[q]);
    }
    top = half_warp_max(top);
    const int old = in && k > K0 ? wf.ex[r] : E_NONE;
    top = max(top, old);
    float n2 = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) n2 += square_scaled(x[q], top - t[q]);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
    if (in && k > K0) n2 += wf.n2[r] * exp2f((float)(2 * max(old - top, -60)));
    while (n2 > UPD_NORM2) { n2 *= 0.25f; ++top; }
    int sq = 0;
    if (in) {
        int e[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) e[q] = top - t[q];
        const int64_t stride = (int64_t)wf.nrt * GROUP;
        char* dst = wf.XS + (int64_t)(r >> 6) * GROUP;
        sq = store_digits<UPD_DB, UPD_FB>(x, e, dst + (k - K0) / KB * stride, stride, r & 63, ch);
        if (top > old)
            for (int c = K0; c < k; c += NB) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    x[q] = src[c + q];
                    e[q] = lu ? top - sign * wf.tk[c - K0 + j0 + q] : top;
                }
                sq += store_digits<UPD_DB, UPD_FB>(x, e, dst + (c - K0) / KB * stride, stride, r & 63, ch);
            }
    }
    sq = half_warp_sum(sq);                              // (every lane has read the old exponent)
    if (in && ch == 0) {
        wf.ex[r] = top;
        wf.n2[r] = n2;
        wf.sq[r] = k > K0 && top == old ? wf.sq[r] + sq : sq;
    }
    if (!ok) mark_bad(f.node, err, bad_front);
    else if (lu && in && top > row_scale(f, r, blockIdx.z, lu_scaling(sw), de) + SPREAD_MAX) err[ERR_SPREAD] = 1;
}

// ---- the GEMM ------------------------------------------------------------------------------

// tile `g` of a launch: its task, 128-row tile and W-column tile.  Lower tasks (C's lower
// triangle) have min(ntn, c0 + m q) tiles in row tile q, m = 128 / W, c0 = m (tm0 + 1) - tn0.
template <int W>
__device__ __forceinline__ int f64_tile(const F64Task* __restrict__ tasks, int ntask, int g, int* tm, int* tn) {
    constexpr int m = BM / W;
    int lo = 0, hi = ntask - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tasks[mid].tile_begin <= g) lo = mid; else hi = mid - 1;
    }
    const F64Task& t = tasks[lo];
    const int l = g - t.tile_begin;
    int q, c;
    if (t.lower) {
        const int c0 = m * (t.tm0 + 1) - t.tn0;
        auto before = [&](int r) { return c0 * r + m / 2 * r * (r - 1); };    // tiles of row tiles 0 .. r - 1
        const int qs = max(0, (t.ntn - c0 + m - 1) / m);                       // the first with all ntn
        if (l < before(qs)) {
            const float b = (float)c0 - 0.5f * m;
            q = (int)((sqrtf(b * b + 2.0f * m * (float)l) - b) / m);
            q = max(0, min(q, qs - 1));
            while (q > 0 && before(q) > l) --q;
            while (q + 1 < qs && before(q + 1) <= l) ++q;
            c = l - before(q);
        } else {
            q = qs + (l - before(qs)) / t.ntn;
            c = (l - before(qs)) % t.ntn;
        }
    } else {
        q = l / t.ntn;
        c = l % t.ntn;
    }
    *tm = t.tm0 + q;
    *tn = t.tn0 + c;
    return lo;
}

__device__ __forceinline__ void tmem_ld(uint32_t a, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}

__device__ __forceinline__ void tmem_ld(uint32_t a, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(a));
}

// SOLVE = false: C -= A B^T.  SOLVE = true: C = A B^T.  W: tile columns.
template <bool SOLVE, int W>
__global__ void __launch_bounds__(F64_THREADS, 1)
k_gemm_f64_tc(const F64Task* __restrict__ tasks, int ntask, int n_tiles, int* __restrict__ err) {
    extern __shared__ unsigned char smem_raw[];
    constexpr int B_BYTES = F64Smem<W>::B_BYTES, A_ST = F64Smem<W>::A_ST;
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023) & ~1023u;                // two K blocks of B, A_ST x 16 KB of A, barriers
    const uint32_t sA = base + 2 * B_BYTES, bars = sA + A_ST * A_BYTES;
    const uint32_t b_full = bars, b_empty = bars + 16, a_full = bars + 32, a_empty = a_full + 8 * A_ST;
    const uint32_t acc_full = a_empty + 8 * A_ST, acc_empty = acc_full + 8;
    uint32_t* tmem_slot = (uint32_t*)(smem_raw + (acc_empty + 8 - raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int q = 0; q < 2; ++q) { mbar_init(b_full + 8 * q, 1); mbar_init(b_empty + 8 * q, 1); }
        for (int q = 0; q < A_ST; ++q) { mbar_init(a_full + 8 * q, 1); mbar_init(a_empty + 8 * q, 1); }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, F64_THREADS - 64);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(ND * W) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    bool ok = true;                          // no wait of this thread has given up
    if (warp == 0) {
        if (lane == 0) {
            uint32_t ia = 0, ib = 0;
            for (int g = blockIdx.x; g < n_tiles && ok; g += gridDim.x) {
                int tm, tn;
                const F64Task& t = tasks[f64_tile<W>(tasks, ntask, g, &tm, &tn)];
                const char* A = t.A + (int64_t)(2 * tm) * GROUP;
                const int br = tn * W - t.b_c0;                  // B's first row
                const char* B = t.B + (int64_t)(br / TN) * GROUP + (br % TN) * 128;
                const int64_t sa = (int64_t)t.a_nrt * GROUP, sb = (int64_t)t.b_nrt * GROUP;
                const int nkb = t.nkb;
                for (int kb = 0; kb < nkb && ok; ++kb, ++ib) {
                    const uint32_t q = ib & 1;
                    if (!mbar_wait(b_empty + 8 * q, ((ib >> 1) & 1) ^ 1, err)) { ok = false; break; }
                    mbar_expect_tx(b_full + 8 * q, B_BYTES);
                    if constexpr (W == TN) {
                        bulk_load(base + q * B_BYTES, B + kb * sb, B_BYTES, b_full + 8 * q);
                    } else {
#pragma unroll
                        for (int d = 0; d < ND; ++d)
                            bulk_load(base + q * B_BYTES + d * W * 128, B + kb * sb + d * BLK, W * 128, b_full + 8 * q);
                    }
                    for (int i = 0; i < ND; ++i, ++ia) {
                        const uint32_t s = ia % A_ST;
                        if (!mbar_wait(a_empty + 8 * s, ((ia / A_ST) & 1) ^ 1, err)) { ok = false; break; }
                        mbar_expect_tx(a_full + 8 * s, A_BYTES);
                        const char* a = A + kb * sa + i * BLK;
                        bulk_load(sA + s * A_BYTES, a, BLK, a_full + 8 * s);
                        bulk_load(sA + s * A_BYTES + BLK, a + GROUP, BLK, a_full + 8 * s);
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            uint32_t ia = 0, ib = 0, it = 0;
            for (int g = blockIdx.x; g < n_tiles && ok; g += gridDim.x, ++it) {
                int tm, tn;
                const int nkb = tasks[f64_tile<W>(tasks, ntask, g, &tm, &tn)].nkb;
                if (!mbar_wait(acc_empty, (it & 1) ^ 1, err)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int kb = 0; kb < nkb && ok; ++kb, ++ib) {
                    const uint32_t q = ib & 1;
                    if (!mbar_wait(b_full + 8 * q, (ib >> 1) & 1, err)) { ok = false; break; }
                    for (int i = 0; i < ND; ++i, ++ia) {
                        const uint32_t s = ia % A_ST;
                        if (!mbar_wait(a_full + 8 * s, (ia / A_ST) & 1, err)) { ok = false; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        // digit i of A times digits j of B, j < 8 - i, into the sums d = i + j
                        constexpr int JN = 256 / W;              // digits of B per MMA, at most
                        for (int j = 0; j < ND - i; j += JN) {
                            const uint32_t idesc = idesc_of(0u, W * min(JN, ND - i - j));
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                mma_f16(tmem + (i + j) * W, smem_desc(sA + s * A_BYTES + kk * 32),
                                        smem_desc(base + q * B_BYTES + j * W * 128 + kk * 32), idesc, (kb | i | kk) != 0);
                        }
                        mma_commit(a_empty + 8 * s);
                    }
                    if (ok) mma_commit(b_empty + 8 * q);
                }
                mma_commit(acc_full);
            }
        }
    } else {
        constexpr int CW = W / (EPI_WARPS / 4), GW = CW < 8 ? CW : 8;   // columns per thread, per load
        constexpr int DB = SOLVE ? SLV_DB : UPD_DB, S = 4 * DB;
        constexpr int E0 = 14 * DB - 7 * DB - 2 * (SOLVE ? SLV_FB : UPD_FB);   // exponent of the sum d = 7
        const int quarter = warp & 3, part = (warp - 2) >> 2, row = quarter * 32 + lane;
        uint32_t it = 0;
        for (int g = blockIdx.x; g < n_tiles; g += gridDim.x, ++it) {
            int tm, tn;
            const F64Task& t = tasks[f64_tile<W>(tasks, ntask, g, &tm, &tn)];
            const int gr = tm * BM + row, c_base = tn * W + part * CW;
            const int r_lo = t.r_lo, r_hi = t.r_hi, c_lo = t.c_lo, s = t.s;
            const int c_hi = t.lower ? min(t.c_hi, gr + 1) : t.c_hi;
            const bool in = gr >= r_lo && gr < r_hi && c_base < c_hi && c_base + CW > c_lo;
            const int ea = in ? t.ea[gr] : 0;
            const int* eb = t.eb + (c_base - t.b_c0);
            double* P = t.P + (int64_t)gr * t.ldp;
            double* U = t.U + (int64_t)(gr - s) * t.ldu - s;
            if (!SOLVE && in && c_base >= c_lo) asm volatile("prefetch.global.L2 [%0];" ::"l"(c_base < s ? P + c_base : U + c_base));
            if (!__all_sync(0xffffffffu, mbar_wait(acc_full, it & 1, err))) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            long long a1[CW];
            uint32_t a0[CW];
#pragma unroll
            for (int q = 0; q < CW / GW; ++q)
#pragma unroll
                for (int lowhalf = 0; lowhalf < 2; ++lowhalf) {
                    uint32_t v[4][GW];
#pragma unroll
                    for (int d = 0; d < 4; ++d)
                        tmem_ld(tmem + ((uint32_t)(quarter * 32) << 16) + (4 * lowhalf + d) * W + part * CW + q * GW, v[d]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int c = 0; c < GW; ++c) {
                        int n[4];
#pragma unroll
                        for (int d = 0; d < 4; ++d) n[d] = __float2int_rn(__uint_as_float(v[d][c]));
                        const long long sum = (long long)n[0] * (1 << 3 * DB) + (long long)n[1] * (1 << 2 * DB) + (long long)n[2] * (1 << DB) + n[3];
                        if (!lowhalf) {
                            a1[GW * q + c] = sum;
                        } else {
                            a1[GW * q + c] += sum >> S;
                            a0[GW * q + c] = (uint32_t)(sum & ((1ll << S) - 1));
                        }
                    }
                }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty) : "memory");
            if (!in) continue;
            if (!SOLVE && t.sq && gr >= c_base && gr < c_base + CW) {       // C's diagonal
                const uint32_t add = (uint32_t)(t.sq[gr] + 64) >> 7;
#pragma unroll
                for (int c = 0; c < CW; ++c)
                    if (gr == c_base + c) {
                        a0[c] += add;
                        a1[c] += a0[c] >> (S & 31);
                        a0[c] &= (1u << (S & 31)) - 1u;
                    }
            }
#pragma unroll
            for (int q = 0; q < CW / GW; ++q) {
                const int c0 = c_base + GW * q;
                if (c0 >= c_hi || c0 + GW <= c_lo) continue;
                double* C = c0 >= s ? U : P;
                if (c0 >= c_lo && c0 + GW <= c_hi && (c0 + GW <= s || (c0 >= s && !(s & 1)))) {
                    double2* C2 = reinterpret_cast<double2*>(C + c0);
                    double2 v[GW / 2];
                    if constexpr (!SOLVE)
#pragma unroll
                        for (int c = 0; c < GW / 2; ++c) v[c] = C2[c];
#pragma unroll
                    for (int c = 0; c < GW / 2; ++c) {
                        const int k = GW * q + 2 * c;
                        const double x = from_fixed<S>(a1[k], a0[k], ea + __ldg(eb + k) + E0);
                        const double y = from_fixed<S>(a1[k + 1], a0[k + 1], ea + __ldg(eb + k + 1) + E0);
                        C2[c] = SOLVE ? make_double2(x, y) : make_double2(v[c].x - x, v[c].y - y);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < GW; ++c) {
                        const int cc = c0 + c;
                        if (cc < c_lo || cc >= c_hi) continue;
                        const double x = from_fixed<S>(a1[GW * q + c], a0[GW * q + c], ea + __ldg(eb + GW * q + c) + E0);
                        double* p = (cc >= s ? U : P) + cc;
                        *p = SOLVE ? x : *p - x;
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    const bool gave_up = __syncthreads_or(!ok);
    if (warp == 1) {
        if (gave_up) settle_in_flight();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ND * W) : "memory");
    }
}

size_t al(size_t v) { return (v + 1023) & ~(size_t)1023; }
int row_tiles(int N) { return 2 * ((N + BM - 1) / BM); }

size_t front_bytes(int N) {
    const size_t g = (size_t)row_tiles(N) * GROUP;
    return (WP / KB + 2) * g + 4 * (size_t)GROUP + 4 * al(sizeof(int) * (size_t)N) + al(sizeof(int) * NB) + al(sizeof(int) * WP);
}

// tiles of W columns covering the task's rows and columns
int64_t set_tiles(F64Task& t, int W) {
    t.tm0 = t.r_lo / BM; t.ntm = (t.r_hi + BM - 1) / BM - t.tm0;
    t.tn0 = t.c_lo / W; t.ntn = (t.c_hi + W - 1) / W - t.tn0;
    if (!t.lower) return (int64_t)t.ntm * t.ntn;
    int64_t n = 0;
    for (int q = 0; q < t.ntm; ++q) n += std::min(t.ntn, BM / W * (t.tm0 + q + 1) - t.tn0);
    return n;
}

}  // namespace

int launch_lu_scale(Handle& h) {
    cudaStream_t st = h.stream;
    const int pi = prof_begin(h, K_ASSEMBLE, st);
    RSD_CUDA_TRY(cudaMemsetAsync(h.d_lu_scale + h.n, 0x80, sizeof(int) * LU_SCALE_EXTRA, st));       // far below any exponent
    k_lu_diag_exp<<<(unsigned)((h.n + 255) / 256), 256, 0, st>>>(h.n, h.d_rowptr, h.d_col, h.d_val, h.d_lu_scale);
    k_lu_spread<<<(unsigned)std::min((h.n + 7) / 8, 8 * h.num_sms), 256, 0, st>>>(h.n, h.d_rowptr, h.d_col, h.d_val, h.d_lu_scale,
                                                                                h.d_lu_scale + h.n);
    count_launch(2);
    prof_end(h, pi, 0.0, 12.0 * h.nnz, st);
    RSD_CUDA_TRY(cudaGetLastError());
    return RSD_OK;
}

// Workspace of a level: the digits of one 512-wide panel of every front at once where that
// fits the cap (groups of fronts then take turns), of one front at least.  The cap is far
// above what fills the chip: 4 GiB hold over 100 fronts of 4000 rows, thousands of tiles.
size_t f64_tc_workspace(const std::vector<int>& rows, bool lu, size_t* least) {
    const size_t cap = (size_t)4 << 30;
    size_t sum = 0, most = 0;
    for (int N : rows) { sum += (lu ? 2 : 1) * front_bytes(N); most = std::max(most, (lu ? 2 : 1) * front_bytes(N)); }
    *least = std::max(*least, most);
    return std::min(sum, std::max(cap, most));
}

// Partial Cholesky (all steps of factor.cu) or LU (of factor_lu.cu) of every FP64 front of
// level li, 512-wide panels: per 128-wide block column the update by the panel's earlier
// columns, the diagonal block, the split and the solve of the rows below; per panel the
// update of everything right of it (P and U; PU), K = the panel's width.  Nonsymmetric
// fronts run every step on [L; X] and [U^T; Y^T] (side 0 and 1) in one launch:
// P -= P PU^T, PU -= PU P^T, U -= X Y.
int factor_level_f64_tc(Handle& h, int li) {
    Level& L = h.levels[li];
    cudaStream_t st = h.stream;
    const int nf_all = (int)L.fronts.size(), sides = h.lu ? 2 : 1;
    struct Launch { size_t off; int n, tiles, solve, few; double flops, bytes; };
    struct Group { int f0, nf, max_s; };
    std::vector<Group> groups;
    std::vector<F64Front> wk((size_t)nf_all * sides);
    for (int f0 = 0; f0 < nf_all;) {
        Group g{f0, 0, 0};
        size_t off = 0;
        while (f0 + g.nf < nf_all) {
            const FrontDesc& f = L.fronts[f0 + g.nf];
            const size_t need = front_bytes(f.N);
            if (g.nf && off + sides * need > h.f64_ws_bytes) break;
            if (sides * need > h.f64_ws_bytes) return RSD_ERR_ARG;
            for (int sd = 0; sd < sides; ++sd) {
                F64Front& w = wk[(size_t)(f0 + g.nf) * sides + sd];
                char* p = h.f64_ws + off;
                w.nrt = row_tiles(f.N);
                w.XS = p; p += (size_t)(WP / KB) * w.nrt * GROUP;
                w.AS = p; p += (size_t)2 * w.nrt * GROUP;
                w.DS = p; p += (size_t)4 * GROUP;
                w.ex = (int*)p; p += al(sizeof(int) * (size_t)f.N);
                w.sq = (int*)p; p += al(sizeof(int) * (size_t)f.N);
                w.n2 = (float*)p; p += al(sizeof(float) * (size_t)f.N);
                w.aex = (int*)p; p += al(sizeof(int) * (size_t)f.N);
                w.dex = (int*)p; p += al(sizeof(int) * NB);
                w.tk = sd ? wk[(size_t)(f0 + g.nf) * sides].tk : (int*)p;      // both sides' columns
                off += need;
            }
            g.max_s = std::max(g.max_s, f.s);
            ++g.nf;
        }
        f0 += g.nf;
        groups.push_back(g);
    }
    // every launch's task list, uploaded once
    std::vector<F64Task> tasks;
    std::vector<Launch> launches;
    // Launches of few 128 x 64 tiles take 16-column tiles: a tile is a serial chain (the loads
    // and MMAs of its K, then an epilogue of 16 columns a thread), about 28 us at K = 128 with
    // most SMs idle; with four columns a thread and a quarter of the MMAs 14 us.  With more than
    // half a wave of wide tiles the narrow ones, which load A four times as often, gain nothing.
    auto finish = [&]() {
        if (launches.empty()) return;
        Launch& l = launches.back();
        if (l.tiles * 2 > h.num_sms) return;
        l.few = 1;
        l.tiles = 0;
        for (int i = 0; i < l.n; ++i) {
            F64Task& t = tasks[l.off + i];
            t.tile_begin = l.tiles;
            l.tiles += (int)set_tiles(t, TN_FEW);
        }
    };
    auto begin = [&](int solve) {
        finish();
        launches.push_back({tasks.size(), 0, 0, solve, 0, 0, 0});
    };
    auto add = [&](F64Task t) {
        Launch& l = launches.back();
        t.tile_begin = l.tiles;
        l.tiles += (int)set_tiles(t, TN);
        ++l.n;
        const double m = t.r_hi - t.r_lo, n = t.c_hi - t.c_lo;
        const double c = t.lower ? m * n - 0.5 * n * (n - 1) : m * n;
        l.flops += 2.0 * c * t.nkb * KB;
        l.bytes += 16.0 * c + 16.0 * m * t.nkb * KB;
        tasks.push_back(t);
    };
    for (const Group& g : groups) {
        for (int k = 0; k < g.max_s; k += NB) {
            const int K0 = k / WP * WP;
            // rows [r0, N) and columns [c0, c1) of front q (side sd): C -= X X^T, X Y^T or Y X^T
            auto update = [&](int q, int sd, int r0, int c0, int c1, int nkb, bool lower) {
                const FrontDesc& f = L.fronts[g.f0 + q];
                const F64Front& a = wk[(size_t)(g.f0 + q) * sides + sd];
                const F64Front& b = wk[(size_t)(g.f0 + q) * sides + (sides - 1 - sd)];
                F64Task t{};
                t.A = a.XS; t.B = b.XS;
                t.a_nrt = t.b_nrt = a.nrt;
                t.ea = a.ex; t.eb = b.ex;
                t.sq = sides == 1 ? a.sq : nullptr;
                t.P = (double*)(sd ? f.PU : f.P); t.U = (double*)f.U;
                t.ldp = f.ldp; t.ldu = f.ldu; t.s = f.s;
                t.r_lo = r0; t.r_hi = f.N; t.c_lo = c0; t.c_hi = c1;
                t.nkb = nkb;
                t.lower = lower;
                add(t);
            };
            if (k > K0) {                                  // the block column from the panel's earlier ones
                begin(0);
                for (int q = 0; q < g.nf; ++q) {
                    const FrontDesc& f = L.fronts[g.f0 + q];
                    if (f.s <= k) continue;
                    for (int sd = 0; sd < sides; ++sd) update(q, sd, k, k, std::min(k + NB, f.s), (k - K0) / KB, true);
                }
            }
            begin(1);                                      // the rows below the diagonal block
            for (int q = 0; q < g.nf; ++q) {
                const FrontDesc& f = L.fronts[g.f0 + q];
                const int wd = std::min(NB, f.s - k);
                if (f.s <= k || f.N <= k + wd) continue;
                for (int sd = 0; sd < sides; ++sd) {
                    const F64Front& w = wk[(size_t)(g.f0 + q) * sides + sd];
                    F64Task t{};
                    t.A = w.AS; t.B = w.DS;
                    t.a_nrt = w.nrt; t.b_nrt = 2;
                    t.ea = w.aex; t.eb = w.dex;
                    t.P = (double*)(sd ? f.PU : f.P); t.U = (double*)f.U;
                    t.ldp = f.ldp; t.ldu = f.ldu; t.s = f.s;
                    t.r_lo = k + wd; t.r_hi = f.N; t.c_lo = k; t.c_hi = k + wd;
                    t.b_c0 = k;
                    t.nkb = (wd + KB - 1) / KB;
                    add(t);
                }
            }
            if (k + NB < std::min(K0 + WP, g.max_s)) continue;
            begin(0);                                      // everything right of the panel
            for (int q = 0; q < g.nf; ++q) {
                const FrontDesc& f = L.fronts[g.f0 + q];
                const int c0 = std::min(K0 + WP, f.s), nkb = (c0 - K0 + KB - 1) / KB;
                if (f.s <= K0 || f.N <= c0) continue;
                if (sides == 1) {
                    update(q, 0, c0, c0, f.N, nkb, true);
                    continue;
                }
                if (f.s > c0)
                    for (int sd = 0; sd < 2; ++sd) update(q, sd, c0, c0, f.s, nkb, true);
                if (f.b) update(q, 0, f.s, f.s, f.N, nkb, false);
            }
        }
    }
    finish();
    const size_t o_tasks = al(sizeof(F64Front) * wk.size()), total = o_tasks + sizeof(F64Task) * tasks.size();
    char* meta = nullptr;
    RSD_CUDA_TRY(cudaMallocAsync((void**)&meta, total, st));
    struct Free { char* p; cudaStream_t s; ~Free() { cudaFreeAsync(p, s); } } fr{meta, st};
    RSD_CUDA_TRY(cudaMemcpyAsync(meta, stage_host(h, wk.data(), sizeof(F64Front) * wk.size()), sizeof(F64Front) * wk.size(), cudaMemcpyHostToDevice, st));
    if (!tasks.empty())
        RSD_CUDA_TRY(cudaMemcpyAsync(meta + o_tasks, stage_host(h, tasks.data(), sizeof(F64Task) * tasks.size()),
                                     sizeof(F64Task) * tasks.size(), cudaMemcpyHostToDevice, st));
    const F64Front* d_wk = (const F64Front*)meta;
    const F64Task* d_tasks = (const F64Task*)(meta + o_tasks);
    using Kernel = void (*)(const F64Task*, int, int, int*);
    static constexpr Kernel kern[2][2] = {{k_gemm_f64_tc<false, TN>, k_gemm_f64_tc<true, TN>},
                                          {k_gemm_f64_tc<false, TN_FEW>, k_gemm_f64_tc<true, TN_FEW>}};
    static constexpr int smem[2] = {F64Smem<TN>::TOTAL, F64Smem<TN_FEW>::TOTAL};
    for (int few = 0; few < 2; ++few)
        for (int sv = 0; sv < 2; ++sv)
            RSD_CUDA_TRY(cudaFuncSetAttribute(kern[few][sv], cudaFuncAttributeMaxDynamicSharedMemorySize, smem[few]));
    const int* de = h.lu ? h.d_lu_scale : nullptr;
    const int* sw = h.lu ? h.d_lu_scale + h.n : nullptr;
    size_t li_ = 0;
    auto run = [&]() -> int {
        const Launch& l = launches[li_++];
        if (!l.tiles) return RSD_OK;
        const int pi = prof_begin(h, K_GEMM_TC16, st);
        const unsigned grid = (unsigned)std::min(l.tiles, h.num_sms);
        kern[l.few][l.solve]<<<grid, F64_THREADS, smem[l.few], st>>>(d_tasks + l.off, l.n, l.tiles, h.d_err);
        count_launch();
        prof_end(h, pi, l.flops, l.bytes, st);
        RSD_CUDA_TRY(cudaGetLastError());
        return RSD_OK;
    };
    for (const Group& g : groups) {
        const FrontDesc* d_fr = L.d_fronts + g.f0;
        if (g.max_s == 0) continue;
        for (int k = 0; k < g.max_s; k += NB) {
            const int K0 = k / WP * WP;
            if (k > K0) RSD_TRY(run());
            RSD_TRY(launch_diag_f64(h, li, g.f0, g.nf, k, st));
            double bytes = 0;
            int rows = 0;                                   // below the diagonal block, at most
            for (int q = 0; q < g.nf; ++q) {
                const FrontDesc& f = L.fronts[g.f0 + q];
                if (f.s <= k) continue;
                const int wd = std::min(NB, f.s - k);
                rows = std::max(rows, f.N - k - wd);
                bytes += 24.0 * sides * (f.N - k - wd) * wd;
            }
            auto split = [&](bool x) -> int {
                if (!rows) return RSD_OK;
                const int pi = prof_begin(h, K_COPY16, st);
                if (x) k_split_x<<<dim3((unsigned)((rows + 15) / 16), (unsigned)g.nf, (unsigned)sides), 256, 0, st>>>(
                           d_fr, d_wk + (size_t)g.f0 * sides, k, K0, de, sw, h.d_err, h.d_front_bad);
                else {
                    // 64 rows a CTA share the load of s_j; with few CTAs 16, for the shorter chain
                    const int nr = (rows + 63) / 64 * g.nf * sides > h.num_sms ? 64 : 16, na = (rows + nr - 1) / nr;
                    k_split_a<<<dim3((unsigned)(na + NB / nr), (unsigned)g.nf, (unsigned)sides), 256, 0, st>>>(
                        d_fr, d_wk + (size_t)g.f0 * sides, k, K0, na, nr, de, sw, h.d_err, h.d_front_bad);
                }
                count_launch();
                prof_end(h, pi, 0.0, bytes, st);
                RSD_CUDA_TRY(cudaGetLastError());
                return RSD_OK;
            };
            RSD_TRY(split(false));
            RSD_TRY(run());
            RSD_TRY(split(true));
            if (k + NB >= std::min(K0 + WP, g.max_s)) RSD_TRY(run());
        }
    }
    return RSD_OK;
}

}  // namespace rsd
