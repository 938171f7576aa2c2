// FP64 diagonal blocks.  Partial Cholesky (step (b) of factor.cu): L_kk L_kk^T =
// P[k:k+w, k:k+w] (w <= NB) written back, L_kk^-1 to Dinv.
//
// The FP64 pipe bounds it: an SM retires 1.65 FP64 FMAs per clock and a warp's FMA takes
// 65 clocks, so the block's 0.7M FMAs are over 200 us on one SM whatever the schedule, and
// a level near the root has few fronts.  A cluster of CL (up to 16) CTAs therefore takes one front:
//   - the 32 x 32 diagonal sub-block is factored and inverted by every CTA (redundantly:
//     cheaper than handing it on), one column per step, lane = row, the columns spread
//     over the eight warps;
//   - CTA q owns the block's rows congruent to q mod CL: their part of the panel
//     L_IJ = A_IJ X_JJ^T, stored into every CTA's copy of L through distributed shared
//     memory, and of the trailing update; the rows of the next diagonal sub-block go to
//     every CTA the same way;
//   - the inverse is spread by columns (four adjacent ones to a CTA), which needs no
//     exchange: X_JK = -X_JJ sum_M L_JM X_MK.
// Measured: one 128-block per launch 0.57 ms at first (one CTA, the block in registers, two
// barriers and a reciprocal square root per column for the factor and again for the
// inverse), 0.16 on 8 CTAs scaling column by column, 0.13 on 16 with the unscaled chain of
// chol_inv32 (four times 22 us of it in the 32 x 32 blocks); 64 fronts on 2 CTAs each 0.25 ms.
// L fills the lower triangle of a 128 x 129 array, X (transposed, one column further
// right) its upper triangle.
#include <algorithm>
#include <atomic>

#include "cluster.cuh"
#include "rsd_internal.cuh"

namespace rsd {
namespace {

constexpr int DT = 256, DW = DT / 32;    // threads, warps
constexpr int SBK = 32;                  // sub-block
constexpr int LD = NB + 1;               // row stride of L / X (odd: lanes over rows hit distinct banks)
constexpr int SLD = SBK + 1;
constexpr size_t DIAG_SMEM = sizeof(double) * ((size_t)NB * LD + 2 * SBK * SLD + 5 * SBK);

__device__ __forceinline__ void cl_st_f64(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// 1 / sqrt(d) for d > 0: an FP32 estimate y of the reduced argument (2^-21) and one
// third-order Householder step, y + y e (1/2 + 3/8 e) with e = 1 - d y^2 (1.5 roundings).
__device__ __forceinline__ double rsqrt_chain(double d) {
    const long long b = __double_as_longlong(d);
    const int ex = (int)(b >> 52) - 1023;
    if (ex < -1000 || ex > 1000) return 1.0 / sqrt(d);
    const int q = ex >> 1;                                         // d = f 4^q, f in [1, 4)
    const float f = __int_as_float(((ex - 2 * q + 127) << 23) | (int)((b >> 29) & 0x7fffff));
    const int yb = __float_as_int(rsqrtf(f));
    const double y = __longlong_as_double(((long long)((yb >> 23) - 127 + 1023 - q) << 52) | ((long long)(yb & 0x7fffff) << 29));
    const double e = fma(-(d * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// 1 / d for finite d != 0: an FP32 estimate y (2^-22) and the third-order hyperpower step
// (Altman, "An optimum cubically convergent iterative method of inverting a linear bounded
// operator", 1960) y + y (e + e^2), e = 1 - d y: three FMAs deep on the chain from pivot to pivot
// (about 260 clocks; 1.0 / d takes 360).  One rounding of 1 / d.
__device__ __forceinline__ double rcp_chain(double d) {
    const long long b = __double_as_longlong(d);
    const int ex = (int)((b >> 52) & 0x7ff) - 1023;
    if (ex < -1000 || ex > 1000) return 1.0 / d;
    const float f = __int_as_float((127 << 23) | (int)((b >> 29) & 0x7fffff));      // |d| = f 2^ex, f in [1, 2)
    float yf;
    asm("rcp.approx.f32 %0, %1;" : "=f"(yf) : "f"(f));
    const int yb = __float_as_int(yf);
    const double y = __longlong_as_double((b & 0x8000000000000000ll) | ((long long)((yb >> 23) - 127 + 1023 - ex) << 52) |
                                          ((long long)(yb & 0x7fffff) << 29));
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// Cholesky of the 32 x 32 block in D (lower part) and its inverse, all eight warps: thread
// (lane, warp) holds row `lane` of columns warp + 8 q of both.  On return D holds L and Y
// the inverse (both with zeros above the diagonal).  Returns 1 on a pivot that is not
// positive or not finite (replaced by 1; 1 / inf would hide an infinite pivot behind zeros).
// The columns are eliminated unscaled, D = L' diag(d) L'^T with L' unit lower: the chain
// from pivot to pivot is one FMA, a reciprocal and a product, every other entry takes one FMA a
// step (of D right of the pivot, of L'^-1 left of it), and the square roots come at the end, all 32
// at once.  The warp that owns column j + 1 updates it first and publishes it while the
// others are still at step j: 22 us a block where scaling by 1 / sqrt(d) step by step took 27
// (its own FMAs wait for those of the other warp of its scheduler).
__device__ int chol_inv32(double* __restrict__ D, double* __restrict__ Y, double* __restrict__ buf, double* __restrict__ piv,
                          int lane, int warp) {
    double a[4], y[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int c = warp + DW * q;
        a[q] = c <= lane ? D[lane * SLD + c] : 0.0;
        y[q] = c == lane ? 1.0 : 0.0;
    }
    int bad = 0;
    // column j (updated by all before it): pivot, then the column and L'_j to buffer j & 1
    auto publish = [&](double& aj, int j) {
        double d = __shfl_sync(0xffffffffu, aj, j);
        if (!(d > 0.0 && d <= 1.7976931348623157e308)) { bad = 1; d = 1.0; }
        double* b = buf + (j & 1) * 2 * SBK;
        b[lane] = aj;
        b[SBK + lane] = lane > j ? aj * rcp_chain(d) : 0.0;
        if (lane == j) { aj = d; piv[j] = d; }
    };
    if (warp == 0) publish(a[0], 0);
#pragma unroll
    for (int jb = 0; jb < 4; ++jb) {
#pragma unroll 1
        for (int jj = 0; jj < DW; ++jj) {
            const int j = DW * jb + jj;
            __syncthreads();
            const double* cj = buf + (j & 1) * 2 * SBK;
            const double li = cj[SBK + lane];
            // the next pivot's column first
            const bool wrap = jj == DW - 1;
            if (!wrap && warp == jj + 1) {
                a[jb] -= li * cj[j + 1];
                publish(a[jb], j + 1);
            }
            if (jb < 3 && wrap && warp == 0) {
                a[jb < 3 ? jb + 1 : 3] -= li * cj[j + 1];
                publish(a[jb < 3 ? jb + 1 : 3], j + 1);
            }
#pragma unroll
            for (int q = jb; q < 4; ++q)
                if (warp + DW * q > j + 1) a[q] -= li * cj[warp + DW * q];
#pragma unroll
            for (int q = 0; q <= jb; ++q) {
                if (warp + DW * q > j) continue;
                y[q] -= li * __shfl_sync(0xffffffffu, y[q], j);          // (li = 0 on rows <= j)
            }
        }
    }
    __syncthreads();
    const double inv = rsqrt_chain(piv[lane]);
    if (warp == 0) buf[lane] = inv;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int c = warp + DW * q;
        D[lane * SLD + c] = c <= lane ? a[q] * buf[c] : 0.0;
        Y[lane * SLD + c] = c <= lane ? y[q] * inv : 0.0;
    }
    __syncthreads();
    return bad;
}

template <int CL>
__device__ __forceinline__ void cluster_or_cta_sync() {
    if constexpr (CL > 1) cl_sync(); else __syncthreads();
}

template <int CL>
__global__ void __launch_bounds__(DT, 1) k_chol_diag_f64(const FrontDesc* __restrict__ fronts, int k, int* __restrict__ err,
                                                       int* __restrict__ bad_front) {
    extern __shared__ __align__(16) unsigned char diag_smem[];
    double* Lf = (double*)diag_smem;             // NB x LD
    double* D = Lf + NB * LD;                    // 32 x SLD: the diagonal sub-block
    double* Y = D + SBK * SLD;                   // 32 x SLD: its inverse
    double* buf = Y + SBK * SLD;                 // two columns, raw and scaled
    double* piv = buf + 4 * SBK;
    const FrontDesc f = fronts[blockIdx.x / CL];
    if (f.s <= k) return;                        // the whole cluster
    const int w = min(NB, f.s - k), nJ = (w + SBK - 1) / SBK;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = CL > 1 ? (int)cl_rank() : 0;
    double* P = (double*)f.P + (int64_t)k * f.ldp + k;
    double* Dg = (double*)f.Dinv + (int64_t)(k / NB) * NB * NB;
    // this CTA's rows, and the first diagonal sub-block (every CTA); identity past the front
    for (int r = rank + CL * warp; r < nJ * SBK; r += CL * DW)
        for (int c = lane; c <= r; c += 32) Lf[r * LD + c] = r < w ? P[(int64_t)r * f.ldp + c] : (r == c ? 1.0 : 0.0);
    for (int e = tid; e < SBK * SBK; e += DT) {
        const int r = e / SBK, c = e % SBK;
        D[r * SLD + c] = c <= r ? (r < w ? P[(int64_t)r * f.ldp + c] : (r == c ? 1.0 : 0.0)) : 0.0;
    }
    cluster_or_cta_sync<CL>();                   // every CTA has read the block before one writes L over it
    int bad = 0;
    for (int J = 0; J < nJ; ++J) {
        const int o = SBK * J, below = SBK * (J + 1), rows = nJ * SBK;
        if (J > 0) cluster_or_cta_sync<CL>();          // the sub-block's rows are in D
        bad |= chol_inv32(D, Y, buf, piv, lane, warp);
        // L_JJ out (one CTA), X_JJ into the columns this CTA owns
        if (rank == J % CL)
            for (int e = tid; e < SBK * SBK; e += DT) {
                const int r = e / SBK, c = e % SBK;
                if (c <= r && o + r < w) P[(int64_t)(o + r) * f.ldp + o + c] = D[r * SLD + c];
            }
        for (int e = tid; e < SBK * SBK; e += DT) {
            const int c = e / SBK, r = e % SBK;
            if (r >= c && ((o + c) >> 2) % CL == rank) Lf[(o + c) * LD + o + r + 1] = Y[r * SLD + c];
        }
        // panel: this CTA's rows below, L_rc = sum_m A_rm Y_cm
        constexpr int UP = (96 / CL + DW - 1) / DW;
        const int r_first = below + ((rank - below) % CL + CL) % CL;      // first own row >= below
        double pv[UP];
#pragma unroll
        for (int u = 0; u < UP; ++u) {
            const int r = r_first + CL * (warp + DW * u);
            double s = 0.0;
            if (r < rows)
#pragma unroll 8
                for (int m = 0; m < SBK; ++m) s += Lf[r * LD + o + m] * Y[lane * SLD + m];
            pv[u] = s;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < UP; ++u) {
            const int r = r_first + CL * (warp + DW * u);
            if (r >= rows) continue;
            double* dst = Lf + r * LD + o + lane;
            *dst = pv[u];
            if constexpr (CL > 1)
                for (int q = 1; q < CL; ++q) cl_st_f64(cl_map(dst, (uint32_t)((rank + q) % CL)), pv[u]);
            if (r < w) P[(int64_t)r * f.ldp + o + lane] = pv[u];
        }
        if (J + 1 < nJ) {
            cluster_or_cta_sync<CL>();                 // the panel is complete in every CTA
            // trailing update of this CTA's rows; a warp takes a row and 32 of its columns, the
            // next diagonal sub-block (first column block of rows below .. below + 31) first,
            // whose results go to every CTA
            int it = 0;
            for (int r = r_first; r < rows; r += CL) {
                const int rb = r / SBK;
                for (int cb = J + 1; cb <= rb; ++cb, ++it) {
                    if (it % DW != warp) continue;
                    const int c = cb * SBK + lane;
                    double s = 0.0;
#pragma unroll 8
                    for (int m = 0; m < SBK; ++m) s += Lf[r * LD + o + m] * Lf[c * LD + o + m];
                    if (c > r) continue;
                    const double v = Lf[r * LD + c] - s;
                    Lf[r * LD + c] = v;
                    if (rb == J + 1) {
                        double* dst = D + (r - below) * SLD + lane;
                        *dst = v;
                        if constexpr (CL > 1)
                            for (int q = 1; q < CL; ++q) cl_st_f64(cl_map(dst, (uint32_t)((rank + q) % CL)), v);
                    }
                }
            }
        } else {
            __syncthreads();
        }
        // block row J of the inverse, this CTA's columns: a warp takes a column c, lane = row;
        // T = sum over blocks M of L_JM X_M,c, then X_J,c = -X_JJ T
        int ic = 0;
        for (int c0 = 4 * rank; c0 < o; c0 += 4 * CL)
            for (int cc = 0; cc < 4; ++cc, ++ic) {
                if (ic % DW != warp) continue;
                const int c = c0 + cc, m0 = c & ~(SBK - 1);
                const double* Lr = Lf + (o + lane) * LD;
                const double* Xc = Lf + c * LD + 1;     // Xc[m] = X[m][c], m >= c
                double t0 = 0.0, t1 = 0.0;
#pragma unroll 4
                for (int m = m0; m < o; m += 2) {
                    t0 += Lr[m] * (m >= c ? Xc[m] : 0.0);
                    t1 += Lr[m + 1] * (m + 1 >= c ? Xc[m + 1] : 0.0);
                }
                const double t = t0 + t1;
                double x = 0.0;
#pragma unroll 8
                for (int m = 0; m < SBK; ++m) x -= Y[lane * SLD + m] * __shfl_sync(0xffffffffu, t, m);
                Lf[c * LD + 1 + o + lane] = x;
            }
    }
    __syncthreads();
    // the inverse's columns of this CTA (zero above the diagonal and past the front)
    for (int e = tid; e < NB * (NB / CL); e += DT) {
        const int r = e / (NB / CL), q = e % (NB / CL);
        const int c = (q >> 2) * 4 * CL + 4 * rank + (q & 3);
        Dg[r * NB + c] = (r >= c && r < w) ? Lf[c * LD + 1 + r] : 0.0;
    }
    if (bad && rank == 0 && lane == 0) {
        atomicExch(&err[ERR_NOT_SPD], 1);
        atomicMin(&err[ERR_NOT_SPD_NODE], f.node);
        bad_front[f.node] = 1;
    }
}

// ---- nonsymmetric fronts ---------------------------------------------------------------
// LU without pivoting of the block (lower part from P, upper part from PU transposed), the
// same division of work: L (unit) to P, U^T to PU, L^-1 to Dinv, (U^T)^-1 to DinvU.  A row of
// the next diagonal sub-block goes to every CTA with all its columns, the block row of U
// is formed by columns (CTA q those congruent to q mod CL).  The two inverses double the
// FP64 work; they live in Dinv and DinvU themselves (each CTA reads back only the columns it
// wrote).  Measured on a 37^3 convection-diffusion system: 0.80 ms a launch before (one CTA,
// three barriers a column, one thread a column of the inverses), 0.24 ms.

// LU and the inverses of L and U^T of the 32 x 32 block at A (row stride LD), all eight warps,
// thread (lane, warp) holding row `lane` of columns warp + 8 q; A keeps L and U, YL = L^-1, YW =
// (U^T)^-1 (lower, zeros above).  Returns 1 on a pivot that is zero or not finite (replaced by 1).
// As in chol_inv32 the next pivot's column goes ahead, and (U^T)^-1 is formed unscaled
// (with U'_ji = u_ji / u_jj) and its rows divided by the pivots at the end.
__device__ int lu_inv32(double* __restrict__ A, double* __restrict__ YL, double* __restrict__ YW, double* __restrict__ buf,
                        double* __restrict__ rcp, int lane, int warp) {
    double a[4], yl[4], yw[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int c = warp + DW * q;
        a[q] = A[lane * LD + c];
        yl[q] = yw[q] = c == lane ? 1.0 : 0.0;
    }
    int bad = 0;
    // column j (updated by all before it): pivot, then L_j to buffer j & 1
    auto publish = [&](double& aj, int j) {
        double d = __shfl_sync(0xffffffffu, aj, j);
        if (!(d != 0.0) || !(fabs(d) <= 1.7976931348623157e308)) {
            bad = 1;
            d = 1.0;
            if (lane == j) aj = 1.0;
        }
        const double r = rcp_chain(d);
        if (lane > j) aj *= r;
        buf[(j & 1) * 2 * SBK + lane] = lane > j ? aj : 0.0;
        if (lane == j) rcp[j] = r;
    };
    if (warp == 0) publish(a[0], 0);
    if (lane == 0) {                                  // row 0 of U
#pragma unroll
        for (int q = 0; q < 4; ++q) buf[SBK + warp + DW * q] = a[q];
    }
#pragma unroll
    for (int jb = 0; jb < 4; ++jb) {
#pragma unroll 1
        for (int jj = 0; jj < DW; ++jj) {
            const int j = DW * jb + jj;
            __syncthreads();
            const double* cj = buf + (j & 1) * 2 * SBK;      // L_j, row j of U
            const double* rj = cj + SBK;
            const double li = cj[lane];
            const bool wrap = jj == DW - 1;
            if (!wrap && warp == jj + 1) {
                a[jb] -= li * rj[j + 1];
                publish(a[jb], j + 1);
            }
            if (jb < 3 && wrap && warp == 0) {
                a[jb < 3 ? jb + 1 : 3] -= li * rj[j + 1];
                publish(a[jb < 3 ? jb + 1 : 3], j + 1);
            }
#pragma unroll
            for (int q = jb; q < 4; ++q)
                if (warp + DW * q > j + 1) a[q] -= li * rj[warp + DW * q];
            if (lane == j + 1) {                             // row j + 1 of U is final
                double* rn = buf + ((j + 1) & 1) * 2 * SBK + SBK;
#pragma unroll
                for (int q = jb; q < 4; ++q) rn[warp + DW * q] = a[q];
            }
            const double ui = lane > j ? rj[lane] * rcp[j] : 0.0;
#pragma unroll
            for (int q = 0; q <= jb; ++q) {
                if (warp + DW * q > j) continue;
                const double xl = __shfl_sync(0xffffffffu, yl[q], j), xw = __shfl_sync(0xffffffffu, yw[q], j);
                yl[q] -= li * xl;
                yw[q] -= ui * xw;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int c = warp + DW * q;
        A[lane * LD + c] = a[q];
        YL[lane * SLD + c] = c <= lane ? yl[q] : 0.0;
        YW[lane * SLD + c] = c <= lane ? yw[q] * rcp[lane] : 0.0;
    }
    __syncthreads();
    return bad;
}

constexpr size_t LU_SMEM = sizeof(double) * ((size_t)NB * LD + 2 * SBK * SLD + 5 * SBK);

template <int CL>
__global__ void __launch_bounds__(DT, 1) k_lu_diag_f64(const FrontDesc* __restrict__ fronts, int k, int* __restrict__ err,
                                                     int* __restrict__ bad_front) {
    extern __shared__ __align__(16) unsigned char diag_smem[];
    double* A = (double*)diag_smem;              // NB x LD: L below the diagonal, U on and above it
    double* YL = A + NB * LD;                    // 32 x SLD: L_JJ^-1
    double* YW = YL + SBK * SLD;                 // 32 x SLD: (U_JJ^T)^-1
    double* buf = YW + SBK * SLD;                // two columns of L and rows of U
    double* rcp = buf + 4 * SBK;                 // reciprocal pivots
    const FrontDesc f = fronts[blockIdx.x / CL];
    if (f.s <= k) return;                        // the whole cluster
    const int w = min(NB, f.s - k), nJ = (w + SBK - 1) / SBK, rows = nJ * SBK;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = CL > 1 ? (int)cl_rank() : 0;
    double* P = (double*)f.P + (int64_t)k * f.ldp + k;
    double* PU = (double*)f.PU + (int64_t)k * f.ldp + k;
    double* Dg = (double*)f.Dinv + (int64_t)(k / NB) * NB * NB;
    double* DUg = (double*)f.DinvU + (int64_t)(k / NB) * NB * NB;
    // this CTA's rows and the first block row; identity past the front
    for (int r = warp; r < rows; r += DW) {
        if (r >= SBK && r % CL != rank) continue;
        for (int c = lane; c < rows; c += 32)
            A[r * LD + c] = (r < w && c < w) ? (c <= r ? P[(int64_t)r * f.ldp + c] : PU[(int64_t)c * f.ldp + r]) : (r == c ? 1.0 : 0.0);
    }
    cluster_or_cta_sync<CL>();                   // read everywhere before L and U are written over it
    int bad = 0;
    for (int J = 0; J < nJ; ++J) {
        const int o = SBK * J, below = SBK * (J + 1);
        if (J > 0) cluster_or_cta_sync<CL>();          // the block row is here
        bad |= lu_inv32(A + o * LD + o, YL, YW, buf, rcp, lane, warp);
        for (int e = tid; e < SBK * SBK; e += DT) {
            const int c = e % SBK, r = e / SBK;
            if (((o + c) >> 2) % CL == rank) {
                Dg[(o + r) * NB + o + c] = YL[r * SLD + c];
                DUg[(o + r) * NB + o + c] = YW[r * SLD + c];
            }
        }
        // own rows below: L_rc = sum_m A_rm W_cm; own columns to the right: U_ic = sum_m X_im A_mc
        constexpr int UP = (96 / CL + DW - 1) / DW;
        const int first = below + ((rank - below) % CL + CL) % CL;        // first own row or column >= below
        double pl[UP], pu[UP];
#pragma unroll
        for (int u = 0; u < UP; ++u) {
            const int r = first + CL * (warp + DW * u);
            double s = 0.0, t = 0.0;
            if (r < rows)
#pragma unroll 8
                for (int m = 0; m < SBK; ++m) {
                    s += A[r * LD + o + m] * YW[lane * SLD + m];
                    t += A[(o + m) * LD + r] * YL[lane * SLD + m];
                }
            pl[u] = s;
            pu[u] = t;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < UP; ++u) {
            const int r = first + CL * (warp + DW * u);
            if (r >= rows) continue;
            double* dl = A + r * LD + o + lane;
            double* du = A + (o + lane) * LD + r;
            *dl = pl[u];
            *du = pu[u];
            if constexpr (CL > 1)
                for (int q = 1; q < CL; ++q) {
                    cl_st_f64(cl_map(dl, (uint32_t)((rank + q) % CL)), pl[u]);
                    cl_st_f64(cl_map(du, (uint32_t)((rank + q) % CL)), pu[u]);
                }
        }
        if (J + 1 < nJ) {
            cluster_or_cta_sync<CL>();                 // panel and block row are complete in every CTA
            int it = 0;
            for (int r = first; r < rows; r += CL)
                for (int cb = J + 1; cb < nJ; ++cb, ++it) {
                    if (it % DW != warp) continue;
                    const int c = cb * SBK + lane;
                    double s = 0.0;
#pragma unroll 8
                    for (int m = 0; m < SBK; ++m) s += A[r * LD + o + m] * A[(o + m) * LD + c];
                    double* dst = A + r * LD + c;
                    const double v = *dst - s;
                    *dst = v;
                    if constexpr (CL > 1)
                        if (r < below + SBK)
                            for (int q = 1; q < CL; ++q) cl_st_f64(cl_map(dst, (uint32_t)((rank + q) % CL)), v);
                }
        } else {
            __syncthreads();
        }
        // block row J of both inverses, this CTA's columns: a warp takes a column, lane = row
        int ic = 0;
        for (int c0 = 4 * rank; c0 < o; c0 += 4 * CL)
            for (int cc = 0; cc < 4; ++cc, ++ic) {
                if (ic % DW != warp) continue;
                const int c = c0 + cc, m0 = c & ~(SBK - 1);
                double tl = 0.0, tw = 0.0;
#pragma unroll 4
                for (int m = m0; m < o; ++m) {
                    tl += A[(o + lane) * LD + m] * Dg[m * NB + c];
                    tw += A[m * LD + o + lane] * DUg[m * NB + c];
                }
                double xl = 0.0, xw = 0.0;
#pragma unroll 8
                for (int m = 0; m < SBK; ++m) {
                    xl -= YL[lane * SLD + m] * __shfl_sync(0xffffffffu, tl, m);
                    xw -= YW[lane * SLD + m] * __shfl_sync(0xffffffffu, tw, m);
                }
                Dg[(o + lane) * NB + c] = xl;
                DUg[(o + lane) * NB + c] = xw;
            }
    }
    __syncthreads();
    // L (unit) and U^T, this CTA's rows; the inverses' zeros above the diagonal and past the front
    for (int r = rank + CL * warp; r < w; r += CL * DW)
        for (int c = lane; c <= r; c += 32) {
            P[(int64_t)r * f.ldp + c] = c < r ? A[r * LD + c] : 1.0;
            PU[(int64_t)r * f.ldp + c] = A[c * LD + r];
        }
    for (int e = tid; e < NB * (NB / CL); e += DT) {
        const int r = e / (NB / CL), q = e % (NB / CL);
        const int c = (q >> 2) * 4 * CL + 4 * rank + (q & 3);
        if (r < c || r >= w || c >= w) Dg[r * NB + c] = DUg[r * NB + c] = 0.0;
    }
    if (bad && rank == 0 && lane == 0) {
        atomicExch(&err[ERR_NOT_SPD], 1);
        atomicMin(&err[ERR_NOT_SPD_NODE], f.node);
        bad_front[f.node] = 1;
    }
}

using DiagKernel = void (*)(const FrontDesc*, int, int*, int*);

int launch_cl(DiagKernel kern, int CL, size_t smem, const FrontDesc* d_fronts, int nf, int k, int* err, int* bad_front, cudaStream_t st) {
    RSD_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (CL > 8) RSD_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nf * CL));
    cfg.blockDim = dim3(DT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    RSD_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, d_fronts, k, err, bad_front));
    count_launch();
    return RSD_OK;
}

}  // namespace

// How many clusters of 16 (more than the portable 8) of the Cholesky or the LU kernel the
// current device holds at once; 0 where it takes none.  (Threads that ask at once store the
// same count.)
static int wide_clusters(DiagKernel kern, size_t smem, bool lu) {
    static std::atomic<int> known[64][2];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 0; }
    int n = known[dev][lu].load(std::memory_order_relaxed);
    if (!n) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16 * 16);
        cfg.blockDim = dim3(DT);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int m = 0;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&m, (void*)kern, &cfg) != cudaSuccess) {
            cudaGetLastError();
            m = 0;
        }
        n = m + 1;
        known[dev][lu].store(n, std::memory_order_relaxed);
    }
    return n - 1;
}

// The largest cluster that still gives every front with rows past k SMs of its own: the
// FP64 pipes it adds are worth more than anything else to a lone block (see above), and
// past one wave a larger cluster only queues.
int launch_diag_f64(Handle& h, int li, int f0, int nf, int k, cudaStream_t st) {
    Level& L = h.levels[li];
    int alive = 0;
    double flops = 0, bytes = 0;
    for (int q = f0; q < f0 + nf; ++q) {
        if (L.fronts[q].s <= k) continue;
        const double w = std::min(NB, L.fronts[q].s - k);
        ++alive;
        flops += (h.lu ? 4.0 : 2.0) * w * w * w / 3.0;
        bytes += (2.0 * w * w + NB * NB) * (h.lu ? 16 : 8);
    }
    if (!alive) return RSD_OK;
    const FrontDesc* fr = L.d_fronts + f0;
    const int pi = prof_begin(h, K_POTRF, st);
    static constexpr DiagKernel kern[2][5] = {
        {k_chol_diag_f64<1>, k_chol_diag_f64<2>, k_chol_diag_f64<4>, k_chol_diag_f64<8>, k_chol_diag_f64<16>},
        {k_lu_diag_f64<1>, k_lu_diag_f64<2>, k_lu_diag_f64<4>, k_lu_diag_f64<8>, k_lu_diag_f64<16>}};
    const size_t smem = h.lu ? LU_SMEM : DIAG_SMEM;
    int lg = alive * 8 <= h.num_sms ? 3 : alive * 4 <= h.num_sms ? 2 : alive * 2 <= h.num_sms ? 1 : 0;
    if (lg == 3 && alive <= wide_clusters(kern[h.lu][4], smem, h.lu)) lg = 4;
    const int rc = launch_cl(kern[h.lu][lg], 1 << lg, smem, fr, nf, k, h.d_err, h.d_front_bad, st);
    prof_end(h, pi, flops, bytes, st);
    return rc;
}

}  // namespace rsd
