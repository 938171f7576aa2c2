// Paper mode with gamma inner GMRES iterations (Sec. 3.2, Algorithms 1 and 2): every
// interface system S~_t u_t = g_t of a tree level is solved approximately by gamma
// GMRES iterations from u = 0 (no restart, modified Gram-Schmidt, no preconditioner),
// all interfaces of the level at once; S~ is never formed.
//
// S-MatVec (Algorithm 1) for interface t:
//     y = K_{I_t I_t} x - sum_{l in V-hat_t} K_{I_t l} K_ll^-1 K_{l I_t} x.
// Setup factors every leaf front [K_ll K_lB; K_Bl .] into L_l and X_l = K_{B_l l} L_l^-T
// (rows: the ancestor DOFs B_l coupled to l), so with R = the rows of X_l that lie in I_t,
//     K_{I_t l} K_ll^-1 K_{l I_t} = (K_{I_t l} L_l^-T)(L_l^-1 K_{l I_t}) = X_l[R] X_l[R]^T:
// the two leaf solves of Algorithm 1 become two streaming products with X_l[R]: t_l =
// X_l[R]^T x (column-parallel), then one row product X_l[row] . t_l per coupling, summed
// per interface DOF over the leaves that touch it in a fixed order.
// V-hat_t is exactly the set of leaves with a nonempty R for t (a leaf couples to its
// ancestors' DOFs only, Eq. 3.1).
//
// Vectors of a level are packed: interface slot i of the level owns positions
// [if_off[i], if_off[i+1]) in I_t order (pk_pos maps a global DOF to its position).
// Every reduction has a fixed order, so results are bitwise reproducible.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "cluster.cuh"
#include "rsd_internal.cuh"

namespace rsd {
namespace {

constexpr int GT = 512;           // threads of the per-interface GMRES kernels
constexpr int GAMMA_MAX = 32;     // largest gamma (inner iterations) the kernels hold

// Block-wide sum in a fixed order; every thread receives the result.
__device__ double block_sum_all(double v, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        double t = lane < nw ? red[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) red[32] = t;
    }
    __syncthreads();
    return red[32];
}

// Products with a leaf's X block accumulate in the block's own precision (A = T): FP32
// blocks of the mixed form in FP32, as the substitution sweeps do, FP64 blocks in FP64.
// With H16 (T = float) they read the leaf's FP16 copy instead: row i of P scaled by the
// power of two rs_i, so exactly the factor's TF32 values down to 2^-27 sqrt(K_ii); x enters
// scaled by ri of its row and a row product is scaled by ri once, at half the bytes.
template <typename T> struct VecOf;
template <> struct VecOf<float> { using V = float4; };
template <> struct VecOf<double> { using V = double2; };

template <typename T, bool H16> struct SmvElems { static constexpr int W = 16 / (int)sizeof(T); };
template <> struct SmvElems<float, true> { static constexpr int W = 8; };

// The W elements of one 16-byte load at p (a row of X, element offset c).
template <typename T, bool H16>
__device__ __forceinline__ void smv_load(const void* p, int64_t off, T (&o)[SmvElems<T, H16>::W]) {
    if constexpr (H16) {
        const uint4 u = __ldg((const uint4*)((const __half*)p + off));
        const __half2* h = reinterpret_cast<const __half2*>(&u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 f = __half22float2(h[k]);
            o[2 * k] = f.x;
            o[2 * k + 1] = f.y;
        }
    } else {
        using V = typename VecOf<T>::V;
        const V v = __ldg((const V*)((const T*)p + off));
        const T* e = (const T*)&v;
#pragma unroll
        for (int k = 0; k < SmvElems<T, H16>::W; ++k) o[k] = e[k];
    }
}

// the same from a 16-byte load already made
template <typename T, bool H16>
__device__ __forceinline__ void smv_unpack(const uint4& u, T (&o)[SmvElems<T, H16>::W]) {
    if constexpr (H16) {
        const __half2* h = reinterpret_cast<const __half2*>(&u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 f = __half22float2(h[k]);
            o[2 * k] = f.x;
            o[2 * k + 1] = f.y;
        }
    } else {
        const T* e = reinterpret_cast<const T*>(&u);
#pragma unroll
        for (int k = 0; k < SmvElems<T, H16>::W; ++k) o[k] = e[k];
    }
}

// t_l = X_l[R_l]^T x for every leaf with rows coupled to the level; one CTA per (leaf, 32 x W
// columns), W columns per lane read with one 16-byte load per row.  The rows' offsets and x
// values are staged in shared memory 256 at a time; the eight warps take every eighth row
// (many loads in flight per column tile instead of one serial walk over the leaf's rows)
// and their partial sums are added in warp order.
template <typename T, bool H16>
__global__ void __launch_bounds__(256) k_smv_leaf(const FrontDesc* __restrict__ leaves, const int* __restrict__ cl_ptr,
                                                  const int* __restrict__ cl_row, const int* __restrict__ cl_pos,
                                                  const int* __restrict__ tl_off, const double* __restrict__ x,
                                                  T* __restrict__ tl) {
    constexpr int W = SmvElems<T, H16>::W, CT = 32 * W;
    __shared__ int s_row[256];
    __shared__ T s_x[256];
    __shared__ T s_red[8][CT];
    const int l = blockIdx.x;
    const int k0 = cl_ptr[l], k1 = cl_ptr[l + 1];
    const int s = leaves[l].s, ldp = leaves[l].ldp;
    const int c0 = blockIdx.y * CT;
    if (k0 == k1 || c0 >= s) return;
    const void* X = H16 ? (const void*)((const __half*)leaves[l].P16 + (int64_t)s * ldp)
                        : (const void*)((const T*)leaves[l].P + (int64_t)s * ldp);
    const float* ri = H16 ? leaves[l].ri + s : nullptr;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = c0 + lane * W;
    T acc[W];
#pragma unroll
    for (int e = 0; e < W; ++e) acc[e] = 0;
    for (int kb = k0; kb < k1; kb += 256) {
        const int nb = min(256, k1 - kb);
        __syncthreads();
        if ((int)threadIdx.x < nb) {
            const int row = cl_row[kb + threadIdx.x];
            s_row[threadIdx.x] = row;
            const T xv = (T)x[cl_pos[kb + threadIdx.x]];
            s_x[threadIdx.x] = H16 ? xv * (T)ri[row] : xv;
        }
        __syncthreads();
        if (c < s) {
#pragma unroll 4
            for (int q = warp; q < nb; q += 8) {
                T e[W];
                smv_load<T, H16>(X, (int64_t)s_row[q] * ldp + c, e);
                const T xv = s_x[q];
#pragma unroll
                for (int u = 0; u < W; ++u) acc[u] += e[u] * xv;
            }
        }
    }
#pragma unroll
    for (int e = 0; e < W; ++e) s_red[warp][lane * W + e] = acc[e];
    __syncthreads();
    T* out = tl + tl_off[l];
    for (int e = threadIdx.x; e < CT; e += blockDim.x) {
        if (c0 + e >= s) break;
        T v = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += s_red[w][e];
        out[c0 + e] = v;
    }
}

// The W entries of t at c (16- or 32-byte aligned: t_l slots start at multiples of 8
// elements and c is a multiple of W).
template <typename T, int W>
__device__ __forceinline__ void smv_tload(const T* t, T (&o)[W]) {
    if constexpr (sizeof(T) * W == 32) {
        const float4 a = __ldg((const float4*)t), b = __ldg((const float4*)t + 1);
        const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int q = 0; q < W; ++q) o[q] = v[q];
    } else {
        using V = typename VecOf<T>::V;
        const V v = __ldg((const V*)t);
        const T* e = (const T*)&v;
#pragma unroll
        for (int q = 0; q < W; ++q) o[q] = e[q];
    }
}

// yl_k = X_l[row_k] . t_l for every coupling k (a row of a leaf's X block that lies in the
// level's interfaces).  One warp per group of R consecutive couplings: couplings are grouped
// by leaf, so a group of one leaf reads each chunk of t_l once for its R rows (16-byte loads
// along the rows); a group that straddles two leaves takes its rows one at a time.  Either
// way a row's sum runs in the same order (lane-strided chunks, the ragged tail, then the
// butterfly), so the result does not depend on the grouping.
template <typename T, bool H16>
__global__ void __launch_bounds__(256) k_smv_rows(int nk, const int* __restrict__ cl_leaf, const int* __restrict__ cl_row,
                                                  const FrontDesc* __restrict__ leaves, const int* __restrict__ tl_off,
                                                  const T* __restrict__ tl, double* __restrict__ yl) {
    constexpr int W = SmvElems<T, H16>::W, R = 4;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t ng = ((int64_t)nk + R - 1) / R;
    for (int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; g < ng; g += warps) {
        const int64_t k0 = g * R;
        const int nr = (int)(nk - k0 < R ? nk - k0 : R);
        const bool shared = nr == R && cl_leaf[k0] == cl_leaf[k0 + R - 1];
        for (int r0 = 0; r0 < nr; r0 += shared ? R : 1) {
            const int m = shared ? R : 1;            // rows summed together
            const int l = cl_leaf[k0 + r0];
            const int s = leaves[l].s, ldp = leaves[l].ldp;
            const void* base = H16 ? (const void*)leaves[l].P16 : (const void*)leaves[l].P;
            const T* t = tl + tl_off[l];
            int64_t roff[R];
            T d[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                roff[r] = r < m ? (int64_t)(s + cl_row[k0 + r0 + r]) * ldp : 0;
                d[r] = 0;
            }
            const int sv = s / W * W;
#pragma unroll 1
            for (int c = lane * W; c < sv; c += 32 * W) {
                T tv[W];
                smv_tload<T, W>(t + c, tv);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (r < m) {
                        T e[W];
                        smv_load<T, H16>(base, roff[r] + c, e);
#pragma unroll
                        for (int q = 0; q < W; ++q) d[r] += e[q] * tv[q];
                    }
                }
            }
            for (int c = sv + lane; c < s; c += 32) {
                const T tv = t[c];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (r < m) {
                        const T v = H16 ? (T)__half2float(((const __half*)base)[roff[r] + c]) : ((const T*)base)[roff[r] + c];
                        d[r] += v * tv;
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) d[r] += __shfl_xor_sync(0xffffffffu, d[r], o);
                if (lane == 0 && r < m) {
                    const int64_t k = k0 + r0 + r;
                    yl[k] = H16 ? (double)(d[r] * (T)leaves[l].ri[s + cl_row[k]]) : (double)d[r];
                }
            }
        }
    }
}

// y_p = (K_{I_t I_t} x)_p - sum of yl_k over the couplings k of position p.  Eight lanes
// per packed position (four positions per warp): the lanes take every eighth entry of the
// row and every eighth coupling, and their partial sums meet in a fixed butterfly, so the
// gathers of four rows are in flight at once.
__global__ void __launch_bounds__(256) k_smv_iface(int S, const int* __restrict__ if_dofs, const int64_t* __restrict__ rowptr,
                                                   const int* __restrict__ col, const double* __restrict__ val,
                                                   const int* __restrict__ owner, const int* __restrict__ pk_pos,
                                                   const int* __restrict__ ci_ptr, const int* __restrict__ ci_k,
                                                   const double* __restrict__ yl, const double* __restrict__ x,
                                                   double* __restrict__ y) {
    const int lane = threadIdx.x & 31, sub = lane & 7;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    // warp-uniform trip count: every lane reaches the shuffles
    for (int64_t pw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; pw * 4 < S; pw += warps) {
        const int64_t p = pw * 4 + (lane >> 3);
        double acc = 0;
        if (p < S) {
            const int dof = if_dofs[p];
            const int o = owner[dof];
            for (int64_t k = rowptr[dof] + sub; k < rowptr[dof + 1]; k += 8) {
                const int j = col[k];
                if (owner[j] == o) acc += val[k] * x[pk_pos[j]];
            }
            for (int q = ci_ptr[p] + sub; q < ci_ptr[p + 1]; q += 8) acc -= yl[ci_k[q]];
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 4);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        if (sub == 0 && p < S) y[p] = acc;
    }
}

// Both products of a leaf in one CTA (small leaves): t_l = X_l[R]^T x in shared memory, then
// yl_k = X_l[row_k] . t_l.  A thread takes one 16-byte chunk of columns and every
// `groups`-th row for t_l, the groups' partial sums being added in order; a warp takes four rows at a time
// for yl.  The leaf's rows come from L2 once and, mostly, from L1 the second time.
template <typename T, bool H16>
__global__ void __launch_bounds__(256) k_smv_both(const FrontDesc* __restrict__ ty, const FrontDesc* __restrict__ tx,
                                                  const int* __restrict__ cl_ptr, const int* __restrict__ cl_row,
                                                  const int* __restrict__ cl_pos, int max_s, const double* __restrict__ x,
                                                  double* __restrict__ yl) {
    constexpr int W = SmvElems<T, H16>::W, R = 4;
    __shared__ int s_row[256];
    __shared__ T s_x[256];
    extern __shared__ __align__(16) unsigned char smv_smem[];
    T* s_t = (T*)smv_smem;                             // max_s rounded up to W
    T* s_red = s_t + (max_s + W - 1) / W * W;          // groups x (nch W)
    const int l = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k0 = cl_ptr[l], k1 = cl_ptr[l + 1];
    if (k0 == k1) return;
    const int s = ty[l].s, ldp = ty[l].ldp;
    const void* Y = H16 ? (const void*)((const __half*)ty[l].P16 + (int64_t)s * ldp) : (const void*)((const T*)ty[l].P + (int64_t)s * ldp);
    const void* X = H16 ? (const void*)((const __half*)tx[l].P16 + (int64_t)s * ldp) : (const void*)((const T*)tx[l].P + (int64_t)s * ldp);
    const float* ri = H16 ? ty[l].ri + s : nullptr;
    const int nch = (s + W - 1) / W, groups = 256 / nch;          // (nch <= 256)
    const int ch = tid % nch, g = tid / nch;
    T acc[W];
#pragma unroll
    for (int e = 0; e < W; ++e) acc[e] = 0;
    for (int kb = k0; kb < k1; kb += 256) {
        const int nb = min(256, k1 - kb);
        __syncthreads();
        if (tid < nb) {
            const int row = cl_row[kb + tid];
            s_row[tid] = row;
            const T xv = (T)x[cl_pos[kb + tid]];
            s_x[tid] = H16 ? xv * (T)ri[row] : xv;
        }
        __syncthreads();
        if (g < groups) {
            constexpr int U = 8;                       // rows in flight per thread
            const char* Yc = (const char*)Y + (int64_t)ch * 16;
            for (int q = g; q < nb; q += U * groups) {
                uint4 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (q + u * groups < nb) v[u] = __ldg((const uint4*)(Yc + (int64_t)s_row[q + u * groups] * ldp * (16 / W)));
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (q + u * groups < nb) {
                        T e[W];
                        smv_unpack<T, H16>(v[u], e);
                        const T xv = s_x[q + u * groups];
#pragma unroll
                        for (int w = 0; w < W; ++w) acc[w] += e[w] * xv;
                    }
            }
        }
    }
    if (g < groups) {
#pragma unroll
        for (int e = 0; e < W; ++e) s_red[(g * nch + ch) * W + e] = acc[e];
    }
    __syncthreads();
    for (int e = tid; e < nch * W; e += 256) {
        T v = 0;
        for (int q = 0; q < groups; ++q) v += s_red[q * nch * W + e];
        s_t[e] = e < s ? v : (T)0;                     // (columns past s: the rows' padding is not read as data)
    }
    __syncthreads();
    for (int k = k0 + warp * R; k < k1; k += 8 * R) {
        const int nr = min(R, k1 - k);
        int64_t off[R];
        T d[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            off[r] = (int64_t)cl_row[k + min(r, nr - 1)] * ldp;
            d[r] = 0;
        }
        for (int c0 = lane; c0 < nch; c0 += 64) {      // two chunks of each row in flight
            uint4 v[2][R];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (c0 + 32 * h < nch) v[h][r] = __ldg((const uint4*)((const char*)X + (off[r] + (int64_t)(c0 + 32 * h) * W) * (16 / W)));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = c0 + 32 * h;
                if (c >= nch) break;
                T tv[W];
#pragma unroll
                for (int q = 0; q < W; ++q) tv[q] = s_t[c * W + q];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    T e[W];
                    smv_unpack<T, H16>(v[h][r], e);
#pragma unroll
                    for (int q = 0; q < W; ++q) d[r] += (c * W + q < s ? e[q] : (T)0) * tv[q];
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) d[r] += __shfl_xor_sync(0xffffffffu, d[r], o);
            if (lane == 0 && r < nr) yl[k + r] = H16 ? (double)(d[r] * (T)ri[cl_row[k + r]]) : (double)d[r];
        }
    }
}

// The GMRES vector kernels give each interface a cluster of GC CTAs, CTA r of the cluster
// holding the r-th contiguous chunk of the interface's entries, so a long interface (the
// root's) is spread over GC SMs instead of one; a level of many short ones takes smaller
// clusters, so that its CTAs still run at once (65^3, 64 interfaces of 631 entries: 37 us
// a step in clusters of 8, 22 in clusters of 4).
constexpr int GC_MAX = 8;
inline int gm_cluster(int n_if, int num_sms) {
    int gc = GC_MAX;
    while (gc > 1 && n_if * gc > 2 * num_sms) gc /= 2;
    return gc;
}

struct GmChunk {
    int i, o, s, lo, hi;        // interface, its offset and size; this CTA's entries [lo, hi)
};

template <int GC>
__device__ __forceinline__ GmChunk gm_chunk(const int* __restrict__ if_off, int i, int r) {
    GmChunk c;
    c.i = i;
    c.o = if_off[i];
    c.s = if_off[i + 1] - c.o;
    const int per = (c.s + GC - 1) / GC;
    c.lo = min(c.s, r * per);
    c.hi = min(c.s, c.lo + per);
    return c;
}

// Sum over the cluster in a fixed order: each CTA's block sum (block_sum_all), then the GC
// partials added in rank order by every CTA, so every thread of the cluster gets the same
// bits.  part[] alternates between calls: a CTA rewrites part[p] only after the barrier of
// the call in between, which every CTA passes after its reads of part[p].
template <int GC>
__device__ double cluster_sum_all(double v, double* red, double* part, double* tot, int& p) {
    const double b = block_sum_all(v, red);
    if (threadIdx.x == 0) part[p] = b;
    cl_sync();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int r = 0; r < GC; ++r) t += cl_ld_f64(cl_map(&part[p], (uint32_t)r));
        *tot = t;
    }
    __syncthreads();
    p ^= 1;
    return *tot;
}

// v_0 = g / beta on every interface of the level (g indexed by global DOF).
template <int GC>
__global__ void __cluster_dims__(GC, 1, 1) __launch_bounds__(GT)
    k_gm_init(const int* __restrict__ if_off, const int* __restrict__ if_dofs, const double* __restrict__ g,
              double* __restrict__ V, double* __restrict__ beta, int* __restrict__ kused) {
    __shared__ double red[33], part[2], tot;
    const int r = (int)cl_rank();
    const GmChunk c = gm_chunk<GC>(if_off, blockIdx.x / GC, r);
    int p = 0;
    double a = 0;
    for (int e = c.lo + threadIdx.x; e < c.hi; e += blockDim.x) { const double v = g[if_dofs[c.o + e]]; a += v * v; }
    const double b = sqrt(cluster_sum_all<GC>(a, red, part, &tot, p));
    if (r == 0 && threadIdx.x == 0) { beta[c.i] = b; kused[c.i] = b > 0.0 ? 0 : -1; }
    const double inv = b > 0.0 ? 1.0 / b : 0.0;
    for (int e = c.lo + threadIdx.x; e < c.hi; e += blockDim.x) V[c.o + e] = g[if_dofs[c.o + e]] * inv;
    cl_sync();                                  // no CTA leaves while a peer reads its partials
}

// Sums of a[0..16) over the warp, merged as they go: lane l gets the sum of a[l >> 1].
__device__ __forceinline__ double warp_sum16_f64(const double (&a)[16], int lane) {
    double b[8], c[4], d[2];
#pragma unroll
    for (int i = 0; i < 8; ++i) b[i] = (lane & 16 ? a[i + 8] : a[i]) + __shfl_xor_sync(0xffffffffu, lane & 16 ? a[i] : a[i + 8], 16);
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i] = (lane & 8 ? b[i + 4] : b[i]) + __shfl_xor_sync(0xffffffffu, lane & 8 ? b[i] : b[i + 4], 8);
#pragma unroll
    for (int i = 0; i < 2; ++i) d[i] = (lane & 4 ? c[i + 2] : c[i]) + __shfl_xor_sync(0xffffffffu, lane & 4 ? c[i] : c[i + 2], 4);
    const double e = (lane & 2 ? d[1] : d[0]) + __shfl_xor_sync(0xffffffffu, lane & 2 ? d[0] : d[1], 2);
    return e + __shfl_xor_sync(0xffffffffu, e, 1);
}

// Arnoldi step j with modified Gram-Schmidt on w = S~ v_j, per interface (a cluster, CTA r
// its r-th chunk): h_qj = <w - sum_{i<q} h_ij v_i, v_q>.  With the products r_q = <w, v_q>
// and the Gram entries G_qi = <v_q, v_i> that is h_q = r_q - sum_{i<q} G_qi h_i, so one pass
// and one cluster sum give every r_q and the new row G_j, and a forward substitution the h's,
// where one sum per q made a step a chain of j + 2 cluster sums (Swirydowicz, Langou,
// Ananthan, Yang, Thomas, "Low synchronization Gram-Schmidt and GMRES algorithms", 2021).
// Then w -= sum h_q v_q, h_{j+1,j} = ||w||, v_{j+1} = w / h_{j+1,j}.
// An interface whose h_{j+1,j} falls to 1e-14 beta (exact breakdown) stops with j + 1
// columns; one that completes min(gamma, s) steps stops with that many.
// (w itself stays a launch of its own: its gathers want more CTAs than the clusters have.)
template <int GC>
__global__ void __cluster_dims__(GC, 1, 1) __launch_bounds__(GT)
    k_gm_step(int j, int gamma, int S, const int* __restrict__ if_off, double* __restrict__ w, double* __restrict__ V,
              double* __restrict__ H, double* __restrict__ G, const double* __restrict__ beta, int* __restrict__ kused) {
    constexpr int QB = 8;                              // products of each kind per pass
    __shared__ double red[33], part[2], tot;
    __shared__ double s_red[GT / 32][2 * QB], s_part[2][2 * QB], s_rg[2][GAMMA_MAX];
    __shared__ double s_G[GAMMA_MAX][GAMMA_MAX + 1], s_h[GAMMA_MAX];
    const int r = (int)cl_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const GmChunk c = gm_chunk<GC>(if_off, blockIdx.x / GC, r);
    const int m = min(gamma, c.s);
    if (kused[c.i] != 0 || j >= m) return;     // the whole cluster
    const bool lead = r == 0 && tid == 0;
    double* Hi = H + (int64_t)c.i * (gamma + 1) * gamma;
    double* Gi = G + (int64_t)c.i * gamma * gamma;
    double* wi = w + c.o;
    const double* vj = V + (int64_t)j * S + c.o;
    for (int e = tid; e < j * j; e += GT) s_G[e / j][e % j] = Gi[(e / j) * gamma + e % j];     // rows 0 .. j - 1
    // r_q and G_jq, q <= j, QB of each per pass
    int pp = 0;
    for (int q0 = 0; q0 <= j; q0 += QB, pp ^= 1) {
        const int nq = min(QB, j + 1 - q0);
        double a[2 * QB];
#pragma unroll
        for (int q = 0; q < 2 * QB; ++q) a[q] = 0;
        for (int e = c.lo + tid; e < c.hi; e += GT) {
            const double we = wi[e], ve = vj[e];
#pragma unroll
            for (int q = 0; q < QB; ++q)
                if (q < nq) {
                    const double vq = V[(int64_t)(q0 + q) * S + c.o + e];
                    a[q] += we * vq;
                    if (q0 + q < j) a[QB + q] += ve * vq;
                }
        }
        const double ws = warp_sum16_f64(a, lane);
        if ((lane & 1) == 0) s_red[warp][lane >> 1] = ws;
        __syncthreads();
        if (tid < 256) {                               // value tid / 16, warp tid % 16
            double v = s_red[tid & 15][tid >> 4];
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if ((tid & 15) == 0) s_part[pp][tid >> 4] = v;
        }
        cl_sync();                                     // (s_part alternates: see cluster_sum_all)
        if (tid < 16 * GC) {                           // value tid / GC, CTA tid % GC
            double v = cl_ld_f64(cl_map(&s_part[pp][tid / GC], (uint32_t)(tid % GC)));
#pragma unroll
            for (int o = GC / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            const int q = tid / GC;
            if (tid % GC == 0 && q % QB < nq) s_rg[q / QB][q0 + q % QB] = v;
        }
        __syncthreads();
    }
    if (warp == 0) {                                   // forward substitution, lane = q
        double rq = lane <= j ? s_rg[0][lane] : 0.0;
        for (int i = 0; i < j; ++i) {
            const double hi = __shfl_sync(0xffffffffu, rq, i);
            const double g = lane > i && lane <= j ? (lane < j ? s_G[lane][i] : s_rg[1][i]) : 0.0;
            rq -= g * hi;
        }
        if (lane <= j) {
            s_h[lane] = rq;
            if (r == 0) {
                Hi[lane * gamma + j] = rq;
                if (lane < j) Gi[j * gamma + lane] = s_rg[1][lane];
            }
        }
    }
    __syncthreads();
    double a = 0;
    for (int e = c.lo + tid; e < c.hi; e += GT) {
        double we = wi[e];
#pragma unroll 4
        for (int q = 0; q <= j; ++q) we -= s_h[q] * V[(int64_t)q * S + c.o + e];
        wi[e] = we;
        a += we * we;
    }
    int p = 0;
    const double nrm = sqrt(cluster_sum_all<GC>(a, red, part, &tot, p));
    if (lead) Hi[(j + 1) * gamma + j] = nrm;
    if (nrm <= 1e-14 * beta[c.i]) {
        if (lead) kused[c.i] = j + 1;
    } else {
        double* vn = V + (int64_t)(j + 1) * S + c.o;
        const double inv = 1.0 / nrm;
        for (int e = c.lo + tid; e < c.hi; e += GT) vn[e] = wi[e] * inv;
        if (j + 1 == m && lead) kused[c.i] = m;
    }
    cl_sync();                                  // no CTA leaves while a peer reads its partials
}

// u_t = V_k y with y the least-squares solution of min || beta e1 - H_k y || (H_k the
// (k+1) x k Hessenberg matrix; Givens rotations), written to z on the interface DOFs.
// Every CTA of an interface solves the small problem itself (the same bits) and writes
// its chunk.  The small problem takes one warp, lane = column (then row): a rotation's
// norm on entries scaled by a power of two, the rest of the rotation one step for all
// columns; one thread alone took 30 us (an FP64 operation's latency is 65 clocks).
__global__ void __launch_bounds__(GT) k_gm_finish(int GC, int gamma, int S, const int* __restrict__ if_off,
                                                  const int* __restrict__ if_dofs, const double* __restrict__ V,
                                                  const double* __restrict__ H, const double* __restrict__ beta,
                                                  const int* __restrict__ kused, double* __restrict__ z) {
    __shared__ double y[GAMMA_MAX];
    __shared__ double R[GAMMA_MAX + 1][GAMMA_MAX + 1];  // rotated Hessenberg
    const int i = blockIdx.x / GC, o = if_off[i], s = if_off[i + 1] - o, per = (s + GC - 1) / GC;
    const int lo = min(s, (int)(blockIdx.x % GC) * per), hi = min(s, lo + per);
    const int ku = kused[i], tid = threadIdx.x, lane = tid & 31;
    const int k = ku < 0 ? 0 : (ku == 0 ? min(gamma, s) : ku);
    const double* Hi = H + (int64_t)i * (gamma + 1) * gamma;
    for (int e = tid; e < (k + 1) * k; e += GT) R[e / k][e % k] = e / k <= e % k + 1 ? Hi[(e / k) * gamma + e % k] : 0.0;
    __syncthreads();
    if (tid < 32 && k > 0) {
        double g0 = beta[i], t = 0.0;                  // the entry of the right-hand side being rotated; row `lane`'s
        for (int c = 0; c < k; ++c) {
            const double a = R[c][c], b = R[c + 1][c];
            const double mx = fmax(fabs(a), fabs(b));
            double cs = 1.0, sn = 0.0, den = mx;
            if (mx > 0.0 && mx <= 1.7976931348623157e308) {
                const int ex = (int)((__double_as_longlong(mx) >> 52) & 0x7ff);
                const int sc = max(-1000, min(1000, 1023 - ex));
                const double as = ldexp(a, sc), bs = ldexp(b, sc);
                const double d2 = as * as + bs * bs, inv = 1.0 / sqrt(d2);
                cs = as * inv;
                sn = bs * inv;
                den = ldexp(d2 * inv, -sc);
            } else if (mx != 0.0) {                    // not finite
                cs = sn = den = a + b;
            }
            double r0 = 0.0, r1 = 0.0;
            if (lane > c && lane < k) { r0 = R[c][lane]; r1 = R[c + 1][lane]; }
            __syncwarp();
            if (lane > c && lane < k) {
                R[c][lane] = cs * r0 + sn * r1;
                R[c + 1][lane] = -sn * r0 + cs * r1;
            }
            if (lane == c) { R[c][c] = den; t = cs * g0; }
            g0 = -sn * g0;
            __syncwarp();
        }
        const double d = lane < k ? R[lane][lane] : 1.0;
        const double rd = d != 0.0 ? 1.0 / d : 0.0;
        for (int r = k - 1; r >= 0; --r) {
            const double yr = __shfl_sync(0xffffffffu, t * rd, r);
            if (lane < r) t -= R[lane][r] * yr;
            if (lane == r) y[r] = yr;
        }
    }
    __syncthreads();
    for (int e = lo + tid; e < hi; e += GT) {
        double u = 0;
        for (int q = 0; q < k; ++q) u += y[q] * V[(int64_t)q * S + o + e];
        z[if_dofs[o + e]] = u;
    }
}

}  // namespace

static int round_up_int(int v, int a) { return (v + a - 1) / a * a; }

// Apply-time launches of one level's inner GMRES: reads g (global DOF order, h.d_pg) on
// the level's interface DOFs and writes u_t = GMRES_gamma(S~_t, g_t) into z there.
int gamma_interface_solve(Handle& h, int li, double* z) {
    GammaLevel& G = h.gamma_levels[li];
    if (G.n_if == 0 || G.S == 0) return RSD_OK;
    const Level& Ll = h.levels.back();
    const int nleaf = (int)Ll.fronts.size();
    // t_l = (L_l^-1 K_{l I})[:, R] x reads Y^T (the backward descriptors) for nonsymmetric
    // leaves; for symmetric ones Y^T = X
    const FrontDesc* ty = Ll.d_fronts_bwd ? Ll.d_fronts_bwd : Ll.d_fronts;
    const bool f64 = is_fp64(Ll.prec);
    // the leaves' FP16 copy when they have one (16-bit operand levels; not the transposed
    // upper factors of nonsymmetric leaves)
    const bool c16 = smv_reads_fp16(Ll);
    const int gam = h.gamma;
    int pi = prof_begin(h, K_GAMMA);
    const int gc = gm_cluster(G.n_if, h.num_sms), lg = gc == 8 ? 3 : gc == 4 ? 2 : gc == 2 ? 1 : 0;
    using Init = void (*)(const int*, const int*, const double*, double*, double*, int*);
    using Step = void (*)(int, int, int, const int*, double*, double*, double*, double*, const double*, int*);
    static constexpr Init init[4] = {k_gm_init<1>, k_gm_init<2>, k_gm_init<4>, k_gm_init<8>};
    static constexpr Step step[4] = {k_gm_step<1>, k_gm_step<2>, k_gm_step<4>, k_gm_step<8>};
    init[lg]<<<G.n_if * gc, GT, 0, h.stream>>>(G.d_if_off, G.d_if_dofs, h.d_pg, h.d_gm_V, h.d_gm_beta, h.d_gm_kused);
    count_launch();
    prof_end(h, pi, 0.0, 0.0);
    const int wcol = f64 ? 2 : (c16 ? 8 : 4);     // columns per lane of k_smv_leaf
    const dim3 gl((unsigned)nleaf, (unsigned)std::max(1, (Ll.max_s + 32 * wcol - 1) / (32 * wcol)));
    const unsigned gi = (unsigned)std::max(1, std::min(h.num_sms * 8, (G.S + 31) / 32));   // 32 positions per CTA
    // One CTA a leaf does both products where the leaves fill the chip and a leaf's rows
    // of the level fit L1 beside those of the CTAs it shares it with (the second reading hits
    // there); larger leaves keep the two kernels, which spread a leaf over many CTAs.
    const int W = 16 / (f64 ? 8 : c16 ? 2 : 4);
    const bool both = nleaf >= h.num_sms && (Ll.max_s + W - 1) / W <= 256 && G.xbytes / 2 <= 192.0 * 1024 * nleaf;
    const size_t both_smem = ((size_t)round_up_int(Ll.max_s, W) + 256 * W) * (f64 ? 8 : 4);
    for (int j = 0; j < gam; ++j) {
        const double* vj = h.d_gm_V + (int64_t)j * G.S;
        const unsigned gr = (unsigned)std::max(1, std::min(h.num_sms * 4, (G.nk + 31) / 32));   // 8 warps of 4 rows
        pi = prof_begin(h, K_GAMMA_SMV);
        if (both) {
            if (f64) k_smv_both<double, false><<<nleaf, 256, both_smem, h.stream>>>(ty, Ll.d_fronts, G.d_cl_ptr, G.d_cl_row, G.d_cl_pos, Ll.max_s, vj, h.d_gm_yl);
            else if (c16) k_smv_both<float, true><<<nleaf, 256, both_smem, h.stream>>>(Ll.d_fronts, Ll.d_fronts, G.d_cl_ptr, G.d_cl_row, G.d_cl_pos, Ll.max_s, vj, h.d_gm_yl);
            else k_smv_both<float, false><<<nleaf, 256, both_smem, h.stream>>>(ty, Ll.d_fronts, G.d_cl_ptr, G.d_cl_row, G.d_cl_pos, Ll.max_s, vj, h.d_gm_yl);
        } else if (f64) {
            k_smv_leaf<double, false><<<gl, 256, 0, h.stream>>>(ty, G.d_cl_ptr, G.d_cl_row, G.d_cl_pos, h.d_tl_off, vj,
                                                                h.d_tl);
            k_smv_rows<double, false><<<gr, 256, 0, h.stream>>>(G.nk, G.d_cl_leaf, G.d_cl_row, Ll.d_fronts, h.d_tl_off,
                                                                h.d_tl, h.d_gm_yl);
        } else if (c16) {
            float* tl32 = (float*)h.d_tl;
            k_smv_leaf<float, true><<<gl, 256, 0, h.stream>>>(Ll.d_fronts, G.d_cl_ptr, G.d_cl_row, G.d_cl_pos, h.d_tl_off,
                                                              vj, tl32);
            k_smv_rows<float, true><<<gr, 256, 0, h.stream>>>(G.nk, G.d_cl_leaf, G.d_cl_row, Ll.d_fronts, h.d_tl_off, tl32,
                                                              h.d_gm_yl);
        } else {
            float* tl32 = (float*)h.d_tl;
            k_smv_leaf<float, false><<<gl, 256, 0, h.stream>>>(ty, G.d_cl_ptr, G.d_cl_row, G.d_cl_pos, h.d_tl_off, vj,
                                                               tl32);
            k_smv_rows<float, false><<<gr, 256, 0, h.stream>>>(G.nk, G.d_cl_leaf, G.d_cl_row, Ll.d_fronts, h.d_tl_off,
                                                               tl32, h.d_gm_yl);
        }
        prof_end(h, pi, 0.0, G.xbytes);
        pi = prof_begin(h, K_GAMMA_IFACE);
        k_smv_iface<<<gi, 256, 0, h.stream>>>(G.S, G.d_if_dofs, h.d_rowptr, h.d_col, h.d_val, h.d_owner, h.d_pk_pos,
                                              G.d_ci_ptr, G.d_ci_k, h.d_gm_yl, vj, h.d_gm_w);
        prof_end(h, pi, 0.0, 0.0);
        pi = prof_begin(h, K_GAMMA);
        step[lg]<<<G.n_if * gc, GT, 0, h.stream>>>(j, gam, G.S, G.d_if_off, h.d_gm_w, h.d_gm_V, h.d_gm_H, h.d_gm_G, h.d_gm_beta,
                                                   h.d_gm_kused);
        prof_end(h, pi, 0.0, 0.0);
        count_launch(both ? 3 : 4);
    }
    pi = prof_begin(h, K_GAMMA);
    k_gm_finish<<<G.n_if * gc, GT, 0, h.stream>>>(gc, gam, G.S, G.d_if_off, G.d_if_dofs, h.d_gm_V, h.d_gm_H, h.d_gm_beta,
                                             h.d_gm_kused, z);
    count_launch();
    prof_end(h, pi, 0.0, 0.0);
    RSD_CUDA_TRY(cudaGetLastError());
    return RSD_OK;
}

}  // namespace rsd
