// dl_sgreal.cu -- kernels of the real least solution S~ of the same-generation equation
// (Sec. 7.2; the two-sided class of Sec. 6.3):
//     S~ = eps (B + P S~ P^T),   eps = 1 / (1 + ||P||_inf^2).
// One step of the fixpoint series X <- eps (B + P X P^T) is two gather passes over the CSR of P
// in FP64 (U = X P^T, then eps (B + P U)); the same passes give the residual
// eps (B + P X P^T) - X of the refinement.  The FP32 helpers serve Smith's doubling for the
// Stein equation on the TF32 tensor cores (the GEMMs themselves are dl_umma.cu's).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dl_internal.h"

namespace dl {

namespace {

// Bound on the change of a series step without FP64 arithmetic.  The series is monotone in
// floating point too (every operation is monotone on non-negative values), so v >= x and
// k = bits(v) - bits(x) >= 0 counts the doubles between them; then v - x < 2^(bitlength(k) +
// exponent(v) - 1075).  Returned as that power plus 4096 (0: no change), for an integer max.
__device__ __forceinline__ unsigned long long change_code(double v, double x) {
    const long long bv = __double_as_longlong(v), bx = __double_as_longlong(x);
    long long k = bv - bx;
    if (k == 0) return 0ull;
    if (k < 0) k = -k;  // not reached by the series; kept as a bound
    const int ev = static_cast<int>((bv >> 52) & 0x7FF);
    return static_cast<unsigned long long>((64 - __clzll(k)) + max(ev, 1) - 1075 + 4096);
}

// U = X P^T:  U[i][j] = sum_{w : P[j][w] = 1} X[i][w].  One block per row i, the row staged in
// shared memory; rows and columns >= n are zero.
__global__ void __launch_bounds__(256) sg_xpt_kernel(const int *__restrict__ ptr, const int *__restrict__ col, int n,
                                                     int np, const double *__restrict__ X, double *__restrict__ U) {
    extern __shared__ double xs[];
    const int i = blockIdx.x;
    const double *xr = X + static_cast<int64_t>(i) * np;
    for (int t = threadIdx.x; t < np; t += blockDim.x) xs[t] = xr[t];
    __syncthreads();
    double *ur = U + static_cast<int64_t>(i) * np;
    for (int j = threadIdx.x; j < np; j += blockDim.x) {
        double s = 0.0;
        if (i < n && j < n) {
            const int q1 = ptr[j + 1];
            for (int q = ptr[j]; q < q1; ++q) s += xs[col[q]];
        }
        ur[j] = s;
    }
}

// V[i][j] = eps (B[i][j] + sum_{y : P[i][y] = 1} U[y][j])  (B = NULL: the identity), and
// D = V - X.  Xn (optional) <- V (a series step); R (optional, FP32) <- D (the residual).
// With R: *dmax = max |D| as the bit pattern of a non-negative double; without: *dmax = the
// max of change_code(V, X).
// Grid: x over columns (256 per block), y over rows.
__global__ void __launch_bounds__(256) sg_pu_kernel(const int *__restrict__ ptr, const int *__restrict__ col, int n,
                                                    int np, double eps, const uint8_t *__restrict__ B,
                                                    const double *__restrict__ U, const double *__restrict__ X,
                                                    double *__restrict__ Xn, float *__restrict__ R,
                                                    unsigned long long *dmax) {
    const int i = blockIdx.y;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long m = 0;
    if (j < np) {
        double v = 0.0;
        if (i < n && j < n) {
            double s = B != nullptr ? static_cast<double>(B[static_cast<int64_t>(i) * n + j] & 1) : (i == j ? 1.0 : 0.0);
            const int q1 = ptr[i + 1];
            for (int q = ptr[i]; q < q1; ++q) s += U[static_cast<int64_t>(col[q]) * np + j];
            v = eps * s;
        }
        const int64_t at = static_cast<int64_t>(i) * np + j;
        if (R != nullptr) {  // the residual: the real difference
            const double d = v - X[at];
            R[at] = static_cast<float>(d);
            m = static_cast<unsigned long long>(__double_as_longlong(d)) & 0x7FFFFFFFFFFFFFFFull;  // |d|
        } else {
            m = change_code(v, X[at]);
        }
        if (Xn != nullptr) Xn[at] = v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, m, o);
        m = other > m ? other : m;
    }
    if ((threadIdx.x & 31) == 0 && m != 0) atomicMax(dmax, m);
}

constexpr int kFusedMaxNp = 16384;  // 1024 threads x 16 columns

// The same step in one pass when every node has few parents:
//   V[i][j] = eps ([B_ij] + sum_{y in P_i} sum_{w in P_j} X[y][w]).
// One block per row i; the rows y of X (the parents of i) go through shared memory one at a
// time and each thread keeps the sums of its columns j = t + THREADS c in registers (512 x 8
// up to np = 4096, two blocks per SM; else 1024 x 16).  A sum starts
// from its first term (no 0 + x) and B's term is added only where it is 1, so a column with one
// parent pair costs one FP64 multiply.
template <int THREADS, int COLS>
__global__ void __launch_bounds__(THREADS)
    sg_fused_kernel(const int *__restrict__ ptr, const int *__restrict__ col, int n, int np, double eps,
                    const uint8_t *__restrict__ B, const double *__restrict__ X, double *__restrict__ Xn,
                    float *__restrict__ R, unsigned long long *dmax) {
    extern __shared__ double xs[];
    const int i = blockIdx.x;
    double acc[COLS];
    unsigned started = 0;  // bit c: column c's sum has a term
#pragma unroll
    for (int c = 0; c < COLS; ++c) acc[c] = 0.0;
    const int q0 = i < n ? ptr[i] : 0, q1 = i < n ? ptr[i + 1] : 0;
    for (int q = q0; q < q1; ++q) {  // parents y of i (block-uniform)
        const double *xr = X + static_cast<int64_t>(col[q]) * np;
        __syncthreads();
        for (int t = threadIdx.x; t < np; t += THREADS) xs[t] = xr[t];
        __syncthreads();
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
            const int j = threadIdx.x + c * THREADS;
            if (j >= n) break;
            int w = ptr[j];
            const int w1 = ptr[j + 1];
            if (w < w1 && !((started >> c) & 1)) {  // a first term is assigned, not added to 0
                acc[c] = xs[col[w]];
                started |= 1u << c;
                ++w;
            }
            for (; w < w1; ++w) acc[c] += xs[col[w]];
        }
    }
    unsigned long long m = 0;
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
        const int j = threadIdx.x + c * THREADS;
        if (j >= np) break;
        double v = 0.0;
        if (i < n && j < n) {
            const bool b = B != nullptr ? (B[static_cast<int64_t>(i) * n + j] & 1) != 0 : i == j;
            double s = acc[c];
            if (b) s = (started >> c) & 1 ? s + 1.0 : 1.0;
            v = eps * s;
        }
        const int64_t at = static_cast<int64_t>(i) * np + j;
        if (Xn != nullptr) Xn[at] = v;
        if (R != nullptr) {  // the residual: the real difference
            const double d = v - X[at];
            R[at] = static_cast<float>(d);
            const unsigned long long ad = static_cast<unsigned long long>(__double_as_longlong(d)) & 0x7FFFFFFFFFFFFFFFull;
            m = ad > m ? ad : m;
        } else if (dmax != nullptr) {  // a series step: the integer bound
            const unsigned long long cc = change_code(v, X[at]);
            m = cc > m ? cc : m;
        }
    }
    if (dmax != nullptr) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xffffffffu, m, o);
            m = other > m ? other : m;
        }
        if ((threadIdx.x & 31) == 0 && m != 0) atomicMax(dmax, m);
    }
}

// A = s P (FP32, np x np, zero padding) and NA = -A.
__global__ void sg_scaled_p_kernel(const uint8_t *__restrict__ P, int n, int np, float s, float *__restrict__ A,
                                   float *__restrict__ NA) {
    const int64_t total = static_cast<int64_t>(np) * np;
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < total;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t i = t / np, j = t - i * np;
        const float v = (i < n && j < n && (P[i * n + j] & 1)) ? s : 0.0f;
        A[t] = v;
        NA[t] = -v;
    }
}

// *out = max over rows of sum_j |A[i][j]| (FP32 bit patterns of non-negative sums, atomicMax).
__global__ void __launch_bounds__(256) row_abs_sum_max_kernel(const float *__restrict__ A, int np, unsigned *out) {
    __shared__ float part[8];
    const int i = blockIdx.x;
    float s = 0.0f;
    for (int j = threadIdx.x; j < np; j += blockDim.x) s += fabsf(A[static_cast<int64_t>(i) * np + j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t += part[w];
        atomicMax(out, __float_as_uint(t));
    }
}

__global__ void negate_f32_kernel(const float *__restrict__ a, float *__restrict__ b, int64_t count) {
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < count;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x)
        b[t] = -a[t];
}

__global__ void add_f32_to_f64_kernel(double *__restrict__ x, const float *__restrict__ d, int64_t count) {
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < count;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x)
        x[t] += static_cast<double>(d[t]);
}

__global__ void bits_or_kernel(uint64_t *__restrict__ dst, const uint64_t *__restrict__ src, int64_t words) {
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < words;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x)
        dst[t] |= src[t];
}

constexpr int kTT = 32;

// dst[c][r] = src[r][c] for an rows x cols block (32 x 32 tiles through shared memory).
template <class T>
__global__ void transpose_tile_kernel(const T *__restrict__ src, int64_t lds, int rows, int cols, T *__restrict__ dst,
                                      int64_t ldd) {
    __shared__ T tile[kTT][kTT + 1];
    const int c0 = blockIdx.x * kTT, r0 = blockIdx.y * kTT;
    for (int y = threadIdx.y; y < kTT; y += blockDim.y) {
        const int r = r0 + y, c = c0 + threadIdx.x;
        if (r < rows && c < cols) tile[y][threadIdx.x] = src[static_cast<int64_t>(r) * lds + c];
    }
    __syncthreads();
    for (int y = threadIdx.y; y < kTT; y += blockDim.y) {
        const int c = c0 + y, r = r0 + threadIdx.x;
        if (r < rows && c < cols) dst[static_cast<int64_t>(c) * ldd + r] = tile[threadIdx.x][y];
    }
}

// ---- the transposed class: X = eps (R1 + R1 X^T) (Sec. 6.2) ----------------------------------
// Two steps of the series without a transpose: the first one forms the *transposed* iterate row by
// row, Y[j][i] = eps (R1[i][j] + sum_{y in succ(i)} X[j][y]) (trans_local_kernel: row j of X is all
// it needs, gathered from shared memory), and the second one gathers rows of it,
// X[i][j] = eps (R1[i][j] + sum_{y in succ(i)} Y[y][j]) (trans_gather_kernel, coalesced).  R1 itself
// is read off the successor lists.  In FP64 a step is bound by GB300's FP64 rate (two lanes per SM:
// nnz n + n^2 operations, 0.15 ms at n = 4096 with 4 facts per row), in FP32 (the correction series
// D = R + L D of the refinement, R the residual) by its bytes.  The constants are relabelled by
// falling number of successors (rank_kernel): the lanes of a warp of the local step, one constant
// each, then have lists of one length; in the given order a warp took its longest list's time, 2.3
// times the mean (FP64 0.46 ms, FP32 0.094 ms a step at n = 4096).  One step was 0.44 ms as a
// transpose and a gather without vector loads, all in FP64.

// A converged solve: the last pair's change is at the FP32 rounding of the iterate (slots[0] the
// bits of max |change|, slots[1] those of max |iterate|; both 0 when that pair was left out).
__device__ __forceinline__ bool trans_converged(const unsigned long long *slots) {
    if (slots == nullptr) return false;
    const float change = __uint_as_float(static_cast<unsigned>(slots[0]));
    return change <= 4.8e-7f * __uint_as_float(static_cast<unsigned>(slots[1]));
}

template <class T, int G>
struct alignas(sizeof(T) * G) RowPack {
    T v[G];
};

// rank[i] += constants k of this CTA's part that come before i (more successors, or as many and a
// smaller number); rank zeroed by the caller.  n^2 comparisons spread over the grid.
constexpr int kRankPart = 512;
__global__ void __launch_bounds__(256) rank_kernel(const int *__restrict__ ptr, int n, int *rank) {
    __shared__ int deg_s[kRankPart];
    const int k0 = blockIdx.y * kRankPart, m = min(kRankPart, n - k0);
    for (int k = threadIdx.x; k < m; k += blockDim.x) deg_s[k] = ptr[k0 + k + 1] - ptr[k0 + k];
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int d = ptr[i + 1] - ptr[i];
    int before = 0;
#pragma unroll 8
    for (int k = 0; k < m; ++k) before += deg_s[k] > d || (deg_s[k] == d && k0 + k < i);
    if (before) atomicAdd(rank + i, before);
}

// perm = the inverse of rank, cnt[a] = the number of successors of constant perm[a].
__global__ void relabel_counts_kernel(const int *__restrict__ ptr, const int *__restrict__ rank, int n, int *perm,
                                      int *cnt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    perm[rank[i]] = i;
    cnt[rank[i]] = ptr[i + 1] - ptr[i];
}

// The successor lists under the new labels (warp per row).
__global__ void __launch_bounds__(256)
    relabel_lists_kernel(const int *__restrict__ ptr, const int *__restrict__ col, const int *__restrict__ rank,
                         const int *__restrict__ perm, const int *__restrict__ ptr2, int n, int *col2) {
    const int a = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (a >= n) return;
    const int i = perm[a], q0 = ptr[i], d = ptr[i + 1] - q0, at = ptr2[a];
    for (int t = threadIdx.x & 31; t < d; t += 32) col2[at + t] = rank[col[q0 + t]];
}

// Rows j0 .. j0 + G of Y: RHS (T = float): RT[j][i] + eps sum, else eps (R1[i][j] + sum); the G rows of
// X interleaved in shared memory so that one gather serves all of them.  X == NULL: X = 0.
template <class T, int G, bool RHS>
__global__ void __launch_bounds__(512)
    trans_local_kernel(const int *__restrict__ ptr, const int *__restrict__ col, int n, int np, T eps,
                       const T *__restrict__ X, const float *__restrict__ RT, T *__restrict__ Y,
                       const unsigned long long *skip) {
    if (trans_converged(skip)) return;
    extern __shared__ __align__(16) uint8_t trans_smem[];
    auto *xs = reinterpret_cast<RowPack<T, G> *>(trans_smem);  // n entries
    const int j0 = blockIdx.x * G;
#pragma unroll 2
    for (int y = threadIdx.x; y < n; y += blockDim.x) {
        RowPack<T, G> r;
#pragma unroll
        for (int g = 0; g < G; ++g) r.v[g] = X != nullptr ? X[static_cast<int64_t>(j0 + g) * np + y] : T(0);
        xs[y] = r;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < np; i += blockDim.x) {
        RowPack<T, G> s;
        unsigned facts = 0;  // bit g: R1[i][j0 + g]
#pragma unroll
        for (int g = 0; g < G; ++g) s.v[g] = T(0);
        if (i < n) {
            const int q0 = ptr[i], q1 = ptr[i + 1];
            int c = q0 < q1 ? col[q0] : 0;
            if (q0 < q1) {  // a first term is assigned, not added to 0
                s = xs[c];
                if (!RHS && static_cast<unsigned>(c - j0) < G) facts |= 1u << (c - j0);
            }
            for (int q = q0 + 1; q < q1; ++q) {
                c = col[q];
                const RowPack<T, G> r = xs[c];
#pragma unroll
                for (int g = 0; g < G; ++g) s.v[g] += r.v[g];
                if (!RHS && static_cast<unsigned>(c - j0) < G) facts |= 1u << (c - j0);
            }
        }
        if (!RHS && facts != 0) {
#pragma unroll
            for (int g = 0; g < G; ++g)
                if ((facts >> g) & 1u) s.v[g] += T(1);
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int64_t at = static_cast<int64_t>(j0 + g) * np + i;
            T v = T(0);
            if (i < n && j0 + g < n) v = RHS ? static_cast<T>(RT[at]) + eps * s.v[g] : eps * s.v[g];
            Y[at] = v;
        }
    }
}

// X from the rows of Y: RHS (T = float) R + eps sum, else eps (R1 + sum).  T = float: slots[0] / [1] =
// bits of max |change| / max |X|; T = double: slots[0] = change_code of the largest change (of two
// steps).  old: the iterate two steps before (X itself, R for a first pair, or NULL: 0).
template <class T, bool RHS>
__global__ void __launch_bounds__(256)
    trans_gather_kernel(const int *__restrict__ ptr, const int *__restrict__ col, int n, int np, T eps,
                        const T *__restrict__ Y, const float *__restrict__ R, const T *old, T *X,
                        unsigned long long *slots, const unsigned long long *skip) {
    if (trans_converged(skip)) return;
    constexpr int V = 16 / sizeof(T);
    using Pack = RowPack<T, V>;
    const int i = blockIdx.y;
    const int j0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
    unsigned long long m0 = 0, m1 = 0;
    if (j0 < np) {
        Pack s, was;
        unsigned facts = 0;  // bit v: R1[i][j0 + v]
#pragma unroll
        for (int v = 0; v < V; ++v) s.v[v] = was.v[v] = T(0);
        const int64_t at = static_cast<int64_t>(i) * np + j0;
        if (old != nullptr) was = *reinterpret_cast<const Pack *>(old + at);
        if (i < n) {
            const int q1 = ptr[i + 1];
            int q = ptr[i];
            auto row = [&](int c) {
                if (!RHS && static_cast<unsigned>(c - j0) < V) facts |= 1u << (c - j0);
                return *reinterpret_cast<const Pack *>(Y + static_cast<int64_t>(c) * np + j0);
            };
            if (q < q1) s = row(col[q++]);
            for (; q + 2 <= q1; q += 2) {  // two rows in flight
                const Pack a = row(col[q]), b = row(col[q + 1]);
#pragma unroll
                for (int v = 0; v < V; ++v) s.v[v] = (s.v[v] + a.v[v]) + b.v[v];
            }
            if (q < q1) {
                const Pack a = row(col[q]);
#pragma unroll
                for (int v = 0; v < V; ++v) s.v[v] += a.v[v];
            }
        }
        if (!RHS && facts != 0) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                if ((facts >> v) & 1u) s.v[v] += T(1);
        }
        Pack x;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            x.v[v] = T(0);
            if (i < n && j0 + v < n) x.v[v] = RHS ? static_cast<T>(R[at + v]) + eps * s.v[v] : eps * s.v[v];
            if (sizeof(T) == 8) {
                const unsigned long long c = change_code(x.v[v], was.v[v]);
                m0 = c > m0 ? c : m0;
            } else {
                const unsigned c = __float_as_uint(fabsf(static_cast<float>(x.v[v]) - static_cast<float>(was.v[v])));
                const unsigned a = __float_as_uint(fabsf(static_cast<float>(x.v[v])));
                m0 = c > m0 ? c : m0;
                m1 = a > m1 ? a : m1;
            }
        }
        *reinterpret_cast<Pack *>(X + at) = x;
    }
    __shared__ unsigned long long part[2][8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, m0, o), b = __shfl_xor_sync(0xffffffffu, m1, o);
        m0 = a > m0 ? a : m0;
        m1 = b > m1 ? b : m1;
    }
    if ((threadIdx.x & 31) == 0) {
        part[0][threadIdx.x >> 5] = m0;
        part[1][threadIdx.x >> 5] = m1;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        unsigned long long m = 0;
        for (int w = 0; w < 8; ++w) m = part[threadIdx.x][w] > m ? part[threadIdx.x][w] : m;
        // (most CTAs find the slot at least as large: a read before the atomic keeps them off it)
        if (m != 0 && m > *reinterpret_cast<volatile unsigned long long *>(slots + threadIdx.x))
            atomicMax(slots + threadIdx.x, m);
    }
}

// R[i][j] = YT[j][i] - X[i][j] (FP64 difference, rounded to FP32), RT = R^T; *rmax = bits of max |R|
// (FP64).  32 x 32 tiles.
__global__ void __launch_bounds__(256)
    trans_residual_kernel(const double *__restrict__ YT, const double *__restrict__ X, int np, float *__restrict__ R,
                          float *__restrict__ RT, unsigned long long *rmax) {
    __shared__ double t[kTT][kTT + 1];
    __shared__ float r[kTT][kTT + 1];
    const int i0 = blockIdx.y * kTT, j0 = blockIdx.x * kTT;
    for (int y = threadIdx.y; y < kTT; y += blockDim.y)
        t[y][threadIdx.x] = YT[static_cast<int64_t>(j0 + y) * np + i0 + threadIdx.x];
    __syncthreads();
    unsigned long long m = 0;
    for (int y = threadIdx.y; y < kTT; y += blockDim.y) {
        const int64_t at = static_cast<int64_t>(i0 + y) * np + j0 + threadIdx.x;
        const double d = t[threadIdx.x][y] - X[at];
        const float f = static_cast<float>(d);
        R[at] = f;
        r[threadIdx.x][y] = f;
        const unsigned long long a = static_cast<unsigned long long>(__double_as_longlong(d)) & 0x7FFFFFFFFFFFFFFFull;
        m = a > m ? a : m;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < kTT; y += blockDim.y)
        RT[static_cast<int64_t>(j0 + y) * np + i0 + threadIdx.x] = r[y][threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, m, o);
        m = other > m ? other : m;
    }
    if (threadIdx.x == 0 && m > *reinterpret_cast<volatile unsigned long long *>(rmax)) atomicMax(rmax, m);
}

// The solution under its own labels: out[i][j] = X[rank[i]][rank[j]] (row stride n, optional) and the
// bits out > 0 (wp words per row).  A CTA per row, staged in shared memory.
__global__ void __launch_bounds__(512)
    trans_finish_kernel(const int *__restrict__ rank, int n, int np, int wp, const double *__restrict__ X,
                        double *__restrict__ out, uint32_t *__restrict__ bits) {
    extern __shared__ double finish_s[];
    const int i = blockIdx.x;
    const double *row = X + static_cast<int64_t>(rank[i]) * np;
    for (int t = threadIdx.x; t < n; t += blockDim.x) finish_s[t] = row[t];
    __syncthreads();
    for (int j = threadIdx.x; j < 64 * wp; j += blockDim.x) {
        const double v = j < n ? finish_s[rank[j]] : 0.0;
        if (out != nullptr && j < n) out[static_cast<int64_t>(i) * n + j] = v;
        const long long b = __double_as_longlong(v);
        const uint32_t pos = __ballot_sync(0xffffffffu, b > 0 && b <= 0x7FF0000000000000ll);
        if ((threadIdx.x & 31) == 0) bits[static_cast<int64_t>(i) * 2 * wp + (j >> 5)] = pos;
    }
}

__global__ void f32_to_f64_kernel(double *__restrict__ x, const float *__restrict__ d, int64_t count) {
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < count;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x)
        x[t] = static_cast<double>(d[t]);
}

unsigned stream_blocks(int64_t count) {
    return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((count + 255) / 256, 152 * 32)));
}

}  // namespace

bool sg_real_fused(int np, unsigned long long max_parents) {
    return np <= kFusedMaxNp && max_parents <= 4;
}

cudaError_t sg_real_step(const int *ptr, const int *col, int n, int np, double eps, const uint8_t *B, const double *X,
                         double *U, double *Xn, float *R, unsigned long long *dmax, bool fused, cudaStream_t s) {
    const size_t smem = sizeof(double) * static_cast<size_t>(np);
    if (fused && np <= 4096) {
        cudaError_t e = allow_all_smem(sg_fused_kernel<512, 8>);
        if (e != cudaSuccess) return e;
        sg_fused_kernel<512, 8><<<static_cast<unsigned>(np), 512, smem, s>>>(ptr, col, n, np, eps, B, X, Xn, R, dmax);
        return cudaGetLastError();
    }
    if (fused) {
        cudaError_t e = allow_all_smem(sg_fused_kernel<1024, 16>);
        if (e != cudaSuccess) return e;
        sg_fused_kernel<1024, 16><<<static_cast<unsigned>(np), 1024, smem, s>>>(ptr, col, n, np, eps, B, X, Xn, R,
                                                                               dmax);
        return cudaGetLastError();
    }
    cudaError_t e = allow_all_smem(sg_xpt_kernel);
    if (e != cudaSuccess) return e;
    sg_xpt_kernel<<<static_cast<unsigned>(np), 256, smem, s>>>(ptr, col, n, np, X, U);
    dim3 grid(static_cast<unsigned>((np + 255) / 256), static_cast<unsigned>(np));
    sg_pu_kernel<<<grid, 256, 0, s>>>(ptr, col, n, np, eps, B, U, X, Xn, R, dmax);
    return cudaGetLastError();
}

cudaError_t sg_scaled_p(const uint8_t *P, int n, int np, float scale, float *A, float *NA, cudaStream_t s) {
    sg_scaled_p_kernel<<<stream_blocks(static_cast<int64_t>(np) * np), 256, 0, s>>>(P, n, np, scale, A, NA);
    return cudaGetLastError();
}

cudaError_t row_abs_sum_max(const float *A, int np, unsigned *out, cudaStream_t s) {
    row_abs_sum_max_kernel<<<static_cast<unsigned>(np), 256, 0, s>>>(A, np, out);
    return cudaGetLastError();
}

cudaError_t negate_f32(const float *a, float *b, int64_t count, cudaStream_t s) {
    negate_f32_kernel<<<stream_blocks(count), 256, 0, s>>>(a, b, count);
    return cudaGetLastError();
}

cudaError_t add_f32_to_f64(double *x, const float *d, int64_t count, cudaStream_t s) {
    add_f32_to_f64_kernel<<<stream_blocks(count), 256, 0, s>>>(x, d, count);
    return cudaGetLastError();
}

cudaError_t bits_or(uint64_t *dst, const uint64_t *src, int64_t words, cudaStream_t s) {
    bits_or_kernel<<<stream_blocks(words), 256, 0, s>>>(dst, src, words);
    return cudaGetLastError();
}

cudaError_t transpose_f32(const float *src, int64_t lds, int rows, int cols, float *dst, int64_t ldd, cudaStream_t s) {
    dim3 grid(static_cast<unsigned>((cols + kTT - 1) / kTT), static_cast<unsigned>((rows + kTT - 1) / kTT));
    transpose_tile_kernel<float><<<grid, dim3(kTT, 8), 0, s>>>(src, lds, rows, cols, dst, ldd);
    return cudaGetLastError();
}

namespace {

// The local step with as many rows per CTA as shared memory holds (up to 16 bytes per entry).
template <class T, bool RHS>
cudaError_t trans_local(const int *ptr, const int *col, int n, int np, T eps, const T *X, const float *RT, T *Y,
                        const unsigned long long *skip, cudaStream_t s) {
    constexpr int GMAX = 16 / static_cast<int>(sizeof(T));
    const size_t row = static_cast<size_t>(n) * sizeof(T);
    const size_t limit = 227 * 1024;
    int g = GMAX;
    while (g > 1 && row * g > limit) g >>= 1;
    if (row * g > limit) return cudaErrorInvalidValue;
    auto launch = [&](auto *kernel) -> cudaError_t {
        const size_t smem = row * g;
        const cudaError_t e = allow_all_smem(kernel);
        if (e != cudaSuccess) return e;
        kernel<<<static_cast<unsigned>(np / g), 512, smem, s>>>(ptr, col, n, np, eps, X, RT, Y, skip);
        return cudaGetLastError();
    };
    if (g == GMAX) return launch(trans_local_kernel<T, GMAX, RHS>);
    if (g == 2) return launch(trans_local_kernel<T, 2, RHS>);
    return launch(trans_local_kernel<T, 1, RHS>);
}

template <class T, bool RHS>
cudaError_t trans_gather(const int *ptr, const int *col, int n, int np, T eps, const T *Y, const float *R, const T *old,
                         T *X, unsigned long long *slots, const unsigned long long *skip, cudaStream_t s) {
    constexpr int V = 16 / static_cast<int>(sizeof(T));
    dim3 grid(static_cast<unsigned>((np / V + 255) / 256), static_cast<unsigned>(np));
    trans_gather_kernel<T, RHS><<<grid, 256, 0, s>>>(ptr, col, n, np, eps, Y, R, old, X, slots, skip);
    return cudaGetLastError();
}

}  // namespace

cudaError_t trans_relabel(const int *ptr, const int *col, int n, int *rank, int *perm, int *cnt, int *ptr2, int *col2,
                          cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(rank, 0, static_cast<size_t>(n) * sizeof(int), s);
    if (e != cudaSuccess) return e;
    const unsigned blocks = static_cast<unsigned>((n + 255) / 256);
    rank_kernel<<<dim3(blocks, static_cast<unsigned>((n + kRankPart - 1) / kRankPart)), 256, 0, s>>>(ptr, n, rank);
    relabel_counts_kernel<<<blocks, 256, 0, s>>>(ptr, rank, n, perm, cnt);
    if ((e = exclusive_scan(cnt, n, ptr2, s)) != cudaSuccess) return e;
    relabel_lists_kernel<<<static_cast<unsigned>((n + 7) / 8), 256, 0, s>>>(ptr, col, rank, perm, ptr2, n, col2);
    return cudaGetLastError();
}

cudaError_t trans_real_steps(const int *ptr, const int *col, int n, int np, double eps, double *X, double *U,
                             unsigned long long *dmax, cudaStream_t s) {
    const cudaError_t e = trans_local<double, false>(ptr, col, n, np, eps, X, nullptr, U, nullptr, s);
    if (e != cudaSuccess) return e;
    return trans_gather<double, false>(ptr, col, n, np, eps, U, nullptr, X, X, dmax, nullptr, s);
}

cudaError_t trans_correction_steps(const int *ptr, const int *col, int n, int np, double eps, const float *R,
                                   const float *RT, const float *D_in, float *D, float *E, unsigned long long *slots,
                                   const unsigned long long *skip, cudaStream_t s) {
    const float e32 = static_cast<float>(eps);
    cudaError_t e;
    if (R == nullptr) {  // the right-hand side eps R1
        if ((e = trans_local<float, false>(ptr, col, n, np, e32, D_in, nullptr, E, skip, s)) != cudaSuccess) return e;
        return trans_gather<float, false>(ptr, col, n, np, e32, E, nullptr, D_in, D, slots, skip, s);
    }
    if ((e = trans_local<float, true>(ptr, col, n, np, e32, D_in, RT, E, skip, s)) != cudaSuccess) return e;
    return trans_gather<float, true>(ptr, col, n, np, e32, E, R, D_in, D, slots, skip, s);
}

cudaError_t trans_residual(const int *ptr, const int *col, int n, int np, double eps, const double *X, double *U,
                           float *R, float *RT, unsigned long long *rmax, cudaStream_t s) {
    const cudaError_t e = trans_local<double, false>(ptr, col, n, np, eps, X, nullptr, U, nullptr, s);
    if (e != cudaSuccess) return e;
    dim3 grid(static_cast<unsigned>(np / kTT), static_cast<unsigned>(np / kTT));
    trans_residual_kernel<<<grid, dim3(kTT, 8), 0, s>>>(U, X, np, R, RT, rmax);
    return cudaGetLastError();
}

cudaError_t trans_last_step(const int *ptr, const int *col, int n, int np, double eps, const double *U, double *X,
                            unsigned long long *dmax, cudaStream_t s) {
    return trans_gather<double, false>(ptr, col, n, np, eps, U, nullptr, X, X, dmax, nullptr, s);
}

cudaError_t trans_finish(const int *rank, int n, int np, int64_t wp, const double *X, double *out, uint64_t *bits,
                         cudaStream_t s) {
    const size_t smem = static_cast<size_t>(n) * sizeof(double);
    const cudaError_t e = allow_all_smem(trans_finish_kernel);
    if (e != cudaSuccess) return e;
    trans_finish_kernel<<<static_cast<unsigned>(n), 512, smem, s>>>(rank, n, np, static_cast<int>(wp), X, out,
                                                                    reinterpret_cast<uint32_t *>(bits));
    return cudaGetLastError();
}

cudaError_t f32_to_f64(double *x, const float *d, int64_t count, cudaStream_t s) {
    f32_to_f64_kernel<<<stream_blocks(count), 256, 0, s>>>(x, d, count);
    return cudaGetLastError();
}

cudaError_t trans_real_step(const int *ptr, const int *col, int n, int np, double eps, const uint8_t *R1,
                            const double *X, double *U, double *Xn, unsigned long long *dmax, cudaStream_t s) {
    dim3 tgrid(static_cast<unsigned>((np + kTT - 1) / kTT), static_cast<unsigned>((np + kTT - 1) / kTT));
    transpose_tile_kernel<double><<<tgrid, dim3(kTT, 8), 0, s>>>(X, np, np, np, U, np);  // U = X^T
    dim3 grid(static_cast<unsigned>((np + 255) / 256), static_cast<unsigned>(np));
    sg_pu_kernel<<<grid, 256, 0, s>>>(ptr, col, n, np, eps, R1, U, X, Xn, nullptr, dmax);
    return cudaGetLastError();
}

}  // namespace dl
