// dl_fp64.cu -- the plain FP64 route: R~ = (I - eps E)^-1 eps E (Proposition 1) by blocked
// Gaussian elimination without pivoting, all in FP64 on the CUDA cores, then threshold > 0
// (Theorem 1).
//
// A = I - eps E is strictly diagonally dominant by rows for 0 < eps <= 1/(1 + ||E||_inf)
// (proof of Proposition 1: eps ||E||_inf <= 1 - eps < 1 = a_ii - |eps e_ii| margin), and so is
// every Schur complement, so block elimination without pivoting exists and every quantity keeps
// its sign.  It runs on the augmented matrix G = [A | eps E] (np x 2np, padded rows/columns:
// identity in A, zero in eps E), in blocks of b = 32.  Per block column k:
//   1. panel:  R_k = S_kk^-1 [A_k,>k | B_k]                  (S_kk^-1: see 2)
//   2. update: [A_i,>k | B_i] -= A_ik R_k for the other block rows i (32 x 32 tiles); its first CTA
//      forms S_k+1,k+1 and its inverse meanwhile, so no step waits for a diagonal block.
// Up to kJordanNp the other rows are all rows (Gauss-Jordan: B ends as X, no backward pass; 3/2 n^3
// FMA, every step a full grid); beyond it they are the rows below (4/3 n^3 FMA), and the backward
// pass is B_i -= A_ik X_k for the rows above, k from the last.
//
// GB300 has two FP64 lanes per SM: 4/3 n^3 FMA are 2.5 ms at n = 1024 whatever the memory does, and
// what matters is that no SM idles.  The triangular solves by one thread per row or column and the
// one-CTA LU of a diagonal block that this replaced took 350-480 us per block column of 64, one
// after the other.  One call before and now: n = 300 2.9 -> 0.66 ms, 1000 10.9 -> 3.45 ms, 2048 33.8 ->
// 21.1 ms, 4096 180 -> 157 ms (the FP64 rate's floor: 155 ms).  Where the line between the two forms
// lies: Gauss-Jordan / elimination with a backward pass measured 3.45 / 3.66 ms at 1000, 6.13 / 6.12
// at 1280, 10.1 / 9.7 at 1536, 174 / 157 at 4096.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dl_internal.h"
#include "dl_ptx.cuh"

namespace dl {

namespace {

constexpr int B = 32;  // block size of the blocked elimination
constexpr int kJordanNp = 1024;  // up to here Gauss-Jordan, beyond it elimination and a backward pass

__global__ void build_kernel(const uint8_t *__restrict__ E, const uint8_t *__restrict__ A, int n, int np, double eps,
                             double *__restrict__ G, int64_t ldg) {
    const int64_t row = blockIdx.y;
    for (int64_t c = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; c < 2 * np;
         c += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double v;
        if (c < np) {
            const double e = (row < n && c < n && E[row * n + c]) ? eps : 0.0;
            v = (c == row ? 1.0 : 0.0) - e;
        } else {
            const int64_t cc = c - np;
            v = (row < n && cc < n && A[row * n + cc]) ? eps : 0.0;
        }
        G[row * ldg + c] = v;
    }
}

// G = [I - eps E | eps F] with a real right-hand side F (n x n FP64, row stride n).
__global__ void build_real_kernel(const uint8_t *__restrict__ E, const double *__restrict__ F, int n, int np,
                                  double eps, double *__restrict__ G, int64_t ldg) {
    const int64_t row = blockIdx.y;
    for (int64_t c = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; c < 2 * np;
         c += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double v;
        if (c < np) {
            const double e = (row < n && c < n && E[row * n + c]) ? eps : 0.0;
            v = (c == row ? 1.0 : 0.0) - e;
        } else {
            const int64_t cc = c - np;
            v = (row < n && cc < n) ? eps * F[row * n + cc] : 0.0;
        }
        G[row * ldg + c] = v;
    }
}

// A group of 64 threads forms a 32 x TN product tile, K = 32:  acc = A Bm with A in shared memory by
// columns (sA[k][row]) and Bm by rows (sB[k][col]); a thread holds 4 rows x TN / 8 columns.  The FP64
// units bound it whatever the tile (2 FMA per clock and SM: 8.6 us for 32 x 32 x 32 on one SM); small
// tiles keep the SMs' shares even.
constexpr int kThreads = 64;                    // of a group
constexpr int kGroups = 8;                      // of a CTA of update_kernel
constexpr int kInvThreads = 288;                // of an inverse: 8 warps of FMAs, one of reciprocals

// Barrier `id` over `threads` threads of the CTA.
__device__ __forceinline__ void group_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <int TN>
__device__ __forceinline__ void tile_product(int t, const double (*sA)[B + 2], const double (*sB)[TN],
                                             double (&acc)[4][TN / 8]) {
    const int tx = t & 7, ty = t >> 3;
#pragma unroll 8
    for (int k = 0; k < B; ++k) {
        const double2 a01 = *reinterpret_cast<const double2 *>(&sA[k][4 * ty]);
        const double2 a23 = *reinterpret_cast<const double2 *>(&sA[k][4 * ty + 2]);
        const double a[4] = {a01.x, a01.y, a23.x, a23.y};
#pragma unroll
        for (int h = 0; h < TN / 16; ++h) {
            const double2 b = *reinterpret_cast<const double2 *>(&sB[k][16 * h + 2 * tx]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[i][2 * h] = fma(a[i], b.x, acc[i][2 * h]);
                acc[i][2 * h + 1] = fma(a[i], b.y, acc[i][2 * h + 1]);
            }
        }
    }
}

// The 32 x 32 block at g into shared memory, by columns (64 threads, t of them).
__device__ __forceinline__ void load_by_columns(int t, const double *g, int64_t ldg, double (*sA)[B + 2]) {
#pragma unroll 4
    for (int q = t; q < B * B / 2; q += kThreads) {
        const int i = q / (B / 2), k = 2 * (q % (B / 2));
        const double2 v = *reinterpret_cast<const double2 *>(g + i * ldg + k);
        sA[k][i] = v.x;
        sA[k + 1][i] = v.y;
    }
}

// The 32 x TN block at g into shared memory, by rows.
template <int TN>
__device__ __forceinline__ void load_by_rows(int t, const double *g, int64_t ldg, double (*sB)[TN]) {
#pragma unroll 4
    for (int q = t; q < B * TN / 2; q += kThreads) {
        const int k = q / (TN / 2), j = 2 * (q % (TN / 2));
        *reinterpret_cast<double2 *>(&sB[k][j]) = *reinterpret_cast<const double2 *>(g + k * ldg + j);
    }
}

// In-place inverse of the 32 x 32 block S in shared memory by Gauss-Jordan without pivoting, by the
// first kInvThreads threads of the CTA (lane = column, warps 0-7 four rows each).  Every element of a
// step is one FMA, a_ij - c_i r_j with r the pivot row over the pivot, the pivot column of a replaced
// by zeros and r_k = 1 / pivot; warp 8 forms the next pivot and its reciprocal meanwhile.  512 cycles
// of FMA per step on the SM's two FP64 lanes.
__device__ void block_inverse(double (*S)[B + 1], double *recip) {
    const int j = threadIdx.x & 31, warp = threadIdx.x >> 5, i0 = 4 * warp;
    if (warp == 8 && j == 0) recip[0] = 1.0 / S[0][0];
    group_sync(1, kInvThreads);
#pragma unroll 1
    for (int k = 0; k < B; ++k) {
        const double p = recip[k & 1];
        if (warp < 8) {
            const double r = j == k ? p : S[k][j] * p;
            double c[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) c[i] = S[i0 + i][k];
            group_sync(1, kInvThreads);  // every thread has read row and column k
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double a = j == k ? 0.0 : S[i0 + i][j];
                S[i0 + i][j] = i0 + i == k ? r : fma(-c[i], r, a);
            }
        } else {
            const int m = min(k + 1, B - 1);
            const double next = fma(-S[m][k], S[k][m] * p, S[m][m]);  // the pivot as this step leaves it
            group_sync(1, kInvThreads);
            if (j == 0 && k + 1 < B) recip[(k + 1) & 1] = 1.0 / next;
        }
        group_sync(1, kInvThreads);
    }
}

// S^-1 of the diagonal block at g (the first one; the later ones are formed by update_kernel).
__global__ void __launch_bounds__(kInvThreads) first_inverse_kernel(const double *g, int64_t ldg, double *Sinv) {
    __shared__ double S[B][B + 1];
    __shared__ double recip[2];
    grid_dep_launch();
    grid_dep_wait();
    for (int t = threadIdx.x; t < B * B; t += kInvThreads) S[t / B][t % B] = g[(t / B) * ldg + t % B];
    __syncthreads();
    block_inverse(S, recip);
    for (int t = threadIdx.x; t < B * B; t += kInvThreads) Sinv[t] = S[t / B][t % B];
}

// R = S^-1 P in place for the block row at g (32 rows, 16 columns per CTA).
__global__ void __launch_bounds__(kThreads) panel_kernel(const double *__restrict__ Sinv, double *g, int64_t ldg) {
    __shared__ __align__(16) double sA[B][B + 2];
    __shared__ __align__(16) double sB[B][16];
    grid_dep_launch();
    grid_dep_wait();
    const int t = threadIdx.x;
    double *p = g + 16 * static_cast<int64_t>(blockIdx.x);
    load_by_columns(t, Sinv, B, sA);
    load_by_rows<16>(t, p, ldg, sB);
    __syncthreads();
    double acc[4][2] = {};
    tile_product<16>(t, sA, sB, acc);
    const int tx = t & 7, ty = t >> 3;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<double2 *>(p + (4 * ty + i) * ldg + 2 * tx) = make_double2(acc[i][0], acc[i][1]);
}

// Block rows [row0, row0 + rows) but k:  G_ij -= G_ik R_j for the columns from col0 (a multiple of
// 32) to the end, R = block row k, in 32 x 32 tiles.  One CTA per SM; the tiles go round the CTAs, and
// the kGroups groups of a CTA take its tiles in turn, so that a group's loads pass under the others'
// products.  With next >= 0 the first CTA instead forms diagonal block `next` as this step leaves it
// and writes its inverse (the block itself is not needed any more): alone on its SM, since its chain
// of dependent FP64 operations would queue behind every other warp's (as one CTA among 13 on an SM it
// ended 25-50 us after them).
struct UpdateSmem {
    double a[kGroups][B][B + 2];
    double b[kGroups][B][B];
    double recip[2];
    int taken, claim[kGroups];
};

__global__ void __launch_bounds__(kThreads *kGroups, 1)
    update_kernel(double *G, int64_t ldg, int k, int row0, int tiles, int64_t col0, int col_tiles, int next,
                  double *Sinv) {
    extern __shared__ __align__(16) uint8_t update_smem[];
    UpdateSmem &sm = *reinterpret_cast<UpdateSmem *>(update_smem);
    grid_dep_launch();
    const int group = threadIdx.x / kThreads, t = threadIdx.x % kThreads, tx = t & 7, ty = t >> 3;
    double (*sA)[B + 2] = sm.a[group];
    double (*sB)[B] = sm.b[group];
    const int64_t kb = static_cast<int64_t>(k) * B;
    const int workers = static_cast<int>(gridDim.x) - (next >= 0 ? 1 : 0);
    const int me = static_cast<int>(blockIdx.x) - (next >= 0 ? 1 : 0);
    if (threadIdx.x == 0) sm.taken = 0;
    __syncthreads();
    grid_dep_wait();
    if (me < 0) {
        if (threadIdx.x >= kInvThreads) return;
        const int64_t nb = static_cast<int64_t>(next) * B;
        double *C = G + nb * ldg + nb;
        double (*S)[B + 1] = reinterpret_cast<double(*)[B + 1]>(&sm.a[1][0][0]);
        if (group == 0) {
            load_by_columns(t, G + nb * ldg + kb, ldg, sA);
            load_by_rows<B>(t, G + kb * ldg + nb, ldg, sB);
            group_sync(2, kThreads);
            double acc[4][4] = {};
            tile_product<B>(t, sA, sB, acc);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int r = 4 * ty + i, c = 16 * (h >> 1) + 2 * tx + (h & 1);
                    S[r][c] = C[r * ldg + c] - acc[i][h];
                }
        }
        group_sync(1, kInvThreads);
        block_inverse(S, sm.recip);
        for (int q = threadIdx.x; q < B * B; q += kInvThreads) Sinv[q] = S[q / B][q % B];
        return;
    }
    for (;;) {
        if (t == 0) sm.claim[group] = atomicAdd(&sm.taken, 1);
        group_sync(1 + group, kThreads);  // the claim; and the last tile's operands have been read
        const int tile = me + workers * sm.claim[group];
        if (tile >= tiles) return;
        int ti = row0 + tile / col_tiles;
        if (ti >= k && row0 <= k) ++ti;  // block row k is left out
        const int64_t c0 = col0 + static_cast<int64_t>(tile % col_tiles) * B;
        const bool other = ti == next && c0 == static_cast<int64_t>(next) * B;  // the first CTA's
        double *C = G + static_cast<int64_t>(ti) * B * ldg + c0;
        if (!other) {
            load_by_columns(t, G + static_cast<int64_t>(ti) * B * ldg + kb, ldg, sA);
            load_by_rows<B>(t, G + kb * ldg + c0, ldg, sB);
        }
        group_sync(1 + group, kThreads);
        if (other) continue;
        double acc[4][4] = {};
        tile_product<B>(t, sA, sB, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                double2 *c = reinterpret_cast<double2 *>(C + (4 * ty + i) * ldg + 16 * h + 2 * tx);
                double2 v = *c;
                v.x -= acc[i][2 * h];
                v.y -= acc[i][2 * h + 1];
                *c = v;
            }
    }
}

// Threshold X > 0 into bits (and count the guard band).
// Spread the 32 bits of x to the even bit positions of a 64-bit word (bit l -> bit 2l).
__device__ __forceinline__ uint64_t spread_even(uint32_t x) {
    uint64_t v = x;
    v = (v | (v << 16)) & 0x0000FFFF0000FFFFull;
    v = (v | (v << 8)) & 0x00FF00FF00FF00FFull;
    v = (v | (v << 4)) & 0x0F0F0F0F0F0F0F0Full;
    v = (v | (v << 2)) & 0x3333333333333333ull;
    v = (v | (v << 1)) & 0x5555555555555555ull;
    return v;
}

constexpr int kThreshWords = 8;  // 64-bit words (512 columns) per warp

// A warp takes kThreshWords consecutive words of one row: every lane issues its 16-byte loads
// (columns 2 lane, 2 lane + 1 of each word) before it tests any, and the even and odd columns'
// ballots are interleaved into the word.  Rows are 16-byte aligned (ldx even).
__global__ void __launch_bounds__(256) thresh_pack_kernel(const double *__restrict__ X, int64_t ldx, int n,
                                                          double tau, uint64_t *__restrict__ bits, int64_t wp,
                                                          unsigned long long *guard) {
    const int lane = threadIdx.x & 31;
    const int64_t words = (n + 63) / 64, groups = (words + kThreshWords - 1) / kThreshWords;
    const int64_t gw = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    if (gw >= static_cast<int64_t>(n) * groups) return;
    const int64_t row = gw / groups, w0 = (gw % groups) * kThreshWords;
    const double *xr = X + row * ldx;
    double2 v[kThreshWords];
#pragma unroll
    for (int q = 0; q < kThreshWords; ++q) {
        const int64_t c = (w0 + q) * 64 + 2 * lane;
        v[q] = c + 1 < n ? __ldcs(reinterpret_cast<const double2 *>(xr + c))
                         : make_double2(c < n ? xr[c] : 0.0, 0.0);
    }
    // the comparisons on the bit patterns (doubles of one sign order like integers): on the FP64 units,
    // two lanes per SM, they took 4 times the reads' time
    constexpr long long kInf = 0x7FF0000000000000ll;
    constexpr long long kNegZero = static_cast<long long>(0x8000000000000000ull);
    constexpr long long kNegInf = static_cast<long long>(0xFFF0000000000000ull);
    const long long tau_bits = __double_as_longlong(tau);  // tau >= 0
    uint32_t gcount = 0;
#pragma unroll
    for (int q = 0; q < kThreshWords; ++q) {
        if (w0 + q >= words) break;
        const long long bx = __double_as_longlong(v[q].x), by = __double_as_longlong(v[q].y);
        const uint32_t ev = __ballot_sync(0xffffffffu, bx > 0 && bx <= kInf);
        const uint32_t od = __ballot_sync(0xffffffffu, by > 0 && by <= kInf);
        // guard band: |X| <= tau or X < 0 (-0 and NaN are neither)
        const bool gx = bx > 0 ? bx <= tau_bits : bx > kNegZero && bx <= kNegInf;
        const bool gy = by > 0 ? by <= tau_bits : by > kNegZero && by <= kNegInf;
        gcount += __popc(__ballot_sync(0xffffffffu, gx)) + __popc(__ballot_sync(0xffffffffu, gy));
        if (lane == q) bits[row * wp + w0 + q] = spread_even(ev) | (spread_even(od) << 1);
    }
    if (lane == 0 && gcount) atomicAdd(guard, static_cast<unsigned long long>(gcount));
}

}  // namespace

cudaError_t fp64_build(const uint8_t *E, const uint8_t *A, int n, int np, double eps, double *G, int64_t ldg,
                       cudaStream_t s) {
    dim3 grid(static_cast<unsigned>((2 * np + 255) / 256 < 64 ? (2 * np + 255) / 256 : 64),
              static_cast<unsigned>(np));
    build_kernel<<<grid, 256, 0, s>>>(E, A, n, np, eps, G, ldg);
    return cudaGetLastError();
}

cudaError_t fp64_build_real(const uint8_t *E, const double *F, int n, int np, double eps, double *G, int64_t ldg,
                            cudaStream_t s) {
    dim3 grid(static_cast<unsigned>((2 * np + 255) / 256 < 64 ? (2 * np + 255) / 256 : 64),
              static_cast<unsigned>(np));
    build_real_kernel<<<grid, 256, 0, s>>>(E, F, n, np, eps, G, ldg);
    return cudaGetLastError();
}

cudaError_t fp64_solve(double *G, int64_t ldg, int np, double *scratch, int *launches, cudaStream_t s) {
    cudaError_t e;
    int L = 0;
    const int nb = np / B;
    const bool jordan = np <= kJordanNp;
    auto update = [&](int k, int row0, int rows, int64_t col0, int next) -> cudaError_t {
        const int col_tiles = static_cast<int>((2 * static_cast<int64_t>(np) - col0) / B);
        const int tiles = rows * col_tiles, first = next >= 0 ? 1 : 0;
        const int grid = std::min(tiles, std::max(1, num_sms() - first)) + first;
        if (grid == 0) return cudaSuccess;
        ++L;
        return launch_programmatic(update_kernel, dim3(static_cast<unsigned>(grid)), dim3(kThreads * kGroups),
                                   sizeof(UpdateSmem), s, G, ldg, k, row0, tiles, col0, col_tiles, next, scratch);
    };
    if ((e = cudaFuncSetAttribute(update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(sizeof(UpdateSmem)))) != cudaSuccess)
        return e;
    ++L;
    if ((e = launch_programmatic(first_inverse_kernel, dim3(1), dim3(kInvThreads), 0, s, static_cast<const double *>(G),
                                 ldg, scratch)) != cudaSuccess)
        return e;
    for (int k = 0; k < nb; ++k) {
        const int64_t kb = static_cast<int64_t>(k) * B;
        const int64_t ncols = 2 * static_cast<int64_t>(np) - kb - B;  // R_k: beyond the block, and the RHS
        ++L;
        if ((e = launch_programmatic(panel_kernel, dim3(static_cast<unsigned>(ncols / 16)), dim3(kThreads), 0, s,
                                     static_cast<const double *>(scratch), G + kb * ldg + kb + B, ldg)) != cudaSuccess)
            return e;
        e = jordan ? update(k, 0, nb - 1, kb + B, k + 1 < nb ? k + 1 : -1)
                   : update(k, k + 1, nb - 1 - k, kb + B, k + 1 < nb ? k + 1 : -1);
        if (e != cudaSuccess) return e;
    }
    if (!jordan)
        for (int k = nb - 1; k > 0; --k)
            if ((e = update(k, 0, k, np, -1)) != cudaSuccess) return e;
    if (launches) *launches += L;
    return cudaSuccess;
}

cudaError_t thresh_pack_f64(const double *X, int64_t ldx, int n, int np, double tau, uint64_t *bits,
                            int64_t wp, unsigned long long *guard, cudaStream_t s) {
    (void)np;
    if (n <= 0) return cudaSuccess;
    if (ldx % 2 != 0 || (reinterpret_cast<uintptr_t>(X) & 15) != 0) return cudaErrorInvalidValue;
    const int64_t groups = ((n + 63) / 64 + kThreshWords - 1) / kThreshWords;
    const int64_t threads = static_cast<int64_t>(n) * groups * 32;
    thresh_pack_kernel<<<static_cast<unsigned>((threads + 255) / 256), 256, 0, s>>>(X, ldx, n, tau, bits, wp,
                                                                                   guard);
    return cudaGetLastError();
}

}  // namespace dl
