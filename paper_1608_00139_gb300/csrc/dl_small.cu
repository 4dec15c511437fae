// dl_small.cu -- the whole AUTO closure of a small relation (n <= 1024) in one launch: ingest, Iteration
// steps on bits, model and certificate in the shared memory of one thread-block cluster.
//
// A small closure was nineteen launches and four host reads (n = 256: 0.205 ms, of which the kernels
// themselves took 0.075): memsets, the pass over E, a scan, the successor lists, sweeps, sometimes a
// squaring, the model.  Its bit matrix is at most 128 KB, so here the rows of E and of the
// candidate M = I | E | ... are spread over the CTAs of a cluster (up to 128 rows each), a step
// reads other CTAs' rows through distributed shared memory, and a step ends with one cluster barrier.
// The result goes to pinned host memory, so the host's only wait is the stream's.
//
// Steps: M_i <- M_i | OR_{k in succ(i)} M_k in place (Sec. 7.1's Iteration; eq. series:trcl), and from
// step kIterations on, for n <= kSquareN, M_i <- M_i | OR_{k in M_i} M_k (a squaring: paths of doubled
// length), until a step changes nothing.  Either way M is then the reflexive closure: it holds I | E,
// every pair in it is a path, and it is closed under one more edge or under composition.  Larger
// relations of long paths are left to the general route, whose single-row Iteration and tensor-core
// squarings they need (a squaring here reads a row per set bit): those still changing after
// kIterations steps, or at step kProbe with most rows growing slowly, before much has been spent.
//
// One call before and now (ER, 5 facts per row): n = 64 0.215 -> 0.046 ms, 256 0.201 -> 0.058 ms, 1000
// 0.211 -> 0.074 ms, of which the kernel is 0.013 / 0.026 / 0.042 ms; at n = 2048 the steps of eight SMs
// (0.10-0.13 ms) no longer beat the launches over all of them.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dl_internal.h"
#include "dl_rows.cuh"

namespace cg = cooperative_groups;

namespace dl {

namespace {

constexpr int kSmallThreads = 1024;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kListCap = 32;     // successors of a row kept as a list; longer rows are read off their bits
constexpr int kIterations = 24;  // steps along edges before the squarings or the general route
constexpr int kSquareN = 256;
constexpr int kProbe = 4, kSlowOnes = 8;  // at step kProbe: more than n / 2 rows changing, fewer than kSlowOnes n ones
constexpr int kMaxSteps = 64;    // never reached (kIterations and one squaring per doubling); a limit all the same
constexpr int kMaxCluster = 8;
constexpr unsigned kAll = 0xffffffffu;

// Shared memory of one CTA, in this order: E's rows, M's rows (R x w words each), the lists
// (R x kListCap 16-bit entries), the row degrees (R, 16-bit), and this.
struct SmallState {
    uint64_t colmask[32];                  // columns with a fact, all CTAs
    uint64_t part[kMaxCluster][32];        // ... of each CTA
    int changed[2][kMaxCluster];           // by parity of the step: whether a CTA's rows changed
    unsigned sum[kMaxCluster][3];          // facts, ones of the model, violations
    int dmax[kMaxCluster];
    unsigned acc[3];                       // ... of this CTA
    unsigned probe[kMaxCluster][2], probe_acc[2];  // rows changing and ones at step kProbe
    int dmax_s, bad_s;                     // bad_s: written by thread 0 alone
};

// A 64-bit word of the shared memory of CTA `rank` at this CTA's address p.
template <int C>
__device__ __forceinline__ uint64_t peer_word(const uint64_t *p, unsigned rank) {
    if (C == 1) return *reinterpret_cast<const volatile uint64_t *>(p);
    uint64_t v;
    asm volatile(
        "{\n\t.reg .u32 a;\n\t"
        "mapa.shared::cluster.u32 a, %1, %2;\n\t"
        "ld.shared::cluster.u64 %0, [a];\n\t}"
        : "=l"(v)
        : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank)
        : "memory");
    return v;
}

template <int C>
__device__ __forceinline__ void cluster_barrier() {
    if (C == 1) __syncthreads();
    else cg::this_cluster().sync();
}

// The 16 columns 16 q .. + 16 of a row of E bytes: their low bits, and *bad for other bytes.  Any
// alignment: the one or two aligned 16-byte chunks that hold them (no other chunk is touched).
__device__ __forceinline__ uint32_t pack16_at(const uint8_t *row, int n, int q, bool *bad) {
    const int c0 = 16 * q;
    if (c0 >= n) return 0u;
    const int m = min(16, n - c0);  // columns that exist
    const uint8_t *a = row + c0;
    const int off = static_cast<int>(reinterpret_cast<uintptr_t>(a) & 15);
    const uint4 x = *reinterpret_cast<const uint4 *>(a - off);
    uint4 y = make_uint4(0u, 0u, 0u, 0u);
    if (off + m > 16) y = *reinterpret_cast<const uint4 *>(a - off + 16);
    const uint32_t ones = (byte_lsbs(x.x) | (byte_lsbs(x.y) << 4) | (byte_lsbs(x.z) << 8) | (byte_lsbs(x.w) << 12)) |
                          ((byte_lsbs(y.x) | (byte_lsbs(y.y) << 4) | (byte_lsbs(y.z) << 8) | (byte_lsbs(y.w) << 12))
                           << 16);
    const uint32_t odd = (byte_bad(x.x) | (byte_bad(x.y) << 4) | (byte_bad(x.z) << 8) | (byte_bad(x.w) << 12)) |
                         ((byte_bad(y.x) | (byte_bad(y.y) << 4) | (byte_bad(y.z) << 8) | (byte_bad(y.w) << 12)) << 16);
    const uint32_t valid = (m == 16 ? 0xFFFFu : (1u << m) - 1u);
    *bad |= ((odd >> off) & valid) != 0u;
    return (ones >> off) & valid;
}

// C CTAs of a cluster, R = 1 << logR rows each, G lanes per row (G >= w words, a power of two).
template <int C>
__global__ void __launch_bounds__(kSmallThreads)
    closure_small_kernel(const uint8_t *__restrict__ E, const uint64_t *__restrict__ Eb, int n, int w, int logR, int G,
                         uint64_t *__restrict__ out, SmallClosure *result) {
    extern __shared__ __align__(16) uint8_t small_smem[];
    const int R = 1 << logR;
    uint64_t *Es = reinterpret_cast<uint64_t *>(small_smem);
    uint64_t *Ms = Es + R * w;
    uint16_t *list = reinterpret_cast<uint16_t *>(Ms + R * w);
    uint16_t *deg = list + R * kListCap;
    SmallState &st = *reinterpret_cast<SmallState *>(deg + R);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned me = C == 1 ? 0u : cg::this_cluster().block_rank();
    const int row0 = static_cast<int>(me) << logR;
    const int rows = max(0, min(R, n - row0));
    if (tid < 32) st.colmask[tid] = 0ull;
    if (tid < 3) st.acc[tid] = 0u;
    if (tid < 2) st.probe_acc[tid] = 0u;
    if (tid == 0) st.dmax_s = 0;
    bool bad = false;
    uint32_t bad_kind = 0;
    // ---- the rows of E as bits ---------------------------------------------------------------
    if (Eb == nullptr) {
        uint16_t *e16 = reinterpret_cast<uint16_t *>(Es);
        const int items = rows * 4 * w;
        for (int t0 = tid; t0 < items; t0 += 4 * kSmallThreads) {  // four loads in flight
            uint32_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = t0 + u * kSmallThreads;
                v[u] = t < items ? pack16_at(E + static_cast<int64_t>(row0 + t / (4 * w)) * n, n, t % (4 * w), &bad) : 0u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = t0 + u * kSmallThreads;
                if (t < items) e16[t] = static_cast<uint16_t>(v[u]);
            }
        }
        bad_kind = ST_BAD_INPUT;
    } else {
        const uint64_t last = (n & 63) ? (1ull << (n & 63)) - 1ull : ~0ull;
        for (int t = tid; t < rows * w; t += kSmallThreads) {
            uint64_t e = Eb[static_cast<int64_t>(row0) * w + t];
            if (t % w == w - 1) {
                bad |= (e & ~last) != 0ull;
                e &= last;
            }
            Es[t] = e;
        }
        bad_kind = ST_BAD_PAD;
    }
    // (the flag has one writer: a store of every thread that met a bad byte would race with its zeroing)
    const int any_bad = __syncthreads_or(bad);
    if (tid == 0) st.bad_s = any_bad ? static_cast<int>(bad_kind) : 0;
    // ---- M = I | E, the successor lists, the columns with a fact --------------------------------
    const int grp = lane / G, lw = lane % G, per_warp = 32 / G;
    const unsigned gmask = G == 32 ? kAll : ((1u << G) - 1u) << (grp * G);
    const bool has = lw < w;
    uint64_t cm = 0ull;
    unsigned facts = 0;
    int dmax = 0;
    for (int r0 = warp * per_warp; r0 < rows; r0 += kSmallWarps * per_warp) {
        const int r = r0 + grp;
        const uint64_t e = has && r < rows ? Es[r * w + lw] : 0ull;
        const int i = row0 + r;
        if (has && r < rows) Ms[r * w + lw] = e | (lw == (i >> 6) ? 1ull << (i & 63) : 0ull);
        cm |= e;
        const int c = __popcll(e);
        int inc = c;  // inclusive scan over the row's lanes
        for (int o = 1; o < G; o <<= 1) {
            const int v = __shfl_up_sync(kAll, inc, o, G);
            if (lw >= o) inc += v;
        }
        const int d = __shfl_sync(kAll, inc, G - 1, G);
        if (r < rows) {
            int at = inc - c;
            for (uint64_t x = e; x != 0ull && at < kListCap; x &= x - 1)
                list[r * kListCap + at++] = static_cast<uint16_t>(64 * lw + __ffsll(static_cast<long long>(x)) - 1);
            if (lw == 0) {
                deg[r] = static_cast<uint16_t>(d);
                facts += d;
                dmax = max(dmax, d);
            }
        }
    }
    // one vote of a warp, then 32-bit atomics (a 64-bit one on shared memory is a loop of compare and swap,
    // and 1024 threads in it took longer than everything else)
    for (int o = G; o < 32; o <<= 1) cm |= __shfl_xor_sync(kAll, cm, o);
    facts = __reduce_add_sync(kAll, facts);
    dmax = __reduce_max_sync(kAll, dmax);
    if (grp == 0 && has && cm != 0ull) {
        unsigned *m = reinterpret_cast<unsigned *>(&st.colmask[lw]);
        const unsigned lo = static_cast<unsigned>(cm), hi = static_cast<unsigned>(cm >> 32);
        if (lo) atomicOr(m, lo);
        if (hi) atomicOr(m + 1, hi);
    }
    if (lane == 0 && facts) {
        atomicAdd(&st.acc[0], facts);
        atomicMax(&st.dmax_s, dmax);
    }
    cluster_barrier<C>();  // every CTA of the cluster is running: its shared memory may be written
    if (C > 1) {  // every CTA's part of the column mask and its bad-input flag to every CTA
        for (int t = tid; t < 32 * C; t += kSmallThreads) {
            SmallState *peer = cg::this_cluster().map_shared_rank(&st, t >> 5);
            peer->part[me][t & 31] = st.colmask[t & 31];
            if ((t & 31) == 0) peer->changed[0][me] = st.bad_s;
        }
        cluster_barrier<C>();
        if (tid < 32) {
            uint64_t m = 0ull;
            for (int c = 0; c < C; ++c) m |= st.part[c][tid];
            st.colmask[tid] = m;
        }
        if (tid == 0)
            for (int c = 0; c < C; ++c) st.bad_s |= st.changed[0][c];
        cluster_barrier<C>();  // (also: changed[0] may be written again)
    }
    const int bad_all = st.bad_s;
    // ---- steps until one changes nothing --------------------------------------------------------
    int steps = 0, squarings = 0;
    bool open = false;  // left to the general route
    const uint64_t cmw = has ? st.colmask[lw] : 0ull;
    // OR of the rows of M named by a row's list (or by the bits `from` when it has none) into acc; stops
    // when the group's row holds all it can.
    auto word_of = [&](int k) { return peer_word<C>(Ms + (k & (R - 1)) * w + lw, static_cast<unsigned>(k >> logR)); };
    auto gather = [&](bool live, int r, int d, bool listed, uint64_t from, uint64_t full, uint64_t acc) {
        if (__any_sync(kAll, live && listed && d > 0)) {
            const int dl = live && listed ? d : 0;
            bool room = true;
            for (int t = 0; __any_sync(kAll, room && t < dl); t += 4) {
                const bool go = room && t < dl;
                uint64_t v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = go && has && t + u < dl ? word_of(list[r * kListCap + t + u]) : 0ull;
                acc |= (v[0] | v[1]) | (v[2] | v[3]);
                const unsigned covered = __ballot_sync(kAll, acc == full);  // (every lane takes part in every vote)
                if ((covered & gmask) == gmask) room = false;
            }
        }
        if (__any_sync(kAll, live && !listed)) {
            uint64_t left = live && !listed && has ? from : 0ull;  // this lane's word of names still to take
            for (;;) {
                const unsigned nz = __ballot_sync(kAll, left != 0ull);
                if (nz == 0u) break;
                const unsigned gz = nz & gmask;
                const int src = gz != 0u ? __ffs(gz) - 1 : lane;
                uint64_t x = __shfl_sync(kAll, left, src);
                if (gz == 0u) x = 0ull;
                const int base = 64 * (src % G);
                uint64_t v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {  // up to four names of that word
                    v[u] = 0ull;
                    if (x != 0ull) {
                        const int k = base + __ffsll(static_cast<long long>(x)) - 1;
                        x &= x - 1;
                        if (has) v[u] = word_of(k);
                    }
                }
                if (lane == src && gz != 0u) left = x;
                acc |= (v[0] | v[1]) | (v[2] | v[3]);
                const unsigned covered = __ballot_sync(kAll, acc == full);
                if ((covered & gmask) == gmask) left = 0ull;  // the row is full
            }
        }
        return acc;
    };
    for (bool more = bad_all == 0; more && steps < kMaxSteps;) {
        const bool square = steps >= kIterations;
        const bool probe = C > 1 && n > kSquareN && steps + 1 == kProbe;
        bool changed = false;
        unsigned rows_changed = 0, ones_now = 0;
        for (int r0 = warp * per_warp; r0 < rows; r0 += kSmallWarps * per_warp) {
            const int r = r0 + grp, i = row0 + r;
            const bool in = r < rows;
            const uint64_t before = has && in ? Ms[r * w + lw] : 0ull;
            const uint64_t full = cmw | (has && in && lw == (i >> 6) ? 1ull << (i & 63) : 0ull);
            const unsigned covered = __ballot_sync(kAll, before == full);
            const bool live = in && (covered & gmask) != gmask;
            const int d = in ? deg[r] : 0;
            const bool listed = !square && d <= kListCap;
            const uint64_t from = square ? before : (has && in ? Es[r * w + lw] : 0ull);
            const uint64_t acc = gather(live, r, d, listed, from, live ? full : before, before);
            if (live && has && acc != before) {
                *reinterpret_cast<volatile uint64_t *>(Ms + r * w + lw) = acc;
                changed = true;
            }
            if (probe) {
                const unsigned diff = __ballot_sync(kAll, acc != before);
                rows_changed += lw == 0 && (diff & gmask) != 0u;
                ones_now += __popcll(acc);
            }
        }
        if (probe) {
            rows_changed = __reduce_add_sync(kAll, rows_changed);
            ones_now = __reduce_add_sync(kAll, ones_now);
            if (lane == 0) {
                atomicAdd(&st.probe_acc[0], rows_changed);
                atomicAdd(&st.probe_acc[1], ones_now);
            }
        }
        ++steps;
        squarings += square;
        const int any = __syncthreads_or(changed);
        if (C == 1) {
            more = any != 0;
        } else {
            if (tid < C) {
                SmallState *peer = cg::this_cluster().map_shared_rank(&st, tid);
                peer->changed[steps & 1][me] = any;
                if (probe) peer->probe[me][0] = st.probe_acc[0], peer->probe[me][1] = st.probe_acc[1];
            }
            cluster_barrier<C>();
            int all = 0;
            for (int c = 0; c < C; ++c) all |= st.changed[steps & 1][c];
            more = all != 0;
            if (probe) {
                unsigned moving = 0, ones = 0;
                for (int c = 0; c < C; ++c) moving += st.probe[c][0], ones += st.probe[c][1];
                open = more && moving > static_cast<unsigned>(n / 2) && ones < static_cast<unsigned>(kSlowOnes * n);
            }
        }
        open |= more && n > kSquareN && steps >= kIterations;
        if (open) break;
    }
    // ---- the model E M, its ones, and the certificate M = I | E M -------------------------------
    unsigned ones = 0, viol = 0;
    if (bad_all == 0 && !open) {
        for (int r0 = warp * per_warp; r0 < rows; r0 += kSmallWarps * per_warp) {
            const int r = r0 + grp, i = row0 + r;
            const bool in = r < rows;
            const int d = in ? deg[r] : 0;
            const uint64_t v = gather(in, r, d, d <= kListCap, has && in ? Es[r * w + lw] : 0ull, cmw, 0ull);
            if (in && has) {
                const uint64_t self = lw == (i >> 6) ? 1ull << (i & 63) : 0ull;
                viol += (v | self) != Ms[r * w + lw];
                ones += __popcll(v);
                out[static_cast<int64_t>(i) * w + lw] = v;
            }
        }
    }
    ones = __reduce_add_sync(kAll, ones);
    viol = __reduce_add_sync(kAll, viol);
    if (lane == 0 && ones) atomicAdd(&st.acc[1], ones);
    if (lane == 0 && viol) atomicAdd(&st.acc[2], viol);
    __syncthreads();
    if (tid == 0) {
        SmallState *root = C == 1 ? &st : cg::this_cluster().map_shared_rank(&st, 0);
        for (int q = 0; q < 3; ++q) root->sum[me][q] = st.acc[q];
        root->dmax[me] = st.dmax_s;
    }
    cluster_barrier<C>();  // no CTA leaves while another reads its rows
    if (me == 0 && tid == 0) {
        unsigned s[3] = {0, 0, 0};
        int dm = 0;
        for (int c = 0; c < C; ++c) {
            for (int q = 0; q < 3; ++q) s[q] += st.sum[c][q];
            dm = max(dm, st.dmax[c]);
        }
        result->nnz = s[0];
        result->ones = s[1];
        result->violations = s[2];
        result->dmax = dm;
        result->status = bad_all;
        result->steps = steps;
        result->squarings = squarings;
        result->open = open ? 1 : 0;
        __threadfence_system();
    }
}

// (within the 48 KB that every kernel may have: no limit to raise)
static_assert(2 * 128 * 16 * 8 + 128 * (kListCap + 1) * 2 + sizeof(SmallState) + 16 <= 48 * 1024, "n = 1024: R = 128, w = 16");

template <int C>
cudaError_t launch_small(const uint8_t *E, const uint64_t *Eb, int n, int logR, uint64_t *out, SmallClosure *result,
                         cudaStream_t s) {
    const int w = (n + 63) / 64, R = 1 << logR;
    int G = 1;
    while (G < w) G <<= 1;
    const size_t smem = static_cast<size_t>(2 * R * w) * 8 + static_cast<size_t>(R) * (kListCap + 1) * 2 +
                        sizeof(SmallState) + 16;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, closure_small_kernel<C>, E, Eb, n, w, logR, G, out, result);
}

}  // namespace

bool closure_small_fits(int n) { return n > 0 && n <= 1024; }

cudaError_t closure_small(const uint8_t *E, const uint64_t *Eb, int n, uint64_t *out, SmallClosure *result,
                          cudaStream_t s) {
    // CTAs and rows per CTA: more CTAs share the ingest and the steps, one needs no cluster barrier
    if (n <= 128) return launch_small<1>(E, Eb, n, 7, out, result, s);
    if (n <= 512) return launch_small<4>(E, Eb, n, 7, out, result, s);
    return launch_small<8>(E, Eb, n, 7, out, result, s);
}

}  // namespace dl
