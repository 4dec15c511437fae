// dl_rows.cuh -- per-row device routines shared by the single-problem and batched kernels:
// ingest of one row of a 0/1 base relation (as e4m3 or as bits), successor lists from bits,
// and one row of the certificate / recheck sweep.
#pragma once
#include <cstdint>

#include "dl_internal.h"

namespace dl {

// One CTA writes padded row `row` of the e4m3 operand (np bytes): 0x38 where the source byte
// is 1, zero elsewhere and in the padding, and 1.0 on the diagonal if add_identity.  The
// calling thread's partial row sum and "bad byte" bits are returned in sum / bad; thread 0
// sets extra = 1 if it added a diagonal one that the source lacked.
__device__ __forceinline__ void ingest_row(const uint8_t *__restrict__ src, int n, int np,
                                           uint8_t *__restrict__ dst, int add_identity, int row,
                                           uint32_t &sum, uint32_t &bad, uint32_t &extra) {
    uint8_t *drow = dst + static_cast<int64_t>(row) * np;
    if (row < n) {
        const uint8_t *srow = src + static_cast<int64_t>(row) * n;
        const bool vec = ((n & 15) == 0) && ((reinterpret_cast<uintptr_t>(src) & 15) == 0) &&
                         ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) && ((np & 15) == 0);
        if (vec) {
            const uint4 *s4 = reinterpret_cast<const uint4 *>(srow);
            uint4 *d4 = reinterpret_cast<uint4 *>(drow);
            for (int q = threadIdx.x; q < n / 16; q += blockDim.x) {
                const uint4 x = s4[q];
                const uint32_t w[4] = {x.x, x.y, x.z, x.w};
                uint32_t o[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    bad |= w[t] & 0xFEFEFEFEu;
                    sum += __popc(w[t] & 0x01010101u);
                    o[t] = (w[t] & 0x01010101u) * 0x38u;  // byte 1 -> 0x38 (e4m3 1.0)
                }
                d4[q] = make_uint4(o[0], o[1], o[2], o[3]);
            }
        } else {
            for (int j = threadIdx.x; j < n; j += blockDim.x) {
                const uint32_t b = srow[j];
                bad |= b & 0xFEu;
                sum += b & 1u;
                drow[j] = static_cast<uint8_t>((b & 1u) * 0x38u);
            }
        }
    }
    const int start = row < n ? n : 0;
    for (int j = start + threadIdx.x; j < np; j += blockDim.x) drow[j] = 0;
    __syncthreads();
    if (add_identity && threadIdx.x == 0) {
        if (row >= n || drow[row] == 0) extra = 1;
        drow[row] = 0x38;
    }
}

// Block-wide sum (of a) and OR (of b); the result is valid in thread 0.
__device__ __forceinline__ void block_reduce_sum_or(uint32_t &a, uint32_t &b) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b |= __shfl_xor_sync(0xffffffffu, b, o);
    }
    __shared__ uint32_t s_a[32], s_b[32];
    const int warps = (blockDim.x + 31) >> 5;
    if ((threadIdx.x & 31) == 0) {
        s_a[threadIdx.x >> 5] = a;
        s_b[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t ta = 0, tb = 0;
        for (int w = 0; w < warps; ++w) {
            ta += s_a[w];
            tb |= s_b[w];
        }
        a = ta;
        b = tb;
    }
}

// Warp-uniform read of a counter another warp may be incrementing.
__device__ __forceinline__ unsigned long long warp_read_u64(const unsigned long long *p) {
    unsigned long long v = (threadIdx.x & 31) == 0 ? *reinterpret_cast<const volatile unsigned long long *>(p) : 0ull;
    return __shfl_sync(0xffffffffu, v, 0);
}

// Lanes own words lane, lane+32, ... of a row (up to kSweepWpl per lane per pass; wider
// rows take several passes over the E row).
constexpr int kSweepWpl = 8;

// One warp processes row `row` of the sweep over bit matrix M (wp 64-bit words per row):
//   mode 0: out_row = OR_{k : E[row][k]} M_k;  violation iff (out_row | e_row) != M_row
//   mode 1: out_row = M_row | E_row | OR_{k : E[row][k]} M_k;  violation iff it changed
// (out may equal M in mode 1).  viol and cnt (ones in out_row) are warp-uniform on return.
__device__ __forceinline__ void sweep_row(const uint8_t *__restrict__ erow, int n, const uint64_t *M,
                                          uint64_t *out, int64_t wp, int mode, int row, int lane,
                                          bool &viol_out, uint32_t &cnt_out) {
    const uint64_t *mrow = M + static_cast<int64_t>(row) * wp;
    bool viol = false;
    uint32_t cnt = 0;
    // A row whose accumulator already holds all n columns cannot change any more: stop its
    // scan (single-pass rows only).  Most rows of a closure with a giant component are full.
    const bool single_pass = wp <= 32 * kSweepWpl;
    uint64_t full[kSweepWpl];
#pragma unroll
    for (int q = 0; q < kSweepWpl; ++q) {
        const int64_t w = lane + 32 * q;
        const int64_t lo = w * 64;
        full[q] = (w >= wp || lo >= n) ? 0ull : (n - lo >= 64 ? ~0ull : ((1ull << (n - lo)) - 1ull));
    }
    for (int64_t w0 = 0; w0 < wp; w0 += 32 * kSweepWpl) {
        uint64_t acc[kSweepWpl];
#pragma unroll
        for (int t = 0; t < kSweepWpl; ++t) acc[t] = 0;
        bool saturated = false;
        if (single_pass && mode == 1) {  // the row itself may already be full
            bool mine = true;
#pragma unroll
            for (int q = 0; q < kSweepWpl; ++q) {
                const int64_t w = lane + 32 * q;
                if (w < wp) acc[q] = mrow[w];
                mine &= acc[q] == full[q];
            }
            saturated = __all_sync(0xffffffffu, mine);
        }
        for (int c0 = 0; c0 < n && !saturated; c0 += 512) {
            // lane looks at bytes c0 + 16*lane .. +15
            uint32_t mask = 0;
            const int base = c0 + 16 * lane;
#pragma unroll
            for (int t = 0; t < 16; ++t)
                if (base + t < n && erow[base + t]) mask |= 1u << t;
            uint32_t who = __ballot_sync(0xffffffffu, mask != 0);
            while (who) {
                const int src = __ffs(who) - 1;
                who &= who - 1;
                uint32_t m = __shfl_sync(0xffffffffu, mask, src);
                while (m) {
                    const int t = __ffs(m) - 1;
                    m &= m - 1;
                    const int k = c0 + 16 * src + t;
                    const uint64_t *mk = M + static_cast<int64_t>(k) * wp;
#pragma unroll
                    for (int q = 0; q < kSweepWpl; ++q) {
                        const int64_t w = w0 + lane + 32 * q;
                        if (w < wp) acc[q] |= mk[w];
                    }
                    if (mode == 1) {  // the fact E[i][k] itself
                        const int64_t rel = (k >> 6) - w0;  // word index within this pass
                        if (rel >= 0 && rel < 32 * kSweepWpl && (rel & 31) == lane) {
                            const int qk = static_cast<int>(rel >> 5);
#pragma unroll
                            for (int q = 0; q < kSweepWpl; ++q)
                                if (q == qk) acc[q] |= 1ull << (k & 63);
                        }
                    }
                    if (single_pass) {
                        bool mine = true;
#pragma unroll
                        for (int q = 0; q < kSweepWpl; ++q) mine &= acc[q] == full[q];
                        if (__all_sync(0xffffffffu, mine)) {
                            saturated = true;
                            m = 0;
                            who = 0;
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kSweepWpl; ++q) {
            const int64_t w = w0 + lane + 32 * q;
            if (w >= wp) continue;
            const uint64_t old = mrow[w];
            uint64_t v = acc[q];
            if (mode == 0) {
                const uint64_t self = (w == (row >> 6)) ? (1ull << (row & 63)) : 0ull;
                if ((v | self) != old) viol = true;
                out[static_cast<int64_t>(row) * wp + w] = v;
            } else {
                v |= old;
                if (v != old) {
                    viol = true;
                    out[static_cast<int64_t>(row) * wp + w] = v;
                } else if (out != M) {
                    out[static_cast<int64_t>(row) * wp + w] = v;
                }
            }
            cnt += __popcll(v);
        }
    }
    viol_out = __any_sync(0xffffffffu, viol);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    cnt_out = cnt;
}

// Low bits of the four bytes of x as a 4-bit mask (byte b -> bit b).
__device__ __forceinline__ uint32_t byte_lsbs(uint32_t x) { return ((x & 0x01010101u) * 0x01020408u) >> 24; }
// Bytes of x with any of bits 1..7 set, as a 4-bit mask.
__device__ __forceinline__ uint32_t byte_bad(uint32_t x) {
    const uint32_t t = (x >> 1) & 0x7F7F7F7Fu;
    return byte_lsbs(((t + 0x7F7F7F7Fu) | t) >> 7);
}

// Sixteen bytes that are 0 or 1 as 16 bits, byte b -> bit b, in five operations: a product with a
// multiplier of four powers of two gathers a word's bytes in its top four bits (no lower sum
// carries), a second word's land above them.  Any byte that is neither 0 nor 1 is left in `bad`, and
// the bits are then of no use.
__device__ __forceinline__ uint32_t pack16(const uint4 &x, uint32_t &bad) {
    bad |= (x.x | x.y | x.z | x.w) & 0xFEFEFEFEu;
    const uint32_t lo = x.x * 0x01020408u + x.y * 0x10204080u, hi = x.z * 0x01020408u + x.w * 0x10204080u;
    return __byte_perm(lo, hi, 0x73) & 0xFFFFu;
}
// The bytes of x outside [lo, hi) cleared.
__device__ __forceinline__ uint4 keep_bytes(const uint4 &x, int lo, int hi) {
    auto word = [&](uint32_t v, int at) {
        const int a = min(4, max(0, lo - at)), b = min(4, max(0, hi - at));
        const uint32_t below_b = b == 4 ? 0xFFFFFFFFu : (1u << (8 * b)) - 1u;
        const uint32_t below_a = a == 4 ? 0xFFFFFFFFu : (1u << (8 * a)) - 1u;
        return v & below_b & ~below_a;
    };
    return make_uint4(word(x.x, 0), word(x.y, 4), word(x.z, 8), word(x.w, 12));
}

// *word |= e on shared memory, as 32-bit operations on the halves that have bits (a 64-bit one is a loop
// of compare and swap).
__device__ __forceinline__ void or_shared(uint64_t *word, uint64_t e) {
    unsigned *h = reinterpret_cast<unsigned *>(word);
    const unsigned lo = static_cast<unsigned>(e), hi = static_cast<unsigned>(e >> 32);
    if (lo != 0u) atomicOr(h, lo);
    if (hi != 0u) atomicOr(h + 1, hi);
}

// The bits of the rows [r0, r1) of an n x n 0/1 byte matrix (any alignment) by one CTA.  The rows are
// one run of bytes, so they are read as such: coalesced 16-byte pieces, eight in flight a thread, packed
// to a run of bits in `buf` (tile_words words of shared memory), from which word w of row r is read at
// its bit offset and handed to put(r, w, facts).  Bound by the read: what a row costs beyond its bytes (a
// warp to a row, pieces at the row's own misalignment) took more issue slots than the 6 operations a
// piece (1.43 GB of rows of about 1 KB: 547 us with a warp to a row, 304 us so).  A byte that is neither 0
// nor 1 sets *bad for some thread; bytes outside the matrix are cleared (only the first and the last row's
// pieces can hold any).  Ends with the CTA's threads in their put calls: no barrier behind them.
constexpr int kTileBytes = 32768;       // a tile where there are many
constexpr int kTileBytesSmall = 8192;   // and of one matrix of at most kTileSmallN rows (512 tiles at 2048)
constexpr int kTileSmallN = 4096;
constexpr int kTileRows = 64;
__host__ __device__ inline int tile_rows(int64_t n, int bytes = kTileBytes) {
    const int64_t r = n > 0 ? bytes / n : kTileRows;
    return static_cast<int>(r < 1 ? 1 : r > kTileRows ? kTileRows : r);
}
__host__ __device__ inline size_t tile_words(int64_t n, int rows) {
    return static_cast<size_t>((rows * n + 15 + 127) / 64 + 1);
}

template <class Put>
__device__ __forceinline__ void pack_tile(const uint8_t *__restrict__ E, int n, int wp, int r0, int r1, uint64_t *buf,
                                          bool *bad, Put put) {
    constexpr int kFly = 8;
    const uint8_t *a = E + static_cast<int64_t>(r0) * n;
    const int off = static_cast<int>(reinterpret_cast<uintptr_t>(a) & 15);
    const int lim = off + (r1 - r0) * n;  // the rows are the bytes [off, lim) from the aligned address below
    const uint4 *src = reinterpret_cast<const uint4 *>(a - off);
    const int pieces = (lim + 15) >> 4;
    const bool edge = r0 == 0 || r1 == n;
    uint32_t odd = 0;
    for (int p0 = threadIdx.x; p0 < pieces; p0 += kFly * blockDim.x) {
        uint4 x[kFly];
#pragma unroll
        for (int j = 0; j < kFly; ++j) {
            const int p = p0 + j * blockDim.x;
            x[j] = p < pieces ? __ldg(src + p) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int j = 0; j < kFly; ++j) {
            const int p = p0 + j * blockDim.x;
            if (p >= pieces) break;
            if (edge && (16 * p < off || 16 * p + 16 > lim)) x[j] = keep_bytes(x[j], off - 16 * p, lim - 16 * p);
            reinterpret_cast<uint16_t *>(buf)[p] = static_cast<uint16_t>(pack16(x[j], odd));
        }
    }
    *bad = odd != 0;
    __syncthreads();
    for (int t = threadIdx.x; t < (r1 - r0) * wp; t += blockDim.x) {
        const int i = t / wp, w = t - i * wp;
        const int left = n - 64 * w;  // columns from this word on
        uint64_t e = 0ull;
        if (left > 0) {
            const int at = off + i * n + 64 * w, sh = at & 63;
            e = buf[at >> 6] >> sh;
            if (sh) e |= buf[(at >> 6) + 1] << (64 - sh);
            if (left < 64) e &= (1ull << left) - 1ull;
        }
        put(r0 + i, w, e);
    }
}

// One warp writes the successor list of row r into col[pos0 .. pos1) from its packed bits
// (I + E: the identity bit belongs to E only when the row holds pos1 - pos0 ones).
__device__ __forceinline__ void fill_row_from_bits(const uint64_t *row, int wp, int r, int pos0, int pos1, int *col,
                                                   int lane) {
    int ones = 0;
    for (int w = lane; w < wp; w += 32) ones += __popcll(row[w]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ones += __shfl_xor_sync(0xffffffffu, ones, o);
    const bool self = ones == pos1 - pos0;
    int pos = pos0;
    for (int w0 = 0; w0 < wp; w0 += 32) {
        const int w = w0 + lane;
        uint64_t x = w < wp ? row[w] : 0ull;
        if (!self && w == (r >> 6)) x &= ~(1ull << (r & 63));
        const int c = __popcll(x);
        int inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        int p = pos + inc - c;
        while (x) {
            const int b = __ffsll(static_cast<long long>(x)) - 1;
            x &= x - 1;
            col[p++] = 64 * w + b;
        }
        pos += __shfl_sync(0xffffffffu, inc, 31);
    }
}

// Single-row Iteration (eq. series:trcl on one row vector x_i, x <- min1(e_i + x E) for the
// successor relation), semi-naive: one warp keeps the row's bits in shared memory (`bits`:
// wp words, then two frontiers of kRowFront ints and a counter) and expands only the nodes
// that entered x in the last step, lanes taking frontier nodes and setting their successors'
// bits with shared-memory atomicOr.  ptr/col: the CSR with column indices local to the
// problem (ptr may be offset so that ptr[k] is local row k).  When the frontier empties, x
// is the exact row i of the reflexive closure; a frontier larger than kRowFront or more than
// kRowSteps steps (long paths are left to squarings) ends the row early.  Either way the bits
// reached (all reachable from i) go to mrow; returns whether the row is exact.
constexpr int kRowFront = 256;
constexpr int kRowSteps = 64;

__device__ __forceinline__ bool iterate_row(const int *__restrict__ ptr, const int *__restrict__ col, int i, int wp,
                                            uint64_t *bits, uint64_t *mrow, int lane) {
    int *front = reinterpret_cast<int *>(bits + wp);  // two frontiers of kRowFront
    int *next_cnt = front + 2 * kRowFront;
    for (int w = lane; w < wp; w += 32) bits[w] = w == (i >> 6) ? 1ull << (i & 63) : 0ull;
    if (lane == 0) front[0] = i;
    int cur = 0, cnt = 1, steps = 0;
    bool ok = true;
    __syncwarp();
    while (cnt > 0) {
        if (++steps > kRowSteps) {
            ok = false;
            break;
        }
        if (lane == 0) *next_cnt = 0;
        __syncwarp();
        const int *fc = front + cur * kRowFront;
        int *fn = front + (cur ^ 1) * kRowFront;
        for (int f = lane; f < cnt; f += 32) {
            const int k = fc[f];
            const int q1 = ptr[k + 1];
            for (int q = ptr[k]; q < q1; ++q) {
                const int j = col[q];
                const unsigned b = 1u << (j & 31);  // (32-bit halves: a 64-bit shared atomic is a loop)
                if (!(atomicOr(reinterpret_cast<unsigned *>(bits) + (j >> 5), b) & b)) {
                    const int pos = atomicAdd(next_cnt, 1);
                    if (pos < kRowFront) fn[pos] = j;
                }
            }
        }
        __syncwarp();
        cnt = *next_cnt;
        __syncwarp();  // every lane has read the count before lane 0 clears it
        if (cnt > kRowFront) {
            ok = false;
            break;
        }
        cur ^= 1;
    }
    __syncwarp();
    for (int w = lane; w < wp; w += 32) mrow[w] = bits[w];
    return ok;
}

}  // namespace dl
