// Bit-packed kernels: rows of R are uint64 bit codes (paper Sec. 3.2, bit j
// of row i = R_ij, least significant bit first).
//
//  * product_m4rm / product_gather  one Boolean product on bitsets,
//                 C_i = OR_{k : A_ik = 1} B_k, optionally OR-ed with A_i; with
//                 A = B = R that is one squaring step of Eq. 4:
//                 C_i = R_i | OR_{k : R_ik = 1} R_k. Dense words: tiles of 256
//                 rows x 1,024 columns, per word of A 16 shared-memory tables
//                 of the ORs of 4 rows of B (Four Russians), one lookup per
//                 nibble; few bits per word: one warp per row gathers the
//                 named rows of B.
//  * wcsr_build   the nonzero words of every row (word index + value), so
//                 that frontier expansion touches only words that hold bits.
//  * smp_packed   the selective product of Eq. 5 / Algorithm 2 per query row:
//                 D = v; V = 0; repeat N = (OR_{k in D} R_k) & ~V; V |= N;
//                 D = N until D is empty; out = V = v R+.
//                 One warp per query row, frontier and next bitsets in shared
//                 memory, the visited set in the query's output row, all
//                 frontier levels of a query in one launch
//                 (queries are independent, so no grid-wide step is needed;
//                 a warp takes the next query from a global counter when its
//                 query has converged).
//  * indexed_rows P + A B through the word indexes of A and B: the sparse first
//                 squarings of a closure (A = B = P), a sparse composition's product.
//  * smp_rows     Algorithm 2 for a few query rows straight from R's rows, one
//                 thread-block cluster per row.
//  * smp_sliced   Algorithm 2 for 64 sources at once, bit-sliced, for relations
//                 too large for the tile form of frontier.cu.
//  * insert_fact  one new fact into a transitive closure (rank-1 update).
#include <algorithm>
#include <atomic>

#include "internal.h"
#include "ptx.cuh"

namespace bmlp {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

__device__ __forceinline__ void or4(uint4& a, const uint4& b) {
    a.x |= b.x;
    a.y |= b.y;
    a.z |= b.z;
    a.w |= b.w;
}

// Ones and nonzero words of two output words (a uint4), and a block's totals added into pstat[0] / pstat[1]
// (called by every thread of the block: one pair of atomics per block, since all blocks add to the same two words).
__device__ __forceinline__ void count_words(const uint4& v, unsigned long long& ones, unsigned long long& words) {
    ones += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
    words += ((v.x | v.y) != 0u ? 1u : 0u) + ((v.z | v.w) != 0u ? 1u : 0u);
}
__device__ __forceinline__ void block_add_counts(unsigned long long* pstat, unsigned long long ones,
                                                 unsigned long long words) {
    __shared__ unsigned long long part[2][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ones += __shfl_xor_sync(FULL, ones, off);
        words += __shfl_xor_sync(FULL, words, off);
    }
    if (lane == 0) {
        part[0][warp] = ones;
        part[1][warp] = words;
    }
    __syncthreads();
    if (warp == 0) {
        const int nw = static_cast<int>(blockDim.x >> 5);
        ones = lane < nw ? part[0][lane] : 0ull;
        words = lane < nw ? part[1][lane] : 0ull;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            ones += __shfl_xor_sync(FULL, ones, off);
            words += __shfl_xor_sync(FULL, words, off);
        }
        if (lane == 0 && (ones | words) != 0ull) {
            atomicAdd(pstat, ones);
            atomicAdd(pstat + 1, words);
        }
    }
}

// ---- one Boolean product on bit rows by gathering the named rows
// C_i = (A_i if or_a) OR (OR over the set bits k of A_i of B_k): one warp per row i; the set bits of A_i are found
// with warp ballots and find-first-set, and row k is ORed in with coalesced 128-bit loads (two rows in flight).
// Its work is nnz(A_i) rows of B per row: the form for rows with few bits per nonzero word.
template <int VEC>
__global__ void __launch_bounds__(256) product_gather_kernel(const uint64_t* __restrict__ A, const uint64_t* __restrict__ B,
                                                             uint64_t* __restrict__ dst, int64_t n, int64_t ldw, int or_a,
                                                             int* changed, Deadline dl,
                                                             unsigned long long* __restrict__ pstat) {
    const int lane = threadIdx.x & 31;
    const int64_t warp_id = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const int64_t chunk_words = 64 * VEC;  // 32 lanes x VEC x 2 words
    uint32_t any = 0;
    unsigned long long ones = 0, words = 0;  // of the rows written
    for (int64_t i = warp_id; i < n; i += nwarps) {
        if (dl.budget_ns && __shfl_sync(FULL, lane == 0 ? static_cast<int>(dl.past()) : 0, 0)) break;
        const uint64_t* arow = A + i * ldw;
        for (int64_t c0 = 0; c0 < ldw; c0 += chunk_words) {
            uint4 acc[VEC];
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                const int64_t w = c0 + 2 * (lane + 32 * v);
                acc[v] = (or_a && w < ldw) ? *reinterpret_cast<const uint4*>(arow + w) : make_uint4(0, 0, 0, 0);
            }
            for (int64_t wb = 0; wb < ldw; wb += 32) {
                const uint64_t aw = (wb + lane < ldw) ? arow[wb + lane] : 0ull;
                unsigned m = __ballot_sync(FULL, aw != 0ull);
                while (m) {
                    const int sl = __ffs(m) - 1;
                    m &= m - 1;
                    uint64_t bits = __shfl_sync(FULL, aw, sl);
                    const int64_t kbase = (wb + sl) * 64;
                    while (bits) {
                        const int b0 = __ffsll(static_cast<long long>(bits)) - 1;
                        bits &= bits - 1;
                        int b1 = -1;
                        if (bits) {
                            b1 = __ffsll(static_cast<long long>(bits)) - 1;
                            bits &= bits - 1;
                        }
                        const uint64_t* r0 = B + (kbase + b0) * ldw + c0;
                        const uint64_t* r1 = B + (kbase + (b1 < 0 ? b0 : b1)) * ldw + c0;
                        uint4 x0[VEC], x1[VEC];
#pragma unroll
                        for (int v = 0; v < VEC; ++v) {
                            const int64_t w = 2 * (lane + 32 * v);
                            if (c0 + w < ldw) {
                                x0[v] = __ldg(reinterpret_cast<const uint4*>(r0 + w));
                                x1[v] = __ldg(reinterpret_cast<const uint4*>(r1 + w));
                            } else {
                                x0[v] = make_uint4(0, 0, 0, 0);
                                x1[v] = x0[v];
                            }
                        }
#pragma unroll
                        for (int v = 0; v < VEC; ++v) {
                            or4(acc[v], x0[v]);
                            or4(acc[v], x1[v]);
                        }
                    }
                }
            }
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                const int64_t w = c0 + 2 * (lane + 32 * v);
                if (w < ldw) {
                    const uint4 o = *reinterpret_cast<const uint4*>(arow + w);  // A_i: the squaring's old row
                    any |= (o.x ^ acc[v].x) | (o.y ^ acc[v].y) | (o.z ^ acc[v].z) | (o.w ^ acc[v].w);
                    *reinterpret_cast<uint4*>(dst + i * ldw + w) = acc[v];
                    if (pstat != nullptr) count_words(acc[v], ones, words);
                }
            }
        }
    }
    if (__any_sync(FULL, any != 0) && lane == 0) atomicOr(changed, 1);
    if (pstat != nullptr) block_add_counts(pstat, ones, words);
}

// ---- one Boolean product on bit rows by the method of Four Russians (Arlazarov, Dinic, Kronrod, Faradzev 1970)
// C_i = (A_i if or_a) OR (OR over the set bits k of A_i of B_k). A CTA owns a tile of kM4Rows rows and kM4Cols
// words (64 kM4Cols columns) of C and walks k one word of A (64 values of k) at a time. For each nibble h of that
// word it tabulates, in shared memory, the 16 ORs of the four B rows 64 kw + 4 h .. 64 kw + 4 h + 3 over the tile's
// columns; a row then ORs in one table entry per nibble of each nonzero word of A_i instead of one B row per set
// bit. So an output word costs at most n / 4 shared-memory reads however dense A is, where gathering the named
// rows costs nnz(A_i) reads of B through L2. Every nibble of a nonzero word is looked up, zero or not (measured
// faster than testing each: the loads issue back to back). The tables are double buffered (one barrier per word
// of A), and the B words of the next table are loaded while the current one is read.
// Thread layouts: a table is built by thread (h = tid / 16, column word c = tid % 16), entry x at T[h][x][c]; a
// lookup thread owns row slot r = tid / 8 (rows r, r + 32, ..., r + 224 of the tile) and the column words
// 2 (tid % 8), 2 (tid % 8) + 1, so each row slot reads one whole 128-byte entry per lookup (no bank conflicts).
constexpr int kM4Threads = 256;
constexpr int kM4Cols = 16;
constexpr int kM4Rows = 256;
constexpr int kM4RowsPerThread = kM4Rows / (kM4Threads / 8);
constexpr int kM4TableWords = 16 * 16 * kM4Cols;  // one buffer: 16 nibbles x 16 values x kM4Cols words (32 KiB)
constexpr size_t kM4Smem = 2 * kM4TableWords * sizeof(uint64_t);

__global__ void __launch_bounds__(kM4Threads, 2) product_m4rm_kernel(const uint64_t* __restrict__ A,
                                                                     const uint64_t* __restrict__ B,
                                                                     uint64_t* __restrict__ dst, int64_t n,
                                                                     int64_t ldw, int or_a, int* changed, Deadline dl,
                                                                     unsigned long long* __restrict__ pstat) {
    extern __shared__ __align__(16) uint64_t m4t[];
    const int tid = threadIdx.x;
    const int64_t nch = (ldw + kM4Cols - 1) / kM4Cols;
    const int64_t row0 = (static_cast<int64_t>(blockIdx.x) / nch) * kM4Rows;
    const int64_t c0 = (static_cast<int64_t>(blockIdx.x) % nch) * kM4Cols;
    const int64_t kwn = (n + 63) >> 6;  // words of A that hold columns < n
    // table building: B words of column c0 + bc for rows 64 kw + 4 bh + q
    const int bh = tid >> 4, bc = tid & 15;
    const bool bcol = c0 + bc < ldw;
    auto load_b = [&](int64_t kw, uint64_t (&b)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t k = kw * 64 + bh * 4 + q;
            b[q] = (bcol && k < n) ? B[k * ldw + c0 + bc] : 0ull;
        }
    };
    auto build = [&](int buf, const uint64_t (&b)[4]) {
        uint64_t* t = m4t + buf * kM4TableWords + bh * 16 * kM4Cols + bc;
        const uint64_t e3 = b[0] | b[1], e5 = b[2] | b[0], e6 = b[2] | b[1], e7 = b[2] | e3;
        t[0 * kM4Cols] = 0ull;
        t[1 * kM4Cols] = b[0];
        t[2 * kM4Cols] = b[1];
        t[3 * kM4Cols] = e3;
        t[4 * kM4Cols] = b[2];
        t[5 * kM4Cols] = e5;
        t[6 * kM4Cols] = e6;
        t[7 * kM4Cols] = e7;
        t[8 * kM4Cols] = b[3];
        t[9 * kM4Cols] = b[3] | b[0];
        t[10 * kM4Cols] = b[3] | b[1];
        t[11 * kM4Cols] = b[3] | e3;
        t[12 * kM4Cols] = b[3] | b[2];
        t[13 * kM4Cols] = b[3] | e5;
        t[14 * kM4Cols] = b[3] | e6;
        t[15 * kM4Cols] = b[3] | e7;
    };
    // lookups: rows row0 + lr + 32 j, words c0 + 2 lc, c0 + 2 lc + 1
    const int lr = tid >> 3, lc = tid & 7;
    const int64_t wcol = c0 + 2 * lc;  // ldw is even, so wcol < ldw covers both words
    uint4 acc[kM4RowsPerThread];
#pragma unroll
    for (int j = 0; j < kM4RowsPerThread; ++j) {
        const int64_t i = row0 + lr + 32 * j;
        acc[j] = (or_a && i < n && wcol < ldw) ? *reinterpret_cast<const uint4*>(A + i * ldw + wcol)
                                               : make_uint4(0, 0, 0, 0);
    }
    uint64_t bq[4];
    if (kwn > 0) {
        load_b(0, bq);
        build(0, bq);
    }
    for (int64_t kw = 0; kw < kwn; ++kw) {
        int stop = 0;
        if (tid == 0 && dl.budget_ns && (kw & 63) == 0) stop = dl.past() ? 1 : 0;
        // table kw is complete, and every thread is done with table kw - 1, whose buffer the next build reuses
        if (__syncthreads_or(stop)) return;
        if (kw + 1 < kwn) load_b(kw + 1, bq);
        uint64_t aw[kM4RowsPerThread];
#pragma unroll
        for (int j = 0; j < kM4RowsPerThread; ++j) {
            const int64_t i = row0 + lr + 32 * j;
            aw[j] = i < n ? A[i * ldw + kw] : 0ull;
        }
        const char* tb = reinterpret_cast<const char*>(m4t + (kw & 1) * kM4TableWords) + lc * 16;
#pragma unroll
        for (int j = 0; j < kM4RowsPerThread; ++j) {
            if (aw[j] == 0ull) continue;
#pragma unroll
            for (int h = 0; h < 16; ++h) {
                const uint32_t half = h < 8 ? static_cast<uint32_t>(aw[j]) : static_cast<uint32_t>(aw[j] >> 32);
                const uint32_t x = (half >> (4 * (h & 7))) & 15u;  // entry 0 is zero: no test needed
                const uint4 v = *reinterpret_cast<const uint4*>(tb + (h * 16 + x) * (kM4Cols * 8));
                acc[j].x |= v.x;
                acc[j].y |= v.y;
                acc[j].z |= v.z;
                acc[j].w |= v.w;
            }
        }
        if (kw + 1 < kwn) build(static_cast<int>((kw + 1) & 1), bq);
    }
    uint32_t any = 0;
    unsigned long long ones = 0, words = 0;
#pragma unroll
    for (int j = 0; j < kM4RowsPerThread; ++j) {
        const int64_t i = row0 + lr + 32 * j;
        if (i < n && wcol < ldw) {
            const uint4 o = *reinterpret_cast<const uint4*>(A + i * ldw + wcol);  // A_i: the squaring's old row
            any |= (o.x ^ acc[j].x) | (o.y ^ acc[j].y) | (o.z ^ acc[j].z) | (o.w ^ acc[j].w);
            *reinterpret_cast<uint4*>(dst + i * ldw + wcol) = acc[j];
            if (pstat != nullptr) count_words(acc[j], ones, words);
        }
    }
    if (__any_sync(FULL, any != 0) && (tid & 31) == 0) atomicOr(changed, 1);
    if (pstat != nullptr) block_add_counts(pstat, ones, words);
}

// ---- word-CSR of packed rows
// Entries of row k of a word index: [x, y).
__device__ __forceinline__ longlong2 wcsr_row(const int64_t* __restrict__ wptr, int64_t k) {
    return *reinterpret_cast<const longlong2*>(wptr + 2 * k);
}

// The word index of P in one launch: a warp per row, eight rows per block and step. A pass over the row's words keeps
// only which of them are nonzero (bit k of a lane's mask: word 32 k + lane of a chunk of 1,024); the counts give the
// row's place among the block's eight, whose entries start where the running total ptr[2 n] stood (zero beforehand, as
// ptr[2 n + 1], which receives the largest row's count). The nonzero words are then read again, from L2, and written in
// order. The ranges of the steps lie in the order in which the blocks came: every reader goes by a row's own range, so
// no prefix over all rows is needed. Bound by HBM, one read of P. Counts, a prefix over them and a second whole read of P
// took four launches and 62 us at n = 32,768 (134 MB), 24 us at 14,541, 183 us at 65,536; this kernel 47, 9 and 99 us
// (5.2 TB/s). Holding the rows in registers between the two passes was slower (203 us at 65,536: two blocks per SM),
// and a fixed place for every eight rows instead of the running total did not help that form (220 us).
constexpr int kIndexChunk = 1024;  // words whose nonzero mask a lane holds

__device__ __forceinline__ uint32_t wcsr_mask(const uint64_t* __restrict__ row, int64_t c0, int64_t wpr, uint64_t last,
                                              int lane) {
    uint32_t nz = 0;
    for (int k0 = 0; k0 < 32 && c0 + 32 * k0 < wpr; k0 += 8) {  // eight loads in flight per lane
        uint64_t v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int64_t x = c0 + 32 * (k0 + q) + lane;
            v[q] = x < wpr ? row[x] : 0ull;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (c0 + 32 * (k0 + q) + lane == wpr - 1) v[q] &= last;
            nz |= (v[q] != 0ull ? 1u : 0u) << (k0 + q);
        }
    }
    return nz;
}

__device__ __forceinline__ void wcsr_build_rows(const uint64_t* __restrict__ P, int64_t n, int64_t ldw,
                                                int64_t* __restrict__ wptr, int32_t* __restrict__ widx,
                                                uint64_t* __restrict__ wval, int64_t block, int64_t blocks) {
    __shared__ int s_cnt[8];
    __shared__ unsigned long long s_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int64_t wpr = (n + 63) >> 6;
    const uint64_t last = (n & 63) ? (1ull << (n & 63)) - 1ull : ~0ull;  // columns < n of a row's last word
    for (int64_t i0 = block * 8; i0 < n; i0 += blocks * 8) {  // the same steps in all warps of the block
        const int64_t i = i0 + warp;
        const uint64_t* row = P + i * ldw;
        uint32_t nz = 0;
        int c = 0;
        if (i < n) {
            if (wpr <= kIndexChunk) {
                nz = wcsr_mask(row, 0, wpr, last, lane);
                c = __popc(nz);
            } else {
                for (int64_t c0 = 0; c0 < wpr; c0 += kIndexChunk) c += __popc(wcsr_mask(row, c0, wpr, last, lane));
            }
        }
        const int count = static_cast<int>(__reduce_add_sync(FULL, static_cast<unsigned>(c)));
        if (lane == 0) s_cnt[warp] = count;
        __syncthreads();
        if (threadIdx.x == 0) {
            int total = 0, top = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                total += s_cnt[k];
                top = max(top, s_cnt[k]);
            }
            auto* totals = reinterpret_cast<unsigned long long*>(wptr + 2 * n);
            s_base = total > 0 ? atomicAdd(totals, static_cast<unsigned long long>(total)) : 0ull;
            if (top > 0) atomicMax(totals + 1, static_cast<unsigned long long>(top));
        }
        __syncthreads();
        int64_t o = static_cast<int64_t>(s_base);
        for (int k = 0; k < warp; ++k) o += s_cnt[k];
        __syncthreads();  // the counts are rewritten in the next step
        if (i >= n) continue;
        if (lane == 0) *reinterpret_cast<longlong2*>(wptr + 2 * i) = make_longlong2(o, o + count);
        for (int64_t c0 = 0; c0 < wpr; c0 += kIndexChunk) {
            if (wpr > kIndexChunk) nz = wcsr_mask(row, c0, wpr, last, lane);
            uint32_t any = __reduce_or_sync(FULL, nz);  // groups of 32 words that hold a nonzero one
            while (any) {                               // four of them at a time
                int g[4];
                uint64_t v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    g[q] = any ? __ffs(any) - 1 : -1;
                    any &= any - 1u;
                    const int64_t x = c0 + 32 * g[q] + lane;
                    v[q] = g[q] >= 0 && ((nz >> g[q]) & 1u) ? row[x] : 0ull;
                    if (x == wpr - 1) v[q] &= last;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (g[q] < 0) break;  // uniform
                    const unsigned m = __ballot_sync(FULL, v[q] != 0ull);
                    if (v[q]) {
                        const int64_t e = o + __popc(m & below);
                        widx[e] = static_cast<int32_t>(c0 + 32 * g[q] + lane);
                        wval[e] = v[q];
                    }
                    o += __popc(m);
                }
            }
        }
    }
}

__global__ void __launch_bounds__(256) wcsr_build_kernel(const uint64_t* __restrict__ P, int64_t n, int64_t ldw,
                                                         int64_t* __restrict__ wptr, int32_t* __restrict__ widx,
                                                         uint64_t* __restrict__ wval) {
    wcsr_build_rows(P, n, ldw, wptr, widx, wval, blockIdx.x, gridDim.x);
}

// Bit-matrix transpose of n x n packed rows (ldw words each), one 64 x 64
// tile per 64-thread block: out row c, word bi = bit c of the tile's rows.
__device__ __forceinline__ void bit_transpose_tile(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                                   int64_t n, int64_t ldw, int64_t bi, int64_t bj, uint64_t* t) {
    const int tid = threadIdx.x;
    const int64_t r = bi * 64 + tid;
    t[tid] = r < n ? in[r * ldw + bj] : 0ull;
    __syncthreads();
    uint64_t o = 0;
#pragma unroll 8
    for (int k = 0; k < 64; ++k) o |= ((t[k] >> tid) & 1ull) << k;
    const int64_t c = bj * 64 + tid;
    if (c < n) out[c * ldw + bi] = o;
    __syncthreads();  // t is reused by the block's next tile
}

// The whole-matrix transpose, a tile of 256 rows (4 groups of 64) x 8 words (512 columns) per block: the tile is
// read with sector-wide loads into shared memory, transposed 64 x 64 at a time as four 32 x 32 blocks in registers
// (five shuffles each; two ballots and two selects per column, as before, bound the kernel by its instructions: 57 us
// at n = 14,541, 26 MB each way, against 16.5 us now), and written as 512 output rows x 4 words (one 32-byte sector
// each). Every word of out, padding words included, is written; bits
// at columns >= n are ignored (their output rows do not exist).
constexpr int kTrRows = 256, kTrWords = 8;
__global__ void __launch_bounds__(256) bit_transpose_kernel(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                                            int64_t n, int64_t ldw) {
    __shared__ uint64_t ti[kTrRows][kTrWords + 1];
    __shared__ uint64_t to[kTrWords * 64][5];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = static_cast<int64_t>(blockIdx.y) * kTrRows;   // first input row
    const int64_t w0 = static_cast<int64_t>(blockIdx.x) * kTrWords;  // first input word
    uint64_t v[kTrRows * kTrWords / 256];  // all of a thread's loads in flight at once
#pragma unroll
    for (int j = 0; j < kTrRows * kTrWords / 256; ++j) {
        const int k = tid + 256 * j, r = k >> 3, w = k & 7;
        const int64_t gr = r0 + r, gw = w0 + w;
        v[j] = (gr < n && gw < ldw) ? in[gr * ldw + gw] : 0ull;
    }
#pragma unroll
    for (int j = 0; j < kTrRows * kTrWords / 256; ++j) {
        const int k = tid + 256 * j;
        ti[k >> 3][k & 7] = v[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kTrWords / 2; ++j) {
        const int b = warp + 8 * j, g = b / kTrWords, w = b % kTrWords;
        const uint64_t a0 = ti[64 * g + lane][w], a1 = ti[64 * g + lane + 32][w];
        // output row lane (of the word's 64) holds rows 0 .. 31 of the group in its low half, 32 .. 63 in its high one
        const uint32_t l0 = warp_transpose32(static_cast<uint32_t>(a0), lane);
        const uint32_t l1 = warp_transpose32(static_cast<uint32_t>(a1), lane);
        const uint32_t h0 = warp_transpose32(static_cast<uint32_t>(a0 >> 32), lane);
        const uint32_t h1 = warp_transpose32(static_cast<uint32_t>(a1 >> 32), lane);
        to[64 * w + lane][g] = static_cast<uint64_t>(l0) | (static_cast<uint64_t>(l1) << 32);
        to[64 * w + lane + 32][g] = static_cast<uint64_t>(h0) | (static_cast<uint64_t>(h1) << 32);
    }
    __syncthreads();
    for (int k = tid; k < kTrWords * 64 * 4; k += 256) {
        const int orow = k >> 2, ow = k & 3;
        const int64_t gr = w0 * 64 + orow, gw = static_cast<int64_t>(blockIdx.y) * 4 + ow;
        if (gr < n && gw < ldw) out[gr * ldw + gw] = to[orow][ow];
    }
}

// Direction of a level, by the words each would touch: a push ORs the nonzero words of every frontier
// constant's row (w_out per constant on average); a pull scans an unvisited constant's column words (rows of
// R^T, w_in on average) until one meets the frontier, which on a frontier of nf constants spread over n takes
// about n / nf words, plus PULL_OVERHEAD words' worth of row-range loads per constant. A level pulls when
// nf w_out > nu (PULL_OVERHEAD + min(w_in, n / nf)).
constexpr float PULL_OVERHEAD = 1.0f;

// ---- selective product per query row
// Per warp in shared memory: D, N (ldw words each), FL, the list of the
// frontier's nonzero words (ldw 16-bit word indices), and GM, 64 bytes that
// map a rank to the index of a touched word group. The visited set V is the
// query's own output row in global memory (only its warp touches it). The
// stride is rounded up to 16 bytes so every warp's uint64 arrays stay aligned.
__host__ __device__ __forceinline__ int64_t smp_warp_bytes(int64_t ldw) {
    return (18 * ldw + 64 + 16 + 15) & ~int64_t(15);
}

// N[x] |= v in shared memory, as its nonzero 32-bit halves: OR without return value is one instruction there at 32 bits
// and a compare-and-swap loop at 64, and most words of a sparse relation have one bit.
__device__ __forceinline__ void or_word(uint64_t* N, int64_t x, uint64_t v) {
    unsigned* at = reinterpret_cast<unsigned*>(N + x);
    const unsigned lo = static_cast<unsigned>(v), hi = static_cast<unsigned>(v >> 32);
    if (lo) atomicOr(at, lo);
    if (hi) atomicOr(at + 1, hi);
}

// The same, and grew = 1 if N[x] lacks one of the bits: looked at until this lane has found one. (A bit that is missing when
// it is looked for was missing from the start, and whoever finds it missing sets it, so the answers of all lanes together
// say whether a word grew.)
__device__ __forceinline__ void or_grow(uint64_t* N, int64_t x, uint64_t v, uint64_t& grew) {
    if (grew == 0ull && (v & ~N[x]) != 0ull) grew = 1ull;
    or_word(N, x, v);
}

// Rows of up to NQ frontier constants per lane (k < 0: none) ORed into N:
// their nonzero words, by shared-memory atomics without return value. The row
// ranges and the first four entries of every light row (<= kLightRow nonzero words)
// are loaded before the first atomic; heavy rows are walked by the whole warp, four entries a lane in flight.
// tm collects the word groups written (bit x >> gshift for word x), or without kGroups whether a word grew (1).
constexpr int kLightRow = 16;
template <int NQ, bool kGroups = true>
__device__ __forceinline__ void push_rows(const int (&k)[NQ], int lane, const int64_t* __restrict__ wptr,
                                          const int32_t* __restrict__ widx, const uint64_t* __restrict__ wval,
                                          uint64_t* N, int gshift, uint64_t& tm) {
    int64_t e0[NQ];
    int len[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const longlong2 r = wcsr_row(wptr, k[q] >= 0 ? k[q] : 0);  // an in-range index even where the value is dropped
        e0[q] = r.x;
        len[q] = k[q] >= 0 ? static_cast<int>(r.y - r.x) : 0;
    }
    // entries e, e + step, ... (four; those at or beyond `left` are not the row's)
    const auto four = [&](int64_t e, int step, int left) {
        int y[4];
        uint64_t yv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool in = step * j < left;
            y[j] = in ? widx[e + step * j] : -1;
            yv[j] = in ? wval[e + step * j] : 0ull;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (y[j] >= 0) {
                if (kGroups) {
                    or_word(N, y[j], yv[j]);
                    tm |= 1ull << (y[j] >> gshift);
                } else {
                    or_grow(N, y[j], yv[j], tm);
                }
            }
    };
    int x[NQ][4];
    uint64_t val[NQ][4];
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool in = len[q] <= kLightRow && j < len[q];
            x[q][j] = in ? widx[e0[q] + j] : -1;
            val[q][j] = in ? wval[e0[q] + j] : 0ull;
        }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (x[q][j] >= 0) {
                if (kGroups) {
                    or_word(N, x[q][j], val[q][j]);
                    tm |= 1ull << (x[q][j] >> gshift);
                } else {
                    or_grow(N, x[q][j], val[q][j], tm);
                }
            }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
        if (len[q] <= kLightRow)
            for (int f = 4; f < len[q]; f += 4) four(e0[q] + f, 1, len[q] - f);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        unsigned hm = __ballot_sync(FULL, len[q] > kLightRow);
        while (hm) {
            const int sl = __ffs(hm) - 1;
            hm &= hm - 1;
            const int64_t h0 = __shfl_sync(FULL, e0[q], sl);
            const int hl = __shfl_sync(FULL, len[q], sl);
            for (int f = lane; f < hl; f += 128) four(h0 + f, 32, hl - f);
        }
    }
}

// One push step of a lane on its own frontier word d (the constants of word w): up to NQ of its set bits.
template <int NQ>
__device__ __forceinline__ void push_step(uint64_t& d, int64_t w, int lane, const int64_t* __restrict__ wptr,
                                          const int32_t* __restrict__ widx, const uint64_t* __restrict__ wval,
                                          uint64_t* N, int gshift, uint64_t& tm) {
    int k[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        k[q] = -1;
        if (d) {
            const int b = __ffsll(static_cast<long long>(d)) - 1;
            d &= d - 1;
            k[q] = static_cast<int>(w) * 64 + b;
        }
    }
    push_rows<NQ>(k, lane, wptr, widx, wval, N, gshift, tm);
}

// Position of the set bit of rank r (r < popcount) in x.
__device__ __forceinline__ int select_bit(uint64_t x, int r) {
    int pos = 0;
    int c = __popc(static_cast<unsigned>(x));
    if (r >= c) {
        r -= c;
        x >>= 32;
        pos = 32;
    }
    unsigned v = static_cast<unsigned>(x);
    c = __popc(v & 0xFFFFu);
    if (r >= c) { r -= c; v >>= 16; pos += 16; }
    c = __popc(v & 0xFFu);
    if (r >= c) { r -= c; v >>= 8; pos += 8; }
    c = __popc(v & 0xFu);
    if (r >= c) { r -= c; v >>= 4; pos += 4; }
    c = __popc(v & 0x3u);
    if (r >= c) { r -= c; v >>= 2; pos += 2; }
    if (r >= static_cast<int>(v & 1u)) pos += 1;
    return pos;
}

// Push of a chunk of frontier words (lane l holds word d of index w) with the set bits dealt out to the
// lanes in rank order, two per lane per step: a word with many bits (a band of a squared path, a dense
// frontier) is shared by the whole warp instead of being walked by one lane.
template <int NQ, bool kGroups = true>
__device__ __forceinline__ void push_balanced(uint64_t d, int w, int lane, const int64_t* __restrict__ wptr,
                                              const int32_t* __restrict__ widx, const uint64_t* __restrict__ wval,
                                              uint64_t* N, int gshift, uint64_t& tm) {
    const int c = __popcll(d);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(FULL, incl, 31);
    const int excl = incl - c;
    for (int base = 0; base < total; base += 32 * NQ) {
        int k[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int r = base + q * 32 + lane;
            int owner = 0;  // the lane whose bits hold rank r: the first with inclusive count > r
#pragma unroll
            for (int st = 16; st >= 1; st >>= 1) {
                const int v = __shfl_sync(FULL, incl, owner + st - 1);
                if (v <= r) owner += st;
            }
            const uint64_t od = __shfl_sync(FULL, d, owner);
            const int ow = __shfl_sync(FULL, w, owner);
            const int oex = __shfl_sync(FULL, excl, owner);
            k[q] = r < total ? ow * 64 + select_bit(od, r - oex) : -1;
        }
        push_rows<NQ, kGroups>(k, lane, wptr, widx, wval, N, gshift, tm);
    }
}

// Algorithm 2 for one query row: the frontier expansion from the source row srcw(0 .. ) (words, bits >= n
// ignored), visited set and result in V (ldw_out words), D / N / FL / GM the warp's shared-memory arrays
// (sized for at least ldw words). With `from` it goes on where the query-row kernel stopped after `lv` levels: from holds the
// frontier and the visited set (ceil(n / 64) words each). Returns the levels run (the deepest BFS level + 1). Called by a
// whole warp.
template <class SrcWord>
__device__ __forceinline__ int smp_expand_row(SrcWord srcw, uint64_t* __restrict__ V, int64_t ldw_out, int reflexive,
                                              const int64_t* __restrict__ wptr, const int32_t* __restrict__ widx,
                                              const uint64_t* __restrict__ wval, int64_t n, int64_t ldw,
                                              int max_levels, const Deadline& dl, const int64_t* __restrict__ wptrT,
                                              const int32_t* __restrict__ widxT, const uint64_t* __restrict__ wvalT,
                                              uint64_t* D, uint64_t* N, uint16_t* FL, uint8_t* GM, int lane,
                                              const uint64_t* __restrict__ from = nullptr, int lv = 0) {
    const unsigned lt = (1u << lane) - 1u;  // lanes below this one
    const int64_t wpr = (n + 63) / 64;
    // words of N form at most 64 groups of 2^gshift words; a push records the groups it wrote
    int gshift = 0;
    while ((int64_t(64) << gshift) < wpr) ++gshift;
    const int ngroups = static_cast<int>((wpr + (int64_t(1) << gshift) - 1) >> gshift);
    const uint64_t all_groups = ngroups >= 64 ? ~0ull : (1ull << ngroups) - 1ull;
    const float w_out = wptrT != nullptr ? static_cast<float>(wptr[2 * n]) / static_cast<float>(n) : 0.f;
    const float w_in = wptrT != nullptr ? static_cast<float>(wptrT[2 * n]) / static_cast<float>(n) : 0.f;
    // D = sources; FL = their nonzero words (ballot compaction); V = 0
    int fcount = 0, visited = 0;
    for (int64_t w0 = 0; w0 < ldw; w0 += 32) {
        const int64_t w = w0 + lane;
        uint64_t s = 0, v = 0;
        if (w < wpr) {
            s = from != nullptr ? from[w] : srcw(w);
            if (from != nullptr) v = from[wpr + w];
            visited += __popcll(v);
            const int64_t valid = n - w * 64;
            if (valid < 64) s &= (1ull << valid) - 1ull;
        }
        if (w < ldw) {
            D[w] = s;
            N[w] = 0;
        }
        if (w < ldw_out) V[w] = v;
        const unsigned m = __ballot_sync(FULL, s != 0ull);
        if (s) FL[fcount + __popc(m & lt)] = static_cast<uint16_t>(w);
        fcount += __popc(m);
    }
    __syncwarp();
    bool pull = false;
    int64_t nu = n - static_cast<int64_t>(__reduce_add_sync(FULL, static_cast<unsigned>(visited)));  // unvisited constants
    while (true) {
        if (dl.budget_ns && __shfl_sync(FULL, lane == 0 ? static_cast<int>(dl.past()) : 0, 0)) break;
        uint64_t gm = all_groups;  // groups of N that may be nonzero after this expansion
        if (pull) {
            // pull: unvisited j joins the next frontier iff some word of column j (row j of R^T) meets D;
            // each lane owns whole words of N (no atomics)
            for (int64_t w = lane; w < wpr; w += 32) {
                uint64_t nw = 0;
                {
                    uint64_t u = ~V[w];
                    const int64_t valid = n - w * 64;
                    if (valid < 64) u &= (1ull << valid) - 1ull;
                    while (u) {
                        // two unvisited constants at a time: their column ranges, then the first two
                        // entries of each, all loads in flight before the first test
                        int bs[2];
                        int64_t s0[2], s1[2];
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            bs[q] = -1;
                            if (u) {
                                bs[q] = __ffsll(static_cast<long long>(u)) - 1;
                                u &= u - 1;
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const int64_t j = w * 64 + (bs[q] < 0 ? 0 : bs[q]);
                            const longlong2 r = wcsr_row(wptrT, j);
                            s0[q] = bs[q] < 0 ? 0 : r.x;
                            s1[q] = bs[q] < 0 ? 0 : r.y;
                        }
                        int xi[2][2];
                        uint64_t xv[2][2];
#pragma unroll
                        for (int q = 0; q < 2; ++q)
#pragma unroll
                            for (int r = 0; r < 2; ++r) {
                                const bool in = s0[q] + r < s1[q];
                                xi[q][r] = in ? widxT[s0[q] + r] : 0;
                                xv[q][r] = in ? wvalT[s0[q] + r] : 0ull;
                            }
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            if (bs[q] < 0) continue;
                            bool hit = (xv[q][0] & D[xi[q][0]]) != 0ull || (xv[q][1] & D[xi[q][1]]) != 0ull;
                            for (int64_t e = s0[q] + 2; !hit && e < s1[q]; ++e) hit = (wvalT[e] & D[widxT[e]]) != 0ull;
                            if (hit) nw |= 1ull << bs[q];
                        }
                    }
                    N[w] = nw;
                }
            }
        } else {
            // push: OR the nonzero words of every frontier row into N (no return values, so the
            // atomics are reductions); each lane records the word groups it wrote
            uint64_t tm = 0;
            for (int i0 = 0; i0 < fcount; i0 += 32) {
                const int i = i0 + lane;
                const int64_t w = i < fcount ? FL[i] : 0;
                uint64_t d = i < fcount ? D[w] : 0ull;  // FL[i] for i < fcount <= ldw only
                // at most two constants per word: each lane takes its own; else the bits are dealt out
                if (__reduce_max_sync(FULL, static_cast<unsigned>(__popcll(d))) <= 2u)
                    push_step<2>(d, w, lane, wptr, widx, wval, N, gshift, tm);
                else
                    push_balanced<2>(d, w, lane, wptr, widx, wval, N, gshift, tm);
            }
            gm = static_cast<uint64_t>(__reduce_or_sync(FULL, static_cast<unsigned>(tm))) |
                 (static_cast<uint64_t>(__reduce_or_sync(FULL, static_cast<unsigned>(tm >> 32))) << 32);
        }
        __syncwarp();
        // D := 0 on the old frontier words, then D := N & ~V on the touched groups (V |= D, N := 0);
        // the words that come out nonzero become the new frontier list FL
        for (int i = lane; i < fcount; i += 32) D[FL[i]] = 0;
        __syncwarp();
        int nf = 0, fnew = 0;
        // GM[r] = index of the r-th set group of gm; candidates are the words of those groups
        for (int b = lane; b < 64; b += 32)
            if ((gm >> b) & 1ull) GM[__popcll(gm & ((1ull << b) - 1ull))] = static_cast<uint8_t>(b);
        __syncwarp();
        const int cand = __popcll(gm) << gshift;
        const int gmask = (1 << gshift) - 1;
        for (int c0 = 0; c0 < cand; c0 += 32) {
            const int c = c0 + lane;
            int w = static_cast<int>(wpr);
            if (c < cand) w = (static_cast<int>(GM[c >> gshift]) << gshift) + (c & gmask);
            uint64_t nw = 0;
            if (w < wpr) {
                nw = N[w] & ~V[w];
                N[w] = 0;
                if (nw) {
                    V[w] |= nw;
                    D[w] = nw;
                }
            }
            const unsigned m = __ballot_sync(FULL, nw != 0ull);
            if (nw) FL[fnew + __popc(m & lt)] = static_cast<uint16_t>(w);
            fnew += __popc(m);
            nf += __popcll(nw);
        }
        nf = __reduce_add_sync(FULL, nf);
        fcount = fnew;
        __syncwarp();
        nu -= nf;
        ++lv;
        if (nf == 0 || lv > max_levels) break;
        // direction of the next level: the cheaper one by the words it touches (nf > 0 here)
        pull = wptrT != nullptr &&
               static_cast<float>(nf) * w_out >
                   static_cast<float>(nu) * (PULL_OVERHEAD + fminf(w_in, static_cast<float>(n) / static_cast<float>(nf)));
    }
    if (reflexive)
        for (int64_t w = lane; w < wpr; w += 32) {
            uint64_t s = srcw(w);
            const int64_t valid = n - w * 64;
            if (valid < 64) s &= (1ull << valid) - 1ull;
            V[w] |= s;
        }
    return lv;
}

__global__ void __launch_bounds__(256, 4) smp_packed_kernel(const int64_t* __restrict__ wptr, const int32_t* __restrict__ widx,
                                                         const uint64_t* __restrict__ wval, int64_t n, int64_t ldw,
                                                         const uint64_t* __restrict__ src, int64_t ldw_src, int64_t q,
                                                         uint64_t* __restrict__ out, int64_t ldw_out, int* levels_max,
                                                         unsigned long long* qcounter, int reflexive, int max_levels,
                                                         Deadline dl, const int64_t* __restrict__ wptrT,
                                                         const int32_t* __restrict__ widxT,
                                                         const uint64_t* __restrict__ wvalT, RowState from) {
    extern __shared__ uint64_t sm[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    uint64_t* D = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(sm) + wib * smp_warp_bytes(ldw));
    uint64_t* N = D + ldw;
    uint16_t* FL = reinterpret_cast<uint16_t*>(N + ldw);
    uint8_t* GM = reinterpret_cast<uint8_t*>(FL + ldw);
    while (true) {
        unsigned long long qi = 0;
        if (lane == 0) qi = atomicAdd(qcounter, 1ull);
        qi = __shfl_sync(FULL, qi, 0);
        if (qi >= static_cast<unsigned long long>(q)) break;
        const uint64_t* srow = src + static_cast<int64_t>(qi) * ldw_src;
        uint64_t* V = out + static_cast<int64_t>(qi) * ldw_out;
        const uint64_t* at = nullptr;
        int lv = 0;
        if (from.words != nullptr) {
            lv = from.levels[qi];
            if (lv == 0) continue;  // finished
            const int64_t wpr = (n + 63) / 64;
            at = from.words + static_cast<int64_t>(qi) * 3 * wpr;
            srow = at + 2 * wpr;
        }
        lv = smp_expand_row([srow](int64_t w) { return srow[w]; }, V, ldw_out, reflexive, wptr, widx, wval, n, ldw,
                            max_levels, dl, wptrT, widxT, wvalT, D, N, FL, GM, lane, at, lv);
        if (lane == 0) atomicMax(levels_max, lv);
        __syncwarp();
    }
}

// ---- closures by frontier expansion of many small relations in one launch (grouped batch)
// Transpose and word index of R and of R^T for every job: blockIdx.y = job; one launch builds the transposes, the next
// the word indexes of both matrices (blockIdx.z = matrix).
__global__ void __launch_bounds__(64) frontier_transpose_kernel(const FrontierJob* __restrict__ jobs) {
    __shared__ uint64_t t[64];
    const FrontierJob& J = jobs[blockIdx.y];
    const int64_t wpr = (J.n + 63) / 64;
    for (int64_t tile = blockIdx.x; tile < wpr * wpr; tile += gridDim.x)
        bit_transpose_tile(J.P, J.PT, J.n, J.ldw, tile / wpr, tile % wpr, t);
    // the totals of the two word indexes that the next launch builds, and padding words of the transpose's rows
    if (blockIdx.x == 0 && threadIdx.x < 2) J.wptr[2 * J.n + threadIdx.x] = J.wptrT[2 * J.n + threadIdx.x] = 0;
    for (int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; r < J.n;
         r += static_cast<int64_t>(gridDim.x) * blockDim.x)
        for (int64_t w = wpr; w < J.ldw; ++w) J.PT[r * J.ldw + w] = 0ull;
}

__global__ void __launch_bounds__(256) frontier_wcsr_kernel(const FrontierJob* __restrict__ jobs) {
    const FrontierJob& J = jobs[blockIdx.y];
    if (blockIdx.z == 0) wcsr_build_rows(J.P, J.n, J.ldw, J.wptr, J.widx, J.wval, blockIdx.x, gridDim.x);
    else wcsr_build_rows(J.PT, J.n, J.ldw, J.wptrT, J.widxT, J.wvalT, blockIdx.x, gridDim.x);
}

// Every row of every job as one query: the rows of all jobs are numbered job by job (job j owns rows
// jobs[j].first .. jobs[j].first + n - 1), warps take them from *counter; the source of row i is constant i.
__global__ void __launch_bounds__(256, 4) frontier_group_kernel(const FrontierJob* __restrict__ jobs, int njobs,
                                                                int64_t total, int64_t ldw_max,
                                                                unsigned long long* counter) {
    extern __shared__ uint64_t sm[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    uint64_t* D = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(sm) + wib * smp_warp_bytes(ldw_max));
    uint64_t* N = D + ldw_max;
    uint16_t* FL = reinterpret_cast<uint16_t*>(N + ldw_max);
    uint8_t* GM = reinterpret_cast<uint8_t*>(FL + ldw_max);
    const Deadline none{0, nullptr, nullptr};
    while (true) {
        unsigned long long qi = 0;
        if (lane == 0) qi = atomicAdd(counter, 1ull);
        qi = __shfl_sync(FULL, qi, 0);
        if (qi >= static_cast<unsigned long long>(total)) break;
        int lo = 0, hi = njobs - 1;
        while (lo < hi) {  // the last job whose first row is <= qi
            const int mid = (lo + hi + 1) >> 1;
            if (jobs[mid].first <= static_cast<int64_t>(qi)) lo = mid; else hi = mid - 1;
        }
        const FrontierJob& J = jobs[lo];
        const int64_t i = static_cast<int64_t>(qi) - J.first;
        const int64_t wi = i >> 6;
        const uint64_t bi = 1ull << (i & 63);
        const int lv = smp_expand_row([wi, bi](int64_t w) { return w == wi ? bi : 0ull; }, J.out + i * J.ldw, J.ldw, 0,
                                      J.wptr, J.widx, J.wval, J.n, J.ldw, static_cast<int>(J.n + 1), none, J.wptrT,
                                      J.widxT, J.wvalT, D, N, FL, GM, lane);
        if (lane == 0) atomicMax(J.levels, lv);
        __syncwarp();
    }
}

// ---- incremental closure: one new fact r(u, v) on a transitive R+ (packed rows)
// (R + E_uv)+ = R+ + X Y^T with X = {i : i = u or R+_iu} (the constants that
// reach u) and Y = R+_v + e_v (what v reaches, and v): every row in X gains Y.
// A warp owns each row it updates, so membership (bit u of its own row) is
// read before that row changes; row v itself only gains bit v, which every
// reader adds anyway. When R+_uv already holds, every member row already
// contains Y (transitivity) and no word is written.
__global__ void insert_fact_kernel(uint64_t* __restrict__ P, int64_t n, int64_t ldw, int64_t u, int64_t v) {
    const int lane = threadIdx.x & 31;
    const int64_t wu = u >> 6, wv = v >> 6;
    const uint64_t bu = 1ull << (u & 63), bv = 1ull << (v & 63);
    const int64_t wpr = (n + 63) >> 6;
    const uint64_t* Y = P + v * ldw;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        uint64_t* row = P + i * ldw;
        const bool member = (i == u) || (row[wu] & bu) != 0ull;  // uniform across the warp
        if (!member) continue;
        __syncwarp();
        for (int64_t w = lane; w < wpr; w += 32) {
            uint64_t y = Y[w];
            if (w == wv) y |= bv;
            const uint64_t r = row[w];
            if ((r | y) != r) row[w] = r | y;
        }
    }
}

// ---- incremental closure: a chunk of up to kInsertChunk facts at once on a transitive R+ (three launches)
// With Y_k = R+_{v_k} + e_{v_k} and the links k -> l iff v_k = u_l or R+ holds (v_k, u_l), everything the grown
// relation derives from v_k is W_k = Y_k OR (OR of Y_l over the facts l that k reaches along links), and row i gains W_k
// for every k with i = u_k or R+ holds (i, u_k). One launch per fact, as before, costs a launch's latency each (4 to
// 6 us) and reads one word of all n rows; a chunk reads every row once. Bound by HBM/L2 reads of the n rows when few
// rows change, else by the words that the rows gain: n = 14,541 and 1,000 facts, 6,180 us before, 140 us now.
// R+ is transitive, so a fact whose v_k is already in a row adds nothing that the row's other facts do not bring: if
// i reaches v_k, it also reaches every u_l that v_k links to. The same holds for Y_l inside W_k.
constexpr int kInsertWarps = 8;

// Links of the chunk: bit l of row k of G (mw words per row). A block per fact k.
__global__ void __launch_bounds__(kInsertWarps * 32) insert_links_kernel(const uint64_t* __restrict__ P, int64_t ldw,
                                                                         const int32_t* __restrict__ pairs, int m, int mw,
                                                                         uint32_t* __restrict__ G) {
    const int k = blockIdx.x;
    const int64_t v = pairs[2 * k + 1];
    const uint64_t* row = P + v * ldw;
    for (int l = threadIdx.x; l < mw * 64; l += blockDim.x) {  // whole warps run: mw * 64 is a multiple of 32
        const int64_t u = l < m ? pairs[2 * l] : 0;
        const unsigned b = __ballot_sync(FULL, l < m && (u == v || ((row[u >> 6] >> (u & 63)) & 1ull) != 0ull));
        if ((l & 31) == 0) G[static_cast<int64_t>(k) * 2 * mw + (l >> 5)] = b;
    }
}

// W_k, a warp per fact: the facts that k reaches along links by a search on G (all of it in shared memory, a lane per
// word of the reached set), then the OR of their Y rows.
__global__ void __launch_bounds__(kInsertWarps * 32) insert_reach_kernel(const uint64_t* __restrict__ P, int64_t n,
                                                                         int64_t ldw, const int32_t* __restrict__ pairs,
                                                                         int m, int mw, const uint64_t* __restrict__ G,
                                                                         uint64_t* W) {
    extern __shared__ uint64_t ins_g[];
    for (int x = threadIdx.x; x < m * mw; x += blockDim.x) ins_g[x] = G[x];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int k = blockIdx.x * kInsertWarps + (threadIdx.x >> 5);
    if (k >= m) return;
    uint64_t reach = lane < mw ? ins_g[k * mw + lane] : 0ull;  // mw <= 32
    uint64_t todo = reach;
    while (true) {
        const unsigned any = __ballot_sync(FULL, todo != 0ull);
        if (any == 0u) break;
        const int src = __ffs(any) - 1;
        const int bit = __ffsll(static_cast<long long>(__shfl_sync(FULL, todo, src))) - 1;
        if (lane == src) todo &= todo - 1ull;
        const uint64_t more = lane < mw ? ins_g[(src * 64 + bit) * mw + lane] & ~reach : 0ull;
        reach |= more;
        todo |= more;
    }
    const int64_t wpr = (n + 63) >> 6;
    uint64_t* w = W + static_cast<int64_t>(k) * ldw;
    const auto add = [&](int l, bool first) {
        const int64_t v = pairs[2 * l + 1];
        if (!first && ((w[v >> 6] >> (v & 63)) & 1ull)) return;  // uniform: every lane reads the same word
        const uint64_t* y = P + v * ldw;
        __syncwarp();
        for (int64_t x = lane; x < wpr; x += 32)
            w[x] = (first ? 0ull : w[x]) | y[x] | (x == (v >> 6) ? 1ull << (v & 63) : 0ull);
        __syncwarp();
    };
    add(k, true);
    for (int src = 0; src < mw; ++src) {
        uint64_t bits = __shfl_sync(FULL, reach, src);
        while (bits) {
            add(src * 64 + __ffsll(static_cast<long long>(bits)) - 1, false);
            bits &= bits - 1ull;
        }
    }
}

// Row i gains W_k for every fact k with i = u_k or (i, u_k) in the row; a warp per row, the facts tested 32 at a time.
__global__ void __launch_bounds__(kInsertWarps * 32) insert_rows_kernel(uint64_t* P, int64_t n, int64_t ldw,
                                                                        const int32_t* __restrict__ pairs, int m,
                                                                        const uint64_t* __restrict__ W) {
    const int lane = threadIdx.x & 31;
    const int64_t wpr = (n + 63) >> 6;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * kInsertWarps;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * kInsertWarps + (threadIdx.x >> 5); i < n; i += warps) {
        uint64_t* row = P + i * ldw;
        for (int k0 = 0; k0 < m; k0 += 32) {
            const int k = k0 + lane;
            const int64_t u = k < m ? pairs[2 * k] : 0;
            unsigned hit = __ballot_sync(FULL, k < m && (u == i || ((row[u >> 6] >> (u & 63)) & 1ull) != 0ull));
            while (hit) {
                const int kk = k0 + __ffs(hit) - 1;
                hit &= hit - 1u;
                const int64_t v = pairs[2 * kk + 1];
                const bool has = ((row[v >> 6] >> (v & 63)) & 1ull) != 0ull;  // uniform
                __syncwarp();
                if (has) continue;
                const uint64_t* w = W + static_cast<int64_t>(kk) * ldw;
                for (int64_t x = lane; x < wpr; x += 32) {
                    const uint64_t r = row[x], g = r | w[x];
                    if (g != r) row[x] = g;
                }
                __syncwarp();
            }
        }
    }
}

// ---- passes over a word index with a warp per row
// Rows are dealt to the warps of all blocks; a row with many times the mean of entries (a power-law relation's, a thousand
// against three) would keep one warp busy long after the others are done, so a block puts such rows into a queue and walks
// them with all of its warps at the end (a full queue: the warp walks the row after all). Measured on power-law relations,
// with a warp for every row and with the queue (one pass):
//                                  n = 14,000        20,011          65,536
//     square_growth_kernel                 -       98 -> 46 us    131 -> 80 us
//     indexed_rows_kernel       364 -> 69 us            (two products of a closure; 8 x and 64 against 16 x and 192:
//     indexed_cost_kernel        54 -> 26 us             2,317 against 2,376 us for that closure)
constexpr int kRowQueue = 64;

// Entries of a row from which it is queued: eight times the mean, at least 64.
__device__ __forceinline__ int64_t long_row(const WordIndex& A, int64_t n) {
    const int64_t mean8 = 8 * A.ptr[2 * n] / n;
    return mean8 > 64 ? mean8 : 64;
}

// Calls row(i, range, false) for this warp's rows that are not queued, then row(i, range, true) with all warps of the block
// in step for the queued ones. One call site: the body is large, and two copies of it took more registers than fit.
template <class Row>
__device__ __forceinline__ void rows_of_index(const WordIndex& A, int64_t n, Row&& row) {
    __shared__ int s_queue[kRowQueue];
    __shared__ int s_queued;
    const int lane = threadIdx.x & 31;
    const int64_t nw = blockDim.x >> 5, warps = static_cast<int64_t>(gridDim.x) * nw;
    if (threadIdx.x == 0) s_queued = 0;
    __syncthreads();
    const int64_t limit = long_row(A, n);
    int64_t next = static_cast<int64_t>(blockIdx.x) * nw + (threadIdx.x >> 5);
    bool together = false;
    for (int queued = 0, k = 0;;) {
        int64_t i;
        longlong2 range;
        if (!together) {
            if (next >= n) {
                __syncthreads();
                together = true;
                queued = s_queued < kRowQueue ? s_queued : kRowQueue;
                continue;
            }
            i = next;
            next += warps;
            range = wcsr_row(A.ptr, i);
            if (range.y - range.x > limit) {
                int at = 0;
                if (lane == 0) at = atomicAdd(&s_queued, 1);
                at = __shfl_sync(FULL, at, 0);
                if (at < kRowQueue) {
                    if (lane == 0) s_queue[at] = static_cast<int>(i);
                    continue;
                }
            }
        } else {
            if (k >= queued) break;
            i = s_queue[k++];
            range = wcsr_row(A.ptr, i);
        }
        row(i, range, together);
    }
}

__device__ __forceinline__ void sync_row(bool together) {
    if (together) __syncthreads();
    else __syncwarp();
}

// ---- one product on packed rows through word indexes: C_i = P_i | OR_{k in A_i} B_k, where row k contributes only its
// nonzero words (push_balanced), so the cost follows the indexes, not n / 64 words per k. With A = B = P = R that is one
// squaring step. The row is assembled in shared memory (ldw words per warp). The kernel waits for L2 (a range, then its
// words, at random), so it is as fast as it has loads in flight: 32-bit lengths and one named row a lane at a time leave 48
// registers and five blocks an SM (n = 14,000, 1.5 entries a row, the four products of a closure: 801 us with two rows a
// lane, 64 registers and 64-bit shared-memory atomics, 532 now; six blocks spill and lose on power-law relations). *changed (or null) is raised when C_i != P_i.
__global__ void __launch_bounds__(256, 5) indexed_rows_kernel(const WordIndex A, const WordIndex B,
                                                           const uint64_t* __restrict__ P, int64_t n, int64_t ldw,
                                                           uint64_t* __restrict__ C, int* __restrict__ changed) {
    extern __shared__ __align__(16) uint64_t sq_sm[];
    const int lane = threadIdx.x & 31;
    uint64_t tm = 0;  // whether a row grew
    rows_of_index(A, n, [&](int64_t i, const longlong2& range, bool together) {
        const int nw = together ? blockDim.x >> 5 : 1, warp = threadIdx.x >> 5;  // together: the warps take entries in turn
        const int first = together ? threadIdx.x : lane, step = 32 * nw;
        uint64_t* S = together ? sq_sm : sq_sm + warp * ldw;
        // the row in 16-byte pieces (ldw is even) by asynchronous copies, all in flight without registers: one word at a time
        // through them a row of few entries took twice the time of its bytes (n = 32,768, 4 entries a row, 268 MB: 99 us,
        // 52 now)
        const ulonglong2* Pi = reinterpret_cast<const ulonglong2*>(P + i * ldw);
        ulonglong2* Si = reinterpret_cast<ulonglong2*>(S);
        const int pieces = static_cast<int>(ldw >> 1);
        for (int v = first; v < pieces; v += step)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(Si + v)), "l"(Pi + v) : "memory");
        asm volatile("cp.async.wait_all;" ::: "memory");
        sync_row(together);
        for (int64_t b0 = range.x; b0 < range.y; b0 += step) {
            const int64_t e = b0 + (together ? lane * nw + warp : lane);
            const int64_t ee = e < range.y ? e : range.x;
            const uint64_t d = e < range.y ? A.val[ee] : 0ull;
            const int w = e < range.y ? A.idx[ee] : 0;
            push_balanced<1, false>(d, w, lane, B.ptr, B.idx, B.val, S, 30, tm);
        }
        sync_row(together);
        ulonglong2* Ci = reinterpret_cast<ulonglong2*>(C + i * ldw);
        for (int v = first; v < pieces; v += step) Ci[v] = Si[v];
        sync_row(together);
    });
    if (changed != nullptr && __any_sync(FULL, tm != 0) && lane == 0) atomicOr(changed, 1);
}

// Sum over the block (every thread calls it; thread 0 gets it).
__device__ __forceinline__ unsigned long long block_sum(unsigned long long x) {
    __shared__ unsigned long long part[32];
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(FULL, x, off);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = x;
    __syncthreads();
    x = 0;
    if (threadIdx.x == 0)
        for (int k = 0; k < static_cast<int>(blockDim.x >> 5); ++k) x += part[k];
    __syncthreads();
    return x;
}

// ---- the work of such a product: for every set bit k of every row of A, the nonzero words of row k of B (what
// indexed_rows_kernel ORs into that row). cost[0] += the total, cost[1] = max over rows (one warp or block assembles a
// row, so the largest row bounds the step from below). Two 64-bit atomics per block. Bits at or beyond n are zero in every
// row, so k < n.
__global__ void __launch_bounds__(256) indexed_cost_kernel(const WordIndex A, const WordIndex B, int64_t n,
                                                           unsigned long long* __restrict__ cost) {
    const int lane = threadIdx.x & 31;
    unsigned long long total = 0, top = 0;  // lane 0's (a queued row: thread 0's)
    const auto words_of = [&](int64_t e) {
        unsigned long long c = 0;
        uint64_t d = A.val[e];
        const int64_t base = static_cast<int64_t>(A.idx[e]) << 6;
        while (d) {  // up to four rows' ranges in flight
            longlong2 r[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                r[q] = make_longlong2(0, 0);
                if (d) {
                    r[q] = wcsr_row(B.ptr, base + (__ffsll(static_cast<long long>(d)) - 1));
                    d &= d - 1ull;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) c += static_cast<unsigned long long>(r[q].y - r[q].x);
        }
        return c;
    };
    rows_of_index(A, n, [&](int64_t, const longlong2& range, bool together) {
        unsigned long long c = 0;
        const int first = together ? threadIdx.x : lane, step = together ? blockDim.x : 32;
        for (int64_t e = range.x + first; e < range.y; e += step) c += words_of(e);
        if (together) {
            c = block_sum(c);
            if (threadIdx.x != 0) c = 0;
        } else {
            for (int off = 16; off > 0; off >>= 1) c += __shfl_xor_sync(FULL, c, off);
        }
        if (lane == 0) {
            total += c;
            top = c > top ? c : top;
        }
    });
    if (lane == 0 && total != 0ull) atomicMax(cost + 1, top);
    total = block_sum(total);
    if (threadIdx.x == 0 && total != 0ull) atomicAdd(cost, total);
}

// ---- the next squaring step's nonzero words without forming it: per row, the union of the row's own word indices and
// those of every row k it names (R + R R), in a shared-memory bitmap of ldw bits.
// out[0] += the total nonzero words of R + R R, out[1] += the word ORs the squaring would issue.
__global__ void __launch_bounds__(256, 6) square_growth_kernel(const WordIndex A, int64_t n, int64_t ldw,
                                                            unsigned long long* __restrict__ out,
                                                            unsigned long long* __restrict__ bits_out) {
    extern __shared__ uint32_t growth_bm[];
    const int lane = threadIdx.x & 31;
    const int bw = static_cast<int>((ldw + 31) / 32);  // bitmap words per warp
    unsigned long long words = 0, ors = 0, ones = 0;
    const auto mark = [&](uint32_t* bm, int64_t e) {
        const int x = A.idx[e];
        atomicOr(&bm[x >> 5], 1u << (x & 31));
        uint64_t d = A.val[e];
        ones += static_cast<unsigned long long>(__popcll(d));
        const int64_t base = static_cast<int64_t>(x) << 6;
        while (d) {
            const longlong2 r = wcsr_row(A.ptr, base + (__ffsll(static_cast<long long>(d)) - 1));
            d &= d - 1ull;
            ors += static_cast<unsigned long long>(r.y - r.x);
            for (int64_t f = r.x; f < r.y; f += 4) {  // four of the named row's entries in flight
                int y[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) y[q] = f + q < r.y ? A.idx[f + q] : -1;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (y[q] >= 0) atomicOr(&bm[y[q] >> 5], 1u << (y[q] & 31));
            }
        }
    };
    rows_of_index(A, n, [&](int64_t, const longlong2& range, bool together) {
        uint32_t* bm = together ? growth_bm : growth_bm + (threadIdx.x >> 5) * bw;
        const int first = together ? threadIdx.x : lane, step = together ? blockDim.x : 32;
        for (int j = first; j < bw; j += step) bm[j] = 0u;
        sync_row(together);
        for (int64_t e = range.x + first; e < range.y; e += step) mark(bm, e);
        sync_row(together);
        for (int j = first; j < bw; j += step) words += static_cast<unsigned long long>(__popc(bm[j]));
        sync_row(together);  // the bitmap is cleared for the next row
    });
    words = block_sum(words);
    ors = block_sum(ors);
    ones = block_sum(ones);
    if (threadIdx.x == 0 && (words | ors) != 0ull) {
        atomicAdd(out, words);
        atomicAdd(out + 1, ors);
    }
    if (threadIdx.x == 0 && bits_out != nullptr && ones != 0ull) atomicAdd(bits_out, ones);
}

// Ones of a run of words, 16 bytes a lane.
__global__ void __launch_bounds__(256) packed_ones_kernel(const uint64_t* __restrict__ P, int64_t words,
                                                          unsigned long long* __restrict__ out) {
    unsigned long long c = 0;
    for (int64_t k = blockIdx.x * 256ll + threadIdx.x; 2 * k < words; k += gridDim.x * 256ll) {
        const uint4 v = reinterpret_cast<const uint4*>(P)[k];
        c += static_cast<unsigned long long>(__popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w));
    }
    c = block_sum(c);
    if (threadIdx.x == 0 && c) atomicAdd(out, c);
}

// Bit rows of R^T from the word index of R (out cleared beforehand): warp per row i of R, a lane per nonzero word;
// each set bit (i, j) ORs bit i into word i / 64 of row j. Rows i of one 64-row group hit the same words of R^T,
// on different bits.
__global__ void __launch_bounds__(256) scatter_transpose_kernel(const int64_t* __restrict__ wptr,
                                                                const int32_t* __restrict__ widx,
                                                                const uint64_t* __restrict__ wval, int64_t n,
                                                                int64_t ldw, unsigned long long* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        const unsigned long long bit = 1ull << (i & 63);
        const int64_t wi = i >> 6;
        const longlong2 range = wcsr_row(wptr, i);
        for (int64_t e = range.x + lane; e < range.y; e += 32) {
            uint64_t d = wval[e];
            const int64_t base = static_cast<int64_t>(widx[e]) << 6;
            while (d) {
                const int64_t j = base + (__ffsll(static_cast<long long>(d)) - 1);
                d &= d - 1ull;
                if (j < n) atomicOr(out + j * ldw + wi, bit);  // a caller's bits beyond column n are not columns
            }
        }
    }
}

// ---- frontier expansion of 64 sources at once (closures whose rows reach most constants)
// Algorithm 2 for the 64 query rows e_s0 .. e_s0+63 together, bit-sliced: word w of V, D and Dn holds, in bit j,
// whether constant w is visited by / in the frontier of / in the next frontier of source s0 + j. A level pulls:
// Dn[w] = (OR of D[v] over the in-neighbours v of w, i.e. the set bits of row w of R^T) AND NOT V[w], skipping every
// w already reached from all sources whose frontier is not empty (A, the OR of all D words). One traversal of R^T
// serves 64 sources, and no word is written by two threads. V, D and Dn live in the CTA's slice of `scratch` (3 n words); the CTA takes batches from
// a global counter and, after the last level, writes its 64 output rows through 64 x 64 bit transposes (ballots).
// Threads per CTA and CTAs per SM of the sliced kernel: each CTA holds 3 n words of state, so the number of CTAs
// in flight sets the working set that has to stay in L2.
constexpr int kSlicedThreads = 1024;
constexpr int kSlicedPerSm = 1;

__global__ void __launch_bounds__(kSlicedThreads) smp_sliced_kernel(const int64_t* __restrict__ wptrT,
                                                         const int32_t* __restrict__ widxT,
                                                         const uint64_t* __restrict__ wvalT, int64_t n, int64_t nbatch,
                                                         uint64_t* __restrict__ scratch, uint64_t* __restrict__ out,
                                                         int64_t ldw_out, unsigned long long* bcounter,
                                                         int* levels_max, int max_levels, Deadline dl) {
    __shared__ unsigned long long s_batch;
    __shared__ unsigned long long s_active;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    uint64_t* const V = scratch + static_cast<int64_t>(blockIdx.x) * 3 * n;
    while (true) {
        if (tid == 0) s_batch = atomicAdd(bcounter, 1ull);
        __syncthreads();
        const int64_t b = static_cast<int64_t>(s_batch);
        __syncthreads();
        if (b >= nbatch) break;
        const int64_t s0 = b * 64;
        const int cnt = static_cast<int>(n - s0 < 64 ? n - s0 : 64);
        const uint64_t full = cnt == 64 ? ~0ull : (1ull << cnt) - 1ull;
        uint64_t* D = V + n;
        uint64_t* Dn = V + 2 * n;
        for (int64_t w = tid; w < n; w += blockDim.x) {
            V[w] = 0ull;
            D[w] = (w >= s0 && w < s0 + cnt) ? (1ull << (w - s0)) : 0ull;
        }
        if (tid == 0) s_active = 0ull;
        uint64_t act = full;  // sources whose frontier is not empty
        __syncthreads();
        int lv = 0;
        while (true) {
            int stop = 0;
            if (tid == 0 && dl.budget_ns) stop = dl.past() ? 1 : 0;
            if (__syncthreads_or(stop)) break;
            uint64_t grown = 0ull;
            // two constants per thread at a time, w and w + blockDim.x, whose in-lists are walked in lockstep so
            // that their chains of dependent loads (row range, in-word, frontier words) overlap
            const int64_t stride = blockDim.x;
            for (int64_t wa = tid; wa < n; wa += 2 * stride) {
                const int64_t wb = wa + stride;
                const bool hb = wb < n;
                const uint64_t va = V[wa];
                const uint64_t vb = hb ? V[wb] : ~0ull;
                const uint64_t needa = act & ~va;  // active sources that have not reached the constant
                const uint64_t needb = act & ~vb;
                uint64_t acca = 0ull, accb = 0ull;
                int64_t ea = 0, ea1 = 0, eb = 0, eb1 = 0;
                if (needa) {
                    const longlong2 r = wcsr_row(wptrT, wa);
                    ea = r.x;
                    ea1 = r.y;
                }
                if (needb) {
                    const longlong2 r = wcsr_row(wptrT, wb);
                    eb = r.x;
                    eb1 = r.y;
                }
                while (true) {
                    const bool ta = ea < ea1 && (acca & needa) != needa;
                    const bool tb = eb < eb1 && (accb & needb) != needb;
                    if (!ta && !tb) break;
                    uint64_t ba = ta ? wvalT[ea] : 0ull;
                    uint64_t bb = tb ? wvalT[eb] : 0ull;
                    const int64_t basea = ta ? static_cast<int64_t>(widxT[ea]) << 6 : 0;
                    const int64_t baseb = tb ? static_cast<int64_t>(widxT[eb]) << 6 : 0;
                    while (ba | bb) {
                        if (ba) {
                            const int64_t v = basea + (__ffsll(static_cast<long long>(ba)) - 1);
                            ba &= ba - 1ull;
                            acca |= D[v];
                        }
                        if (bb) {
                            const int64_t v = baseb + (__ffsll(static_cast<long long>(bb)) - 1);
                            bb &= bb - 1ull;
                            accb |= D[v];
                        }
                    }
                    ea += ta ? 1 : 0;
                    eb += tb ? 1 : 0;
                }
                const uint64_t nna = acca & needa;
                Dn[wa] = nna;
                if (nna) V[wa] = va | nna;
                grown |= nna;
                if (hb) {
                    const uint64_t nnb = accb & needb;
                    Dn[wb] = nnb;
                    if (nnb) V[wb] = vb | nnb;
                    grown |= nnb;
                }
            }
            const unsigned glo = __reduce_or_sync(FULL, static_cast<unsigned>(grown));
            const unsigned ghi = __reduce_or_sync(FULL, static_cast<unsigned>(grown >> 32));
            if (lane == 0 && (glo | ghi)) atomicOr(&s_active, static_cast<unsigned long long>(glo) |
                                                                (static_cast<unsigned long long>(ghi) << 32));
            __syncthreads();
            act = s_active;
            __syncthreads();
            if (tid == 0) s_active = 0ull;
            ++lv;
            uint64_t* t = D;
            D = Dn;
            Dn = t;
            if (act == 0ull || lv > max_levels) break;
        }
        if (tid == 0) atomicMax(levels_max, lv);
        // rows s0 .. s0 + cnt - 1 of the output: word wd of row s0 + j = bit j of V[64 wd .. 64 wd + 63]
        const int64_t wpr = (n + 63) >> 6;
        for (int64_t wd = tid >> 5; wd < wpr; wd += blockDim.x >> 5) {
            const int64_t w0 = wd * 64 + lane, w1 = w0 + 32;
            const uint64_t v0 = w0 < n ? V[w0] : 0ull;
            const uint64_t v1 = w1 < n ? V[w1] : 0ull;
            uint64_t mine0 = 0ull, mine1 = 0ull;
#pragma unroll 8
            for (int j = 0; j < 32; ++j) {
                const unsigned lo = __ballot_sync(FULL, ((v0 >> j) & 1ull) != 0ull);
                const unsigned hi = __ballot_sync(FULL, ((v1 >> j) & 1ull) != 0ull);
                if (j == lane) mine0 = static_cast<uint64_t>(lo) | (static_cast<uint64_t>(hi) << 32);
            }
#pragma unroll 8
            for (int j = 32; j < 64; ++j) {
                const unsigned lo = __ballot_sync(FULL, ((v0 >> j) & 1ull) != 0ull);
                const unsigned hi = __ballot_sync(FULL, ((v1 >> j) & 1ull) != 0ull);
                if (j - 32 == lane) mine1 = static_cast<uint64_t>(lo) | (static_cast<uint64_t>(hi) << 32);
            }
            if (lane < cnt) out[(s0 + lane) * ldw_out + wd] = mine0;
            if (lane + 32 < cnt) out[(s0 + lane + 32) * ldw_out + wd] = mine1;
        }
        __syncthreads();
    }
}

// ---- Algorithm 2 for a few query rows, straight from R's bit rows
// One cluster of C CTAs per query row (the largest of 16, 8, 4, 2 whose clusters are all resident at once). Every CTA holds the whole frontier D; CTA
// r ORs the rows of the frontier constants k = r mod C, four in flight per warp, into its own partial N; after a cluster
// barrier it gathers its share of the words from every CTA's N, removes the visited constants and stores the new words
// into every CTA's D; a second barrier ends the level. A query reads the row of each constant it reaches once, so it is
// bound by the two barriers and the row latency per level (2.7 us at n = 5,000, 7 to 10 at 65,536) or, from some tens of
// thousands of constants on, by the rows' bytes; no word index, no transpose and no column is needed. One warp per query over the word indexes of R
// and R^T, which a call has to build first, took 302 us for a call with one query on n = 5,000 constants with 50 facts
// each, 48 us now; n = 65,536 power law 6.1 ms, 0.55 ms now, and 16 queries 5.2 and 1.29 ms. For larger batches the indexes
// are shared and the forms that use them stay.
// Two kinds of rows would be slower here than over the indexes, and are not known from the start:
// * A narrow frontier on its way through many levels (a path: one constant a level). Up to kNarrowN constants one warp
//   then goes on alone, the words of a row in its lanes, without barriers (0.75 us a level). A path from its beginning, by
//   levels of the cluster, over the indexes and so: n = 500: 1,336, 740 and 418 us; 5,000: 13.6, 6.8 and 3.8 ms.
// * Beyond that size, deep or wide rows on large relations, whose levels or bytes cost more than building the indexes and
//   going on there: the cluster writes down its frontier and visited set and stops (RowQueryPlan says when), and the call
//   goes on from them over the indexes (where these have no room on the device, from the sources again, without stopping).
constexpr int kRowsThreads = 512;
constexpr int kRowsWarps = kRowsThreads / 32;
constexpr int kRowsMaxCtas = 16;
constexpr int kNarrowWords = 4;                          // words of a row in a lane of the warp that goes on alone
constexpr int64_t kNarrowN = 32 * 64 * kNarrowWords;
constexpr int kNarrowFrom = 8, kNarrowUntil = 16;       // constants of a frontier that it takes over, and gives back,
constexpr int kNarrowAfter = 6;                          // and levels before it (most rows of dense relations end earlier)

struct RowQueryArgs {
    const uint64_t* R;  // packed rows (bits at columns >= n ignored)
    int64_t ld_r;
    int64_t n;
    const uint64_t* src;  // query rows
    int64_t ld_src;
    uint64_t* out;
    int64_t ld_out;
    int* levels_max;
    int max_levels;
    int reflexive;
    RowQueryPlan plan;
    RowState state;  // where a row that stops leaves its frontier, visited set and source (words null: none stops, and with
                     // levels only the rows that stopped before are expanded)
    int* stopped;    // raised when one does
    Deadline dl;
};

// Levels of a narrow frontier by one warp: until it is empty, has more than kNarrowUntil constants, or the levels or the time
// are used up. The frontier and the visited constants are in its registers, lane l words l, l + 32, ... of a row; they come
// from this CTA's frontier d_s and from every CTA's share of the visited ones, v_s (addresses in shared memory), and go back to
// all of them. Returns the constants of the last frontier; *levels counts on, *stop: out of time. (Not inlined:
// within the kernel's body it makes calls of few levels slower, 52 us instead of 46.)
__device__ __noinline__ int narrow_levels(const uint64_t* __restrict__ R, int64_t ld_r, int n, int wpr, int share, int ctas,
                                          uint32_t d_s, uint32_t v_s, int max_levels, Deadline dl, int* levels, int* stop) {
    const int lane = threadIdx.x & 31;
    uint64_t D[kNarrowWords], V[kNarrowWords], valid[kNarrowWords];
#pragma unroll
    for (int v = 0; v < kNarrowWords; ++v) {
        const int w = 32 * v + lane, left = n - 64 * w;  // what lies beyond column n of a row is not a fact
        D[v] = w < wpr ? ld_dsmem_u64(mapa_shared(d_s + 8u * w, 0)) : 0ull;
        V[v] = w < wpr ? ld_dsmem_u64(mapa_shared(v_s + 8u * (w % share), w / share)) : 0ull;
        valid[v] = left >= 64 ? ~0ull : left > 0 ? (1ull << left) - 1ull : 0ull;
    }
    int found = 0, lv = *levels;
    do {
        uint64_t acc[kNarrowWords];
#pragma unroll
        for (int v = 0; v < kNarrowWords; ++v) acc[v] = 0ull;
#pragma unroll
        for (int u = 0; u < kNarrowWords; ++u) {
            unsigned m = __ballot_sync(FULL, D[u] != 0ull);
            uint64_t bits = 0ull;
            int kb = 0;
            while (m != 0u || bits != 0ull) {
                const uint64_t* row[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    row[q] = nullptr;
                    if (bits == 0ull && m != 0u) {
                        const int sl = __ffs(static_cast<int>(m)) - 1;
                        m &= m - 1u;
                        bits = __shfl_sync(FULL, D[u], sl);
                        kb = (32 * u + sl) * 64;
                    }
                    if (bits != 0ull) {
                        row[q] = R + static_cast<int64_t>(kb + __ffsll(static_cast<long long>(bits)) - 1) * ld_r + lane;
                        bits &= bits - 1ull;
                    }
                }
                uint64_t x[4][kNarrowWords];
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int v = 0; v < kNarrowWords; ++v)
                        x[q][v] = row[q] != nullptr && 32 * v + lane < wpr ? __ldg(row[q] + 32 * v) : 0ull;
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int v = 0; v < kNarrowWords; ++v) acc[v] |= x[q][v];
            }
        }
        unsigned c = 0;
#pragma unroll
        for (int v = 0; v < kNarrowWords; ++v) {
            D[v] = acc[v] & valid[v] & ~V[v];
            V[v] |= D[v];
            c += static_cast<unsigned>(__popcll(D[v]));
        }
        found = static_cast<int>(__reduce_add_sync(FULL, c));
        ++lv;
        if ((lv & 15) == 0 && dl.budget_ns) *stop = __shfl_sync(FULL, lane == 0 ? static_cast<int>(dl.past()) : 0, 0);
    } while (found > 0 && found <= kNarrowUntil && lv <= max_levels && *stop == 0);
#pragma unroll
    for (int v = 0; v < kNarrowWords; ++v) {
        const int w = 32 * v + lane;
        if (w < wpr) {
            st_dsmem_u64(mapa_shared(v_s + 8u * (w % share), w / share), V[v]);
            for (int c = 0; c < ctas; ++c) st_dsmem_u64(mapa_shared(d_s + 8u * w, c), D[v]);
        }
    }
    *levels = lv;
    return found;
}

// kNarrow: narrow frontiers go on in one warp (n <= kNarrowN); else rows may stop. (Two kernels: with both in one, unused, the
// wide levels were 4 to 5 % slower.)
template <bool kNarrow>
__global__ void __launch_bounds__(kRowsThreads) smp_rows_kernel(const RowQueryArgs a) {
    extern __shared__ uint64_t rq_sm[];
    __shared__ int s_flag[2][kRowsMaxCtas];  // by level parity, by each CTA: 4 x the new constants it found, + 1: out of time, + 2: stop
    __shared__ int s_found[2];               // by level parity: this CTA's new constants
    __shared__ int s_narrow[3];              // after narrow levels: levels, constants of the frontier, out of time
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = static_cast<int>(cluster_ctarank()), ctas = static_cast<int>(cluster_nctarank());
    const int wpr = static_cast<int>((a.n + 63) >> 6);
    const int share = (wpr + ctas - 1) / ctas;
    const int base = rank * share;
    const int own = base >= wpr ? 0 : min(share, wpr - base);
    uint64_t* D = rq_sm;
    uint64_t* N[2] = {rq_sm + wpr, rq_sm + 2 * wpr};
    uint64_t* V = rq_sm + 3 * wpr;  // visited, own words
    const uint64_t* src = a.src + static_cast<int64_t>(cluster_id_x()) * a.ld_src;
    uint64_t* out = a.out + static_cast<int64_t>(cluster_id_x()) * a.ld_out;
    // finished by an earlier launch: the whole cluster leaves
    if (!kNarrow && a.state.words == nullptr && a.state.levels != nullptr && a.state.levels[cluster_id_x()] == 0) return;
    const auto valid = [&](int w) {
        const int64_t v = a.n - 64ll * w;
        return v < 64 ? (1ull << v) - 1ull : ~0ull;
    };
    for (int w = tid; w < wpr; w += kRowsThreads) {
        D[w] = src[w] & valid(w);
        N[0][w] = N[1][w] = 0ull;
    }
    for (int w = tid; w < own; w += kRowsThreads) V[w] = 0ull;
    if (tid < 2) s_found[tid] = 0;
    uint64_t mine = 0ull;  // this CTA's constants of a word: bits rank, rank + ctas, ... (ctas divides 64)
    for (int b = rank; b < 64; b += ctas) mine |= 1ull << b;
    cluster_sync();
    int lv = 0, visited = 0, total = 0;  // constants reached, and those of the last level, of the whole relation
    bool stopped = false;
    int p = 0;
    while (true) {
        bool narrow = false;
        for (;; p ^= 1) {
            uint64_t* Np = N[p];
            for (int c0 = 0; c0 < wpr; c0 += 256) {  // 256 words of the rows at a time: 8 per lane
                uint64_t acc[8];
#pragma unroll
                for (int v = 0; v < 8; ++v) acc[v] = 0ull;
                bool any = false;
                for (int w0 = warp; w0 < wpr; w0 += kRowsThreads) {  // lane l: word w0 + kRowsWarps l
                    const int w = w0 + kRowsWarps * lane;
                    const uint64_t d = w < wpr ? D[w] & mine : 0ull;
                    unsigned m = __ballot_sync(FULL, d != 0ull);
                    any |= m != 0u;
                    uint64_t bits = 0ull;
                    int kb = 0;
                    while (m != 0u || bits != 0ull) {
                        const uint64_t* row[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            row[q] = nullptr;
                            if (bits == 0ull && m != 0u) {
                                const int sl = __ffs(m) - 1;
                                m &= m - 1u;
                                bits = __shfl_sync(FULL, d, sl);
                                kb = (w0 + kRowsWarps * sl) * 64;
                            }
                            if (bits != 0ull) {
                                row[q] = a.R + (kb + __ffsll(static_cast<long long>(bits)) - 1) * a.ld_r + c0 + lane;
                                bits &= bits - 1ull;
                            }
                        }
                        uint64_t x[4][8];
#pragma unroll
                        for (int q = 0; q < 4; ++q)
#pragma unroll
                            for (int v = 0; v < 8; ++v)
                                x[q][v] = row[q] != nullptr && c0 + 32 * v + lane < wpr ? __ldg(row[q] + 32 * v) : 0ull;
#pragma unroll
                        for (int q = 0; q < 4; ++q)
#pragma unroll
                            for (int v = 0; v < 8; ++v) acc[v] |= x[q][v];
                    }
                }
                if (any) {
#pragma unroll
                    for (int v = 0; v < 8; ++v)
                        if (acc[v] != 0ull)  // zero beyond wpr
                            atomicOr(reinterpret_cast<unsigned long long*>(&Np[c0 + 32 * v + lane]),
                                     static_cast<unsigned long long>(acc[v]));
                }
            }
            cluster_sync();  // every CTA's N is complete, and nobody reads D any more
            unsigned found = 0;
            const uint32_t n_s = smem_u32(Np + base), d_s = smem_u32(D + base);
            for (int i = tid; i < own; i += kRowsThreads) {
                uint64_t x = 0ull;
#pragma unroll
                for (int c = 0; c < kRowsMaxCtas; ++c)
                    if (c < ctas) x |= ld_dsmem_u64(mapa_shared(n_s + 8u * i, c));
                x &= valid(base + i) & ~V[i];
                V[i] |= x;
                found += static_cast<unsigned>(__popcll(x));
                for (int c = 0; c < ctas; ++c) st_dsmem_u64(mapa_shared(d_s + 8u * i, c), x);
            }
            // the other N was last read before the previous barrier; the next level fills it
            for (int w = tid; w < wpr; w += kRowsThreads) N[p ^ 1][w] = 0ull;
            found = __reduce_add_sync(FULL, found);
            if (lane == 0 && found != 0u) atomicAdd(&s_found[p], static_cast<int>(found));
            __syncthreads();
            if (tid < ctas) {
                int stop = rank == 0 && a.dl.budget_ns && a.dl.past() ? 1 : 0;
                // every 16 levels, by the counts after the level before this one: too deep, or another row has stopped (the
                // indexes are built then, and would wait for this one)
                if (!kNarrow && rank == 0 && a.state.words != nullptr && lv > 0 && (lv & 15) == 0 &&
                    (*static_cast<volatile int*>(a.stopped) != 0 || a.plan.too_deep(a.n, lv, total, visited)))
                    stop |= 2;
                st_dsmem_s32(mapa_shared(smem_u32(&s_flag[p][rank]), tid), 4 * s_found[p] + stop);
            }
            if (tid == 0) s_found[p ^ 1] = 0;
            cluster_sync();  // the new D and the flags are in place
            const unsigned flags = lane < ctas ? static_cast<unsigned>(s_flag[p][lane]) : 0u;
            const unsigned stop = __reduce_or_sync(FULL, flags & 3u);
            total = static_cast<int>(__reduce_add_sync(FULL, flags >> 2));
            visited += total;
            ++lv;
            if (total == 0 || (stop & 1u) != 0u || lv > a.max_levels) break;  // the same in every CTA: no barrier is left open
            if (kNarrow && lv >= kNarrowAfter && total <= kNarrowFrom) {
                narrow = true;
                break;
            }
            if (!kNarrow && a.state.words != nullptr && (stop != 0u || visited > a.plan.most)) {
                stopped = true;
                break;
            }
        }
        if (!kNarrow || !narrow) break;
        // one warp goes on; the others wait at the barrier (each level of its loop ends)
        if (rank == 0 && warp == 0) {
            int levels = lv, out_of_time = 0;
            const int last = narrow_levels(a.R, a.ld_r, static_cast<int>(a.n), wpr, share, ctas, smem_u32(D), smem_u32(V),
                                           a.max_levels, a.dl, &levels, &out_of_time);
            if (lane < ctas) {
                st_dsmem_s32(mapa_shared(smem_u32(&s_narrow[0]), lane), levels);
                st_dsmem_s32(mapa_shared(smem_u32(&s_narrow[1]), lane), last);
                st_dsmem_s32(mapa_shared(smem_u32(&s_narrow[2]), lane), out_of_time);
            }
            __syncwarp();
        }
        cluster_sync();
        lv = s_narrow[0];
        if (s_narrow[1] == 0 || s_narrow[2] != 0 || lv > a.max_levels) break;
        p ^= 1;  // (N of the last level is cleared by the next one)
    }
    if (!kNarrow && stopped) {
        uint64_t* at = a.state.words + static_cast<int64_t>(cluster_id_x()) * 3 * wpr;
        for (int i = tid; i < own; i += kRowsThreads) {
            at[base + i] = D[base + i];
            at[wpr + base + i] = V[i];
            at[2 * wpr + base + i] = src[base + i] & valid(base + i);
        }
        if (rank == 0 && tid == 0) {
            a.state.levels[cluster_id_x()] = lv;
            atomicOr(a.stopped, 1);
        }
        return;
    }
    if (!kNarrow && a.state.words != nullptr && rank == 0 && tid == 0) a.state.levels[cluster_id_x()] = 0;
    if (rank == 0 && tid == 0) atomicMax(a.levels_max, lv);
    for (int i = tid; i < own; i += kRowsThreads)
        out[base + i] = V[i] | (a.reflexive ? src[base + i] & valid(base + i) : 0ull);
    if (rank == ctas - 1)
        for (int64_t w = wpr + tid; w < a.ld_out; w += kRowsThreads) out[w] = 0ull;
}

inline int warps_grid(int64_t rows, int sms) {
    int64_t blocks = (rows + 7) / 8;  // 8 warps of 256 threads
    const int64_t cap = static_cast<int64_t>(sms) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return static_cast<int>(blocks);
}

}  // namespace

cudaError_t launch_product_packed(const uint64_t* A, const uint64_t* B, uint64_t* dst, int64_t n, int64_t ldw,
                                  int or_a, int* changed, int sms, cudaStream_t s, Deadline dl,
                                  unsigned long long* pstat, bool tables) {
    if (n <= 0) return cudaSuccess;
    if (!tables) {
        const int grid = warps_grid(n, sms);
        if (ldw <= 128)
            product_gather_kernel<2><<<grid, 256, 0, s>>>(A, B, dst, n, ldw, or_a, changed, dl, pstat);
        else if (ldw <= 256)
            product_gather_kernel<4><<<grid, 256, 0, s>>>(A, B, dst, n, ldw, or_a, changed, dl, pstat);
        else
            product_gather_kernel<8><<<grid, 256, 0, s>>>(A, B, dst, n, ldw, or_a, changed, dl, pstat);
        return cudaGetLastError();
    }
    const int64_t grid = ((n + kM4Rows - 1) / kM4Rows) * ((ldw + kM4Cols - 1) / kM4Cols);
    const cudaError_t e = allow_smem(product_m4rm_kernel, kM4Smem);
    if (e != cudaSuccess) return e;
    product_m4rm_kernel<<<static_cast<unsigned>(grid), kM4Threads, kM4Smem, s>>>(A, B, dst, n, ldw, or_a, changed,
                                                                                   dl, pstat);
    return cudaGetLastError();
}

cudaError_t launch_insert_fact(uint64_t* P, int64_t n, int64_t ldw, int64_t u, int64_t v, int sms, cudaStream_t s) {
    insert_fact_kernel<<<warps_grid(n, sms), 256, 0, s>>>(P, n, ldw, u, v);
    return cudaGetLastError();
}

int64_t insert_chunk_words(int64_t ldw) { return kInsertChunk * (kInsertChunk / 64 + ldw); }

cudaError_t launch_insert_chunk(uint64_t* P, int64_t n, int64_t ldw, const int32_t* pairs, int m, uint64_t* scratch,
                                int sms, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    if (m > kInsertChunk) return cudaErrorInvalidValue;
    const int mw = (m + 63) / 64;
    uint64_t* G = scratch;
    uint64_t* W = scratch + kInsertChunk * (kInsertChunk / 64);
    const int smem = m * mw * 8;  // at most 128 KiB
    const cudaError_t e = allow_smem(insert_reach_kernel, kInsertChunk * (kInsertChunk / 64) * 8);
    if (e != cudaSuccess) return e;
    insert_links_kernel<<<m, kInsertWarps * 32, 0, s>>>(P, ldw, pairs, m, mw, reinterpret_cast<uint32_t*>(G));
    insert_reach_kernel<<<(m + kInsertWarps - 1) / kInsertWarps, kInsertWarps * 32, smem, s>>>(P, n, ldw, pairs, m, mw, G,
                                                                                              W);
    insert_rows_kernel<<<warps_grid(n, sms), kInsertWarps * 32, 0, s>>>(P, n, ldw, pairs, m, W);
    return cudaGetLastError();
}

cudaError_t launch_wcsr_build(const uint64_t* P, int64_t n, int64_t ldw, const WordIndex& x, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(x.ptr + 2 * n, 0, 2 * sizeof(int64_t), s);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (n + 7) / 8;  // one step each: the next block's reads overlap this one's writes
    wcsr_build_kernel<<<static_cast<unsigned>(blocks), 256, 0, s>>>(P, n, ldw, x.ptr, x.idx, x.val);
    return cudaGetLastError();
}

int smp_packed_max_words() { return 7168; }

// Most shared memory of a warp's arrays, and so of a block of the kernels that choose their warps by it.
constexpr size_t kMostWarpSmem = 200 * 1024;

cudaError_t launch_indexed_rows(const WordIndex& A, const WordIndex& B, const uint64_t* P, int64_t n, int64_t ldw,
                                uint64_t* C, int sms, cudaStream_t s, int* changed) {
    // rows are read and written in 16-byte pieces
    if ((ldw & 1) != 0 || ((reinterpret_cast<uintptr_t>(P) | reinterpret_cast<uintptr_t>(C)) & 15) != 0)
        return cudaErrorInvalidValue;
    int warps = 8;
    while (warps > 1 && warps * ldw * 8 > 32 * 1024) warps >>= 1;
    const size_t smem = static_cast<size_t>(warps) * static_cast<size_t>(ldw) * 8;
    if (smem > kMostWarpSmem) return cudaErrorInvalidValue;
    if (smem > 48 * 1024) {
        const cudaError_t e = allow_smem(indexed_rows_kernel, kMostWarpSmem);
        if (e != cudaSuccess) return e;
    }
    int64_t blocks = (n + warps - 1) / warps;
    // One round of resident blocks, whose rows then end together, is the best for rows of few entries, the first steps of
    // most closures: 5, 10 and 16 blocks an SM: n = 32,768, 4 entries a row 52, 55 and 57 us; 16,000 20, 23 and 25; a grid
    // of 20,000 23, 27 and 29. Rows that have widened prefer more and shorter turns: the third step of n = 14,000 with 2 entries
    // a row 147, 122 and 128 us, of a power-law relation of 30,000 408, 322 and 320. The entries are not known here.
    const int64_t cap = static_cast<int64_t>(sms) * 5;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    indexed_rows_kernel<<<static_cast<int>(blocks), warps * 32, smem, s>>>(A, B, P, n, ldw, C, changed);
    return cudaGetLastError();
}

int64_t smp_sliced_grid(int64_t n, int sms) {
    const int64_t nbatch = (n + 63) / 64;
    const int64_t cap = static_cast<int64_t>(sms) * kSlicedPerSm;
    return nbatch < cap ? nbatch : cap;
}

cudaError_t launch_smp_sliced(const WordIndex& T, int64_t n, uint64_t* scratch, uint64_t* out, int64_t ldw_out, unsigned long long* bcounter,
                              int* levels, int max_levels, int sms, cudaStream_t s, Deadline dl) {
    const int64_t grid = smp_sliced_grid(n, sms);
    smp_sliced_kernel<<<static_cast<int>(grid), kSlicedThreads, 0, s>>>(T.ptr, T.idx, T.val, n, (n + 63) / 64, scratch, out,
                                                             ldw_out, bcounter, levels, max_levels, dl);
    return cudaGetLastError();
}

namespace {
size_t smp_rows_smem(int64_t n, int ctas) {
    const int64_t wpr = (n + 63) / 64;
    return static_cast<size_t>(3 * wpr + (wpr + ctas - 1) / ctas) * 8;
}

cudaLaunchConfig_t smp_rows_config(int64_t n, int64_t q, int ctas, cudaStream_t s, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(q * ctas), 1, 1);
    cfg.blockDim = dim3(kRowsThreads, 1, 1);
    cfg.dynamicSmemBytes = smp_rows_smem(n, ctas);
    cfg.stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = static_cast<unsigned>(ctas);
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// Shared memory of a CTA in steps of kRowsSmemStep, of which it has at most kRowsSmemSteps.
constexpr size_t kRowsSmemStep = 16384, kRowsSmemSteps = 13;

using RowsKernel = void (*)(RowQueryArgs);
RowsKernel rows_kernel(int64_t n) { return n <= kNarrowN ? smp_rows_kernel<true> : smp_rows_kernel<false>; }

cudaError_t smp_rows_attributes(RowsKernel kernel) {
    const cudaError_t e = allow_smem(kernel, kRowsSmemStep * kRowsSmemSteps);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}
}  // namespace

static int rows_ctas(int64_t n, int64_t q) {
    // resident clusters by (device, cluster size, steps of shared memory), asked once each since the query costs more than
    // the launch (0: not asked; else the count + 1); written by any thread, always with the same value
    static std::atomic<unsigned char> known[16][4][kRowsSmemSteps + 1] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (q > kRowsMaxQueries) return 0;
    for (int h = 0; h < 4; ++h) {
        const int ctas = kRowsMaxCtas >> h;
        const size_t step = (smp_rows_smem(n, ctas) + kRowsSmemStep - 1) / kRowsSmemStep;
        if (step > kRowsSmemSteps) return 0;
        const bool keyed = dev >= 0 && dev < 16;
        int clusters = keyed ? static_cast<int>(known[dev][h][step].load(std::memory_order_relaxed)) - 1 : -1;
        if (clusters < 0) {
            cudaLaunchAttribute at;
            cudaLaunchConfig_t cfg = smp_rows_config(n, 1, ctas, nullptr, &at);
            cfg.dynamicSmemBytes = step * kRowsSmemStep;
            clusters = 0;
            if (smp_rows_attributes(rows_kernel(n)) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&clusters, rows_kernel(n), &cfg) != cudaSuccess) {
                cudaGetLastError();
                continue;  // asked again by the next call
            }
            if (clusters > 200) clusters = 200;
            if (keyed) known[dev][h][step].store(static_cast<unsigned char>(clusters + 1), std::memory_order_relaxed);
        }
        if (q <= clusters) return ctas;
    }
    return 0;
}

// When a row stops, from query rows of uniform random, power-law, grid and path relations of 500 to 262,144 constants. Here a
// level takes 2.3 us + 0.1 ns n (half as much again with several clusters) + 3e-16 s n^2, and all rows' bytes come at 9.2 TB/s
// or 98 GB/s a CTA; over the indexes it is 60 us + 1.3e-13 s n^2 to build them, 1.35 us a level and 40 ns a reached constant.
// A row stops when going on is predicted to cost more by twice the build, and not before it has cost 15 % of what it would have
// cost there: narrow rows on large relations end within a few levels, where the build alone is 0.6 ms at n = 65,536
// and 9 ms at 262,144. Calls that never stop, that stop, and over the indexes from the start:
//     63 rows, uniform random, n = 131,072, 3 facts a row    16.1     8.9     8.0 ms
//     63 rows, uniform random, n = 262,144, 2 facts a row    57.8    21.9    18.9 ms
//     63 rows, grid, n = 65,536                              10.0     6.0     4.8 ms
//     1 row, path, n = 65,536                                 502      92      91 ms
// and where the prediction fails: 63 rows, uniform random, n = 65,536, 1.2 facts a row 1.9, 2.6 and 2.1 ms; 1 row of a
// grid, n = 131,072, 8.8, 10.3 and 9.5 ms.
RowQueryPlan smp_rows_plan(int64_t n, int64_t q) {
    RowQueryPlan p{};
    p.ctas = rows_ctas(n, q);
    p.may_stop = p.ctas > 0 && n > kNarrowN;
    if (!p.may_stop) return p;
    const double nn = static_cast<double>(n);
    const double build = 60e-6 + 1.3e-13 * nn * nn, index_level = 1.35e-6, index_row = 40e-9;
    const double level = 2.3e-6 + 0.1e-9 * nn * (q > 1 ? 1.5 : 1.0) + 3e-16 * nn * nn;
    const double ctas = static_cast<double>(q) * p.ctas, row = nn / 8.0 * static_cast<double>(q) / std::min(9.2e12, 98e9 * ctas);
    const double least = 0.15 * (build + nn * index_row);
    p.level_gain = static_cast<float>(level - index_level);
    p.row_gain = static_cast<float>(row - index_row);
    p.need = static_cast<float>(2.0 * build);
    p.first_level = std::max(32, static_cast<int>(least / level));
    p.most = nn * (row - index_row) >= 2.0 * build ? static_cast<int>(least / row) : 0x7FFFFFFF;
    return p;
}

cudaError_t launch_smp_rows(const uint64_t* R, int64_t ld_r, int64_t n, const uint64_t* src, int64_t ld_src, int64_t q,
                            uint64_t* out, int64_t ld_out, int reflexive, int* levels, int max_levels, const RowQueryPlan& plan,
                            RowState state, int* stopped, cudaStream_t s, Deadline dl) {
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = smp_rows_config(n, q, plan.ctas, s, &at);
    const cudaError_t e = smp_rows_attributes(rows_kernel(n));
    if (e != cudaSuccess) return e;
    const RowQueryArgs a{R, ld_r, n, src, ld_src, out, ld_out, levels, max_levels, reflexive, plan, state, stopped, dl};
    return cudaLaunchKernelEx(&cfg, rows_kernel(n), a);
}

cudaError_t launch_square_growth(const WordIndex& x, int64_t n, int64_t ldw, unsigned long long* out, int sms, cudaStream_t s,
                                 unsigned long long* bits_out) {
    const size_t smem = static_cast<size_t>(8) * ((ldw + 31) / 32) * 4;
    if (smem > 48 * 1024) return cudaErrorInvalidValue;
    square_growth_kernel<<<warps_grid(n, sms), 256, smem, s>>>(x, n, ldw, out, bits_out);
    return cudaGetLastError();
}

cudaError_t launch_scatter_transpose(const WordIndex& x, int64_t n, int64_t ldw, uint64_t* out, int sms, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(out, 0, static_cast<size_t>(n) * static_cast<size_t>(ldw) * 8, s);
    if (e != cudaSuccess) return e;
    scatter_transpose_kernel<<<warps_grid(n, sms), 256, 0, s>>>(x.ptr, x.idx, x.val, n, ldw,
                                                                reinterpret_cast<unsigned long long*>(out));
    return cudaGetLastError();
}

cudaError_t launch_indexed_cost(const WordIndex& A, const WordIndex& B, int64_t n, unsigned long long* cost, int sms,
                                cudaStream_t s) {
    indexed_cost_kernel<<<warps_grid(n, sms), 256, 0, s>>>(A, B, n, cost);
    return cudaGetLastError();
}

cudaError_t launch_smp_packed(const WordIndex& x, const WordIndex& T, int64_t n, int64_t ldw, const uint64_t* src,
                              int64_t ldw_src, int64_t q, uint64_t* out, int64_t ldw_out, int* levels, int* qcounter,
                              int reflexive, int sms, cudaStream_t s, Deadline dl, RowState from) {
    // blocks of 1-8 warps, chosen so that as many warps as possible fit an SM's shared memory
    const int64_t per_warp = smp_warp_bytes(ldw);
    if (per_warp > static_cast<int64_t>(kMostWarpSmem)) return cudaErrorInvalidValue;
    int warps = 8;
    while (warps > 1 && warps * per_warp > 32 * 1024) warps >>= 1;
    const size_t smem = static_cast<size_t>(warps) * per_warp;
    const cudaError_t e = allow_smem(smp_packed_kernel, kMostWarpSmem);
    if (e != cudaSuccess) return e;
    int64_t blocks = (q + warps - 1) / warps;
    int per_sm = static_cast<int>((220 * 1024) / (smem + 1024));
    if (per_sm < 1) per_sm = 1;
    if (blocks > static_cast<int64_t>(sms) * per_sm) blocks = static_cast<int64_t>(sms) * per_sm;
    if (blocks < 1) blocks = 1;
    const int max_levels = static_cast<int>(n + 1 < 0x7FFFFFFF ? n + 1 : 0x7FFFFFFF);
    smp_packed_kernel<<<static_cast<int>(blocks), warps * 32, smem, s>>>(
        x.ptr, x.idx, x.val, n, ldw, src, ldw_src, q, out, ldw_out, levels,
        reinterpret_cast<unsigned long long*>(qcounter), reflexive, max_levels, dl, T.ptr, T.idx, T.val, from);
    return cudaGetLastError();
}

cudaError_t launch_packed_ones(const uint64_t* P, int64_t words, unsigned long long* ones, int sms, cudaStream_t s) {
    packed_ones_kernel<<<static_cast<int>(std::min<int64_t>((words + 511) / 512, sms * 8)), 256, 0, s>>>(P, words, ones);
    return cudaGetLastError();
}

cudaError_t launch_bit_transpose(const uint64_t* in, uint64_t* out, int64_t n, int64_t ldw, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const dim3 grid(static_cast<unsigned>((ldw + kTrWords - 1) / kTrWords), static_cast<unsigned>((ldw + 3) / 4));
    bit_transpose_kernel<<<grid, 256, 0, s>>>(in, out, n, ldw);
    return cudaGetLastError();
}

cudaError_t launch_frontier_group(const FrontierJob* jobs, int njobs, int64_t max_n, int64_t max_ldw, int64_t total,
                                  unsigned long long* counter, int sms, cudaStream_t s) {
    if (njobs <= 0) return cudaSuccess;
    const int64_t per_warp = smp_warp_bytes(max_ldw);
    if (per_warp > static_cast<int64_t>(kMostWarpSmem) || njobs > 65535) return cudaErrorInvalidValue;
    const unsigned nj = static_cast<unsigned>(njobs);
    const int64_t wpr = (max_n + 63) / 64;
    int64_t tb = wpr * wpr;
    if (tb > 4096) tb = 4096;
    frontier_transpose_kernel<<<dim3(static_cast<unsigned>(tb < 1 ? 1 : tb), nj), 64, 0, s>>>(jobs);
    const int rows_grid = warps_grid(max_n, sms) / 8 + 1;  // the jobs of a launch share the GPU
    frontier_wcsr_kernel<<<dim3(static_cast<unsigned>(rows_grid), nj, 2), 256, 0, s>>>(jobs);
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    int warps = 8;
    while (warps > 1 && warps * per_warp > 32 * 1024) warps >>= 1;
    const size_t smem = static_cast<size_t>(warps) * per_warp;
    e = allow_smem(frontier_group_kernel, kMostWarpSmem);
    if (e != cudaSuccess) return e;
    int per_sm = static_cast<int>((220 * 1024) / (smem + 1024));
    if (per_sm < 1) per_sm = 1;
    int64_t blocks = (total + warps - 1) / warps;
    if (blocks > static_cast<int64_t>(sms) * per_sm) blocks = static_cast<int64_t>(sms) * per_sm;
    if (blocks < 1) blocks = 1;
    frontier_group_kernel<<<static_cast<int>(blocks), warps * 32, smem, s>>>(jobs, njobs, total, max_ldw, counter);
    return cudaGetLastError();
}

}  // namespace bmlp
