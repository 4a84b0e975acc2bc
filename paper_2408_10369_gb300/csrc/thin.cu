// A squaring R <- R + R R (Eq. 4, Algorithm 1) restricted to the entries of R that are still zero.
//
// R' = R | C with C = R R can differ from R only where R is 0. Let B be any set of columns and Rb the rows that
// have a zero outside B; every zero of R then lies in a column of B or a row of Rb, so
//     C[:, b] = OR_{k : R[k][b] = 1} R[:, k]   (b in B: row b of R'^T gains row k of R^T for each such k)
//     C[r, :] = OR_{k : R[r][k] = 1} R[k, :]   (r in Rb)
// give every entry of R' that can change. With B = the columns holding fewer than n / 2 ones (or very few), a matrix close
// to its closure (the squaring that only confirms the fixpoint, and the one before it on many graphs) has few such
// columns and rows, and they hold few ones: the step costs a few row ORs on bit rows instead of a dense product.
// The result is the same R', so the count of products and the fixpoint test are those of Algorithm 1.
//
// The same holds for any S between R and R': the zeros of S are the entries still open, and C there is computed from
// R. A squaring that is not yet the last ones' kind starts with a product over a slice of k only (S = R + R[:, K] R[K, :]
// for some constants K): when most rows and columns of R are dense, that sets nearly every entry that R' has, and the
// rows and columns that still hold zeros afterwards are the sparse ones.
//
// All of this works on bit rows, which the squaring kernel's epilogue writes beside (or instead of) its E2M1 operands.
#include "internal.h"

namespace bmlp {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

// Ones of a bit row of ldw words (a multiple of 4), by a whole warp; every lane returns them.
__device__ __forceinline__ int row_ones(const uint64_t* __restrict__ row, int64_t ldw, int lane) {
    int c = 0;
#pragma unroll 4
    for (int64_t w = 2 * lane; w < ldw; w += 64) {
        const uint4 v = *reinterpret_cast<const uint4*>(row + w);
        c += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
    }
    return static_cast<int>(__reduce_add_sync(FULL, static_cast<unsigned>(c)));
}

// The ones of each of the n rows of PT into colcnt, and of SrcT into srccnt (blockIdx.y = 1, when the two differ); a warp
// per row.
__global__ void __launch_bounds__(256) bits_count_kernel(const uint64_t* __restrict__ PT, const uint64_t* __restrict__ SrcT,
                                                         int64_t ldw, int64_t n, int32_t* __restrict__ colcnt,
                                                         int32_t* __restrict__ srccnt) {
    const int lane = threadIdx.x & 31;
    const uint64_t* M = blockIdx.y == 0 ? PT : SrcT;
    int32_t* cnt = blockIdx.y == 0 ? colcnt : srccnt;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        const int c = row_ones(M + i * ldw, ldw, lane);
        if (lane == 0) cnt[i] = c;
    }
}

// Columns of B: those with fewer than n / 2 ones in S (colcnt), and those with at most kThinCap in R (srccnt), which cost
// little and may miss many rows (a constant that few others reach within R: a slice of k misses some of its column in
// thousands of dense rows); none that S has filled. A thread per column of the ldw words: Bmask gets their bits, blist
// the columns (in no particular order); stat[0] += |B|, stat[2] += their ones in R and stat[4] = the most of one, an
// entry counting at most kThinCap.
__global__ void __launch_bounds__(256) thin_columns_kernel(const int32_t* __restrict__ colcnt,
                                                           const int32_t* __restrict__ srccnt, int64_t n, int64_t ldw,
                                                           uint32_t* __restrict__ Bmask, int32_t* __restrict__ blist,
                                                           unsigned long long* __restrict__ stat) {
    const int lane = threadIdx.x & 31;
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= ldw * 64) return;  // whole warps: ldw * 64 is a multiple of 32
    const int64_t c = j < n ? colcnt[j] : n;
    const int src = j < n ? srccnt[j] : 0;
    const bool in = c < n && (2 * c < n || src <= kThinCap);
    const unsigned m = __ballot_sync(FULL, in);
    if (lane == 0) Bmask[j >> 5] = m;
    if (m == 0u) return;
    const unsigned ones = in ? static_cast<unsigned>(min(src, kThinCap)) : 0u;
    const unsigned sum = __reduce_add_sync(FULL, ones), top = __reduce_max_sync(FULL, ones);
    unsigned long long at = 0;
    if (lane == 0) {
        at = atomicAdd(&stat[0], static_cast<unsigned long long>(__popc(m)));
        atomicAdd(&stat[2], static_cast<unsigned long long>(sum));
        atomicMax(&stat[4], static_cast<unsigned long long>(top));
    }
    at = __shfl_sync(FULL, at, 0);
    if (in) blist[at + __popc(m & ((1u << lane) - 1u))] = static_cast<int32_t>(j);
}

// Rows of Rb: a zero of P at some column j < n outside B. rlist gets them, Smask (cleared beforehand) those with at most
// kThinCap ones in Src; stat[1] += |Rb|, stat[3] += their ones in Src and stat[5] = the most of one, an entry counting at
// most kThinCap.
__global__ void __launch_bounds__(256) thin_rows_kernel(const uint64_t* __restrict__ P, int64_t ldw, int64_t n,
                                                        const uint64_t* __restrict__ Src,
                                                        const uint64_t* __restrict__ Bmask,
                                                        int32_t* __restrict__ rlist, unsigned int* __restrict__ Smask,
                                                        unsigned long long* __restrict__ stat) {
    const int lane = threadIdx.x & 31;
    const int64_t wpr = (n + 63) >> 6;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    const int64_t first = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    unsigned long long ones = 0;
    int top = 0;
    for (int64_t i = first; i < n; i += warps) {
        bool gap = false;
#pragma unroll 4
        for (int64_t w = lane; w < wpr; w += 32) {
            const int64_t valid = n - w * 64;
            const uint64_t cols = valid < 64 ? (1ull << valid) - 1ull : ~0ull;  // columns j < n of this word
            gap |= ((P[i * ldw + w] | Bmask[w]) & cols) != cols;
        }
        if (__any_sync(FULL, gap)) {
            const int c = row_ones(Src + i * ldw, ldw, lane);
            if (lane == 0) {
                rlist[atomicAdd(&stat[1], 1ull)] = static_cast<int32_t>(i);
                if (c <= kThinCap) atomicOr(&Smask[i >> 5], 1u << (i & 31));
            }
            ones += min(c, kThinCap);
            top = max(top, min(c, kThinCap));
        }
    }
    if (lane == 0 && ones != 0ull) {
        atomicAdd(&stat[3], ones);
        atomicMax(&stat[5], static_cast<unsigned long long>(top));
    }
}

// Of `rows` rows of P spread evenly over its n rows: stat[0] = the most ones of one with at least n / 2 ones,
// stat[1] = the most zeros (among columns < n) of such a row; ones[r] (or null) = the ones of each (warp per row).
__global__ void __launch_bounds__(256) thin_sample_kernel(const uint64_t* __restrict__ P, int64_t ldw, int64_t n, int rows,
                                                          unsigned long long* __restrict__ stat,
                                                          int* __restrict__ ones) {
    const int lane = threadIdx.x & 31;
    const int r = static_cast<int>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= rows) return;
    const unsigned long long c =
        static_cast<unsigned long long>(row_ones(P + static_cast<int64_t>(r) * n / rows * ldw, ldw, lane));
    if (lane != 0) return;
    if (ones != nullptr) ones[r] = static_cast<int>(c);
    if (2 * c >= static_cast<unsigned long long>(n)) {
        atomicMax(&stat[0], c);
        atomicMax(&stat[1], static_cast<unsigned long long>(n) - c);
    }
}

// T[l] = the OR of the rows that the set bits of list entry l's own row name: SrcT rows for the columns of B
// (l < |B| = stat[0]), Src rows for the rows of Rb (the stat[1] entries after them). A warp owns kOrWords words of one
// entry, in registers (ORing into T in memory cost a read and a write of it per named row); the set bits of 32 words at a
// time are dealt into a list in shared memory, so that four named rows are in flight whether a word holds one bit or
// sixty. Bound by the latency of those loads for few entries, by L2 reads for many.
//
// An entry with more than kThinCap ones is there for zeros that its dense row fills within a few named rows (if it is
// going to): it stops when none of them is open, where a row's are those outside B (the columns of B see to the others)
// and a column's those outside the rows of Smask (which are done in full). Stopping after kThinCap rows bounds the step:
// a saturated row of n = 32,768 names 26,000 others, 16 ms for its warp.
constexpr int kOrWords = 256;
__global__ void __launch_bounds__(256) thin_row_or_kernel(int64_t n, const uint64_t* __restrict__ P,
                                                          const uint64_t* __restrict__ PT,
                                                          const uint64_t* __restrict__ Src,
                                                          const uint64_t* __restrict__ SrcT, int64_t ldw,
                                                          const uint64_t* __restrict__ Bmask,
                                                          const uint64_t* __restrict__ Smask,
                                                          const int32_t* __restrict__ blist,
                                                          const int32_t* __restrict__ rlist,
                                                          const unsigned long long* __restrict__ stat,
                                                          uint64_t* __restrict__ T, int* __restrict__ incomplete) {
    __shared__ uint16_t s_named[8][2048];
    const int lane = threadIdx.x & 31;
    uint16_t* named = s_named[threadIdx.x >> 5];
    const int64_t nb = static_cast<int64_t>(stat[0]), entries = nb + static_cast<int64_t>(stat[1]);
    const int64_t chunks = (ldw + kOrWords - 1) / kOrWords;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    for (int64_t item = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
         item < entries * chunks; item += warps) {
        const int64_t l = item / chunks, c0 = (item % chunks) * kOrWords + 2 * lane;
        const bool column = l < nb;
        const uint64_t* M = column ? SrcT : Src;
        const int64_t x = column ? blist[l] : rlist[l - nb];
        const uint64_t* row = M + x * ldw;
        const bool dense = row_ones(row, ldw, lane) > kThinCap;
        uint4 acc[kOrWords / 64];
#pragma unroll
        for (int v = 0; v < kOrWords / 64; ++v) acc[v] = make_uint4(0, 0, 0, 0);
        // whether some zero that this (dense) entry is there for is still open in the warp's words
        const auto open = [&]() {
            bool o = false;
#pragma unroll
            for (int v = 0; v < kOrWords / 64; ++v) {
                const int64_t w = c0 + 64 * v;
                if (w < ldw) {
                    const uint4 h = *reinterpret_cast<const uint4*>((column ? PT : P) + x * ldw + w);
                    const uint4 m = *reinterpret_cast<const uint4*>((column ? Smask : Bmask) + w);
                    const uint64_t lo = (static_cast<uint64_t>(h.y | m.y | acc[v].y) << 32) | (h.x | m.x | acc[v].x);
                    const uint64_t hi = (static_cast<uint64_t>(h.w | m.w | acc[v].w) << 32) | (h.z | m.z | acc[v].z);
                    const int64_t v0 = n - 64 * w, v1 = v0 - 64;
                    const uint64_t c_lo = v0 >= 64 ? ~0ull : v0 > 0 ? (1ull << v0) - 1ull : 0ull;
                    const uint64_t c_hi = v1 >= 64 ? ~0ull : v1 > 0 ? (1ull << v1) - 1ull : 0ull;
                    o |= (~lo & c_lo) != 0ull || (~hi & c_hi) != 0ull;
                }
            }
            return __any_sync(FULL, o) != 0;
        };
        int done = 0;
        bool stop = false;
        for (int64_t wb = 0; wb < ldw && !stop; wb += 32) {
            uint64_t b = wb + lane < ldw ? row[wb + lane] : 0ull;
            if (!__any_sync(FULL, b != 0ull)) continue;
            const int cnt = __popcll(b);
            int at = cnt;  // inclusive prefix
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, at, o);
                if (lane >= o) at += y;
            }
            const int total = __shfl_sync(FULL, at, 31);
            at -= cnt;
            while (b) {
                named[at++] = static_cast<uint16_t>(lane * 64 + (__ffsll(static_cast<long long>(b)) - 1));
                b &= b - 1ull;
            }
            __syncwarp();
            for (int g = 0; g < total; g += 4) {
                uint4 r[4][kOrWords / 64];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int k = named[g + q < total ? g + q : g];  // past the end: the first again
                    const uint64_t* src = M + (wb * 64 + k) * ldw + c0;
#pragma unroll
                    for (int v = 0; v < kOrWords / 64; ++v)
                        r[q][v] = c0 + 64 * v < ldw ? __ldg(reinterpret_cast<const uint4*>(src + 64 * v))
                                                    : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int v = 0; v < kOrWords / 64; ++v) {
                        acc[v].x |= r[q][v].x;
                        acc[v].y |= r[q][v].y;
                        acc[v].z |= r[q][v].z;
                        acc[v].w |= r[q][v].w;
                    }
                done += 4;
                if (dense && (done & 31) == 0) {  // uniform
                    const bool left = open();
                    stop = !left || done >= kThinCap;
                    if (left && stop && lane == 0) atomicOr(incomplete, 1);
                    if (stop) break;
                }
            }
            __syncwarp();  // the list is rewritten for the next words
        }
#pragma unroll
        for (int v = 0; v < kOrWords / 64; ++v)
            if (c0 + 64 * v < ldw) *reinterpret_cast<uint4*>(T + l * ldw + c0 + 64 * v) = acc[v];
    }
}

// One set entry (row, col) of an E2M1 matrix (ld4 bytes per row), ORed into its 32-bit word.
__device__ __forceinline__ void set_nibble(uint8_t* Q, int64_t ld4, int64_t row, int64_t col) {
    const int64_t byte = row * ld4 + (col >> 1);
    const uint32_t bit = static_cast<uint32_t>((byte & 3) * 8 + (col & 1) * 4 + 1);
    atomicOr(reinterpret_cast<unsigned int*>(Q + (byte & ~int64_t(3))), 1u << bit);
}

// The new ones into S (Q and the bit rows P) and S^T (QT and PT): for entry l with index x and computed row T[l], the
// bits of T[l] that row x of P (a row of Rb) or of PT (a column of B) lacks. Rows and columns are handled together, so
// every write is an atomic OR; an entry found by both is written twice. Raises *changed when anything is new. Does
// nothing when `hold` is given and raised.
__global__ void __launch_bounds__(256) thin_apply_kernel(uint64_t* P, uint64_t* PT, const uint64_t* __restrict__ T,
                                                         int64_t ldw, const int32_t* __restrict__ blist,
                                                         const int32_t* __restrict__ rlist,
                                                         const unsigned long long* __restrict__ stat,
                                                         uint8_t* __restrict__ Q, uint8_t* __restrict__ QT, int64_t ld4,
                                                         int* __restrict__ changed, const int* __restrict__ hold) {
    if (hold != nullptr && *hold != 0) return;
    const int64_t nb = static_cast<int64_t>(stat[0]), entries = nb + static_cast<int64_t>(stat[1]);
    const int lane = threadIdx.x & 31;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    bool any = false;
    for (int64_t l = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); l < entries; l += warps) {
        const bool transposed = l < nb;
        const int64_t x = transposed ? blist[l] : rlist[l - nb];
        uint64_t* Cur = (transposed ? PT : P) + x * ldw;
        uint64_t* Other = transposed ? P : PT;
        for (int64_t w = lane; w < ldw; w += 32) {
            uint64_t nb_ = T[l * ldw + w] & ~Cur[w];
            if (!nb_) continue;
            any = true;
            atomicOr(reinterpret_cast<unsigned long long*>(Cur + w), static_cast<unsigned long long>(nb_));
            while (nb_) {
                const int64_t j = w * 64 + (__ffsll(static_cast<long long>(nb_)) - 1);
                nb_ &= nb_ - 1ull;
                const int64_t r = transposed ? j : x, c = transposed ? x : j;  // the new entry is (r, c)
                if (Q != nullptr) {
                    set_nibble(Q, ld4, r, c);
                    set_nibble(QT, ld4, c, r);
                }
                atomicOr(reinterpret_cast<unsigned long long*>(Other + j * ldw + (x >> 6)), 1ull << (x & 63));
            }
        }
    }
    if (__syncthreads_or(any) && threadIdx.x == 0) atomicOr(changed, 1);
}

int rows_grid(int64_t rows, int sms) {
    int64_t blocks = (rows + 7) / 8;
    const int64_t cap = static_cast<int64_t>(sms) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return static_cast<int>(blocks);
}

}  // namespace

cudaError_t launch_thin_sample(const uint64_t* P, int64_t ldw, int64_t n, int rows, unsigned long long* stat, int* ones,
                               cudaStream_t s) {
    if (rows < 1) return cudaSuccess;
    thin_sample_kernel<<<(rows + 7) / 8, 256, 0, s>>>(P, ldw, n, rows, stat, ones);
    return cudaGetLastError();
}

size_t thin_aux_bytes(int64_t n, int64_t ldw) { return static_cast<size_t>(2 * ldw * 8 + 4 * n * 4); }

ThinLists thin_lists(void* aux, int64_t n, int64_t ldw) {
    ThinLists t;
    t.Bmask = static_cast<uint64_t*>(aux);
    t.Smask = t.Bmask + ldw;
    t.colcnt = reinterpret_cast<int32_t*>(t.Smask + ldw);
    t.srccnt = t.colcnt + n;
    t.blist = t.srccnt + n;
    t.rlist = t.blist + n;
    return t;
}

cudaError_t launch_thin_stats(int64_t n, const uint64_t* P, const uint64_t* PT, const uint64_t* Src, const uint64_t* SrcT,
                              int64_t ldw, const ThinLists& t, unsigned long long* stat, int sms, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(stat, 0, 6 * sizeof(unsigned long long), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(t.Smask, 0, static_cast<size_t>(ldw) * 8, s);
    if (e != cudaSuccess) return e;
    const bool two = SrcT != PT;
    bits_count_kernel<<<dim3(rows_grid(n, sms), two ? 2 : 1), 256, 0, s>>>(PT, SrcT, ldw, n, t.colcnt, t.srccnt);
    thin_columns_kernel<<<static_cast<int>((ldw * 64 + 255) / 256), 256, 0, s>>>(
        t.colcnt, two ? t.srccnt : t.colcnt, n, ldw, reinterpret_cast<uint32_t*>(t.Bmask), t.blist, stat);
    thin_rows_kernel<<<rows_grid(n, sms), 256, 0, s>>>(P, ldw, n, Src, t.Bmask, t.rlist,
                                                       reinterpret_cast<unsigned int*>(t.Smask), stat);
    return cudaGetLastError();
}

cudaError_t launch_thin_squaring(int64_t n, uint64_t* P, uint64_t* PT, const uint64_t* Src, const uint64_t* SrcT,
                                 int64_t ldw, const ThinLists& t, const unsigned long long* stat, int64_t entries,
                                 uint64_t* T, uint8_t* Q, uint8_t* QT, int64_t ld4, int* changed, int* incomplete,
                                 bool all_or_none, int sms, cudaStream_t s) {
    // every new one is found from R before any is written
    const int64_t chunks = (ldw + kOrWords - 1) / kOrWords;
    thin_row_or_kernel<<<rows_grid(entries * chunks, sms), 256, 0, s>>>(n, P, PT, Src, SrcT, ldw, t.Bmask, t.Smask, t.blist,
                                                                        t.rlist, stat, T, incomplete);
    thin_apply_kernel<<<rows_grid(entries, sms), 256, 0, s>>>(P, PT, T, ldw, t.blist, t.rlist, stat, Q, QT, ld4, changed,
                                                              all_or_none ? incomplete : nullptr);
    return cudaGetLastError();
}

}  // namespace bmlp
