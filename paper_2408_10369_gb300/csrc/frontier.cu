// Algorithm 2 for many rows at once over a relation whose rows widen fast: closures (the identity's rows) and query
// batches, bit-sliced, with the whole frontier of a batch in one SM's shared memory.
//
// A CTA expands a batch of W rows (W = 64, 32 or 16): word D[v] holds, in bit j, whether constant v is in the frontier of
// row j. A level pulls: Dn[w] = (OR of D[v] over the in-neighbours v of w) AND NOT V[w] for every w that some active row
// has not reached. What bounds it is the issue of a few instructions per in-neighbour around the gather of D at random
// places of shared memory (32 words a warp instruction, about 6 cycles for 64-bit words and 4 for narrower ones). The same
// gather through distributed shared memory (a cluster of CTAs holding D between them, which this replaces) ran at a fifth
// of that, and through L2 slower still.
//
// The lists are laid out for that gather. The constants are renumbered by descending in-degree, so that the constants of a
// warp's tile (one per lane; two per lane, packed into a word, for W = 16) have lists of nearly the same length, and the
// lists of a tile are stored interleaved, four 16-bit neighbours per constant and step (coalesced 256- or 512-byte loads
// from L2). Shorter lists are filled up with the constant itself, whose frontier bits are all visited ones after level 0,
// so that no length is tested then. Constants with more than kHeavy in-neighbours come first (rounded up to whole tiles)
// and are walked by a whole warp each. The lists are built from the word index of R by two passes over its ones (count,
// fill) and a counting sort; no transpose of R is formed.
// Two things keep work out of the levels. A constant that nothing reaches is in no frontier after level 0: such constants
// come last in the new numbers and have no place in D, V and the lists, and their facts are visited directly when they are
// sources. And in a closure a row with one fact, c -> d, is d's row and d: only the rows at the ends of such chains are
// expanded (batches from a list of rows), the others are copied afterwards. Their depths follow from the expanded row's,
// except where the deepest constants of that row all lie on chains to it and the other row's chain has more than one step
// (lists_rows_kernel, derived_rows_kernel): such rows are expanded after all if they could be the deepest. Rows one step from
// a hub that only they lead to, n = 30,000: 795 us, 1,573 with those rows expanded too; n = 4,200: 223 and 280 us.
// Measured: closure of a power-law relation, n = 20,011 (32 levels; 64 % of the rows have one fact and 22 % of the
// constants are not reached), the whole call: 6,590 us with clusters, 1,690 with every row expanded, 680 now; 4,096 query
// rows on n = 65,536 (30 levels) 4,290, 1,740 (16 rows a batch) and 1,375 us (32 rows, one round of the SMs).
#include "internal.h"
#include "ptx.cuh"

namespace bmlp {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int kHeavy = 64;       // in-degree above which a constant's list is walked by a warp
constexpr int kBins = 1024;      // degree bins of the counting sort (the last holds all larger ones)
constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kPrepThreads = 256;
constexpr int kMaxHops = 32;             // longest chain of one-fact rows that a row is derived over
constexpr int kEmptyRoot = 1 << 30;      // in hops: the row at the end is empty
constexpr int kUnclear = 1 << 30;        // in info: the row's deepest constants all have this row as their root,
constexpr int kRootOnly = 1 << 29;       // and the only one is the row's own

// Layout of the work areas: int32 words, then the 16-bit neighbour numbers.
struct Lists {
    // `prep`, filled before the sizes are known on the host
    int32_t* deg;       // in-degree of each constant
    int32_t* meta;      // [0] heavy constants
    int32_t* root;      // of each constant: the constant whose row its own follows from (itself: its row is expanded)
    int32_t* hops;      // steps to it; -1: the row is empty
    int32_t* rows;      // the rows to expand
    int32_t* info;      // of each expanded row: its depth, and kUnclear, kRootOnly
    // `scratch`
    int32_t* red;       // in-degree over constants that are reached themselves; counted down to 0 by the fill
    int32_t* rank;      // new number of each constant
    int32_t* rdeg;      // reduced in-degree by new number
    int32_t* rroot;     // root by new number
    int32_t* hist;      // kBins: constants per bin, then where the bin's next constant goes
    int32_t* start;     // by new number: a heavy constant's first entry; start[heavy + t]: tile t's first step
    uint16_t* ids;      // lists
};

__host__ __device__ inline int64_t align64(int64_t x) { return (x + 63) & ~int64_t(63); }

// Words of D, V and Dn: whole tiles of up to 64 constants behind the heavy ones.
__host__ __device__ inline int64_t tile_pitch(int64_t n) { return align64(n) + 64; }

Lists lists_of(void* prep, void* scratch, int64_t n) {
    Lists l;
    int32_t* p = static_cast<int32_t*>(prep);
    l.deg = p;
    l.meta = l.deg + align64(n);  // deg and meta are cleared together
    l.root = l.meta + 64;
    l.hops = l.root + align64(n);
    l.rows = l.hops + align64(n);
    l.info = l.rows + align64(n);
    p = static_cast<int32_t*>(scratch);
    l.red = p;
    l.hist = l.red + align64(n);  // red and hist are cleared together
    l.rank = l.hist + kBins;
    l.rdeg = l.rank + align64(n);
    l.rroot = l.rdeg + align64(n);
    l.start = l.rroot + align64(n);
    l.ids = reinterpret_cast<uint16_t*>(l.start + align64(n + n / 32 + 2));
    return l;
}

// fn(i, j) for every one (i, j) of the indexed relation: a warp per row, a lane per nonzero word; rows of more than kLong
// words by the whole block afterwards (a power-law row of a thousand facts kept its warp busy for the whole pass: the list
// fill of one took 46 us at n = 20,011 and 58 at 65,536, and takes 14 and 21).
constexpr int kLong = 64, kLongQueue = 64;
template <class Fn>
__device__ __forceinline__ void for_ones(const WordIndex& x, int64_t n, Fn&& fn) {
    __shared__ int s_queue[kLongQueue];
    __shared__ int s_queued;
    const int lane = threadIdx.x & 31;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    const auto row = [&](int64_t i, const longlong2& r, int64_t first, int64_t step) {
        for (int64_t e = r.x + first; e < r.y; e += step) {
            uint64_t d = x.val[e];
            const int base = x.idx[e] << 6;
            while (d) {
                fn(static_cast<int>(i), base + (__ffsll(static_cast<long long>(d)) - 1));
                d &= d - 1ull;
            }
        }
    };
    if (threadIdx.x == 0) s_queued = 0;
    __syncthreads();
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        const longlong2 r = *reinterpret_cast<const longlong2*>(x.ptr + 2 * i);
        if (r.y - r.x > kLong) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_queued, 1);
            at = __shfl_sync(FULL, at, 0);
            if (at < kLongQueue) {
                if (lane == 0) s_queue[at] = static_cast<int>(i);
                continue;
            }
        }
        row(i, r, lane, 32);
    }
    __syncthreads();
    const int queued = min(s_queued, kLongQueue);
    for (int k = 0; k < queued; ++k)
        row(s_queue[k], *reinterpret_cast<const longlong2*>(x.ptr + 2 * static_cast<int64_t>(s_queue[k])), threadIdx.x,
            blockDim.x);
}

__global__ void __launch_bounds__(kPrepThreads) lists_degree_kernel(const WordIndex x, int64_t n, Lists l) {
    for_ones(x, n, [&](int, int j) { atomicAdd(&l.deg[j], 1); });
}

// The one fact of constant c's row, if it has one fact, to another constant; else -1 (*empty: it has none).
__device__ __forceinline__ int only_fact(const WordIndex& x, int c, bool* empty) {
    const longlong2 r = *reinterpret_cast<const longlong2*>(x.ptr + 2 * static_cast<int64_t>(c));
    *empty = r.y == r.x;
    if (r.y - r.x != 1) return -1;
    const uint64_t d = x.val[r.x];
    if (d & (d - 1ull)) return -1;
    const int j = (x.idx[r.x] << 6) + __ffsll(static_cast<long long>(d)) - 1;
    return j != c ? j : -1;
}

// counts[0] = constants that something reaches, counts[1] = rows to expand, counts[3] = the largest in-degree; and with `derive` which
// rows those are: a row with one fact, c -> d, is d's row and d, so only the rows at the ends of such chains are expanded,
// if they have facts at all. (A chain of more than kMaxHops, or a cycle, is expanded from its beginning.)
__global__ void __launch_bounds__(kPrepThreads) lists_rows_kernel(const WordIndex x, int n, Lists l, int derive, int* counts) {
    __shared__ int s_reached, s_expand, s_base, s_top;
    if (threadIdx.x == 0) s_reached = s_expand = s_top = 0;
    __syncthreads();
    const int c = blockIdx.x * kPrepThreads + threadIdx.x;
    int mine = -1;
    if (c < n) {
        const int d = l.deg[c];
        if (d > 0) {
            atomicAdd(&s_reached, 1);
            atomicMax(&s_top, d);
        }
        int at = c, hops = 0;
        bool empty = false;
        if (derive) {
            for (int j; hops <= kMaxHops && (j = only_fact(x, at, &empty)) >= 0; ++hops) at = j;
            if (hops > kMaxHops) {
                at = c;
                hops = 0;
                empty = false;
            }
        }
        l.root[c] = at;
        l.hops[c] = empty ? (hops | kEmptyRoot) : hops;
        if (at == c && !empty) mine = atomicAdd(&s_expand, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_reached) atomicAdd(counts, s_reached);
        s_base = s_expand ? atomicAdd(counts + 1, s_expand) : 0;
        if (s_top) atomicMax(counts + 3, s_top);
    }
    __syncthreads();
    if (mine >= 0) l.rows[s_base + mine] = c;
}

__global__ void __launch_bounds__(kPrepThreads) lists_reduced_kernel(const WordIndex x, int64_t n, Lists l) {
    for_ones(x, n, [&](int i, int j) {
        if (l.deg[i] > 0) atomicAdd(&l.red[j], 1);
    });
}

// Sort key: constants that nothing reaches come last.
__device__ __forceinline__ int list_key(const Lists& l, int c) { return l.deg[c] > 0 ? min(l.red[c] + 1, kBins - 1) : 0; }

// Constants per bin of the key, per block in shared memory, then added up.
__global__ void __launch_bounds__(kPrepThreads) lists_hist_kernel(int n, Lists l) {
    __shared__ int h[kBins];
    for (int b = threadIdx.x; b < kBins; b += kPrepThreads) h[b] = 0;
    __syncthreads();
    for (int c = blockIdx.x * kPrepThreads + threadIdx.x; c < n; c += gridDim.x * kPrepThreads) atomicAdd(&h[list_key(l, c)], 1);
    __syncthreads();
    for (int b = threadIdx.x; b < kBins; b += kPrepThreads)
        if (h[b]) atomicAdd(&l.hist[b], h[b]);
}

// Exclusive prefix over a block of kBins threads (one value each); total to *sum.
__device__ __forceinline__ int block_prefix(int v, int* warp_tot, int* sum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += y;
    }
    __syncthreads();  // warp_tot may still be read from the previous call
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int t = warp_tot[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(FULL, t, d);
            if (lane >= d) t += y;
        }
        warp_tot[lane] = t;
    }
    __syncthreads();
    *sum = warp_tot[31];
    return incl - v + (warp > 0 ? warp_tot[warp - 1] : 0);
}

// Constants of a tile, and 4-entry groups of a step of one.
__host__ __device__ constexpr int tile_constants(int width) { return width == 16 ? 64 : 32; }

// Where each bin starts (larger degrees first), and the number of heavy constants (whole tiles of them). One block of
// kBins threads.
__global__ void __launch_bounds__(kBins) lists_bins_kernel(int n1, int C, Lists l) {
    __shared__ int warp_tot[32];
    const int b = kBins - 1 - static_cast<int>(threadIdx.x);
    int sum = 0;
    const int at = block_prefix(l.hist[b], warp_tot, &sum);
    if (b == kHeavy) l.meta[0] = min((at + C - 1) / C * C, n1);  // the constants of the bins above kHeavy
    __syncthreads();
    l.hist[b] = at;
}

// New numbers: each block takes a run of its bins' places.
__global__ void __launch_bounds__(kPrepThreads) lists_rank_kernel(int n, Lists l) {
    __shared__ int h[kBins];
    const int c = blockIdx.x * kPrepThreads + threadIdx.x;
    for (int b = threadIdx.x; b < kBins; b += kPrepThreads) h[b] = 0;
    __syncthreads();
    const int b = c < n ? list_key(l, c) : 0;
    const int mine = c < n ? atomicAdd(&h[b], 1) : 0;
    __syncthreads();
    for (int k = threadIdx.x; k < kBins; k += kPrepThreads)
        if (h[k]) h[k] = atomicAdd(&l.hist[k], h[k]);
    __syncthreads();
    if (c < n) {
        const int r = h[b] + mine;
        l.rank[c] = r;
        l.rdeg[r] = l.red[c];
        l.rroot[r] = l.root[c];
    }
}

// Place of entry `slot` of the list of the constant of new number r: the heavy lists (first entries in units of 4), then
// the tiles (first steps in units of 4 C entries: 4 entries of each of the C constants).
__device__ __forceinline__ int64_t list_place(const Lists& l, int heavy, int C, int r, int slot) {
    if (r < heavy) return static_cast<int64_t>(l.start[r]) * 4 + slot;
    const int t = (r - heavy) / C, k = (r - heavy) % C;
    return (static_cast<int64_t>(l.start[heavy + t]) + (slot >> 2)) * (4 * C) + k * 4 + (slot & 3);
}

__global__ void __launch_bounds__(kBins) lists_start_kernel(int n1, int C, Lists l) {
    __shared__ int warp_tot[32];
    const int heavy = l.meta[0];
    int base = 0, sum = 0;
    for (int r0 = 0; r0 < heavy; r0 += kBins) {
        const int r = r0 + static_cast<int>(threadIdx.x);
        const int at = block_prefix(r < heavy ? (l.rdeg[r] + 3) / 4 : 0, warp_tot, &sum);
        if (r < heavy) l.start[r] = base + at;
        base += sum;
    }
    base = (base + C - 1) / C;  // tiles start on a step
    const int tiles = (n1 - heavy + C - 1) / C;
    for (int t0 = 0; t0 < tiles; t0 += kBins) {
        const int t = t0 + static_cast<int>(threadIdx.x);
        const int at = block_prefix(t < tiles ? (l.rdeg[heavy + C * t] + 3) / 4 : 0, warp_tot, &sum);
        if (t < tiles) l.start[heavy + t] = base + at;
        base += sum;
    }
    if (threadIdx.x == 0) l.start[heavy + tiles] = base;
}

__global__ void __launch_bounds__(kPrepThreads) lists_fill_kernel(const WordIndex x, int64_t n, int n1, int C, Lists l) {
    const int heavy = l.meta[0];
    for_ones(x, n, [&](int i, int j) {
        if (l.deg[i] == 0) return;  // in no frontier after level 0
        const int slot = atomicSub(&l.red[j], 1) - 1;
        l.ids[list_place(l, heavy, C, l.rank[j], slot)] = static_cast<uint16_t>(l.rank[i]);
    });
    // the rest of each tile list: the constant itself; the places of the last tile beyond n1 (which need nothing): constant 0
    const int tiles = (n1 - heavy + C - 1) / C;
    for (int r = heavy + static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x); r < heavy + C * tiles;
         r += static_cast<int>(gridDim.x * blockDim.x)) {
        const int t = (r - heavy) / C;
        const int end = 4 * (l.start[heavy + t + 1] - l.start[heavy + t]);
        for (int slot = r < n1 ? l.rdeg[r] : 0; slot < end; ++slot)
            l.ids[list_place(l, heavy, C, r, slot)] = static_cast<uint16_t>(r < n1 ? r : 0);
    }
}

struct TileArgs {
    Lists l;
    WordIndex x;
    const uint64_t* src;  // query rows, or null: the rows are those of the constants in l.rows
    int64_t ld_src;
    int n, n1;            // constants, and how many of them something reaches (the first n1 new numbers)
    const int* count;     // rows (on the device)
    int64_t rows;         // rows when `count` is null
    int* info;            // depths of the rows, or null
    uint64_t* out;
    int64_t ld_out;
    void* scratch;        // per CTA: V and Dn, where shared memory does not hold them
    int in_smem;          // how many of V, Dn lie in shared memory behind D (0, 1, 2)
    unsigned long long* counter;
    int* levels_max;
    int max_levels;
    int reflexive;
    Deadline dl;
};

template <class T>
__device__ __forceinline__ T or_warp(T x) {
    if (sizeof(T) == 8) {
        const uint64_t v = static_cast<uint64_t>(x);
        return static_cast<T>(static_cast<uint64_t>(__reduce_or_sync(FULL, static_cast<unsigned>(v))) |
                              (static_cast<uint64_t>(__reduce_or_sync(FULL, static_cast<unsigned>(v >> 32))) << 32));
    }
    return static_cast<T>(__reduce_or_sync(FULL, static_cast<unsigned>(x)));
}

// Per row width: a word of D (T), what a lane holds of a tile's V (Word: P constants' words), and its neighbours of a step.
template <int W>
struct Tile;
template <>
struct Tile<64> {
    using T = unsigned long long;
    using Word = unsigned long long;
    using Ids = uint2;
    static constexpr int P = 1;
};
template <>
struct Tile<32> {
    using T = uint32_t;
    using Word = uint32_t;
    using Ids = uint2;
    static constexpr int P = 1;
};
template <>
struct Tile<16> {
    using T = uint16_t;
    using Word = uint32_t;
    using Ids = uint4;
    static constexpr int P = 2;
};

// The OR of D over four neighbours.
template <class T>
__device__ __forceinline__ T gather4(const T* D, uint32_t a, uint32_t b) {
    return static_cast<T>(D[a & 0xFFFFu] | D[a >> 16] | D[b & 0xFFFFu] | D[b >> 16]);
}
// The same over the first `left` of them only.
template <class T>
__device__ __forceinline__ T gather4(const T* D, uint32_t a, uint32_t b, int left) {
    T x = 0;
    if (left > 0) x |= D[a & 0xFFFFu];
    if (left > 1) x |= D[a >> 16];
    if (left > 2) x |= D[b & 0xFFFFu];
    if (left > 3) x |= D[b >> 16];
    return x;
}
// A lane's neighbours of a step, for its constant or for both (d0, d1: list entries left, when LIMIT).
template <bool LIMIT, class T>
__device__ __forceinline__ T gather_step(const T* D, const uint2& q, int d0, int) {
    return LIMIT ? gather4(D, q.x, q.y, d0) : gather4(D, q.x, q.y);
}
template <bool LIMIT>
__device__ __forceinline__ uint32_t gather_step(const uint16_t* D, const uint4& q, int d0, int d1) {
    const uint32_t lo = LIMIT ? gather4(D, q.x, q.y, d0) : gather4(D, q.x, q.y);
    const uint32_t hi = LIMIT ? gather4(D, q.z, q.w, d1) : gather4(D, q.z, q.w);
    return lo | (hi << 16);
}

// What a warp needs of a tile: each lane's V word and the first two steps of its list. Loaded two tiles ahead: with each
// L2 round trip of a tile waited for in turn a level of n = 65,536 constants took 77 us, with these in flight and two constants per lane 30 us.
template <int W>
struct TileLoad {
    typename Tile<W>::Word v;
    int len;
    const typename Tile<W>::Ids* list;
    typename Tile<W>::Ids q0, q1;
};

template <int W>
struct TileState {
    using T = typename Tile<W>::T;
    using Word = typename Tile<W>::Word;
    using Ids = typename Tile<W>::Ids;
    static constexpr int P = Tile<W>::P;
    static constexpr int C = 32 * P;
    const TileArgs& a;
    T *D, *V, *Dn;
    int* start;
    unsigned char* fresh;
    int n1, heavy, tiles, lane, warp;

    __device__ __forceinline__ void load(int t, TileLoad<W>& x) const {
        x.v = ~Word(0);
        x.len = 0;
        if (t >= tiles) return;
        const int st = start[t];
        x.len = start[t + 1] - st;
        x.list = reinterpret_cast<const Ids*>(a.l.ids) + static_cast<int64_t>(st) * 32 + lane;
        // the pitch of V covers whole tiles; what lies beyond n1 is never written and reads as reached after level 0
        x.v = *reinterpret_cast<const Word*>(V + heavy + C * t + P * lane);
        if (x.len > 0) x.q0 = __ldg(x.list);
        if (x.len > 1) x.q1 = __ldg(x.list + 32);
    }

    // One level; returns the OR of the new words that this warp found (both constants' for P = 2). FIRST: level 0, whose
    // sources are not visited constants, so the entries that fill a list up are left out by its length.
    template <bool FIRST>
    __device__ __forceinline__ Word level(Word act) const {
        Word grown = 0;
        TileLoad<W> x0, x1;
        load(warp, x0);
        load(warp + kWarps, x1);
        for (int r = warp; r < heavy; r += kWarps) {
            const T v = V[r], need = static_cast<T>(static_cast<T>(act) & ~v);
            T acc = 0;
            if (need) {  // uniform
                const int d = a.l.rdeg[r];
                const uint2* list = reinterpret_cast<const uint2*>(a.l.ids) + a.l.start[r];
                for (int e0 = 0; e0 < d; e0 += 128) {
                    const int e = e0 + 4 * lane;
                    const uint2 q = e < d ? list[e >> 2] : make_uint2(0, 0);
                    acc |= gather4(D, q.x, q.y, d - e);
                    if (static_cast<T>(or_warp(acc) & need) == need) break;
                }
                acc = static_cast<T>(or_warp(acc) & need);
            }
            __syncwarp();  // every lane has read V
            if (lane == 0) {
                Dn[r] = acc;
                if (acc) V[r] = static_cast<T>(v | acc);
            }
            grown |= acc;
        }
        for (int t = warp; t < tiles; t += kWarps) {
            TileLoad<W> x = x0;
            x0 = x1;
            load(t + 2 * kWarps, x1);
            const Word need = act & ~x.v;
            bool any_new = false;
            if (x.len > 0 && __any_sync(FULL, need != 0)) {
                const int r = heavy + C * t + P * lane;
                int d0 = 0, d1 = 0;
                if (FIRST) {
                    d0 = r < n1 ? a.l.rdeg[r] : 0;
                    d1 = P > 1 && r + 1 < n1 ? a.l.rdeg[r + 1] : 0;
                }
                Word acc = gather_step<FIRST>(D, x.q0, d0, d1);
                if (x.len > 1) {
                    acc |= gather_step<FIRST>(D, x.q1, d0 - 4, d1 - 4);
                    for (int g = 2; g < x.len; ++g) {
                        // stop once no lane is missing a row that it could still gain
                        const Ids q = __ldg(x.list + g * 32);
                        if (!__any_sync(FULL, (need & ~acc) != 0)) break;
                        acc |= gather_step<FIRST>(D, q, d0 - 4 * g, d1 - 4 * g);
                    }
                }
                const Word nn = acc & need;
                any_new = __any_sync(FULL, nn != 0) != 0;
                if (any_new) {
                    *reinterpret_cast<Word*>(Dn + r) = nn;
                    if (nn) *reinterpret_cast<Word*>(V + r) = x.v | nn;
                }
                grown |= nn;
            }
            if (lane == 0) fresh[t] = any_new ? 1 : 0;
        }
        return grown;
    }
};

// V[r] |= m (V in shared or global memory).
__device__ __forceinline__ void or_place(unsigned long long* V, int r, unsigned long long m) { atomicOr(V + r, m); }
__device__ __forceinline__ void or_place(uint32_t* V, int r, uint32_t m) { atomicOr(V + r, m); }
__device__ __forceinline__ void or_place(uint16_t* V, int r, uint16_t m) {
    atomicOr(reinterpret_cast<uint32_t*>(V) + (r >> 1), static_cast<uint32_t>(m) << (16 * (r & 1)));
}

// Level 0 of a source that nothing reaches (it has no place in D): its facts are reached by the rows of m. A warp calls it;
// returns whether there is one.
template <class T>
__device__ __forceinline__ bool push_source(const TileArgs& a, T* V, int c, T m) {
    const longlong2 e = *reinterpret_cast<const longlong2*>(a.x.ptr + 2 * static_cast<int64_t>(c));
    for (int64_t k = e.x + (threadIdx.x & 31); k < e.y; k += 32) {
        uint64_t d = a.x.val[k];
        const int base = a.x.idx[k] << 6;
        while (d) {
            or_place(V, a.l.rank[base + __ffsll(static_cast<long long>(d)) - 1], m);
            d &= d - 1ull;
        }
    }
    return e.y > e.x;
}

template <int W>
__global__ void __launch_bounds__(kThreads, 1) smp_tile_kernel(const TileArgs a) {
    using S = TileState<W>;
    using T = typename S::T;
    using Word = typename S::Word;
    extern __shared__ __align__(16) unsigned char ti_sm[];
    __shared__ long long s_batch;
    __shared__ unsigned long long s_active, s_pushed, s_clear, s_more;
    __shared__ int s_stop, s_row[64];
    constexpr int VEC = 16 / static_cast<int>(sizeof(T));  // words of a 16-byte copy
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = a.n, n1 = a.n1;
    const int wpr = (n + 63) >> 6;
    const int64_t rows = a.count != nullptr ? *a.count : a.rows;
    const int64_t batches = (rows + W - 1) / W;
    const int pitch = static_cast<int>(tile_pitch(n1));
    T* D = reinterpret_cast<T*>(ti_sm);  // pitch words; then V and Dn as far as they fit
    T* spill = static_cast<T*>(a.scratch) + static_cast<int64_t>(blockIdx.x) * 2 * pitch;
    S st{a, D, a.in_smem >= 1 ? D + pitch : spill, a.in_smem >= 2 ? D + 2 * pitch : spill + pitch,
         reinterpret_cast<int*>(D + (1 + a.in_smem) * pitch), nullptr, n1, a.l.meta[0], 0, lane, warp};
    st.tiles = (n1 - st.heavy + S::C - 1) / S::C;
    st.fresh = reinterpret_cast<unsigned char*>(st.start + n1 / S::C + 2);
    T *V = st.V, *Dn = st.Dn;
    const int heavy = st.heavy;
    for (int t = tid; t <= st.tiles; t += kThreads) st.start[t] = a.l.start[heavy + t];
    while (true) {
        __syncthreads();
        if (tid == 0) s_batch = static_cast<long long>(atomicAdd(a.counter, 1ull));
        __syncthreads();
        if (s_batch >= batches) break;
        const int64_t s0 = s_batch * W;
        const int cnt = static_cast<int>(rows - s0 < W ? rows - s0 : W);
        for (int k = tid; k < pitch / VEC; k += kThreads) {  // nothing is visited
            reinterpret_cast<uint4*>(V)[k] = make_uint4(0, 0, 0, 0);
            reinterpret_cast<uint4*>(D)[k] = make_uint4(0, 0, 0, 0);
        }
        if (tid < cnt) s_row[tid] = a.src == nullptr ? a.l.rows[s0 + tid] : static_cast<int>(s0) + tid;
        if (tid == 0) s_pushed = 0ull;
        __syncthreads();
        // level 0: bit j of D[rank(c)] = constant c is a source of row j of the batch; sources without a place in D at once
        T pushed = 0;
        if (a.src == nullptr) {
            for (int j = warp; j < cnt; j += kWarps) {
                const int c = s_row[j], r = a.l.rank[c];
                const T m = static_cast<T>(T(1) << j);
                if (r < n1) {
                    if (lane == 0) D[r] = m;
                } else if (push_source(a, V, c, m)) {
                    pushed |= m;
                }
            }
        } else {
            for (int wd = warp; wd < wpr; wd += kWarps) {
                const uint64_t r0 = lane < cnt ? a.src[(s0 + lane) * a.ld_src + wd] : 0ull;
                const uint64_t r1 = lane + 32 < cnt ? a.src[(s0 + lane + 32) * a.ld_src + wd] : 0ull;
                if (!__any_sync(FULL, (r0 | r1) != 0)) continue;
                uint64_t c0 = warp_transpose32(static_cast<uint32_t>(r0), lane);  // constants 64 wd + lane and + 32
                uint64_t c1 = warp_transpose32(static_cast<uint32_t>(r0 >> 32), lane);
                if (W > 32) {
                    c0 |= static_cast<uint64_t>(warp_transpose32(static_cast<uint32_t>(r1), lane)) << 32;
                    c1 |= static_cast<uint64_t>(warp_transpose32(static_cast<uint32_t>(r1 >> 32), lane)) << 32;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c = wd * 64 + 32 * h + lane;
                    const T m = c < n ? static_cast<T>(h == 0 ? c0 : c1) : T(0);
                    const int r = m ? a.l.rank[c] : n;
                    if (r < n1) D[r] = m;
                    unsigned far = __ballot_sync(FULL, m && r >= n1);
                    while (far) {
                        const int sl = __ffs(static_cast<int>(far)) - 1;
                        far &= far - 1u;
                        const T mm = static_cast<T>(__shfl_sync(FULL, m, sl));
                        if (push_source(a, V, __shfl_sync(FULL, c, sl), mm)) pushed |= mm;
                    }
                }
            }
        }
        if (lane == 0 && pushed) atomicOr(&s_pushed, static_cast<unsigned long long>(pushed));
        T act = static_cast<T>(cnt == 64 ? ~0ull : (1ull << cnt) - 1ull);  // rows whose frontier may be nonempty
        int lv = 0;
        while (true) {
            if (tid == 0) {
                s_active = s_clear = s_more = 0ull;
                s_stop = a.dl.budget_ns && a.dl.past() ? 1 : 0;
            }
            __syncthreads();  // D, V, the tiles' starts and the flags are in place
            if (s_stop) break;
            const Word both = S::P == 1 ? static_cast<Word>(act) : static_cast<Word>(act) | (static_cast<Word>(act) << 16);
            Word grown = lv == 0 ? st.template level<true>(both) : st.template level<false>(both);
            grown = or_warp(grown);
            if (S::P > 1) grown = (grown | (grown >> 16)) & 0xFFFFu;
            if (lane == 0 && grown) atomicOr(&s_active, static_cast<unsigned long long>(grown));
            __syncthreads();  // Dn is complete, and nobody reads D any more
            const T before = act;
            act = static_cast<T>(lv == 0 ? s_active | s_pushed : s_active);
            const T ended = static_cast<T>(before & ~act);
            if (a.info != nullptr && ended) {
                // rows whose deepest constants are those of D (found one level ago): whether one of them has another root, and
                // whether one of this root is another constant than it
                T other = 0, more = 0;
                if (lv > 0)
                    for (int k = tid; k < n1; k += kThreads) {
                        unsigned long long w = static_cast<unsigned long long>(D[k] & ended);
                        if (w) {
                            const int root = a.l.rroot[k];
                            for (unsigned long long x = w; x; x &= x - 1ull) {
                                const int j = __ffsll(static_cast<long long>(x)) - 1;
                                if (s_row[j] == root) {
                                    w &= ~(1ull << j);
                                    if (a.l.rank[root] != k) more |= static_cast<T>(T(1) << j);
                                }
                            }
                            other |= static_cast<T>(w);
                        }
                    }
                other = or_warp(other);
                more = or_warp(more);
                if (lane == 0 && other) atomicOr(&s_clear, static_cast<unsigned long long>(other));
                if (lane == 0 && more) atomicOr(&s_more, static_cast<unsigned long long>(more));
                __syncthreads();
                if (tid < cnt && ((static_cast<unsigned long long>(ended) >> tid) & 1ull))
                    a.info[s_row[tid]] = lv > 0 && !((s_clear >> tid) & 1ull)
                                             ? lv | kUnclear | ((s_more >> tid) & 1ull ? 0 : kRootOnly)
                                             : lv;
            }
            ++lv;
            if (act == 0 || lv > a.max_levels) break;
            if (lv == 1) {  // what level 0 found is what is visited; from here on the places beyond n1 count as reached
                for (int k = tid; k < pitch / VEC; k += kThreads) {
                    reinterpret_cast<uint4*>(D)[k] = reinterpret_cast<const uint4*>(V)[k];
#pragma unroll
                    for (int x = k * VEC; x < (k + 1) * VEC; ++x)
                        if (x >= n1) {
                            D[x] = 0;
                            V[x] = static_cast<T>(~T(0));
                        }
                }
            } else {
                for (int k = tid; k < pitch / VEC; k += kThreads) {  // a vector lies in one tile, or among the heavy constants
                    const int r = k * VEC;
                    const bool any = r < heavy || (r < n1 && st.fresh[(r - heavy) / S::C] != 0);
                    reinterpret_cast<uint4*>(D)[k] = any ? reinterpret_cast<const uint4*>(Dn)[k] : make_uint4(0, 0, 0, 0);
                }
            }
            __syncthreads();  // s_active is cleared for the next level
        }
        if (tid == 0) atomicMax(a.levels_max, lv);
        __syncthreads();  // V is complete
        // output words: word wd of row s0 + j = bit j of V over the constants 64 wd .. 64 wd + 63
        for (int wd = warp; wd < wpr; wd += kWarps) {
            const int c = wd * 64 + lane;
            const int k0 = c < n ? a.l.rank[c] : n, k1 = c + 32 < n ? a.l.rank[c + 32] : n;
            const uint64_t v0 = k0 < n1 ? static_cast<uint64_t>(V[k0]) : 0ull;
            const uint64_t v1 = k1 < n1 ? static_cast<uint64_t>(V[k1]) : 0ull;
            uint64_t m0 = warp_transpose32(static_cast<uint32_t>(v0), lane) |
                          (static_cast<uint64_t>(warp_transpose32(static_cast<uint32_t>(v1), lane)) << 32);
            uint64_t m1 = 0ull;
            if (W > 32)
                m1 = warp_transpose32(static_cast<uint32_t>(v0 >> 32), lane) |
                     (static_cast<uint64_t>(warp_transpose32(static_cast<uint32_t>(v1 >> 32), lane)) << 32);
            if (a.reflexive && a.src != nullptr) {
                const int valid = n - wd * 64;
                const uint64_t m = valid < 64 ? (1ull << valid) - 1ull : ~0ull;
                if (lane < cnt) m0 |= a.src[(s0 + lane) * a.ld_src + wd] & m;
                if (lane + 32 < cnt) m1 |= a.src[(s0 + lane + 32) * a.ld_src + wd] & m;
            }
            if (lane < cnt) a.out[static_cast<int64_t>(s_row[lane]) * a.ld_out + wd] = m0;
            if (lane + 32 < cnt) a.out[static_cast<int64_t>(s_row[lane + 32]) * a.ld_out + wd] = m1;
        }
        for (int64_t w = wpr + tid; w < a.ld_out; w += kThreads)  // words of a row beyond n
            for (int j = 0; j < cnt; ++j) a.out[static_cast<int64_t>(s_row[j]) * a.ld_out + w] = 0ull;
    }
}

// Level count of a row of `hops` steps to an expanded row of info d, if it is certain, else an upper bound. The chain reaches
// each of its constants within its steps, the expanded row's others come behind it. One step reaches the root alone: where the
// root is the only constant of the deepest level, the level before it counts (it holds others), else that level does.
__device__ __forceinline__ int derived_levels(int hops, int d, bool* certain) {
    *certain = (d & kUnclear) == 0 || hops == 1;
    return hops + (d & ~(kUnclear | kRootOnly)) + 1 - ((d & kRootOnly) != 0 ? 1 : 0);
}

// Rows that follow from an expanded row or from none: that row and the constants of the chain to it, a warp per row.
// *levels: the largest level count of those whose depth is certain; counts[2] that of the others if it were what their
// chain adds to the expanded row's (it is less when the deepest constants of that row all lie on their chain).
__global__ void __launch_bounds__(kPrepThreads) derived_rows_kernel(const WordIndex x, int n, Lists l, uint64_t* out,
                                                                    int64_t ld_out, int* levels, int* counts) {
    const int lane = threadIdx.x & 31;
    int top = 0, unclear = 0;
    for (int i = static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 5); i < n;
         i += static_cast<int>((gridDim.x * blockDim.x) >> 5)) {
        const int root = l.root[i], h = l.hops[i], hops = h & ~kEmptyRoot;
        const bool empty = (h & kEmptyRoot) != 0;
        if (root == i && !empty) continue;  // expanded
        uint64_t* row = out + static_cast<int64_t>(i) * ld_out;
        const uint64_t* from = out + static_cast<int64_t>(root) * ld_out;
        for (int64_t w = lane; w < ld_out; w += 32) row[w] = empty ? 0ull : from[w];
        int at = i, mine = -1;
        bool e = false;
        for (int k = 0; k < hops; ++k) {
            at = only_fact(x, at, &e);
            if (k == lane) mine = at;
        }
        __syncwarp();
        if (mine >= 0) atomicOr(reinterpret_cast<unsigned long long*>(row) + (mine >> 6), 1ull << (mine & 63));
        bool certain = true;
        const int lv = derived_levels(hops, empty ? 0 : l.info[root], &certain);
        if (certain) top = max(top, lv);
        else unclear = max(unclear, lv);
    }
    if (lane == 0) {
        if (top > 0) atomicMax(levels, top);
        if (unclear > 0) atomicMax(counts + 2, unclear);
    }
}

// The derived rows of uncertain depth that could still be deeper than *levels, to be expanded after all: counts[1] of them.
__global__ void __launch_bounds__(kPrepThreads) unclear_rows_kernel(int n, Lists l, const int* levels, int* counts) {
    const int i = blockIdx.x * kPrepThreads + threadIdx.x;
    if (i >= n || l.root[i] == i || (l.hops[i] & kEmptyRoot)) return;
    bool certain = true;
    if (derived_levels(l.hops[i], l.info[l.root[i]], &certain) > *levels && !certain) l.rows[atomicAdd(counts + 1, 1)] = i;
}

// Shared memory of a CTA with `kept` of V, Dn in it.
size_t tile_smem(int64_t n, int width, int kept) {
    const int C = tile_constants(width);
    return static_cast<size_t>((1 + kept) * tile_pitch(n) * (width / 8) + 4 * (n / C + 2) + n / C + 1);
}
constexpr size_t kTileSmem = 226 * 1024;

int tile_kept(int64_t n, int width) {
    int kept = 2;
    while (kept > 0 && tile_smem(n, width, kept) > kTileSmem) --kept;
    return kept;
}

template <int W>
cudaError_t launch_tiles(const TileArgs& a, int grid, size_t smem, cudaStream_t s) {
    const cudaError_t e = allow_smem(smp_tile_kernel<W>, kTileSmem);
    if (e != cudaSuccess) return e;
    smp_tile_kernel<W><<<grid, kThreads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Rows per batch: the width whose frontier fits shared memory and whose rounds over the SMs cost least (a gather of
// 64-bit words takes about half as long again as one of narrower ones); the wider one on a tie.
int smp_tile_width(int64_t n1, int64_t rows, int sms) {
    int best = 0;
    double best_cost = 0.0;
    for (int width = 64; width >= 16; width >>= 1) {
        if (tile_smem(n1, width, 0) > kTileSmem) continue;
        const int64_t batches = (rows + width - 1) / width;
        const double cost = static_cast<double>((batches + sms - 1) / sms) * (width == 64 ? 1.5 : 1.0);
        if (best == 0 || cost < best_cost) {
            best = width;
            best_cost = cost;
        }
    }
    return best;
}

size_t smp_tile_prep_bytes(int64_t n) { return static_cast<size_t>(5 * align64(n) + 64) * 4; }

size_t smp_tile_bytes(int64_t n, int64_t n1, int64_t ones, int width, int sms) {
    // words of the work area, lists (each tile's longest list, rounded up to a step), V and Dn of every CTA
    const int64_t ints = 4 * align64(n) + align64(n + n / 32 + 2) + kBins;
    const int64_t ids = ones + 4 * n + 64 * (kHeavy + 4) + 512 + 4 * 64 * (n / 32 + 2);
    return static_cast<size_t>(align64(ints) * 4 + align64(ids) * 2) +
           static_cast<size_t>(sms) * 2 * static_cast<size_t>(tile_pitch(n1)) * (width / 8);
}

cudaError_t launch_smp_tile_prep(const WordIndex& x, int64_t n, void* prep, int* counts, bool derive, int sms, cudaStream_t s) {
    const Lists l = lists_of(prep, nullptr, n);
    cudaError_t e = cudaMemsetAsync(l.deg, 0, static_cast<size_t>(align64(n) + 64) * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(counts, 0, 4 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    const int rows_grid = static_cast<int>((n + 7) / 8 < sms * 8 ? (n + 7) / 8 : sms * 8);
    const int each = static_cast<int>((n + kPrepThreads - 1) / kPrepThreads);
    lists_degree_kernel<<<rows_grid, kPrepThreads, 0, s>>>(x, n, l);
    lists_rows_kernel<<<each, kPrepThreads, 0, s>>>(x, static_cast<int>(n), l, derive ? 1 : 0, counts);
    return cudaGetLastError();
}

cudaError_t launch_smp_tiles(const WordIndex& x, int64_t n, int64_t n1, int64_t ones, const uint64_t* src, int64_t ld_src,
                             int64_t rows, uint64_t* out, int64_t ld_out, int reflexive, int width, void* prep, void* scratch,
                             bool derive, bool again, int* counts, unsigned long long* counter, int* levels, int max_levels,
                             int sms, cudaStream_t s, Deadline dl) {
    const Lists l = lists_of(prep, scratch, n);
    const int C = tile_constants(width), nn = static_cast<int>(n), nn1 = static_cast<int>(n1);
    const int rows_grid = static_cast<int>((n + 7) / 8 < sms * 8 ? (n + 7) / 8 : sms * 8);
    const int each = static_cast<int>((n + kPrepThreads - 1) / kPrepThreads);
    cudaError_t e = cudaSuccess;
    if (again) {
        e = cudaMemsetAsync(counts + 1, 0, sizeof(int), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, sizeof(*counter), s);
        if (e != cudaSuccess) return e;
        unclear_rows_kernel<<<each, kPrepThreads, 0, s>>>(nn, l, levels, counts);
    } else {
        e = cudaMemsetAsync(l.red, 0, static_cast<size_t>(align64(n) + kBins) * 4, s);
        if (e != cudaSuccess) return e;
        lists_reduced_kernel<<<rows_grid, kPrepThreads, 0, s>>>(x, n, l);
        lists_hist_kernel<<<each < sms ? each : sms, kPrepThreads, 0, s>>>(nn, l);
        lists_bins_kernel<<<1, kBins, 0, s>>>(nn1, C, l);
        lists_rank_kernel<<<each, kPrepThreads, 0, s>>>(nn, l);
        lists_start_kernel<<<1, kBins, 0, s>>>(nn1, C, l);
        lists_fill_kernel<<<rows_grid, kPrepThreads, 0, s>>>(x, n, nn1, C, l);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the rows expanded after all are as many as the device finds, up to all of them
    const int64_t batches = ((again ? n : rows) + width - 1) / width;
    const int grid = static_cast<int>(batches < sms ? batches : sms);
    TileArgs a{};
    a.l = l;
    a.x = x;
    a.src = src;
    a.ld_src = ld_src;
    a.n = nn;
    a.n1 = nn1;
    a.rows = rows;
    a.count = src == nullptr ? counts + 1 : nullptr;
    a.info = derive && !again ? l.info : nullptr;
    a.out = out;
    a.ld_out = ld_out;
    const int64_t state = static_cast<int64_t>(smp_tile_bytes(n, n1, ones, width, 0));  // V and Dn come last
    a.scratch = static_cast<unsigned char*>(scratch) + state;
    a.in_smem = tile_kept(n1, width);
    a.counter = counter;
    a.levels_max = levels;
    a.max_levels = max_levels;
    a.reflexive = reflexive;
    a.dl = dl;
    const size_t smem = tile_smem(n1, width, a.in_smem);
    if (grid > 0) {
        if (width == 64) e = launch_tiles<64>(a, grid, smem, s);
        else if (width == 32) e = launch_tiles<32>(a, grid, smem, s);
        else e = launch_tiles<16>(a, grid, smem, s);
    }
    if (e == cudaSuccess && derive && !again) {
        derived_rows_kernel<<<rows_grid, kPrepThreads, 0, s>>>(x, nn, l, out, ld_out, levels, counts);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace bmlp
