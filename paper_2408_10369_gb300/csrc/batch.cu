// Grouped batch runner: many independent linear recursive programs of uneven
// sizes (closures, paper Sec. 3.3 program P2, and two-relation compositions,
// Sec. 3.4 Thm. 1) evaluated together.
//
// Two CUDA graph WHILE nodes hold the squaring steps R <- R + R R. In the
// first ONE launch per iteration (packed_group_kernel) squares, on bit rows,
// the problems that the autotuner put there and every other one for as long as
// that is cheaper than its share of a grouped tensor-core product; in the
// second ONE persistent tensor-core launch (tc_group_kernel) squares the
// problems handed over, over a device work list of (problem, tile) items. A
// single-block planner after each retires problems whose changed flag stayed 0
// (or that reached their cap), flips the ping-pong parity of the others,
// rebuilds the work lists and sets the node's condition. Encoding, the
// iterations, the final products of compositions and decoding are one graph
// launch; the host reads back the per-problem iteration counts once at the end.
//
// Problems large enough to fill the GPU on their own (n >= solo_n) run in the
// same graph as device-driven single-problem pipelines, on up to four
// parallel branches: squarings on word-indexed bit rows while the next one costs less than a
// tensor-core product (the same cost model and the same switch as the
// single-problem path, decided by a one-thread kernel that sets the
// condition of a WHILE node), then squarings on packed E2M1 operands on the
// tensor cores in a second WHILE node, two products per iteration with a
// guard word so that the second is skipped once the first changed nothing,
// then the decode (closures) or I + R2+ and the final product with R1
// (compositions). No host round trip per squaring.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"

namespace bmlp {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int TILE = 64;

// ------------------------------------------------------------ encoding --
// Columns c0 .. c0 + 15 of row r of n packed rows (padding bits zero).
__device__ __forceinline__ uint32_t src_bits16(const uint64_t* in, int64_t ldw, int64_t n, int64_t r, int64_t c0) {
    if (r >= n || c0 >= n) return 0;
    return static_cast<uint32_t>((in[r * ldw + (c0 >> 6)] >> (c0 & 63)) & 0xFFFFu);
}

__device__ __forceinline__ uint4 expand16(uint32_t m) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t v = 0;
#pragma unroll
        for (int x = 0; x < 4; ++x) v |= (((m >> (4 * q + x)) & 1u) ? static_cast<uint32_t>(BMLP_E4M3_ONE) : 0u) << (8 * x);
        w[q] = v;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// R and R^T (ld x ld E4M3 bytes, zero padding) of n packed rows, tiles
// strided over the blocks of this problem.
__device__ void encode_e4m3(const uint64_t* in, int64_t ldw, int64_t n, uint8_t* R, uint8_t* RT, int64_t ld,
                            uint16_t (*masks)[TILE / 16 + 1]) {
    const int tid = threadIdx.x;
    const int r = tid >> 2, cseg = (tid & 3) * 16;
    const int64_t tiles1 = ld / TILE;
    for (int64_t t = blockIdx.x; t < tiles1 * tiles1; t += gridDim.x) {
        const int64_t row0 = (t / tiles1) * TILE, col0 = (t % tiles1) * TILE;
        const uint32_t m = src_bits16(in, ldw, n, row0 + r, col0 + cseg);
        masks[r][tid & 3] = static_cast<uint16_t>(m);
        *reinterpret_cast<uint4*>(R + (row0 + r) * ld + col0 + cseg) = expand16(m);
        __syncthreads();
        uint32_t tb = 0;
#pragma unroll
        for (int x = 0; x < 16; ++x) tb |= ((masks[cseg + x][r >> 4] >> (r & 15)) & 1u) << x;
        *reinterpret_cast<uint4*>(RT + (col0 + r) * ld + row0 + cseg) = expand16(tb);
        __syncthreads();
    }
}

// A caller matrix as n packed rows of ldw words (a warp per row, padding bits and words zero); its ones are added into
// *ones and the most of one row goes into *top (null: not counted).
__device__ void pack_rows(const void* in, int fmt, int64_t n, uint64_t* P, int64_t ldw, unsigned long long* ones,
                          int* top) {
    const int lane = threadIdx.x & 31;
    const int64_t wpr = (n + 63) / 64;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    unsigned long long sum = 0;
    unsigned most = 0;
    for (int64_t r = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n; r += warps) {
        unsigned c = 0;
        for (int64_t w0 = 0; w0 < ldw; w0 += 32) {
            uint64_t bits = 0;
            const int64_t w = w0 + lane;
            if (fmt == BMLP_FMT_U8) {
                const uint8_t* row = static_cast<const uint8_t*>(in) + r * n;
                for (int64_t x = w0; x < w0 + 32 && x < wpr; ++x) {  // 64 bytes of the row per step, a byte per lane
                    const int64_t j = x * 64 + lane;
                    const unsigned lo = __ballot_sync(FULL, j < n && row[j] != 0);
                    const unsigned hi = __ballot_sync(FULL, j + 32 < n && row[j + 32] != 0);
                    if (x == w) bits = static_cast<uint64_t>(lo) | (static_cast<uint64_t>(hi) << 32);
                }
            } else if (w < wpr) {
                bits = static_cast<const uint64_t*>(in)[r * wpr + w];
                const int64_t valid = n - w * 64;
                if (valid < 64) bits &= (1ull << valid) - 1ull;
            }
            if (w < ldw) P[r * ldw + w] = bits;
            c += __popcll(bits);
        }
        c = __reduce_add_sync(FULL, c);
        sum += c;
        most = c > most ? c : most;
    }
    if (ones != nullptr && lane == 0 && sum != 0ull) {
        atomicAdd(ones, sum);
        atomicMax(top, static_cast<int>(most));
    }
}

// blockIdx.y = problem. 256 threads. Every problem starts as packed rows.
__global__ void __launch_bounds__(256) batch_encode_kernel(const GroupProblem* probs, const GroupState* st) {
    const GroupProblem& g = probs[blockIdx.y];
    if (g.n == 0) return;
    pack_rows(g.kind == 1 ? g.in2 : g.in1, g.fmt, g.n, g.P[0], g.ldw, &st->ones[blockIdx.y], &st->top[blockIdx.y]);
    if (g.kind == 1) pack_rows(g.in1, g.fmt, g.n, g.PR1, g.ldw, nullptr, nullptr);
}

// Tensor-core operands of the problems that the bit rows handed over.
__global__ void __launch_bounds__(256) batch_operands_kernel(const GroupProblem* probs, const GroupState* st) {
    __shared__ uint16_t masks[TILE][TILE / 16 + 1];
    const GroupProblem& g = probs[blockIdx.y];
    if (g.n == 0 || st->phase[blockIdx.y] == 0) return;
    encode_e4m3(g.P[st->ppar[blockIdx.y]], g.ldw, g.n, g.M[0], g.T[0], g.ld, masks);
    if (g.kind == 1) encode_e4m3(g.PR1, g.ldw, g.n, g.X, g.R1T, g.ld, masks);  // X is scratch here
}

// ------------------------------------------------------------- planner --
// Whether the next squaring of a tensor-core problem is cheaper on its bit rows: every one of R names a row of ldw words
// (L2 reads over the whole GPU), and the row with the most ones is one warp's work; against its share of a grouped
// tensor-core product (ld^3 at the E4M3 kernel's rate). Relations of a knowledge graph with fewer constants than triples
// stay sparse up to their closure: their dense products were 7.2 ms of a batch, their bit rows are 0.5 ms.
__device__ __forceinline__ bool rows_cheaper(const GroupProblem& g, unsigned long long ones, int top) {
    const double ld = static_cast<double>(g.ld);
    return top <= 192 && static_cast<double>(ones) * static_cast<double>(g.ldw) * 1.5e-12 < 2.0 * ld * ld * ld / 2.4e15;
}

// mode 0: start (every squaring problem on bit rows, except the tensor-core ones whose bit rows are too full); mode 1:
// after a bit-row squaring; mode 3: start of the tensor-core loop (the problems handed over); mode 4: after a tensor-core
// product (1 and 4: retire, flip parity, count; 1 also hands over); mode 2: final products of compositions.
__global__ void __launch_bounds__(1024) batch_plan_kernel(const GroupProblem* probs, const GroupState* st, int nprob,
                                                          int mode, cudaGraphConditionalHandle h, int set_cond) {
    __shared__ unsigned long long warp_sum[32];
    const int t = threadIdx.x, lane = t & 31;
    const int per = (nprob + 1023) / 1024;
    const int a = t * per, b = min(a + per, nprob);
    int stc = 0, spk = 0;
    for (int p = a; p < b; ++p) {
        const GroupProblem& g = probs[p];
        if (mode == 0) {
            // frontier-engine problems (engine 2) take no part in the squaring loop; their closure rows are
            // written into P[1] by the grouped frontier launch
            st->parity[p] = g.engine == 2 ? 1 : 0;
            st->iters[p] = 0;
            st->notconv[p] = 0;
            st->phase[p] = g.n > 0 && g.engine == 0 && !rows_cheaper(g, st->ones[p], st->top[p]) ? 1 : 0;
            st->active[p] = (g.n > 0 && g.engine != 2 && st->phase[p] == 0) ? 1 : 0;
        } else if (mode == 1 || mode == 4) {
            if (st->active[p]) {
                st->iters[p] += 1;
                st->parity[p] ^= 1;
                if (!st->changed[p]) {
                    st->active[p] = 0;
                } else if (st->iters[p] >= g.cap) {
                    st->active[p] = 0;
                    st->notconv[p] = 1;
                } else if (mode == 1 && g.engine == 0 && !rows_cheaper(g, st->ones[p], st->top[p])) {
                    st->active[p] = 0;
                    st->phase[p] = 1;
                }
            }
        } else if (mode == 3) {
            st->ppar[p] = st->parity[p];
            st->active[p] = st->phase[p];
            if (st->phase[p]) st->parity[p] = 0;
        } else {
            st->active[p] = (g.kind == 1 && g.n > 0 && st->phase[p] == 1) ? 1 : 0;
        }
        if (mode <= 1) {
            st->ones[p] = 0ull;
            st->top[p] = 0;
        }
        st->changed[p] = 0;
        const int act = st->active[p];
        const int ctc = (act && mode >= 2) ? g.m_tiles * g.n_tiles : 0;
        const int cpk = (act && mode <= 1) ? static_cast<int>(g.n) : 0;
        st->tc_offs[p] = ctc;
        st->pk_offs[p] = cpk;
        stc += ctc;
        spk += cpk;
    }
    // exclusive prefixes over the threads, both at once (each total is below 2^31): in registers, since the plan runs between
    // any two steps of all problems and a scan through shared memory with its twenty barriers was a third of its 5 us
    const unsigned long long mine = (static_cast<unsigned long long>(stc) << 32) | static_cast<unsigned>(spk);
    unsigned long long incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long v = __shfl_up_sync(FULL, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) warp_sum[t >> 5] = incl;
    __syncthreads();
    if (t < 32) {
        unsigned long long w = warp_sum[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long v = __shfl_up_sync(FULL, w, off);
            if (lane >= off) w += v;
        }
        warp_sum[lane] = w;
    }
    __syncthreads();
    const unsigned long long before = incl - mine + (t >= 32 ? warp_sum[(t >> 5) - 1] : 0ull);
    int rt = static_cast<int>(before >> 32), rp = static_cast<int>(before & 0xFFFFFFFFull);
    for (int p = a; p < b; ++p) {
        const int ct = st->tc_offs[p], cp = st->pk_offs[p];
        st->tc_offs[p] = rt;
        st->pk_offs[p] = rp;
        rt += ct;
        rp += cp;
    }
    if (t == 0) {
        const int tt = static_cast<int>(warp_sum[31] >> 32), tp = static_cast<int>(warp_sum[31] & 0xFFFFFFFFull);
        st->tc_offs[nprob] = tt;
        st->pk_offs[nprob] = tp;
        *st->tc_total = tt;
        *st->pk_total = tp;
        if (set_cond) cudaGraphSetConditional(h, (tt + tp) > 0 ? 1u : 0u);
    }
}

// ------------------------------------------------ packed squaring step --
// C_i = A_i' | OR_{k : A_ik = 1} B_k for one row, by a whole warp (A_i' = init, a row of ldw words), in chunks of 64 words
// (two per lane), four named rows in flight. A row of up to 16 or 32 words takes a quarter or half of the lanes, so the
// warp's groups of 8 or 16 take its nonzero words in turn (a batch of 1,000 entities: six launches of 226 us in all, 128 now;
// the batch 594 and 494 us). Returns the ones written; *grew: C_i != init.
__device__ __forceinline__ unsigned gather_row(const uint64_t* __restrict__ arow, const uint64_t* __restrict__ B,
                                               const uint64_t* __restrict__ init, uint64_t* __restrict__ out, int64_t ldw,
                                               int lane, bool* grew) {
    unsigned ones = 0;
    uint32_t any = 0;
    const int gs = ldw <= 16 ? 8 : ldw <= 32 ? 16 : 32, groups = 32 / gs, group = lane / gs;
    for (int64_t c0 = 0; c0 < ldw; c0 += 64) {
        const int64_t w = c0 + 2 * (lane & (gs - 1));
        const bool in = w < ldw;  // ldw is even: both words
        const uint4 old = in ? *reinterpret_cast<const uint4*>(init + w) : make_uint4(0, 0, 0, 0);
        uint4 acc = old;
        for (int64_t wb = 0; wb < ldw; wb += 32) {
            const uint64_t aw = wb + lane < ldw ? arow[wb + lane] : 0ull;
            unsigned m = __ballot_sync(FULL, aw != 0ull);
            if (groups > 1) {  // this group's share of the nonzero words (at most 32 words: one pass)
                const int turn = __popc(m & ((1u << lane) - 1u)) & (groups - 1);
                unsigned share = 0;
                for (int q = 0; q < groups; ++q) {
                    const unsigned x = __ballot_sync(FULL, aw != 0ull && turn == q);
                    if (q == group) share = x;
                }
                m = share;
            }
            uint64_t bits = 0ull;
            int64_t kb = 0;
            while (__any_sync(FULL, m != 0u || bits != 0ull)) {
                uint4 x[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const bool word = bits == 0ull && m != 0u;
                    const int sl = word ? __ffs(static_cast<int>(m)) - 1 : 0;
                    const uint64_t next = __shfl_sync(FULL, aw, sl);
                    if (word) {
                        m &= m - 1u;
                        bits = next;
                        kb = (wb + sl) * 64;
                    }
                    x[q] = make_uint4(0, 0, 0, 0);
                    if (bits != 0ull) {
                        const int64_t k = kb + __ffsll(static_cast<long long>(bits)) - 1;
                        bits &= bits - 1ull;
                        if (in) x[q] = *reinterpret_cast<const uint4*>(B + k * ldw + w);
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    acc.x |= x[q].x;
                    acc.y |= x[q].y;
                    acc.z |= x[q].z;
                    acc.w |= x[q].w;
                }
            }
        }
        for (int off = gs; off < 32; off <<= 1) {
            acc.x |= __shfl_xor_sync(FULL, acc.x, off);
            acc.y |= __shfl_xor_sync(FULL, acc.y, off);
            acc.z |= __shfl_xor_sync(FULL, acc.z, off);
            acc.w |= __shfl_xor_sync(FULL, acc.w, off);
        }
        if (in && group == 0) {
            *reinterpret_cast<uint4*>(out + w) = acc;
            any |= (old.x ^ acc.x) | (old.y ^ acc.y) | (old.z ^ acc.z) | (old.w ^ acc.w);
            ones += __popc(acc.x) + __popc(acc.y) + __popc(acc.z) + __popc(acc.w);
        }
    }
    *grew = __any_sync(FULL, any != 0u) != 0;
    return __reduce_add_sync(FULL, ones);
}

// One warp per active row of every problem on bit rows: R' = R | R R.
__global__ void __launch_bounds__(256) packed_group_kernel(const GroupProblem* probs, const GroupState* st, int nprob) {
    const int lane = threadIdx.x & 31;
    const int64_t warp_id = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const int total = *st->pk_total;
    const int* offs = st->pk_offs;
    // a run of consecutive rows per warp, so that the problem of the first is searched for once
    const int64_t per = (total + nwarps - 1) / nwarps;
    const int64_t first = warp_id * per, end = first + per < total ? first + per : total;
    if (first >= end) return;
    int lo = 0, hi = nprob - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (offs[mid] <= first) lo = mid; else hi = mid - 1;
    }
    for (int64_t item = first; item < end; ++item) {
        while (offs[lo + 1] <= item) ++lo;  // offs[nprob] = total > item
        const GroupProblem& g = probs[lo];
        const int par = st->parity[lo];
        const int64_t i = item - offs[lo];
        const uint64_t* src = g.P[par];
        bool grew = false;
        const unsigned ones = gather_row(src + i * g.ldw, src, src + i * g.ldw, g.P[par ^ 1] + i * g.ldw, g.ldw, lane, &grew);
        if (lane == 0) {
            if (grew) atomicOr(&st->changed[lo], 1);
            if (ones != 0u) {
                atomicAdd(&st->ones[lo], static_cast<unsigned long long>(ones));
                atomicMax(&st->top[lo], static_cast<int>(ones));
            }
        }
    }
}

// Compositions whose closure ended on bit rows: (I + R2+) R1 into the other packed buffer, a warp per row.
__global__ void __launch_bounds__(256) batch_compose_rows_kernel(const GroupProblem* probs, const GroupState* st) {
    const GroupProblem& g = probs[blockIdx.y];
    if (g.kind != 1 || g.n == 0 || st->phase[blockIdx.y] != 0) return;
    const int lane = threadIdx.x & 31;
    const int par = st->ppar[blockIdx.y];
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); i < g.n; i += warps) {
        bool grew = false;
        gather_row(g.P[par] + i * g.ldw, g.PR1, g.PR1 + i * g.ldw, g.P[par ^ 1] + i * g.ldw, g.ldw, lane, &grew);
    }
}

// I + R2+ for the compositions (diagonal of the closure buffer).
__global__ void batch_compose_prep_kernel(const GroupProblem* probs, const GroupState* st) {
    const GroupProblem& g = probs[blockIdx.y];
    if (g.kind != 1 || g.n == 0 || st->phase[blockIdx.y] == 0) return;
    uint8_t* R = g.M[st->parity[blockIdx.y]];
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < g.n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        R[i * g.ld + i] = BMLP_E4M3_ONE;
}

// Results into the callers' output buffers.
__global__ void __launch_bounds__(256) batch_decode_kernel(const GroupProblem* probs, const GroupState* st) {
    const GroupProblem& g = probs[blockIdx.y];
    if (g.n == 0) return;
    const int64_t n = g.n, wpr = (n + 63) / 64;
    const int refl = (g.kind == 0) ? g.reflexive : 0;
    const int lane = threadIdx.x & 31;
    const bool tc = st->phase[blockIdx.y] == 1;
    const uint8_t* M = (g.kind == 1) ? g.X : g.M[st->parity[blockIdx.y]];
    const uint64_t* P = g.P[st->ppar[blockIdx.y] ^ (g.kind == 1 ? 1 : 0)];
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    // a warp per row: words of 64 columns, or bytes, from the E4M3 bytes of a row or from its words
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        if (g.fmt == BMLP_FMT_U8) {
            uint8_t* out = static_cast<uint8_t*>(g.out) + i * n;
            for (int64_t j = lane; j < n; j += 32) {
                const bool b = tc ? M[i * g.ld + j] != 0 : ((P[i * g.ldw + (j >> 6)] >> (j & 63)) & 1ull) != 0ull;
                out[j] = (b || (refl && i == j)) ? 1 : 0;
            }
        } else {
            uint64_t* out = static_cast<uint64_t*>(g.out) + i * wpr;
            for (int64_t w0 = 0; w0 < wpr; w0 += 32) {
                const int64_t w = w0 + lane;
                uint64_t bits = 0;
                if (!tc) {
                    bits = w < wpr ? P[i * g.ldw + w] : 0ull;
                } else {
                    for (int64_t x = w0; x < w0 + 32 && x < wpr; ++x) {  // ld is a multiple of 256: both bytes exist
                        const uint8_t* b = M + i * g.ld + x * 64 + lane;
                        const unsigned lo = __ballot_sync(FULL, b[0] != 0);
                        const unsigned hi = __ballot_sync(FULL, b[32] != 0);
                        if (x == w) bits = static_cast<uint64_t>(lo) | (static_cast<uint64_t>(hi) << 32);
                    }
                    const int64_t valid = n - w * 64;
                    if (valid < 64) bits &= valid > 0 ? (1ull << valid) - 1ull : 0ull;
                }
                if (refl && (i >> 6) == w) bits |= 1ull << (i & 63);
                if (w < wpr) out[w] = bits;
            }
        }
    }
}

// ------------------------------------------- device-driven large problems --
// Control words of one large problem (ints; 64-bit words at SW_COST, SW_SMP and SW_TSTAT, 8-byte aligned).
enum SoloWord : int {
    SW_ITERS = 0,     // squarings issued so far
    SW_NOTDONE = 1,   // 1 while the closure is not finished on bit rows
    SW_NOTCONV = 2,   // stopped at the cap while still changing
    SW_CHANGED = 3,   // set by the squaring kernels
    SW_GC = 4,        // guard of the first tensor-core product of a loop iteration
    SW_G1 = 5,        // guard of the second
    SW_TCHANGED = 6,  // set by a restricted squaring that found new ones
    SW_RES = 7,       // 1: a restricted squaring left the closure in Q1 (else Q0 holds it)
    SW_COST = 8,      // word ORs of the next bit-row squaring: total, largest row (2 x u64)
    SW_THIN_GO = 12,  // the restricted squaring is cheaper than a product (set inside its statistics' IF)
    SW_STOP = 13,     // a restricted squaring ended the loop
    SW_TOPEN = 14,    // a restricted squaring stopped with zeros open and left R as it was
    SW_SMP = 16,      // the row sample after a product (2 x u64, thin.cu)
    SW_TSTAT = 20,    // the restricted squaring's statistics (6 x u64, thin.cu)
    SW_WORDS = 32
};

// dst = src, 16 bytes per thread and step (sizes are multiples of 16 bytes).
__global__ void solo_copy_kernel(uint4* __restrict__ dst, const uint4* __restrict__ src, int64_t n16) {
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n16;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        dst[i] = src[i];
}

__global__ void solo_init_kernel(int* w) {
    for (int i = 0; i < SW_WORDS; ++i) w[i] = 0;
    w[SW_NOTDONE] = 1;
}

// After the cost pass on the current bit rows: stop if the last squaring changed nothing (the closure is done),
// hand over to the tensor cores if the next squaring is predicted dearer than a tensor-core product or would use
// the last product the cap allows, else run it (same rule as the single-problem path).
__global__ void solo_rows_decide_kernel(int* w, int cap, int first, double step_s, double s_word, double s_row,
                                        double limit, cudaGraphConditionalHandle h) {
    unsigned long long* cost = reinterpret_cast<unsigned long long*>(w + SW_COST);
    if (!first) {
        w[SW_ITERS] += 1;
        if (!w[SW_CHANGED]) {
            w[SW_NOTDONE] = 0;
            cudaGraphSetConditional(h, 0u);
            return;
        }
    }
    const double t = step_s + fmax(static_cast<double>(cost[0]) * s_word, static_cast<double>(cost[1]) * s_row);
    if (w[SW_ITERS] + 1 >= cap || t > limit) {
        cudaGraphSetConditional(h, 0u);
        return;
    }
    w[SW_CHANGED] = 0;
    cost[0] = 0;
    cost[1] = 0;
    cudaGraphSetConditional(h, 1u);
}

__global__ void solo_mid_kernel(int* w, cudaGraphConditionalHandle h) {
    const int go = w[SW_NOTDONE];
    w[SW_GC] = go;
    w[SW_G1] = 0;
    w[SW_CHANGED] = 0;
    cudaGraphSetConditional(h, go ? 1u : 0u);
}

// After tensor-core product `half` (0: Q0 -> Q1, 1: Q1 -> Q0) of a loop iteration. A product that changed nothing
// wrote R' = R, so both buffers hold the closure and either may be decoded.
__global__ void solo_tc_decide_kernel(int* w, int cap, int half, cudaGraphConditionalHandle h) {
    if (!w[half == 0 ? SW_GC : SW_G1]) return;  // that product was skipped
    w[SW_ITERS] += 1;
    bool go = w[SW_CHANGED] != 0;
    w[SW_CHANGED] = 0;
    if (go && w[SW_ITERS] >= cap) {
        w[SW_NOTCONV] = 1;
        go = false;
    }
    if (half == 0) {
        w[SW_G1] = go ? 1 : 0;
        if (!go) {
            w[SW_GC] = 0;
            cudaGraphSetConditional(h, 0u);
        }
    } else {
        w[SW_G1] = 0;
        if (!go) w[SW_GC] = 0;
        cudaGraphSetConditional(h, go ? 1u : 0u);
    }
}

// After tensor-core product `half` (its R in Q[half ^ 1]): whether the next squaring may run only on the rows and
// columns of R that still hold zeros. Only while the loop goes on (the next product's guard is set) and when the
// sampled rows that reach at least n / 2 constants agree in count within spread x n; the sample is cleared for the
// next product. The statistics' IF reads hT; the squaring's IF stays off until they say it is cheaper.
__global__ void solo_thin_gate_kernel(int* w, int half, int64_t n, double spread, cudaGraphConditionalHandle hT) {
    unsigned long long* sm = reinterpret_cast<unsigned long long*>(w + SW_SMP);
    const int next = half == 0 ? w[SW_G1] : w[SW_GC];
    const double sp = static_cast<double>(sm[0]) - (static_cast<double>(n) - static_cast<double>(sm[1]));
    const bool go = next != 0 && sm[0] > 0 && sp <= spread * static_cast<double>(n);
    sm[0] = sm[1] = 0;
    w[SW_THIN_GO] = 0;
    cudaGraphSetConditional(hT, go ? 1u : 0u);
}

// Inside the statistics' IF: the restricted squaring's cost by the bit-row model (the word ORs over the GPU, or one
// warp's heaviest list entry) against a tensor-core product, as on the host loop.
__global__ void solo_thin_decide_kernel(int* w, int64_t ldw, double fixed_s, double s_word, double s_one, double limit) {
    const unsigned long long* st = reinterpret_cast<const unsigned long long*>(w + SW_TSTAT);
    const double words = static_cast<double>(st[2] + st[3]) * static_cast<double>(ldw);
    const double top = static_cast<double>(st[4] > st[5] ? st[4] : st[5]);
    const double t = fixed_s + fmax(words * s_word, top * s_one);
    w[SW_THIN_GO] = t < limit ? 1 : 0;
    w[SW_TCHANGED] = 0;
    w[SW_TOPEN] = 0;
}

__global__ void solo_thin_arm_kernel(const int* w, cudaGraphConditionalHandle hT2) {
    cudaGraphSetConditional(hT2, w[SW_THIN_GO] ? 1u : 0u);
}

// After a restricted squaring that followed product `half` (R in Q[half ^ 1], updated in place): one more squaring
// counted; if it changed nothing that buffer holds the closure, and at the cap while changing the loop stops
// unconverged; either way the guards go off and the loop-control kernel ends the loop.
__global__ void solo_thin_post_kernel(int* w, int half, int cap) {
    w[SW_THIN_GO] = 0;
    if (w[SW_TOPEN]) return;  // R is as it was: the next product squares it
    w[SW_ITERS] += 1;
    bool stop = false;
    if (!w[SW_TCHANGED]) {
        stop = true;
    } else if (w[SW_ITERS] >= cap) {
        w[SW_NOTCONV] = 1;
        stop = true;
    }
    if (stop) {
        w[SW_RES] = half ^ 1;
        w[SW_GC] = 0;
        w[SW_G1] = 0;
        w[SW_STOP] = 1;
    }
}

__global__ void solo_loop_ctl_kernel(const int* w, cudaGraphConditionalHandle hC) {
    if (w[SW_STOP]) cudaGraphSetConditional(hC, 0u);
}

// After the tensor-core loop: the closure into Q0 when a restricted squaring left it in Q1 (16 bytes per thread).
__global__ void solo_result_copy_kernel(const int* w, uint4* __restrict__ q0, const uint4* __restrict__ q1, int64_t n16) {
    if (w[SW_RES] != 1) return;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n16;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        q0[i] = q1[i];
}

// --------------------------------------------------------------- host --
inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

int bucket_of(int64_t n) {
    int b = 0;
    while ((int64_t(1) << b) < n) ++b;
    return b;
}

int log2_ceil(int64_t n) {
    int k = 0;
    while ((int64_t(1) << k) < n) ++k;
    return k;
}

bool on_device(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

uint64_t fnv(uint64_t h, const void* data, size_t len) {
    const unsigned char* p = static_cast<const unsigned char*>(data);
    for (size_t i = 0; i < len; ++i) {
        h ^= p[i];
        h *= 1099511628211ull;
    }
    return h;
}

}  // namespace

// Cached, instantiated batch graph of a context.
struct BatchCache {
    uint64_t key = 0;
    int nprob = 0;
    std::vector<int> order;          // device slot -> caller index
    GroupProblem* d_probs = nullptr;
    GroupState* d_st = nullptr;
    int* d_ints = nullptr;           // ones (u64) | top | parity | active | iters | changed | notconv | tc_offs |
                                      // pk_offs | totals | phase | ppar
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    size_t ws_bytes = 0;
    std::vector<int> h_iters, h_notconv;
    FrontierJob* d_jobs = nullptr;   // closures by frontier expansion (engine 2), then a 64-bit row counter
    std::vector<int> solo;           // caller indices of the device-driven large problems, in run order
    int* d_solo = nullptr;           // SW_WORDS control words per large problem
    std::vector<int> h_solo;
};

void batch_cache_free(bmlp_ctx* ctx) {
    BatchCache* c = static_cast<BatchCache*>(ctx->batch);
    if (!c) return;
    if (c->exec) cudaGraphExecDestroy(c->exec);
    if (c->graph) cudaGraphDestroy(c->graph);
    if (c->d_probs) cudaFree(c->d_probs);
    if (c->d_st) cudaFree(c->d_st);
    if (c->d_ints) cudaFree(c->d_ints);
    if (c->d_solo) cudaFree(c->d_solo);
    if (c->d_jobs) cudaFree(c->d_jobs);
    delete c;
    ctx->batch = nullptr;
}

namespace {

#define BCK(call, what)                                          \
    do {                                                         \
        cudaError_t e_ = (call);                                 \
        if (e_ != cudaSuccess) return cuda_err(ctx, e_, what);   \
    } while (0)

#define BST(call)                      \
    do {                               \
        bmlp_status s_ = (call);       \
        if (s_ != BMLP_OK) return s_;  \
    } while (0)

bmlp_status add_kernel(bmlp_ctx* ctx, cudaGraph_t g, cudaGraphNode_t* node, const cudaGraphNode_t* deps, size_t ndeps,
                       void* func, dim3 grid, dim3 block, size_t smem, void** args) {
    cudaKernelNodeParams kp = {};
    kp.func = func;
    kp.gridDim = grid;
    kp.blockDim = block;
    kp.sharedMemBytes = static_cast<unsigned>(smem);
    kp.kernelParams = args;
    kp.extra = nullptr;
    BCK(cudaGraphAddKernelNode(node, g, deps, ndeps, &kp), "cudaGraphAddKernelNode");
    return BMLP_OK;
}

// 0: tensor-core squarings; 1: squarings on packed rows; 2: frontier expansion of every row (closures only).
int engine_for(bmlp_ctx* ctx, const bmlp_problem& p, int variant) {
    if (p.kind == BMLP_PROBLEM_COMPOSE) return 0;
    const int v = p.variant ? p.variant : variant;
    if (v == BMLP_RMS_TC || v == BMLP_SMP_TC) return 0;
    if (v == BMLP_RMS_PACKED) return 1;
    if (v == BMLP_SMP_PACKED) return 2;
    const int b = bucket_of(p.n);
    if (b < 32 && ctx->tune[b] >= 0) return ctx->tune[b];
    return 0;
}

// Captures the grouped frontier launches into the batch graph after `after`; *tail receives the nodes the next
// node must depend on.
bmlp_status add_frontier_chain(bmlp_ctx* ctx, BatchCache* c, int njobs, int64_t max_n, int64_t max_ldw, int64_t total,
                               cudaGraphNode_t after, std::vector<cudaGraphNode_t>* tail) {
    cudaStream_t cs = nullptr;
    BCK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking), "capture stream");
    struct Stream {
        cudaStream_t a;
        ~Stream() { cudaStreamDestroy(a); }
    } guard_stream{cs};
    BCK(cudaStreamBeginCaptureToGraph(cs, c->graph, &after, nullptr, 1, cudaStreamCaptureModeRelaxed),
        "begin capture of the frontier launches");
    auto* counter = reinterpret_cast<unsigned long long*>(c->d_jobs + njobs);
    cudaError_t e = launch_frontier_group(c->d_jobs, njobs, max_n, max_ldw, total, counter, ctx->sm_count, cs);
    cudaStreamCaptureStatus st;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    if (e == cudaSuccess) e = cudaStreamGetCaptureInfo(cs, &st, nullptr, nullptr, &deps, nullptr, &nd);
    if (e == cudaSuccess) tail->assign(deps, deps + nd);
    cudaGraph_t g = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(cs, &g);
    if (e != cudaSuccess || e2 != cudaSuccess) return cuda_err(ctx, e != cudaSuccess ? e : e2, "frontier launches");
    return BMLP_OK;
}

bool is_solo(const bmlp_problem& p, int variant, int64_t solo_n) {
    if (solo_n <= 0 || p.n < solo_n) return false;
    if (p.kind == BMLP_PROBLEM_COMPOSE) return true;
    const int v = p.variant ? p.variant : variant;
    return v == BMLP_AUTO || v == BMLP_RMS_TC;
}

bmlp_status build_solo(bmlp_ctx* ctx, BatchCache* c, const bmlp_problem* probs, long long wait_cycles);

bmlp_status build_batch(bmlp_ctx* ctx, const bmlp_problem* probs, int64_t count, int variant, long long wait_cycles,
                        uint64_t key, int64_t solo_n, BatchCache** out) {
    batch_cache_free(ctx);
    BatchCache* c = new BatchCache();
    ctx->batch = c;
    c->key = key;
    // large problems first, as device-driven pipelines after the grouped part; the rest grouped, most expensive
    // first (the work lists are then longest-first)
    for (int64_t i = 0; i < count; ++i)
        if (is_solo(probs[i], variant, solo_n)) c->solo.push_back(static_cast<int>(i));
        else c->order.push_back(static_cast<int>(i));
    std::stable_sort(c->solo.begin(), c->solo.end(), [&](int a, int b) { return probs[a].n > probs[b].n; });
    c->nprob = static_cast<int>(c->order.size());
    const int np = c->nprob;
    std::stable_sort(c->order.begin(), c->order.end(),
                     [&](int a, int b) { return probs[a].n > probs[b].n; });
    std::vector<GroupProblem> hp(np);
    std::vector<size_t> offsets(np);
    size_t total = 0;
    auto take = [&](size_t bytes) {
        size_t o = total;
        total += round_up(static_cast<int64_t>(bytes), 1024);
        return o;
    };
    std::vector<size_t> offM0(np), offM1(np), offT0(np), offT1(np), offX(np), offR1T(np), offP0(np), offP1(np);
    std::vector<size_t> offPT(np), offPR1(np), offPtr[2], offIdx[2], offVal[2];
    for (int m = 0; m < 2; ++m) {
        offPtr[m].resize(np);
        offIdx[m].resize(np);
        offVal[m].resize(np);
    }
    for (int s = 0; s < np; ++s) {
        const bmlp_problem& p = probs[c->order[s]];
        GroupProblem& g = hp[s];
        memset(&g, 0, sizeof(g));
        g.n = p.n;
        g.kind = p.kind;
        g.fmt = p.fmt;
        g.reflexive = p.reflexive;
        g.in1 = p.R1;
        g.in2 = p.R2;
        g.out = p.out;
        g.engine = engine_for(ctx, p, variant);
        g.cap = log2_ceil(p.n > 1 ? p.n : 2) + 2;
        if (p.n == 0) continue;
        if (g.engine == 0) {
            g.ld = round_up(p.n, TC_PAD);
            g.m_tiles = static_cast<int32_t>(g.ld / TC_BM);
            g.n_tiles = static_cast<int32_t>(g.ld / TC_BN);
            g.k_blocks = static_cast<int32_t>(g.ld / TC_BK);
            const size_t mat = static_cast<size_t>(g.ld * g.ld);
            offM0[s] = take(mat);
            offM1[s] = take(mat);
            offT0[s] = take(mat);
            offT1[s] = take(mat);
            if (p.kind == BMLP_PROBLEM_COMPOSE) {
                offX[s] = take(mat);
                offR1T[s] = take(mat);
            }
        }
        g.ldw = round_up((p.n + 63) / 64, 2);
        const size_t bytes = static_cast<size_t>(p.n * g.ldw * 8);
        offP0[s] = take(bytes);
        offP1[s] = take(bytes);
        if (p.kind == BMLP_PROBLEM_COMPOSE) offPR1[s] = take(bytes);
        {
            if (g.engine == 2) {  // R^T and the word indexes of R and R^T (entries sized for the dense worst case)
                offPT[s] = take(bytes);
                for (int m = 0; m < 2; ++m) {
                    offPtr[m][s] = take(static_cast<size_t>((2 * p.n + 2) * 8));
                    offIdx[m][s] = take(static_cast<size_t>(p.n * g.ldw * 4));
                    offVal[m][s] = take(bytes);
                }
            }
        }
    }
    void* base = nullptr;
    BST(ws_get(ctx, WS_BATCH, total, &base));
    c->ws_bytes = total;
    uint8_t* b8 = static_cast<uint8_t*>(base);
    for (int s = 0; s < np; ++s) {
        GroupProblem& g = hp[s];
        if (g.n == 0) continue;
        if (g.engine == 0) {
            g.M[0] = b8 + offM0[s];
            g.M[1] = b8 + offM1[s];
            g.T[0] = b8 + offT0[s];
            g.T[1] = b8 + offT1[s];
            for (int par = 0; par < 2; ++par) {
                BST(make_tmap(ctx, &g.mapA[par], g.M[par], g.ld, g.ld, g.ld, TC_BM));
                BST(make_tmap(ctx, &g.mapB[par], g.T[par], g.ld, g.ld, g.ld, TC_BN));
            }
            if (g.kind == 1) {
                g.X = b8 + offX[s];
                g.R1T = b8 + offR1T[s];
                BST(make_tmap(ctx, &g.mapBF, g.R1T, g.ld, g.ld, g.ld, TC_BN));
            }
        }
        g.P[0] = reinterpret_cast<uint64_t*>(b8 + offP0[s]);
        g.P[1] = reinterpret_cast<uint64_t*>(b8 + offP1[s]);
        if (g.kind == 1) g.PR1 = reinterpret_cast<uint64_t*>(b8 + offPR1[s]);
    }
    // frontier jobs (engine 2): every row of the closure as one query, all jobs in one launch
    std::vector<FrontierJob> jobs;
    int64_t fr_total = 0, fr_max_n = 0, fr_max_ldw = 0;
    for (int s = 0; s < np; ++s) {
        const GroupProblem& g = hp[s];
        if (g.n == 0 || g.engine != 2) continue;
        FrontierJob j{};
        j.P = g.P[0];
        j.PT = reinterpret_cast<uint64_t*>(b8 + offPT[s]);
        j.wptr = reinterpret_cast<int64_t*>(b8 + offPtr[0][s]);
        j.widx = reinterpret_cast<int32_t*>(b8 + offIdx[0][s]);
        j.wval = reinterpret_cast<uint64_t*>(b8 + offVal[0][s]);
        j.wptrT = reinterpret_cast<int64_t*>(b8 + offPtr[1][s]);
        j.widxT = reinterpret_cast<int32_t*>(b8 + offIdx[1][s]);
        j.wvalT = reinterpret_cast<uint64_t*>(b8 + offVal[1][s]);
        j.out = g.P[1];
        j.n = g.n;
        j.ldw = g.ldw;
        j.first = fr_total;
        j.levels = nullptr;  // set below, once the state array exists
        jobs.push_back(j);
        fr_total += g.n;
        fr_max_n = std::max(fr_max_n, g.n);
        fr_max_ldw = std::max(fr_max_ldw, g.ldw);
    }
    // device copies
    BCK(cudaMalloc(&c->d_probs, sizeof(GroupProblem) * (np > 0 ? np : 1)), "cudaMalloc(batch problems)");
    BCK(cudaMemcpy(c->d_probs, hp.data(), sizeof(GroupProblem) * np, cudaMemcpyHostToDevice), "copy batch problems");
    const size_t nints = static_cast<size_t>(10 * np + 2 * (np + 1) + 2);
    BCK(cudaMalloc(&c->d_ints, sizeof(int) * nints), "cudaMalloc(batch state)");
    BCK(cudaMemset(c->d_ints, 0, sizeof(int) * nints), "clear batch state");
    GroupState hs;
    hs.ones = reinterpret_cast<unsigned long long*>(c->d_ints);  // the counts that a launch starts from: cleared by it
    hs.top = c->d_ints + 2 * np;
    int* q = c->d_ints + 3 * np;
    hs.parity = q; q += np;
    hs.active = q; q += np;
    hs.iters = q; q += np;
    hs.changed = q; q += np;
    hs.notconv = q; q += np;
    hs.tc_offs = q; q += np + 1;
    hs.pk_offs = q; q += np + 1;
    hs.tc_total = q; q += 1;
    hs.pk_total = q; q += 1;
    hs.phase = q; q += np;
    hs.ppar = q; q += np;
    BCK(cudaMalloc(&c->d_st, sizeof(GroupState)), "cudaMalloc(batch state)");
    BCK(cudaMemcpy(c->d_st, &hs, sizeof(GroupState), cudaMemcpyHostToDevice), "copy batch state");
    if (!jobs.empty()) {
        size_t k = 0;
        for (int s = 0; s < np; ++s)
            if (hp[s].n > 0 && hp[s].engine == 2) jobs[k++].levels = hs.iters + s;
        BCK(cudaMalloc(&c->d_jobs, sizeof(FrontierJob) * jobs.size() + sizeof(unsigned long long)),
            "cudaMalloc(frontier jobs)");
        BCK(cudaMemcpy(c->d_jobs, jobs.data(), sizeof(FrontierJob) * jobs.size(), cudaMemcpyHostToDevice),
            "copy frontier jobs");
    }
    c->h_iters.assign(np, 0);
    c->h_notconv.assign(np, 0);

    // ---- graph
    BCK(prepare_tc_group(), "tensor-core group kernel attributes");
    BCK(cudaGraphCreate(&c->graph, 0), "cudaGraphCreate");
    if (np == 0) {
        BST(build_solo(ctx, c, probs, wait_cycles));
        BCK(cudaGraphInstantiate(&c->exec, c->graph, 0), "cudaGraphInstantiate");
        *out = c;
        return BMLP_OK;
    }
    cudaGraphConditionalHandle hA, hB;  // the bit-row loop and the tensor-core loop
    BCK(cudaGraphConditionalHandleCreate(&hA, c->graph, 0, cudaGraphCondAssignDefault), "conditional handle");
    BCK(cudaGraphConditionalHandleCreate(&hB, c->graph, 0, cudaGraphCondAssignDefault), "conditional handle");
    GroupProblem* dp = c->d_probs;
    GroupState* ds = c->d_st;
    int nprob = np;
    int* err = ctx->d_ctl + CTL_ERROR;
    long long wc = wait_cycles;
    int phase0 = 0, phase1 = 1;
    const int sms = ctx->sm_count;
    const unsigned gy = static_cast<unsigned>(np > 0 ? np : 1);
    bool any_compose = false;
    for (const GroupProblem& g : hp) any_compose |= g.kind == 1 && g.n > 0;
    // Blocks per problem of the passes over rows (a warp per row) and over 64 x 64 tiles: few problems have the GPU to
    // themselves, many share it, and none needs more than the largest has work for. (32 and 64 for all: one problem of 3,000
    // constants with 50 facts a row 436 us, 210 now; 200 problems of 100 270 and 260 us; the 1,482 of a knowledge graph keep 32
    // and 64.)
    int64_t most_n = 1, most_ld = TILE;
    for (const GroupProblem& g : hp) {
        most_n = std::max(most_n, g.n);
        most_ld = std::max(most_ld, g.ld);
    }
    const int64_t share = 64 * sms / np;
    const unsigned row_blocks = static_cast<unsigned>(std::min<int64_t>(std::max<int64_t>(share, 32), (most_n + 7) / 8));
    const unsigned tile_blocks =
        static_cast<unsigned>(std::min<int64_t>(std::max<int64_t>(share, 64), (most_ld / TILE) * (most_ld / TILE)));
    // a node with the problem list and state as its arguments, one block row per problem
    const auto per_problem = [&](cudaGraphNode_t* node, const cudaGraphNode_t* dep, size_t ndep, void* fn, unsigned gx) {
        void* a[] = {&dp, &ds};
        return add_kernel(ctx, c->graph, node, dep, ndep, fn, dim3(gx, gy), dim3(256), 0, a);
    };
    const auto plan = [&](cudaGraph_t g, cudaGraphNode_t* node, const cudaGraphNode_t* dep, size_t ndep, int mode,
                          cudaGraphConditionalHandle h, int set_cond) {
        void* a[] = {&dp, &ds, &nprob, &mode, &h, &set_cond};
        return add_kernel(ctx, g, node, dep, ndep, reinterpret_cast<void*>(&batch_plan_kernel), dim3(1), dim3(1024), 0, a);
    };
    const auto loop = [&](cudaGraphNode_t* node, const cudaGraphNode_t* dep, size_t ndep, cudaGraphConditionalHandle h,
                          cudaGraph_t* body) {
        cudaGraphNodeParams cp = {};
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        BCK(cudaGraphAddNode(node, c->graph, dep, nullptr, ndep, &cp), "while node");
        *body = cp.conditional.phGraph_out[0];
        return BMLP_OK;
    };
    cudaGraphNode_t n_enc, n_init, n_rows, n_hand, n_ops, n_tc, n_last;
    cudaGraph_t body_rows = nullptr, body_tc = nullptr;
    BST(per_problem(&n_enc, nullptr, 0, reinterpret_cast<void*>(&batch_encode_kernel), row_blocks));
    BST(plan(c->graph, &n_init, &n_enc, 1, 0, hA, 1));
    // the closures by frontier expansion: one chain of grouped launches after the planner's start
    std::vector<cudaGraphNode_t> before_while{n_init};
    if (!jobs.empty()) BST(add_frontier_chain(ctx, c, static_cast<int>(jobs.size()), fr_max_n, fr_max_ldw, fr_total,
                                              n_init, &before_while));
    BST(loop(&n_rows, before_while.data(), before_while.size(), hA, &body_rows));
    {
        cudaGraphNode_t n_sq, n_plan;
        void* b[] = {&dp, &ds, &nprob};
        BST(add_kernel(ctx, body_rows, &n_sq, nullptr, 0, reinterpret_cast<void*>(&packed_group_kernel), dim3(sms * 8),
                       dim3(256), 0, b));
        BST(plan(body_rows, &n_plan, &n_sq, 1, 1, hA, 1));
    }
    BST(plan(c->graph, &n_hand, &n_rows, 1, 3, hB, 1));
    BST(per_problem(&n_ops, &n_hand, 1, reinterpret_cast<void*>(&batch_operands_kernel), tile_blocks));
    BST(loop(&n_tc, &n_ops, 1, hB, &body_tc));
    {
        cudaGraphNode_t n_sq, n_plan;
        void* a[] = {&dp, &ds, &nprob, &phase0, &err, &wc};
        BST(add_kernel(ctx, body_tc, &n_sq, nullptr, 0, tc_group_kernel_ptr(), dim3(sms), dim3(TC_THREADS),
                       tc_smem_bytes(), a));
        BST(plan(body_tc, &n_plan, &n_sq, 1, 4, hB, 1));
    }
    n_last = n_tc;
    if (any_compose) {
        cudaGraphNode_t n_prep, n_prod, n_plan2, n_final;
        BST(per_problem(&n_prep, &n_last, 1, reinterpret_cast<void*>(&batch_compose_prep_kernel), 8));
        BST(per_problem(&n_prod, &n_prep, 1, reinterpret_cast<void*>(&batch_compose_rows_kernel), row_blocks));
        BST(plan(c->graph, &n_plan2, &n_prod, 1, 2, hB, 0));
        void* a[] = {&dp, &ds, &nprob, &phase1, &err, &wc};
        BST(add_kernel(ctx, c->graph, &n_final, &n_plan2, 1, tc_group_kernel_ptr(), dim3(sms), dim3(TC_THREADS),
                       tc_smem_bytes(), a));
        n_last = n_final;
    }
    cudaGraphNode_t n_dec;
    BST(per_problem(&n_dec, &n_last, 1, reinterpret_cast<void*>(&batch_decode_kernel), row_blocks));
    if (!c->solo.empty()) BST(build_solo(ctx, c, probs, wait_cycles));
    BCK(cudaGraphInstantiate(&c->exec, c->graph, 0), "cudaGraphInstantiate");
    *out = c;
    return BMLP_OK;
}

// Adds a conditional WHILE node after the current capture dependencies of `cs` and returns its body graph; the
// capture of `cs` continues after the node.
bmlp_status add_conditional(bmlp_ctx* ctx, cudaStream_t cs, cudaGraphConditionalHandle h, cudaGraphConditionalNodeType type,
                            cudaGraph_t* body) {
    cudaStreamCaptureStatus st;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    BCK(cudaStreamGetCaptureInfo(cs, &st, nullptr, &g, &deps, nullptr, &nd), "capture info");
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = type;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    BCK(cudaGraphAddNode(&node, g, deps, nullptr, nd, &cp), "conditional node");
    BCK(cudaStreamUpdateCaptureDependencies(cs, &node, nullptr, 1, cudaStreamSetCaptureDependencies),
        "capture dependencies");
    *body = cp.conditional.phGraph_out[0];
    return BMLP_OK;
}

bmlp_status add_while(bmlp_ctx* ctx, cudaStream_t cs, cudaGraphConditionalHandle h, cudaGraph_t* body) {
    return add_conditional(ctx, cs, h, cudaGraphCondTypeWhile, body);
}

// One lane of the large problems: device-driven single-problem pipelines, one after another on one scratch sized for the
// lane's largest, captured into the batch graph as a branch of its own. `mine`: their places in c->solo. With base null
// only *bytes, the scratch that the lane needs, is computed.
bmlp_status build_lane(bmlp_ctx* ctx, BatchCache* c, const bmlp_problem* probs, long long wait_cycles,
                       const std::vector<int>& mine, uint8_t* base, size_t* bytes) {
    int64_t nmax = 0;
    bool any_compose = false;
    for (int k : mine) {
        nmax = std::max(nmax, probs[c->solo[k]].n);
        any_compose |= probs[c->solo[k]].kind == BMLP_PROBLEM_COMPOSE;
    }
    const int64_t ldw_max = round_up((nmax + 63) / 64, 2);
    const int64_t np_max = round_up(nmax, TC_PAD);
    const size_t pk = static_cast<size_t>(nmax * ldw_max * 8);
    const size_t q = static_cast<size_t>(np_max * np_max / 2);
    size_t total = 0;
    auto take = [&](size_t bytes) {
        size_t o = total;
        total += round_up(static_cast<int64_t>(bytes), 1024);
        return o;
    };
    const size_t oP0 = take(pk), oP1 = take(pk), oPtr = take(static_cast<size_t>((2 * nmax + 2) * 8)),
                 oIdx = take(static_cast<size_t>(nmax * ldw_max * 4)), oVal = take(pk);
    size_t oQ[2], oQT[2];
    for (int k = 0; k < 2; ++k) {
        oQ[k] = take(q);
        oQT[k] = take(q);
    }
    size_t oM0 = 0;
    if (any_compose) oM0 = take(q);  // a composition's final product: scratch for the transposed output
    // the squaring restricted to the rows and columns holding zeros: bit rows of R and R^T (written by the 4-bit
    // squarings' epilogue), its computed rows, and its counts and lists
    const bool thin_any = thin_is_enabled();
    const int64_t ldwt_max = np_max / 64;
    size_t oTP = 0, oTPT = 0, oTT = 0, oTAux = 0;
    if (thin_any) {
        const size_t bits = static_cast<size_t>(np_max * ldwt_max * 8);
        oTP = take(bits);
        oTPT = take(bits);
        oTT = take(2 * bits);
        oTAux = take(thin_aux_bytes(nmax, ldwt_max));
    }
    *bytes = total;
    if (base == nullptr) return BMLP_OK;
    uint8_t* b8 = base;
    uint64_t* P0 = reinterpret_cast<uint64_t*>(b8 + oP0);
    uint64_t* P1 = reinterpret_cast<uint64_t*>(b8 + oP1);
    int64_t* wptr = reinterpret_cast<int64_t*>(b8 + oPtr);
    int32_t* widx = reinterpret_cast<int32_t*>(b8 + oIdx);
    uint64_t* wval = reinterpret_cast<uint64_t*>(b8 + oVal);
    uint8_t* Q[2] = {b8 + oQ[0], b8 + oQ[1]};
    uint8_t* QT[2] = {b8 + oQT[0], b8 + oQT[1]};
    uint8_t* M0 = b8 + oM0;
    uint64_t* TP = reinterpret_cast<uint64_t*>(b8 + oTP);
    uint64_t* TPT = reinterpret_cast<uint64_t*>(b8 + oTPT);
    uint64_t* TT = reinterpret_cast<uint64_t*>(b8 + oTT);
    cudaStream_t cs = nullptr, cb = nullptr, cc = nullptr;
    BCK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking), "capture stream");
    cudaError_t ce = cudaStreamCreateWithFlags(&cb, cudaStreamNonBlocking);
    if (ce == cudaSuccess) ce = cudaStreamCreateWithFlags(&cc, cudaStreamNonBlocking);
    if (ce != cudaSuccess) {
        cudaStreamDestroy(cs);
        if (cb) cudaStreamDestroy(cb);
        return cuda_err(ctx, ce, "capture stream");
    }
    struct Streams {
        cudaStream_t a, b, c;
        ~Streams() {
            cudaStreamDestroy(a);
            cudaStreamDestroy(b);
            cudaStreamDestroy(c);
        }
    } guard_streams{cs, cb, cc};
    BCK(cudaStreamBeginCaptureToGraph(cs, c->graph, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed),
        "begin capture of the large problems");
    bmlp_status status = BMLP_OK;
    auto fail = [&](bmlp_status st) {
        cudaGraph_t g = nullptr;
        cudaStreamEndCapture(cs, &g);
        cudaGetLastError();
        return st;
    };
#define SCK(call, what)                                                   \
    do {                                                                  \
        cudaError_t e_ = (call);                                          \
        if (e_ != cudaSuccess) return fail(cuda_err(ctx, e_, what));      \
    } while (0)
#define SST(call)                                  \
    do {                                           \
        bmlp_status s_ = (call);                   \
        if (s_ != BMLP_OK) return fail(s_);        \
    } while (0)
    const int sms = ctx->sm_count;
    const double s_word = bitrow_s_per_word(), s_row = bitrow_row_s_per_word(), step_s = bitrow_step_s();
    for (int k : mine) {
        const bmlp_problem& p = probs[c->solo[k]];
        int* w = c->d_solo + SW_WORDS * k;
        const int64_t n = p.n, ldw = round_up((n + 63) / 64, 2), n_pad = round_up(n, TC_PAD), ld4 = n_pad / 2;
        const int cap = log2_ceil(n > 1 ? n : 2) + 2;
        const void* src = p.kind == BMLP_PROBLEM_COMPOSE ? p.R2 : p.R1;
        const double limit = tc4_product_s(n_pad);
        // ---- squarings on word-indexed bit rows while they are cheaper than a tensor-core product
        solo_init_kernel<<<1, 1, 0, cs>>>(w);
        if (p.fmt == BMLP_FMT_U8)
            launch_u8_to_packed(static_cast<const uint8_t*>(src), n, P0, ldw, cs);
        else
            launch_packed_copy(static_cast<const uint64_t*>(src), (n + 63) / 64, n, n, P0, ldw, 0, cs);
        const WordIndex x{wptr, widx, wval};
        SCK(launch_wcsr_build(P0, n, ldw, x, cs), "word index build");
        auto* cost = reinterpret_cast<unsigned long long*>(w + SW_COST);
        SCK(launch_indexed_cost(x, x, n, cost, sms, cs), "squaring cost");
        cudaGraph_t g = nullptr;
        cudaStreamCaptureStatus cst;
        SCK(cudaStreamGetCaptureInfo(cs, &cst, nullptr, &g, nullptr, nullptr, nullptr), "capture info");
        cudaGraphConditionalHandle hA, hC;
        SCK(cudaGraphConditionalHandleCreate(&hA, g, 0, cudaGraphCondAssignDefault), "conditional handle");
        SCK(cudaGraphConditionalHandleCreate(&hC, g, 0, cudaGraphCondAssignDefault), "conditional handle");
        solo_rows_decide_kernel<<<1, 1, 0, cs>>>(w, cap, 1, step_s, s_word, s_row, limit, hA);
        cudaGraph_t body = nullptr;
        SST(add_while(ctx, cs, hA, &body));
        SCK(cudaStreamBeginCaptureToGraph(cb, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed),
            "begin capture of the bit-row loop");
        {
            cudaError_t e = launch_indexed_rows(x, x, P0, n, ldw, P1, sms, cb, w + SW_CHANGED);
            if (e == cudaSuccess) {  // the next step reads P0 (ldw is even: rows are whole 16-byte units)
                solo_copy_kernel<<<sms * 4, 256, 0, cb>>>(reinterpret_cast<uint4*>(P0),
                                                           reinterpret_cast<const uint4*>(P1), n * ldw / 2);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess) e = launch_wcsr_build(P0, n, ldw, x, cb);
            if (e == cudaSuccess) e = launch_indexed_cost(x, x, n, cost, sms, cb);
            if (e == cudaSuccess) {
                solo_rows_decide_kernel<<<1, 1, 0, cb>>>(w, cap, 0, step_s, s_word, s_row, limit, hA);
                e = cudaGetLastError();
            }
            cudaGraph_t tmp = nullptr;
            const cudaError_t e2 = cudaStreamEndCapture(cb, &tmp);
            if (e != cudaSuccess || e2 != cudaSuccess) return fail(cuda_err(ctx, e != cudaSuccess ? e : e2, "bit-row loop"));
        }
        // ---- squarings on packed E2M1 operands (R^T as the B operand), two per loop iteration
        launch_packed_to_e2m1(P0, ldw, n, Q[0], QT[0], n_pad, cs);
        solo_mid_kernel<<<1, 1, 0, cs>>>(w, hC);
        CUtensorMap mA[2], mB0[2], mB1[2];
        for (int b = 0; b < 2; ++b) {
            SST(make_tmap(ctx, &mA[b], Q[b], n_pad, ld4, ld4, TC_BM));
            SST(make_tmap(ctx, &mB0[b], QT[b], n_pad, ld4, ld4, TC_BN / 2));
            SST(make_tmap(ctx, &mB1[b], QT[b], n_pad, ld4, ld4, tc4_b1_rows()));
        }
        SST(add_while(ctx, cs, hC, &body));
        // after each product, when R is close to its closure, the next squaring may run only on the rows and columns
        // that still hold zeros: IF nodes inside the loop's body, one for its statistics and one for the squaring
        const int64_t ldw_t = n_pad / 64;
        const bool thin_p = thin_any && thin_fixed_seconds(n_pad) < limit;
        const ThinLists t_lists = thin_lists(b8 + oTAux, n, ldw_t);
        cudaGraphConditionalHandle hT[2], hT2[2];
        if (thin_p) {
            for (int h = 0; h < 2; ++h) {
                SCK(cudaGraphConditionalHandleCreate(&hT[h], body, 0, cudaGraphCondAssignDefault), "conditional handle");
                SCK(cudaGraphConditionalHandleCreate(&hT2[h], body, 0, cudaGraphCondAssignDefault), "conditional handle");
            }
        }
        auto* t_smp = reinterpret_cast<unsigned long long*>(w + SW_SMP);
        auto* t_stat = reinterpret_cast<unsigned long long*>(w + SW_TSTAT);
        // captures one IF body on stream cc: fn() issues its launches
        auto capture_if = [&](cudaGraphConditionalHandle hh, auto fn) -> cudaError_t {
            cudaGraph_t ifb = nullptr;
            if (add_conditional(ctx, cb, hh, cudaGraphCondTypeIf, &ifb) != BMLP_OK) return cudaErrorUnknown;
            cudaError_t e1 = cudaStreamBeginCaptureToGraph(cc, ifb, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
            if (e1 != cudaSuccess) return e1;
            e1 = fn();
            cudaGraph_t tmp = nullptr;
            const cudaError_t e2 = cudaStreamEndCapture(cc, &tmp);
            return e1 != cudaSuccess ? e1 : e2;
        };
        SCK(cudaStreamBeginCaptureToGraph(cb, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed),
            "begin capture of the tensor-core loop");
        {
            cudaError_t e = cudaSuccess;
            for (int half = 0; half < 2 && e == cudaSuccess; ++half) {
                TcParams p4{};
                p4.m_tiles = static_cast<int32_t>(n_pad / TC_BM);
                p4.n_tiles = tc4_tiles(n_pad, sms);
                p4.k_blocks = static_cast<int32_t>(n_pad / 256);
                p4.mode = TC_MODE_RMS;
                p4.ld = ld4;
                p4.old_r = Q[half];
                p4.out_r = Q[half ^ 1];
                p4.out_rt = QT[half ^ 1];
                p4.changed = w + SW_CHANGED;
                p4.error = ctx->d_ctl + CTL_ERROR;
                p4.wait_cycles = wait_cycles;
                p4.guard = w + (half == 0 ? SW_GC : SW_G1);
                if (thin_p) {  // the epilogue keeps R and R^T as bit rows for the restricted squaring
                    p4.out_bits = reinterpret_cast<uint32_t*>(TP);
                    p4.out_bits_t = reinterpret_cast<uint32_t*>(TPT);
                    p4.ldb = 2 * ldw_t;
                }
                e = launch_tc4_product_duo(mA[half], mB0[half], mB1[half], p4, sms, cb);
                if (e == cudaSuccess) {
                    solo_tc_decide_kernel<<<1, 1, 0, cb>>>(w, cap, half, hC);
                    e = cudaGetLastError();
                }
                if (thin_p && e == cudaSuccess) {
                    uint8_t* Qn = Q[half ^ 1];
                    uint8_t* QTn = QT[half ^ 1];
                    e = launch_thin_sample(TP, ldw_t, n, thin_sample_rows(), t_smp, nullptr, cb);
                    if (e == cudaSuccess) {
                        solo_thin_gate_kernel<<<1, 1, 0, cb>>>(w, half, n, thin_row_spread(), hT[half]);
                        e = cudaGetLastError();
                    }
                    if (e == cudaSuccess)
                        e = capture_if(hT[half], [&]() -> cudaError_t {
                            cudaError_t e3 = launch_thin_stats(n, TP, TPT, TP, TPT, ldw_t, t_lists, t_stat, sms, cc);
                            if (e3 != cudaSuccess) return e3;
                            solo_thin_decide_kernel<<<1, 1, 0, cc>>>(w, ldw_t, thin_fixed_seconds(n_pad), thin_word_s(),
                                                                     thin_one_s(), limit);
                            return cudaGetLastError();
                        });
                    if (e == cudaSuccess) {
                        solo_thin_arm_kernel<<<1, 1, 0, cb>>>(w, hT2[half]);
                        e = cudaGetLastError();
                    }
                    if (e == cudaSuccess)
                        e = capture_if(hT2[half], [&]() -> cudaError_t {
                            // |B| + |Rb| is known on the device only: the grids cover up to n entries at once
                            cudaError_t e3 = launch_thin_squaring(n, TP, TPT, TP, TPT, ldw_t, t_lists, t_stat, n, TT, Qn,
                                                                  QTn, ld4, w + SW_TCHANGED, w + SW_TOPEN, true, sms, cc);
                            if (e3 != cudaSuccess) return e3;
                            solo_thin_post_kernel<<<1, 1, 0, cc>>>(w, half, cap);
                            return cudaGetLastError();
                        });
                    if (e == cudaSuccess) {
                        solo_loop_ctl_kernel<<<1, 1, 0, cb>>>(w, hC);
                        e = cudaGetLastError();
                    }
                }
            }
            cudaGraph_t tmp = nullptr;
            const cudaError_t e2 = cudaStreamEndCapture(cb, &tmp);
            if (e != cudaSuccess || e2 != cudaSuccess)
                return fail(cuda_err(ctx, e != cudaSuccess ? e : e2, "tensor-core loop"));
        }
        if (thin_p) {  // a restricted squaring that ended the loop after the first product left the closure in Q1
            solo_result_copy_kernel<<<sms * 4, 256, 0, cs>>>(w, reinterpret_cast<uint4*>(Q[0]),
                                                             reinterpret_cast<const uint4*>(Q[1]), n_pad * ld4 / 16);
            SCK(cudaGetLastError(), "result copy");
        }
        // ---- results: Q[0] holds the closure (a product that changed nothing left both buffers equal)
        if (p.kind == BMLP_PROBLEM_CLOSURE) {
            if (p.fmt == BMLP_FMT_U8) {  // bytes leave through bit rows, in the places of the bit-row squarings
                launch_e2m1_to_packed(Q[0], ld4, n, P0, ldw, 0, cs);
                launch_packed_to_u8(P0, ldw, n, static_cast<uint8_t*>(p.out), p.reflexive, cs);
            } else {
                launch_e2m1_to_packed(Q[0], ld4, n, static_cast<uint64_t*>(p.out), (n + 63) / 64, p.reflexive, cs);
            }
        } else {
            // out = (I + R2+) R1 on 4-bit operands, on the squaring kernel without an old R: A = I + R2+ (Q[0], diagonal
            // set), B^T = R1^T (encoded with R1 into the free pair Q[1], QT[1]); R' = C > 0 goes to Q[1] (R1 is no longer
            // needed), R'^T to the scratch
            launch_set_diag_e2m1(Q[0], ld4, n, cs);
            if (p.fmt == BMLP_FMT_U8) {
                launch_u8_to_packed(static_cast<const uint8_t*>(p.R1), n, P0, ldw, cs);
                launch_packed_to_e2m1(P0, ldw, n, Q[1], QT[1], n_pad, cs);
            } else {
                launch_packed_to_e2m1(static_cast<const uint64_t*>(p.R1), (n + 63) / 64, n, Q[1], QT[1], n_pad, cs);
            }
            CUtensorMap fa, fb0, fb1;
            SST(make_tmap(ctx, &fa, Q[0], n_pad, ld4, ld4, TC_BM));
            SST(make_tmap(ctx, &fb0, QT[1], n_pad, ld4, ld4, TC_BN / 2));
            SST(make_tmap(ctx, &fb1, QT[1], n_pad, ld4, ld4, tc4_b1_rows()));
            TcParams pp{};
            pp.m_tiles = static_cast<int32_t>(n_pad / TC_BM);
            pp.n_tiles = tc4_tiles(n_pad, sms);
            pp.k_blocks = static_cast<int32_t>(n_pad / 256);
            pp.mode = TC_MODE_RMS;
            pp.ld = ld4;
            pp.out_r = Q[1];
            pp.out_rt = M0;
            pp.changed = w + SW_CHANGED;
            pp.error = ctx->d_ctl + CTL_ERROR;
            pp.wait_cycles = wait_cycles;
            SCK(launch_tc4_product_duo(fa, fb0, fb1, pp, sms, cs), "final product");
            if (p.fmt == BMLP_FMT_U8) {  // bytes leave through bit rows, in the places of the bit-row squarings
                launch_e2m1_to_packed(Q[1], ld4, n, P0, ldw, 0, cs);
                launch_packed_to_u8(P0, ldw, n, static_cast<uint8_t*>(p.out), 0, cs);
            } else {
                launch_e2m1_to_packed(Q[1], ld4, n, static_cast<uint64_t*>(p.out), (n + 63) / 64, 0, cs);
            }
        }
        SCK(cudaGetLastError(), "large-problem launches");
    }
#undef SCK
#undef SST
    cudaGraph_t g = nullptr;
    BCK(cudaStreamEndCapture(cs, &g), "end capture of the large problems");
    return status;
}

// Branches of the batch graph that the large problems are dealt out to, besides the branch of the grouped ones. A
// pipeline is a chain of small launches (bit-row squarings, decisions) between tensor-core products that fill the GPU, so
// several chains at once fill each other's gaps (measured on the knowledge-graph batch, 33 closures and 8 compositions
// with n >= 4,096: 37.4 ms on one branch, 32.2 on two, 30.4 on four, 30.4 on twelve). Every lane adds scratch: fewer of
// them where that would be more than kLaneBytes in all, or more than the device has left.
constexpr int kLanes = 4;
constexpr size_t kLaneBytes = size_t(24) << 30;

bmlp_status build_solo(bmlp_ctx* ctx, BatchCache* c, const bmlp_problem* probs, long long wait_cycles) {
    const int ns = static_cast<int>(c->solo.size());
    BCK(cudaMalloc(&c->d_solo, sizeof(int) * SW_WORDS * ns), "cudaMalloc(large-problem state)");
    BCK(cudaMemset(c->d_solo, 0, sizeof(int) * SW_WORDS * ns), "clear large-problem state");
    c->h_solo.assign(static_cast<size_t>(SW_WORDS * ns), 0);
    // longest first, each to the lane with the least predicted time: a product or two of its size, and its launches
    std::vector<int> order(ns);
    for (int k = 0; k < ns; ++k) order[k] = k;
    const auto cost = [&](int k) {
        const bmlp_problem& p = probs[c->solo[k]];
        return 2.0 * tc4_product_s(round_up(p.n, TC_PAD)) + 300e-6;
    };
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost(x) > cost(y); });
    for (int lanes = std::min(kLanes, ns); lanes >= 1; --lanes) {
        std::vector<std::vector<int>> mine(lanes);
        std::vector<double> load(lanes, 0.0);
        for (int k : order) {
            const int l = static_cast<int>(std::min_element(load.begin(), load.end()) - load.begin());
            mine[l].push_back(k);
            load[l] += cost(k);
        }
        std::vector<size_t> bytes(lanes, 0);
        size_t total = 0;
        for (int l = 0; l < lanes; ++l) {
            BST(build_lane(ctx, c, probs, wait_cycles, mine[l], nullptr, &bytes[l]));
            total += bytes[l];
        }
        if (lanes > 1 && total > kLaneBytes) continue;
        void* base = nullptr;
        const bmlp_status got = ws_get(ctx, WS_SOLO, total, &base);
        if (got == BMLP_ERR_OOM && lanes > 1) continue;
        BST(got);
        size_t at = 0;
        for (int l = 0; l < lanes; ++l) {
            size_t unused = 0;
            BST(build_lane(ctx, c, probs, wait_cycles, mine[l], static_cast<uint8_t*>(base) + at, &unused));
            at += bytes[l];
        }
        break;
    }
    return BMLP_OK;
}

uint64_t batch_key(const bmlp_problem* probs, int64_t count, int variant, long long wait_cycles, const int* tune,
                   int64_t solo_n) {
    uint64_t h = 1469598103934665603ull;
    h = fnv(h, &wait_cycles, sizeof(wait_cycles));  // the bound is an argument of the graph's tensor-core kernels
    h = fnv(h, &count, sizeof(count));
    h = fnv(h, &variant, sizeof(variant));
    h = fnv(h, &solo_n, sizeof(solo_n));
    h = fnv(h, tune, sizeof(int) * 32);
    for (int64_t i = 0; i < count; ++i) h = fnv(h, &probs[i], sizeof(bmlp_problem));
    return h;
}

}  // namespace

bmlp_status batch_run_impl(bmlp_ctx* ctx, const bmlp_problem* probs, int64_t count, int variant,
                           long long wait_cycles, int32_t* iters_out, cudaStream_t s, int64_t solo_n) {
    for (int64_t i = 0; i < count; ++i) {
        const bmlp_problem& p = probs[i];
        if (p.kind != BMLP_PROBLEM_CLOSURE && p.kind != BMLP_PROBLEM_COMPOSE)
            return set_err(ctx, BMLP_ERR_INVALID_ARG, "problem %lld: bad kind %d", (long long)i, p.kind);
        if (p.fmt != BMLP_FMT_U8 && p.fmt != BMLP_FMT_PACKED64)
            return set_err(ctx, BMLP_ERR_INVALID_ARG, "problem %lld: bad format %d", (long long)i, p.fmt);
        if (p.n < 0 || p.n > (int64_t(1) << 17))
            return set_err(ctx, BMLP_ERR_INVALID_ARG, "problem %lld: n out of range", (long long)i);
        if (p.n == 0) continue;
        if (!p.R1 || !p.out || (p.kind == BMLP_PROBLEM_COMPOSE && !p.R2))
            return set_err(ctx, BMLP_ERR_INVALID_ARG, "problem %lld: null pointer", (long long)i);
        if (!on_device(p.R1) || !on_device(p.out) || (p.kind == BMLP_PROBLEM_COMPOSE && !on_device(p.R2)))
            return set_err(ctx, BMLP_ERR_INVALID_ARG, "problem %lld: matrices must be device memory", (long long)i);
    }
    if (count > (int64_t(1) << 20)) return set_err(ctx, BMLP_ERR_UNSUPPORTED, "more than 2^20 problems");
    const uint64_t key = batch_key(probs, count, variant, wait_cycles, ctx->tune, solo_n);
    BatchCache* c = static_cast<BatchCache*>(ctx->batch);
    if (c == nullptr || c->key != key) {
        const bmlp_status built = build_batch(ctx, probs, count, variant, wait_cycles, key, solo_n, &c);
        if (built != BMLP_OK) {  // nothing half built is left to be found under the key by the next call
            batch_cache_free(ctx);
            return built;
        }
    }
    BCK(cudaMemsetAsync(ctx->d_ctl, 0, CTL_WORDS * sizeof(int), s), "reset flags");
    ctx->stats.n_pad = static_cast<int64_t>(c->ws_bytes);
    BCK(cudaGraphLaunch(c->exec, s), "cudaGraphLaunch");
    const int np = c->nprob;
    BCK(cudaMemcpyAsync(c->h_iters.data(), c->d_ints + 5 * np, sizeof(int) * np, cudaMemcpyDeviceToHost, s),
        "read iterations");
    BCK(cudaMemcpyAsync(c->h_notconv.data(), c->d_ints + 7 * np, sizeof(int) * np, cudaMemcpyDeviceToHost, s),
        "read convergence");
    const int ns = static_cast<int>(c->solo.size());
    if (ns > 0)
        BCK(cudaMemcpyAsync(c->h_solo.data(), c->d_solo, sizeof(int) * SW_WORDS * ns, cudaMemcpyDeviceToHost, s),
            "read large-problem state");
    BCK(cudaMemcpyAsync(ctx->h_ctl, ctx->d_ctl, CTL_WORDS * sizeof(int), cudaMemcpyDeviceToHost, s), "read flags");
    BCK(host_sync(ctx, s), "synchronise batch");
    if (ctx->h_ctl[CTL_ERROR] != 0)
        return set_err(ctx, BMLP_ERR_TIMEOUT, "in-kernel wait timed out (code 0x%x)", ctx->h_ctl[CTL_ERROR]);
    int maxit = 0, bad = 0;
    for (int sl = 0; sl < np; ++sl) {
        const int i = c->order[sl];
        if (iters_out) iters_out[i] = c->h_iters[sl];
        maxit = std::max(maxit, c->h_iters[sl]);
        bad |= c->h_notconv[sl];
    }
    for (int k = 0; k < ns; ++k) {
        const int* w = c->h_solo.data() + SW_WORDS * k;
        if (iters_out) iters_out[c->solo[k]] = w[SW_ITERS];
        maxit = std::max(maxit, w[SW_ITERS]);
        bad |= w[SW_NOTCONV];
        ctx->stats.launches += 6 + 6 * w[SW_ITERS];
        ctx->stats.product_launches += w[SW_ITERS];
    }
    ctx->stats.iterations = maxit;
    ctx->stats.launches += 4 + 3 * maxit;
    ctx->stats.product_launches += maxit + 1;
    if (bad) return set_err(ctx, BMLP_ERR_NOT_CONVERGED, "a problem did not converge within its cap");
    return BMLP_OK;
}

}  // namespace bmlp
