// Closures and compositions of small relations (up to kSmallN constants) in one launch, on bit rows.
//
// At these sizes a squaring is a few microseconds of work wherever it runs, and the time of a closure is its chain of
// launches, pipelines and waits (a tensor-core product of 512 padded constants takes 12 us, of which the multiplications
// are half of one). Here one grid does all of it: a CTA owns a few rows, keeps them in shared memory from the caller's
// bytes to the result, and between two squarings only publishes its rows in global memory, waits at a grid-wide barrier
// and reads the rows back that changed (up to n^2 / 8 bytes from L2). A squaring ORs the named rows into each own row.
// Each reads the previous matrix only, so the number of products is that of the squarings elsewhere; a row k that row i
// named before and that has not changed since adds nothing to row i and is left out.
// What bounds it: the barrier (1.5 us), the flags and rows read back (1 to 3 us), and shared memory once rows are dense (a
// row OR is one warp access of up to 128 bytes; n = 1,024: 7 rows of up to 1,024 ones a CTA, 6 us). Whole calls, byte
// matrices with 2 facts a row, the tensor-core products issued together and this: n = 300: 120 and 51 us; 512: 118 and
// 59; 768: 160 and 85; 1,024: 130 and 86 (a word of a row lies in a lane, so the form ends there).
#include "internal.h"
#include "ptx.cuh"

namespace bmlp {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int kThreads = 1024;
constexpr int kPieces = 4;   // 16-byte pieces of a matrix that a thread has in flight
constexpr int kWarps = kThreads / 32;
constexpr size_t kMostSmem = 220 * 1024;  // of 227 KiB, beside the lists (n = 1,024 on 152 SMs: 131 KiB)

struct SmallArgs {
    const void* in;       // n x n bytes, or bit rows of words64 64-bit words
    const void* r1;       // composition: its R1 in the same format (else null)
    void* out;
    int bytes;            // 1: in, r1 and out are bytes
    int n, words64;
    int pitch;            // 32-bit words of a row here (a multiple of 4)
    int rows_per;         // rows of a CTA
    int group;            // lanes of a group: the power of two >= the words of a row, at least 8
    int reflexive;
    int max_iters;
    uint32_t* mats;       // three matrices of n x pitch words: R of even and odd squarings, R1
    uint8_t* grown;       // two vectors of n (even and odd squarings): whether the squaring changed the row
    unsigned* arrived;    // arrivals at the barrier; zero at launch
    int* result;          // products, whether the last one changed R
    int* error;
    long long wait_cycles;
};

// All CTAs of the grid have arrived `round` times (they are resident at once: a cooperative launch). False if that takes
// longer than the bound; each CTA waits for its own (one that gave up never arrives, so the others' run out soon after).
__device__ __forceinline__ bool grid_arrive_wait(const SmallArgs& a, unsigned round, int* s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(a.arrived, 1u);
        const unsigned want = round * gridDim.x;
        const long long t0 = clock64();
        int ok = 1;
        while (true) {
            unsigned seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.arrived) : "memory");
            if (seen >= want) break;
            if (clock64() - t0 > a.wait_cycles) {
                atomicExch(a.error, 0x51);
                ok = 0;
                break;
            }
        }
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Rows r0 .. r0 + rows - 1 of a caller's matrix as bit rows (words beyond column n zero).
__device__ __forceinline__ void read_rows(const SmallArgs& a, const void* in, int r0, int rows, uint32_t* own) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = (a.n + 31) >> 5;
    if (a.bytes) {
        const uint8_t* p = static_cast<const uint8_t*>(in);
        for (int x0 = warp; x0 < rows * a.pitch; x0 += 8 * kWarps) {  // eight loads in flight
            uint8_t v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int x = x0 + q * kWarps, r = x / a.pitch, c = 32 * (x - r * a.pitch) + lane;
                v[q] = r < rows && c < a.n ? p[static_cast<int64_t>(r0 + r) * a.n + c] : 0;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const unsigned m = __ballot_sync(FULL, v[q] != 0);
                if (lane == 0 && x0 + q * kWarps < rows * a.pitch) own[x0 + q * kWarps] = m;
            }
        }
    } else {
        const uint64_t* p = static_cast<const uint64_t*>(in);
        for (int x = threadIdx.x; x < rows * a.pitch; x += kThreads) {
            const int r = x / a.pitch, w = x - r * a.pitch;
            uint32_t m = 0;
            if (w < W) {
                const uint64_t v = p[static_cast<int64_t>(r0 + r) * a.words64 + (w >> 1)];
                m = static_cast<uint32_t>(w & 1 ? v >> 32 : v);
                const int valid = a.n - 32 * w;
                if (valid < 32) m &= (1u << valid) - 1u;
            }
            own[x] = m;
        }
    }
}

// next |= for every own row the rows of S that `names` has ones for (a CTA's rows x pitch words each), of which those that
// `had` (may be null) has too count only if they are in `grown`. A warp takes a word of a row: its ones become a list of row
// numbers (a lane per bit, the last one repeated up to a multiple of eight per group), which the warp's groups of lanes go
// through eight at a time. Found one by one with find-first-set in every lane the ones took five cycles a row OR, of which
// shared memory needs one.
__device__ __forceinline__ void or_named(const SmallArgs& a, int rows, const uint32_t* S, const uint32_t* names,
                                         const uint32_t* had, const uint32_t* grown, uint16_t* lists, uint32_t* next) {
    const int W = (a.n + 31) >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = a.group, l = lane & (g - 1), lw = l < W ? l : W - 1;  // a lane without a word repeats the last one
    const int part = lane / g, step = 8 * (32 / g);  // rows per round of the warp
    uint16_t* list = lists + warp * 64;
    for (int r = 0, w = warp; r < rows; w += kWarps) {
        while (w >= W) {
            w -= W;
            ++r;
        }
        if (r >= rows) break;
        uint32_t bits = names[r * a.pitch + w];
        if (had != nullptr) bits &= ~had[r * a.pitch + w] | grown[w];
        if (bits == 0) continue;
        const int count = __popc(bits), full = (count + step - 1) & -step;  // at most 32
        if ((bits >> lane) & 1u) list[__popc(bits & ((1u << lane) - 1u))] = static_cast<uint16_t>(lane);
        if (lane >= count && lane < full) list[lane] = static_cast<uint16_t>(31 - __clz(static_cast<int>(bits)));
        __syncwarp();
        const uint32_t* base = S + 32 * w * a.pitch + lw;
        uint32_t acc = 0;
        for (int c = part * 8; c < full; c += step) {  // eight rows in flight
            const uint4 k = *reinterpret_cast<const uint4*>(list + c);
            const uint32_t x0 = base[(k.x & 0xFFFFu) * a.pitch], x1 = base[(k.x >> 16) * a.pitch];
            const uint32_t x2 = base[(k.y & 0xFFFFu) * a.pitch], x3 = base[(k.y >> 16) * a.pitch];
            const uint32_t x4 = base[(k.z & 0xFFFFu) * a.pitch], x5 = base[(k.z >> 16) * a.pitch];
            const uint32_t x6 = base[(k.w & 0xFFFFu) * a.pitch], x7 = base[(k.w >> 16) * a.pitch];
            acc |= (x0 | x1 | x2 | x3) | (x4 | x5 | x6 | x7);
        }
        if (acc && l < W) atomicOr(&next[r * a.pitch + l], acc);
        __syncwarp();  // the list is free again
    }
}

__global__ void __launch_bounds__(kThreads, 1) small_closure_kernel(const SmallArgs a) {
    extern __shared__ __align__(16) uint32_t sm_rows[];
    __shared__ int s_ok;
    __shared__ __align__(16) uint16_t s_lists[kWarps * 64];
    __shared__ uint32_t s_grown[kSmallN / 32];   // the rows that the squaring before changed
    const int tid = threadIdx.x, pitch = a.pitch, mat = a.n * pitch;
    uint32_t* S = sm_rows;                       // the whole matrix
    uint32_t* own = S + mat;                     // own rows
    uint32_t* next = own + a.rows_per * pitch;   // own rows of R + R R
    uint32_t* had = next + a.rows_per * pitch;   // own rows before the last squaring
    int lg = 0;                                  // 2^lg threads for the 16-byte pieces of a row
    while ((4 << lg) < pitch) ++lg;
    const int r0 = blockIdx.x * a.rows_per;
    const int rows = min(a.rows_per, a.n - r0);  // the grid has ceil(n / rows_per) CTAs
    const int words = rows * pitch;
    const auto publish = [&](uint32_t* m, const uint32_t* from) {
        for (int x = tid; x < words / 4; x += kThreads)
            __stcg(reinterpret_cast<uint4*>(m + r0 * pitch) + x, reinterpret_cast<const uint4*>(from)[x]);
    };
    // rows into S, a thread per 16 bytes of a row in steps of whole rows; every CTA starts at its own rows, not all at one L2
    // slice. Piece q of a round: its place in S, or -1.
    const int per = kThreads >> lg, piece = tid & ((1 << lg) - 1);
    const auto place = [&](int i) {
        if (i >= a.n || piece >= pitch / 4) return -1;
        const int r = i + r0 < a.n ? i + r0 : i + r0 - a.n;
        return r * (pitch / 4) + piece;
    };
    const auto load = [&](const uint32_t* m, const int (&at)[kPieces], uint4 (&v)[kPieces]) {
#pragma unroll
        for (int q = 0; q < kPieces; ++q)
            if (at[q] >= 0) v[q] = __ldcg(reinterpret_cast<const uint4*>(m) + at[q]);
    };
    const auto keep = [&](const int (&at)[kPieces], const uint4 (&v)[kPieces]) {
#pragma unroll
        for (int q = 0; q < kPieces; ++q)
            if (at[q] >= 0) reinterpret_cast<uint4*>(S)[at[q]] = v[q];
    };
    int at[kPieces];
    uint4 v[kPieces];
    const auto fetch = [&](const uint32_t* m, bool all) {  // all rows, or those in s_grown (S holds the others)
        for (int i0 = tid >> lg; i0 < a.n; i0 += kPieces * per) {
#pragma unroll
            for (int q = 0; q < kPieces; ++q) {
                at[q] = place(i0 + q * per);
                if (!all && at[q] >= 0) {
                    const int r = i0 + q * per + r0 < a.n ? i0 + q * per + r0 : i0 + q * per + r0 - a.n;
                    if (!((s_grown[r >> 5] >> (r & 31)) & 1u)) at[q] = -1;
                }
            }
            load(m, at, v);
            keep(at, v);
        }
        __syncthreads();
    };
    const bool one_round = a.n <= kPieces * per;  // then all rows are loaded along with the flags of the grown ones
    if (a.r1 != nullptr) {
        read_rows(a, a.r1, r0, rows, next);
        __syncthreads();
        publish(a.mats + 2 * mat, next);
        __syncthreads();
    }
    read_rows(a, a.in, r0, rows, own);
    __syncthreads();
    publish(a.mats, own);
    int it = 0;
    bool more = true;
    while (true) {
        if (!grid_arrive_wait(a, it + 1, &s_ok)) return;
        const uint32_t* m = a.mats + (it & 1) * mat;
        if (one_round) {
#pragma unroll
            for (int q = 0; q < kPieces; ++q) at[q] = place((tid >> lg) + q * per);
            load(m, at, v);
        }
        if (it > 0) {  // squaring it - 1 is complete everywhere
            const uint8_t* g = a.grown + ((it - 1) & 1) * a.n;
            bool any = false;
            for (int c0 = tid & ~31; c0 < a.n; c0 += kThreads) {
                const int c = c0 + (tid & 31);
                const unsigned m = __ballot_sync(FULL, c < a.n && __ldcg(g + c) != 0);
                if ((tid & 31) == 0) s_grown[c0 >> 5] = m;
                any |= m != 0;
            }
            more = __syncthreads_or(any) != 0;
            if (!more || it == a.max_iters) break;
        }
        if (one_round) keep(at, v);
        else fetch(m, it == 0);
        for (int x = tid; x < words; x += kThreads) next[x] = own[x];
        __syncthreads();
        or_named(a, rows, S, own, it > 0 ? had : nullptr, s_grown, s_lists, next);
        __syncthreads();
        for (int r = tid >> 5; r < rows; r += kWarps) {  // a warp per row (pitch <= 32)
            const int x = r * pitch + (tid & 31);
            bool grew = false;
            if ((tid & 31) < pitch) {
                grew = next[x] != own[x];
                had[x] = own[x];
                own[x] = next[x];
            }
            grew = __any_sync(FULL, grew);
            if ((tid & 31) == 0) __stcg(a.grown + (it & 1) * a.n + r0 + r, static_cast<uint8_t>(grew));
        }
        __syncthreads();
        publish(a.mats + ((it & 1) ^ 1) * mat, own);
        ++it;
    }
    if (blockIdx.x == 0 && tid == 0) {
        a.result[0] = it;
        a.result[1] = more ? 1 : 0;
    }
    const uint32_t* res = own;
    if (a.r1 != nullptr) {  // (I + R2+) R1
        if (more) return;
        fetch(a.mats + 2 * mat, true);
        for (int x = tid; x < words; x += kThreads) next[x] = S[r0 * pitch + x];
        __syncthreads();
        or_named(a, rows, S, own, nullptr, nullptr, s_lists, next);
        __syncthreads();
        res = next;
    }
    if (a.bytes) {
        uint8_t* out = static_cast<uint8_t*>(a.out) + static_cast<int64_t>(r0) * a.n;
        for (int x = tid; x < rows * a.n; x += kThreads) {
            const int r = x / a.n, c = x - r * a.n;
            const uint32_t one = (res[r * pitch + (c >> 5)] >> (c & 31)) & 1u;
            out[x] = static_cast<uint8_t>(one | (a.reflexive && c == r0 + r ? 1u : 0u));
        }
    } else {
        uint64_t* out = static_cast<uint64_t*>(a.out) + static_cast<int64_t>(r0) * a.words64;
        for (int x = tid; x < rows * a.words64; x += kThreads) {
            const int r = x / a.words64, w = x - r * a.words64;
            const uint32_t* p = res + r * pitch + 2 * w;
            uint64_t v = p[0] | (static_cast<uint64_t>(p[1]) << 32);  // (the pitch is even)
            if (a.reflexive && ((r0 + r) >> 6) == w) v |= 1ull << ((r0 + r) & 63);
            out[x] = v;
        }
    }
}

int small_pitch(int64_t n) { return static_cast<int>((n + 127) / 128 * 4); }

}  // namespace

size_t small_closure_bytes(int64_t n) { return static_cast<size_t>(3 * n * small_pitch(n)) * 4 + 2 * static_cast<size_t>(n); }

cudaError_t launch_small_closure(const void* in, const void* r1, void* out, int64_t n, bool bytes, int reflexive,
                                 int max_iters, void* scratch, unsigned* arrived, int* result, int* error,
                                 long long wait_cycles, int sms, cudaStream_t s) {
    if (n < 1 || n > kSmallN || max_iters < 1) return cudaErrorInvalidValue;
    SmallArgs a{};
    a.in = in;
    a.r1 = r1;
    a.out = out;
    a.bytes = bytes ? 1 : 0;
    a.n = static_cast<int>(n);
    a.words64 = static_cast<int>((n + 63) / 64);
    a.pitch = small_pitch(n);
    a.rows_per = static_cast<int>((n + sms - 1) / sms);
    if (a.rows_per < 2) a.rows_per = 2;
    a.group = 8;
    while (a.group * 32 < n) a.group *= 2;
    a.reflexive = reflexive;
    a.max_iters = max_iters;
    a.mats = static_cast<uint32_t*>(scratch);
    a.grown = reinterpret_cast<uint8_t*>(a.mats + 3 * n * a.pitch);
    a.arrived = arrived;
    a.result = result;
    a.error = error;
    a.wait_cycles = wait_cycles;
    const int grid = static_cast<int>((n + a.rows_per - 1) / a.rows_per);
    const size_t smem = (static_cast<size_t>(n) + 3 * static_cast<size_t>(a.rows_per)) * a.pitch * 4;
    if (smem > kMostSmem) return cudaErrorInvalidValue;
    const cudaError_t e = allow_smem(small_closure_kernel, kMostSmem);
    if (e != cudaSuccess) return e;
    void* args[] = {&a};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(small_closure_kernel), dim3(static_cast<unsigned>(grid)),
                                       dim3(kThreads), args, smem, s);
}

}  // namespace bmlp
