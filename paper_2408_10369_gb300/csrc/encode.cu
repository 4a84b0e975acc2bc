// Format converters between the caller's matrix layouts and the kernels'
// internal layouts (paper Sec. 3.2: row i of R is the bit code b_i).
//
//  * u8 / packed rows  ->  E4M3 0/1 bytes R (n_pad x n_pad) and its transpose
//    R^T, the K-major operands of the tensor-core product;
//  * E4M3 / 0-1 bytes  ->  u8 or packed rows;
//  * u8 <-> packed rows; per-block nonzero flags for frontier skipping.
//
// Padding rows and columns are written as zero: zero rows and columns add no
// paths, so padding never changes a closure.
#include "internal.h"
#include "ptx.cuh"

namespace bmlp {
namespace {

constexpr int T = 64;  // square tile edge (bytes) of the transposing encoders

__device__ __forceinline__ uint8_t e4m3_bit(bool b) { return b ? BMLP_E4M3_ONE : 0; }

// Source readers: one tile row segment of 16 logical elements as a 16-bit mask.
struct SrcU8 {
    const uint8_t* p;
    int64_t n;
    bool vec;  // rows are 16-byte aligned (n % 16 == 0 and p aligned)
    __device__ __forceinline__ uint32_t bits16(int64_t r, int64_t c0, int64_t rows) const {
        if (r >= rows || c0 >= n) return 0;
        const uint8_t* row = p + r * n;
        uint32_t m = 0;
        if (vec && c0 + 16 <= n) {
            uint4 v = *reinterpret_cast<const uint4*>(row + c0);
            uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int x = 0; x < 16; ++x) m |= (((w[x >> 2] >> ((x & 3) * 8)) & 0xFFu) != 0 ? 1u : 0u) << x;
        } else {
            for (int x = 0; x < 16; ++x)
                if (c0 + x < n && row[c0 + x] != 0) m |= 1u << x;
        }
        return m;
    }
};

struct SrcPacked {
    const uint64_t* p;
    int64_t ldw;
    int64_t n;
    __device__ __forceinline__ uint32_t bits16(int64_t r, int64_t c0, int64_t rows) const {
        if (r >= rows || c0 >= n) return 0;
        uint64_t w = p[r * ldw + (c0 >> 6)];
        uint32_t m = static_cast<uint32_t>((w >> (c0 & 63)) & 0xFFFFu);
        int64_t valid = n - c0;
        if (valid < 16) m &= (1u << valid) - 1u;
        return m;
    }
};

__device__ __forceinline__ uint4 expand16(uint32_t m) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t v = 0;
#pragma unroll
        for (int x = 0; x < 4; ++x) v |= static_cast<uint32_t>(e4m3_bit((m >> (q * 4 + x)) & 1u)) << (8 * x);
        w[q] = v;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// One 64 x 64 tile per block (256 threads, 16 elements each): writes R and,
// when RT != null, R^T. The grid covers rows_pad x n_pad.
template <class Src>
__global__ void encode_e4m3_tile(Src src, int64_t rows, uint8_t* __restrict__ R, uint8_t* __restrict__ RT,
                                 int64_t n_pad, int64_t rows_pad) {
    __shared__ uint16_t masks[T][T / 16 + 1];
    const int tid = threadIdx.x;
    const int r = tid >> 2, cseg = (tid & 3) * 16;
    const int64_t row0 = static_cast<int64_t>(blockIdx.y) * T, col0 = static_cast<int64_t>(blockIdx.x) * T;
    uint32_t m = src.bits16(row0 + r, col0 + cseg, rows);
    masks[r][tid & 3] = static_cast<uint16_t>(m);
    *reinterpret_cast<uint4*>(R + (row0 + r) * n_pad + col0 + cseg) = expand16(m);
    if (RT == nullptr) return;
    __syncthreads();
    // R^T row (col0 + r), columns row0 + cseg .. +16 = tile column r, rows cseg..cseg+15
    uint32_t t = 0;
#pragma unroll
    for (int x = 0; x < 16; ++x) t |= ((masks[cseg + x][r >> 4] >> (r & 15)) & 1u) << x;
    *reinterpret_cast<uint4*>(RT + (col0 + r) * rows_pad + row0 + cseg) = expand16(t);
}

// ---- packed E2M1 (4-bit) operands: element k of a row in byte k / 2, low
// nibble first; 0b0010 = 1.0.
// 8 bits -> 8 nibbles of {0, one}
__device__ __forceinline__ uint32_t nib_spread8(uint32_t b) {
    uint32_t t = b & 0xFFu;
    t = (t | (t << 12)) & 0x000F000Fu;
    t = (t | (t << 6)) & 0x03030303u;
    t = (t | (t << 3)) & 0x11111111u;
    return t << 1;
}
// 8 nibbles -> 8 bits (nonzero nibble = 1)
__device__ __forceinline__ uint32_t nib_gather8(uint32_t w) {
    uint32_t x = w | (w >> 1);
    x |= x >> 2;
    x &= 0x11111111u;
    x = (x | (x >> 3)) & 0x03030303u;
    x = (x | (x >> 6)) & 0x000F000Fu;
    x = (x | (x >> 12)) & 0xFFu;
    return x;
}

// One 64 x 64 tile per block (256 threads, 16 elements each): packed E2M1 R
// (row stride ld4 bytes) and R^T, as encode_e4m3_tile.
template <class Src>
__global__ void encode_e2m1_tile(Src src, int64_t rows, uint8_t* __restrict__ R, uint8_t* __restrict__ RT, int64_t ld4) {
    __shared__ uint16_t masks[T][T / 16 + 1];
    const int tid = threadIdx.x;
    const int r = tid >> 2, cseg = (tid & 3) * 16;
    const int64_t row0 = static_cast<int64_t>(blockIdx.y) * T, col0 = static_cast<int64_t>(blockIdx.x) * T;
    const uint32_t m = src.bits16(row0 + r, col0 + cseg, rows);
    masks[r][tid & 3] = static_cast<uint16_t>(m);
    *reinterpret_cast<uint2*>(R + (row0 + r) * ld4 + (col0 + cseg) / 2) = make_uint2(nib_spread8(m), nib_spread8(m >> 8));
    __syncthreads();
    uint32_t t = 0;
#pragma unroll
    for (int x = 0; x < 16; ++x) t |= ((masks[cseg + x][r >> 4] >> (r & 15)) & 1u) << x;
    *reinterpret_cast<uint2*>(RT + (col0 + r) * ld4 + (row0 + cseg) / 2) = make_uint2(nib_spread8(t), nib_spread8(t >> 8));
}

__device__ __forceinline__ uint4 nib_spread32(uint32_t b) {
    return make_uint4(nib_spread8(b), nib_spread8(b >> 8), nib_spread8(b >> 16), nib_spread8(b >> 24));
}

// Packed bit rows (ldw words per row, n x n) -> packed E2M1 R and R^T (n_pad x
// n_pad, row stride ld4 = n_pad / 2 bytes, padding zero): one 256 x 256 tile
// per block of 256 threads. Thread t reads row row0 + t (four 64-bit words);
// each warp turns its 32 rows into R^T bits as eight 32 x 32 bit blocks
// transposed in registers. Both bit tiles go through shared memory (rows of 8
// words padded to 9), so that every global store is 8 lanes x 16 bytes = one
// 128-byte line of a row of R or R^T, 4 lines per warp instruction.
__global__ void __launch_bounds__(256) packed_to_e2m1_kernel(const uint64_t* __restrict__ p, int64_t ldw, int64_t n,
                                                             uint8_t* __restrict__ R, uint8_t* __restrict__ RT,
                                                             int64_t ld4, bool vec) {
    __shared__ uint32_t sR[256][9];   // row t of the tile: bits of columns 32 w .. 32 w + 31 in word w
    __shared__ uint32_t sT[256][9];   // row c of the transposed tile: bits of rows 32 w .. 32 w + 31
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row0 = static_cast<int64_t>(blockIdx.y) * 256, col0 = static_cast<int64_t>(blockIdx.x) * 256;
    const int64_t r = row0 + threadIdx.x;
    uint64_t w[4] = {0, 0, 0, 0};
    if (r < n) {
        const uint64_t* src = p + r * ldw + col0 / 64;
        const int64_t words = (n - col0 + 63) / 64;  // words of this row inside the tile that hold columns < n
        if (vec && words >= 4) {
            const uint4 a = reinterpret_cast<const uint4*>(src)[0], b = reinterpret_cast<const uint4*>(src)[1];
            w[0] = (static_cast<uint64_t>(a.y) << 32) | a.x;
            w[1] = (static_cast<uint64_t>(a.w) << 32) | a.z;
            w[2] = (static_cast<uint64_t>(b.y) << 32) | b.x;
            w[3] = (static_cast<uint64_t>(b.w) << 32) | b.z;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < words) w[q] = src[q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t valid = n - (col0 + 64 * q);
            if (valid <= 0) w[q] = 0;
            else if (valid < 64) w[q] &= (1ull << valid) - 1ull;
        }
    }
    uint32_t x[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        x[2 * q] = static_cast<uint32_t>(w[q]);
        x[2 * q + 1] = static_cast<uint32_t>(w[q] >> 32);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        sR[threadIdx.x][k] = x[k];
        sT[32 * k + lane][warp] = warp_transpose32(x[k], lane);  // column 32 k + lane, rows 32 warp + i
    }
    __syncthreads();
    // lanes 8 q .. 8 q + 7 write the 8 pieces (16 bytes = 32 elements each) of one row
    const int piece = lane & 7;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int t = warp * 32 + i * 4 + (lane >> 3);
        *reinterpret_cast<uint4*>(R + (row0 + t) * ld4 + col0 / 2 + piece * 16) = nib_spread32(sR[t][piece]);
        *reinterpret_cast<uint4*>(RT + (col0 + t) * ld4 + row0 / 2 + piece * 16) = nib_spread32(sT[t][piece]);
    }
}

// Packed E2M1 rows -> packed bit rows (ldw_out words, + I if reflexive); one output word per thread.
__global__ void e2m1_to_packed_kernel(const uint8_t* __restrict__ Q, int64_t ld4, int64_t n,
                                      uint64_t* __restrict__ out, int64_t ldw_out, int reflexive) {
    const int64_t wpr = (n + 63) / 64;
    const int64_t total = n * ldw_out;
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < total;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t r = t / ldw_out, w = t % ldw_out;
        uint64_t bits = 0;
        if (w < wpr) {
            const uint4* src = reinterpret_cast<const uint4*>(Q + r * ld4 + w * 32);  // 64 nibbles
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint4 v = src[q];
                const uint64_t b = nib_gather8(v.x) | (nib_gather8(v.y) << 8) | (nib_gather8(v.z) << 16) |
                                   (static_cast<uint64_t>(nib_gather8(v.w)) << 24);
                bits |= b << (32 * q);
            }
            const int64_t valid = n - w * 64;
            if (valid < 64) bits &= (1ull << valid) - 1ull;
            if (reflexive && (r >> 6) == w) bits |= 1ull << (r & 63);
        }
        out[t] = bits;
    }
}

// 1 per nonzero 128 x 128 block of an input matrix (rows x n, padded to the block grid); one block of
// 256 threads per map entry, 16 elements per thread per pass.
template <class Src>
__global__ void input_block_flags_kernel(Src src, int64_t rows, int64_t flags_ld, uint8_t* __restrict__ flags) {
    const int64_t br = blockIdx.y, bc = blockIdx.x;
    const int tid = threadIdx.x;
    uint32_t any = 0;
#pragma unroll 4
    for (int k = 0; k < 4; ++k) {
        const int e = (k * 256 + tid) * 16;  // element offset inside the 128 x 128 block
        any |= src.bits16(br * 128 + e / 128, bc * 128 + e % 128, rows);
    }
    any = __syncthreads_or(any != 0);
    if (tid == 0) flags[br * flags_ld + bc] = any ? 1 : 0;
}

// out[i][j] = (R[i][j] != 0) | (reflexive && i == j); 16 outputs per thread.
__global__ void bytes_to_u8_kernel(const uint8_t* __restrict__ R, int64_t ld, int64_t n, uint8_t* __restrict__ out,
                                   int reflexive, bool vec_out) {
    const int64_t segs = (n + 15) / 16;
    const int64_t total = n * segs;
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < total;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t i = t / segs, j0 = (t % segs) * 16;
        uint4 v = *reinterpret_cast<const uint4*>(R + i * ld + j0);
        uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint8_t b[16];
#pragma unroll
        for (int x = 0; x < 16; ++x) {
            b[x] = ((w[x >> 2] >> ((x & 3) * 8)) & 0xFFu) != 0;
            if (reflexive && j0 + x == i) b[x] = 1;
        }
        uint8_t* o = out + i * n + j0;
        if (vec_out && j0 + 16 <= n) {
            uint32_t q[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                q[k] = b[4 * k] | (b[4 * k + 1] << 8) | (b[4 * k + 2] << 16) | (static_cast<uint32_t>(b[4 * k + 3]) << 24);
            *reinterpret_cast<uint4*>(o) = make_uint4(q[0], q[1], q[2], q[3]);
        } else {
            for (int x = 0; x < 16 && j0 + x < n; ++x) o[x] = b[x];
        }
    }
}

// One output word per thread: bits of R[r][64w .. 64w+63] != 0.
__global__ void bytes_to_packed_kernel(const uint8_t* __restrict__ R, int64_t ld, int64_t rows, int64_t n,
                                       uint64_t* __restrict__ out, int64_t ldw_out, int reflexive) {
    const int64_t wpr = (n + 63) / 64;
    const int64_t total = rows * ldw_out;
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < total;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t r = t / ldw_out, w = t % ldw_out;
        uint64_t bits = 0;
        if (w < wpr) {
            const uint4* src = reinterpret_cast<const uint4*>(R + r * ld + w * 64);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint4 v = src[q];
                uint32_t x4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int k = 0; k < 16; ++k)
                    if ((x4[k >> 2] >> ((k & 3) * 8)) & 0xFFu) bits |= 1ull << (q * 16 + k);
            }
            const int64_t valid = n - w * 64;
            if (valid < 64) bits &= (1ull << valid) - 1ull;
            if (reflexive && r < n && (r >> 6) == w) bits |= 1ull << (r & 63);
        }
        out[t] = bits;
    }
}

// ---- byte matrices <-> bit rows
// Bound by HBM: n^2 bytes one way and n^2 / 8 the other. A byte row starts at any alignment when n is not a multiple
// of 16, so a block takes one contiguous run of the matrix, a few whole rows or kUnitCols columns of a longer row, and
// moves it as the aligned 16-byte chunks that cover it: a chunk's 16 bytes become 16 bits of a bit run in shared
// memory (or are made from it), and a row's words are cut out of that run by funnel shifts at their bit offset. The
// chunks at the two ends, which hold bytes of neighbouring runs, go byte by byte where they leave the matrix (reads) or
// the run (writes). At n = 14,541 (211 MB of bytes, 26 MB of bits) one word per thread with 64 byte loads took 340 us one
// way and one thread per byte, a 64-bit division each, 384 us the other; this form takes 48 us (5.0 TB/s) and 51 us.
constexpr int kUnitBytes = 32768;  // bytes of a run at most
constexpr int kUnitCols = 16384;   // columns of a run of a row longer than that (a multiple of 64)
constexpr int kUnitThreads = 256;
constexpr int kUnitInFlight = kUnitBytes / 16 / kUnitThreads;  // interior chunks per thread

// The run of block `unit`: rows r0 .. r0 + rows - 1 whole (segs == 1), or columns c0 .. c0 + len - 1 of row r0.
struct ByteUnit {
    int64_t r0, c0;
    int rows, len;
    __device__ ByteUnit(int64_t unit, int64_t n, int rows_per, int segs) {
        r0 = segs > 1 ? unit / segs : unit * rows_per;
        c0 = segs > 1 ? (unit % segs) * kUnitCols : 0;
        rows = segs > 1 ? 1 : static_cast<int>(n - r0 < rows_per ? n - r0 : rows_per);
        len = segs > 1 ? static_cast<int>(n - c0 < kUnitCols ? n - c0 : kUnitCols) : rows * static_cast<int>(n);
    }
};

// 4 bytes -> 4 bits (bit k = byte k nonzero): bit 7 of every nonzero byte, gathered by one multiplication whose
// partial products fall on distinct bits.
__device__ __forceinline__ uint32_t bytes_bits4(uint32_t w) {
    const uint32_t t = ((((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) >> 7) & 0x01010101u;
    return (t * 0x10204080u) >> 28;
}
__device__ __forceinline__ uint32_t bytes_bits16(const uint4& v) {
    return bytes_bits4(v.x) | (bytes_bits4(v.y) << 4) | (bytes_bits4(v.z) << 8) | (bytes_bits4(v.w) << 12);
}
// and back: 4 bits -> 4 bytes of 0 / 1
__device__ __forceinline__ uint32_t bits_bytes4(uint32_t b) { return ((b & 0xFu) * 0x00204081u) & 0x01010101u; }
__device__ __forceinline__ uint4 bits_bytes16(uint32_t m) {
    return make_uint4(bits_bytes4(m), bits_bytes4(m >> 4), bits_bytes4(m >> 8), bits_bytes4(m >> 12));
}

// u8 rows (ld = n) -> bit rows of ldw_out words (columns beyond n zero).
__global__ void __launch_bounds__(kUnitThreads) u8_to_packed_kernel(const uint8_t* __restrict__ in, int64_t n,
                                                                    uint64_t* __restrict__ out, int64_t ldw_out,
                                                                    int rows_per, int segs) {
    __shared__ __align__(16) uint32_t run[kUnitBytes / 32 + 8];  // bit x: byte x of the covering chunks; + what funnel
    uint16_t* run16 = reinterpret_cast<uint16_t*>(run);           // shifts read (and mask off) past the last chunk
    const ByteUnit u(blockIdx.x, n, rows_per, segs);
    const uint8_t* first = in + u.r0 * n + u.c0;
    const int mis = static_cast<int>(reinterpret_cast<uintptr_t>(first) & 15);
    const uint8_t* base = first - mis;
    const uint8_t* end = in + n * n;
    const int chunks = (mis + u.len + 15) >> 4;
    uint4 v[kUnitInFlight];  // chunks 1 .. chunks - 2 lie inside the run: all of a thread's loads in flight at once
#pragma unroll
    for (int j = 0; j < kUnitInFlight; ++j) {
        const int k = 1 + static_cast<int>(threadIdx.x) + j * kUnitThreads;
        v[j] = k < chunks - 1 ? __ldg(reinterpret_cast<const uint4*>(base) + k) : make_uint4(0, 0, 0, 0);
    }
    if (threadIdx.x < 2) {
        const int k = threadIdx.x == 0 ? 0 : chunks - 1;
        const uint8_t* c = base + 16 * k;
        uint32_t m = 0;
        for (int x = 0; x < 16; ++x)
            if (c + x >= in && c + x < end && c[x] != 0) m |= 1u << x;
        run16[k] = static_cast<uint16_t>(m);
    }
#pragma unroll
    for (int j = 0; j < kUnitInFlight; ++j) {
        const int k = 1 + static_cast<int>(threadIdx.x) + j * kUnitThreads;
        if (k < chunks - 1) run16[k] = static_cast<uint16_t>(bytes_bits16(v[j]));
    }
    __syncthreads();
    const int wpr = static_cast<int>((n + 63) >> 6), ldw = static_cast<int>(ldw_out);
    // whole rows: all of their words, padding words too; a segment: its words, and the last one the padding words
    const int w0 = static_cast<int>(u.c0 >> 6);
    const int words = segs == 1 ? ldw : (u.c0 + kUnitCols < n ? kUnitCols / 64 : ldw - w0);
    for (int x = threadIdx.x; x < u.rows * words; x += kUnitThreads) {
        const int r = x / words, wl = x - r * words;
        uint64_t bits = 0;
        if (w0 + wl < wpr) {
            const int b = mis + r * static_cast<int>(n) + 64 * wl;  // (a segment has r = 0)
            const int i = b >> 5;
            bits = static_cast<uint64_t>(__funnelshift_r(run[i], run[i + 1], b & 31)) |
                   (static_cast<uint64_t>(__funnelshift_r(run[i + 1], run[i + 2], b & 31)) << 32);
            const int64_t valid = n - 64ll * (w0 + wl);
            if (valid < 64) bits &= (1ull << valid) - 1ull;
        }
        out[(u.r0 + r) * ldw_out + w0 + wl] = bits;
    }
}

// Bit rows (ldw words) -> u8 rows of 0 / 1 (ld = n), the diagonal set when reflexive.
__global__ void __launch_bounds__(kUnitThreads) packed_to_u8_kernel(const uint64_t* __restrict__ in, int64_t ldw,
                                                                    int64_t n, uint8_t* __restrict__ out,
                                                                    int reflexive, int rows_per, int segs) {
    // the run's rows, wpr words each: at most (kUnitBytes + 63 rows) / 64 words for n >= 64, 64 rows of one for less
    __shared__ __align__(16) uint64_t rows[kUnitBytes / 32 + 8];
    const uint32_t* rows32 = reinterpret_cast<const uint32_t*>(rows);
    const ByteUnit u(blockIdx.x, n, rows_per, segs);
    const int w0 = static_cast<int>(u.c0 >> 6);
    const int cols = segs == 1 ? static_cast<int>(n) : u.len;  // of a row of the run
    const int words = (cols + 63) >> 6;
    for (int x = threadIdx.x; x < u.rows * words; x += kUnitThreads) {
        const int r = x / words, wl = x - r * words;
        uint64_t bits = in[(u.r0 + r) * ldw + w0 + wl];
        if (reflexive && ((u.r0 + r) >> 6) == w0 + wl) bits |= 1ull << ((u.r0 + r) & 63);
        rows[x] = bits;
    }
    __syncthreads();
    uint8_t* first = out + u.r0 * n + u.c0;
    const int mis = static_cast<int>(reinterpret_cast<uintptr_t>(first) & 15);
    uint8_t* base = first - mis;
    const int chunks = (mis + u.len + 15) >> 4;
    for (int k = threadIdx.x; k < chunks; k += kUnitThreads) {
        const int p = 16 * k - mis;  // the chunk's first byte within the run (before it: p < 0)
        const int r = p > 0 ? p / cols : 0;
        const int c = p - r * cols;
        if (p >= 0 && c + 16 <= cols) {
            const int i = 2 * r * words + (c >> 5);
            const uint32_t m = __funnelshift_r(rows32[i], rows32[i + 1], c & 31);
            *reinterpret_cast<uint4*>(base + 16 * k) = bits_bytes16(m);
        } else {  // the run's ends, or a chunk across rows
            uint32_t w[4] = {0, 0, 0, 0};
            int rr = r, cc = c < 0 ? 0 : c;
            for (int x = p < 0 ? -p : 0; x < 16 && p + x < u.len; ++x) {
                const uint32_t bit = (rows32[2 * rr * words + (cc >> 5)] >> (cc & 31)) & 1u;
                w[x >> 2] |= bit << (8 * (x & 3));
                if (++cc == cols) {
                    cc = 0;
                    ++rr;
                }
            }
            if (p >= 0 && p + 16 <= u.len) {
                *reinterpret_cast<uint4*>(base + 16 * k) = make_uint4(w[0], w[1], w[2], w[3]);
            } else {
                for (int x = p < 0 ? -p : 0; x < 16 && p + x < u.len; ++x)
                    base[16 * k + x] = static_cast<uint8_t>(w[x >> 2] >> (8 * (x & 3)));
            }
        }
    }
}

// Word w of a packed row with its bits at columns >= n cleared (w < ceil(n / 64)).
__device__ __forceinline__ uint64_t row_word(const uint64_t* row, int64_t w, int64_t n) {
    const int64_t valid = n - w * 64;
    return valid < 64 ? row[w] & ((1ull << valid) - 1ull) : row[w];
}

// The packed element-wise passes: a warp per row, its lanes over the row's words (bound by HBM; a thread per word of
// the whole matrix spent its time on a 64-bit division for the row).
constexpr int kRowThreads = 256;
#define BMLP_FOR_ROWS(i, rows)                                                                                    \
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (kRowThreads / 32) + (threadIdx.x >> 5); i < (rows);      \
         i += static_cast<int64_t>(gridDim.x) * (kRowThreads / 32))

__global__ void __launch_bounds__(kRowThreads) packed_copy_kernel(const uint64_t* in, int64_t ldw_in, int64_t rows,
                                                                  int64_t n, uint64_t* out, int64_t ldw_out,
                                                                  int reflexive) {
    const int64_t wpr = (n + 63) / 64;
    BMLP_FOR_ROWS(r, rows) {
        for (int64_t w0 = threadIdx.x & 31; w0 < ldw_out; w0 += 128) {
            uint64_t v[4];  // four loads in flight (out may be in, so the compiler keeps loads behind earlier stores)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = w0 + 32 * k < wpr ? row_word(in + r * ldw_in, w0 + 32 * k, n) : 0ull;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t w = w0 + 32 * k;
                if (reflexive && r < n && (r >> 6) == w) v[k] |= 1ull << (r & 63);
                if (w < ldw_out) out[r * ldw_out + w] = v[k];
            }
        }
    }
}

// out = A OR B over n packed rows of ceil(n / 64) words (out may be A or B: each word is read and written by one
// thread).
__global__ void __launch_bounds__(kRowThreads) packed_union_kernel(const uint64_t* A, const uint64_t* B, int64_t n,
                                                                   uint64_t* out) {
    const int64_t wpr = (n + 63) / 64;
    BMLP_FOR_ROWS(r, n) {
        for (int64_t w0 = threadIdx.x & 31; w0 < wpr; w0 += 128) {
            uint64_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t w = w0 + 32 * k;
                v[k] = w < wpr ? row_word(A + r * wpr, w, n) | row_word(B + r * wpr, w, n) : 0ull;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (w0 + 32 * k < wpr) out[r * wpr + w0 + 32 * k] = v[k];
        }
    }
}

__global__ void packed_or_kernel(uint64_t* __restrict__ out, int64_t ldw_out, const uint64_t* __restrict__ src,
                                 int64_t ldw_src, int64_t rows, int64_t n) {
    const int64_t wpr = (n + 63) / 64;
    const int64_t total = rows * wpr;
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < total;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t r = t / wpr, w = t % wpr;
        uint64_t s = src[r * ldw_src + w];
        const int64_t valid = n - w * 64;
        if (valid < 64) s &= (1ull << valid) - 1ull;
        out[r * ldw_out + w] |= s;
    }
}

__global__ void identity_packed_kernel(uint64_t* __restrict__ out, int64_t ldw, int64_t n) {
    const int64_t total = n * ldw;
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < total;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t r = t / ldw, w = t % ldw;
        out[t] = ((r >> 6) == w) ? (1ull << (r & 63)) : 0ull;
    }
}

// NEG of Fig. 3 with the type literals of a stratified negation: out[i][j] =
// rows(i) AND cols(j) AND NOT in[i][j] for i, j < n; a null rows / cols
// vector admits every constant. Bits at j >= n stay zero. out may be in.
__global__ void __launch_bounds__(kRowThreads) negate_restrict_kernel(const uint64_t* in, int64_t ldw_in, int64_t n,
                                                                      const uint64_t* __restrict__ rows,
                                                                      const uint64_t* __restrict__ cols, uint64_t* out,
                                                                      int64_t ldw_out) {
    const int64_t wpr = (n + 63) / 64;
    BMLP_FOR_ROWS(r, n) {
        const bool typed = !rows || ((rows[r >> 6] >> (r & 63)) & 1ull);
        for (int64_t w0 = threadIdx.x & 31; w0 < ldw_out; w0 += 128) {
            uint64_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t w = w0 + 32 * k;
                v[k] = 0ull;
                if (w < wpr && typed) {
                    v[k] = ~in[r * ldw_in + w];
                    if (cols) v[k] &= cols[w];
                    const int64_t valid = n - w * 64;
                    if (valid < 64) v[k] &= (1ull << valid) - 1ull;
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (w0 + 32 * k < ldw_out) out[r * ldw_out + w0 + 32 * k] = v[k];
        }
    }
}

// The same two operators on byte matrices in one pass, without bit rows in between (bound by HBM: at n = 14,541 the union
// moves 633 MB in 96 us, 6.6 TB/s, and NEG 422 MB in 84 us; through bit rows they took 1,080 and 740 us). Union: 16 bytes per thread and step where all three
// matrices are 16-byte aligned, else byte by byte. out may be A or B.
__device__ __forceinline__ uint32_t bytes_ones4(uint32_t w) {  // each byte 0 or 1: whether it was nonzero
    return ((((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) >> 7) & 0x01010101u;
}
__global__ void __launch_bounds__(256) u8_union_kernel(const uint8_t* A, const uint8_t* B, int64_t bytes, uint8_t* out,
                                                       bool vec) {
    const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t n16 = vec ? bytes / 16 : 0;
#pragma unroll 4
    for (int64_t t = t0; t < n16; t += stride) {
        const uint4 a = reinterpret_cast<const uint4*>(A)[t], b = reinterpret_cast<const uint4*>(B)[t];
        reinterpret_cast<uint4*>(out)[t] = make_uint4(bytes_ones4(a.x | b.x), bytes_ones4(a.y | b.y),
                                                      bytes_ones4(a.z | b.z), bytes_ones4(a.w | b.w));
    }
    for (int64_t t = 16 * n16 + t0; t < bytes; t += stride) out[t] = (A[t] | B[t]) != 0 ? 1 : 0;
}

// NEG on bytes: a block per run of the matrix (ByteUnit), 16 output bytes per thread and step; the type vectors are bit
// vectors, so 16 columns are cut out of `cols` by a funnel shift. out may be in (each byte is read and written by one
// thread).
__global__ void __launch_bounds__(kUnitThreads) u8_negate_kernel(const uint8_t* in, int64_t n,
                                                                 const uint64_t* __restrict__ rows,
                                                                 const uint64_t* __restrict__ cols, uint8_t* out,
                                                                 int rows_per, int segs) {
    const ByteUnit u(blockIdx.x, n, rows_per, segs);
    const int ncols = segs == 1 ? static_cast<int>(n) : u.len;
    const int64_t off = u.r0 * n + u.c0;
    const int mis = static_cast<int>(reinterpret_cast<uintptr_t>(out + off) & 15);
    const bool vec = ((reinterpret_cast<uintptr_t>(in) ^ reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    const int chunks = (mis + u.len + 15) >> 4;
    const int cwords = static_cast<int>((n + 31) >> 5);  // 32-bit words of a type vector that hold constants
    const uint32_t* cols32 = reinterpret_cast<const uint32_t*>(cols);
    const auto typed = [&](int64_t i) { return !rows || ((rows[i >> 6] >> (i & 63)) & 1ull) != 0ull; };
#pragma unroll 2
    for (int k = threadIdx.x; k < chunks; k += kUnitThreads) {
        const int p = 16 * k - mis;
        const int r = p > 0 ? p / ncols : 0;
        const int c = p - r * ncols;
        if (vec && p >= 0 && c + 16 <= ncols) {
            const uint4 v = *reinterpret_cast<const uint4*>(in + off + p);
            uint32_t m = typed(u.r0 + r) ? 0xFFFFu : 0u;
            if (cols) {
                const int b = static_cast<int>(u.c0) + c, i = b >> 5;
                m &= __funnelshift_r(cols32[i], i + 1 < cwords ? cols32[i + 1] : 0u, b & 31);
            }
            const uint4 ones = bits_bytes16(m);
            *reinterpret_cast<uint4*>(out + off + p) = make_uint4(ones.x & ~bytes_ones4(v.x), ones.y & ~bytes_ones4(v.y),
                                                                  ones.z & ~bytes_ones4(v.z), ones.w & ~bytes_ones4(v.w));
        } else {
            int rr = r, cc = c < 0 ? 0 : c;
            for (int x = p < 0 ? -p : 0; x < 16 && p + x < u.len; ++x) {
                const int64_t j = u.c0 + cc;
                const bool ok = typed(u.r0 + rr) && (!cols || ((cols[j >> 6] >> (j & 63)) & 1ull));
                out[off + p + x] = ok && in[off + p + x] == 0 ? 1 : 0;
                if (++cc == ncols) {
                    cc = 0;
                    ++rr;
                }
            }
        }
    }
}

// Entry (i, i) of a packed E2M1 matrix (ld bytes per row) set to one for i < n: nibble i & 1 of byte i / 2 of row i
// (each row's byte is written by one thread).
__global__ void set_diag_e2m1_kernel(uint8_t* Q, int64_t ld, int64_t n) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n) Q[i * ld + (i >> 1)] |= static_cast<uint8_t>((i & 1) ? 0x20 : 0x02);
}

__global__ void set_diag_kernel(uint8_t* R, int64_t ld, int64_t n) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        R[i * ld + i] = BMLP_E4M3_ONE;
}

// flags[mb * kb_count + kb] = any nonzero byte in the 128 x 128 block (mb, kb).
__global__ void block_flags_kernel(const uint8_t* __restrict__ A, int64_t ld, int64_t kb_count,
                                   uint8_t* __restrict__ flags) {
    const int64_t mb = blockIdx.y, kb = blockIdx.x;
    const int r = threadIdx.x >> 1, half = threadIdx.x & 1;  // 256 threads: 128 rows x 2 halves of 64 bytes
    const uint4* p = reinterpret_cast<const uint4*>(A + (mb * 128 + r) * ld + kb * 128 + half * 64);
    uint32_t any = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint4 v = p[q];
        any |= v.x | v.y | v.z | v.w;
    }
    any = __syncthreads_or(any != 0);
    if (threadIdx.x == 0) flags[mb * kb_count + kb] = any ? 1 : 0;
}

inline int grid_for(int64_t work, int threads) {
    int64_t g = (work + threads - 1) / threads;
    if (g > 152 * 32) g = 152 * 32;
    if (g < 1) g = 1;
    return static_cast<int>(g);
}

}  // namespace

void launch_u8_to_e4m3(const uint8_t* in, int64_t n, uint8_t* R, uint8_t* RT, int64_t n_pad, cudaStream_t s) {
    SrcU8 src{in, n, (n % 16 == 0) && ((reinterpret_cast<uintptr_t>(in) & 15) == 0)};
    dim3 grid(static_cast<unsigned>(n_pad / T), static_cast<unsigned>(n_pad / T));
    encode_e4m3_tile<SrcU8><<<grid, 256, 0, s>>>(src, n, R, RT, n_pad, n_pad);
}

void launch_packed_to_e4m3(const uint64_t* in, int64_t ldw_in, int64_t rows, int64_t n, uint8_t* R, uint8_t* RT,
                           int64_t n_pad, int64_t rows_pad, cudaStream_t s) {
    SrcPacked src{in, ldw_in, n};
    dim3 grid(static_cast<unsigned>(n_pad / T), static_cast<unsigned>(rows_pad / T));
    encode_e4m3_tile<SrcPacked><<<grid, 256, 0, s>>>(src, rows, R, RT, n_pad, rows_pad);
}

void launch_u8_to_e2m1(const uint8_t* in, int64_t n, uint8_t* R, uint8_t* RT, int64_t n_pad, cudaStream_t s) {
    SrcU8 src{in, n, (n % 16 == 0) && ((reinterpret_cast<uintptr_t>(in) & 15) == 0)};
    dim3 grid(static_cast<unsigned>(n_pad / T), static_cast<unsigned>(n_pad / T));
    encode_e2m1_tile<SrcU8><<<grid, 256, 0, s>>>(src, n, R, RT, n_pad / 2);
}

void launch_packed_to_e2m1(const uint64_t* in, int64_t ldw_in, int64_t n, uint8_t* R, uint8_t* RT, int64_t n_pad,
                           cudaStream_t s) {
    // n_pad is a multiple of 256 (TC_PAD); 16-byte row loads when every tile's first word is 16-byte aligned
    const bool vec = (ldw_in % 2 == 0) && ((reinterpret_cast<uintptr_t>(in) & 15) == 0);
    dim3 grid(static_cast<unsigned>(n_pad / 256), static_cast<unsigned>(n_pad / 256));
    packed_to_e2m1_kernel<<<grid, 256, 0, s>>>(in, ldw_in, n, R, RT, n_pad / 2, vec);
}

void launch_e2m1_to_packed(const uint8_t* Q, int64_t ld4, int64_t n, uint64_t* out, int64_t ldw_out, int reflexive,
                           cudaStream_t s) {
    e2m1_to_packed_kernel<<<grid_for(n * ldw_out, 256), 256, 0, s>>>(Q, ld4, n, out, ldw_out, reflexive);
}

void launch_input_block_flags(const void* in, int32_t fmt, int64_t ldw_in, int64_t n, int64_t n_pad, uint8_t* flags,
                              int64_t flags_ld, cudaStream_t s) {
    dim3 grid(static_cast<unsigned>(n_pad / 128), static_cast<unsigned>(n_pad / 128));
    if (fmt == BMLP_FMT_U8) {
        SrcU8 src{static_cast<const uint8_t*>(in), n,
                  (n % 16 == 0) && ((reinterpret_cast<uintptr_t>(in) & 15) == 0)};
        input_block_flags_kernel<SrcU8><<<grid, 256, 0, s>>>(src, n, flags_ld, flags);
    } else {
        SrcPacked src{static_cast<const uint64_t*>(in), ldw_in, n};
        input_block_flags_kernel<SrcPacked><<<grid, 256, 0, s>>>(src, n, flags_ld, flags);
    }
}

void launch_bytes_to_u8(const uint8_t* R, int64_t ld, int64_t n, uint8_t* out, int reflexive, cudaStream_t s) {
    bool vec = (n % 16 == 0) && ((reinterpret_cast<uintptr_t>(out) & 15) == 0);
    int64_t work = n * ((n + 15) / 16);
    bytes_to_u8_kernel<<<grid_for(work, 256), 256, 0, s>>>(R, ld, n, out, reflexive, vec);
}

void launch_bytes_to_packed(const uint8_t* R, int64_t ld, int64_t rows, int64_t n, uint64_t* out, int64_t ldw_out,
                            int reflexive, cudaStream_t s) {
    bytes_to_packed_kernel<<<grid_for(rows * ldw_out, 256), 256, 0, s>>>(R, ld, rows, n, out, ldw_out, reflexive);
}

// Runs of the byte <-> bit converters: whole rows while a row has at most kUnitCols bytes, small enough that the runs
// give each of 152 SMs two blocks (a bound of their size only: any number of SMs takes them in turn), but at least 2 KB.
static int64_t byte_units(int64_t n, int* rows_per, int* segs) {
    if (n > kUnitCols) {
        *rows_per = 1;
        *segs = static_cast<int>((n + kUnitCols - 1) / kUnitCols);
        return n * *segs;
    }
    int64_t bytes = n * n / (2 * 152);
    if (bytes > kUnitBytes) bytes = kUnitBytes;
    if (bytes < 2048) bytes = 2048;
    int64_t rows = bytes / n;
    if (rows < 1) rows = 1;
    if (rows > n) rows = n;
    *rows_per = static_cast<int>(rows);
    *segs = 1;
    return (n + rows - 1) / rows;
}

void launch_u8_to_packed(const uint8_t* in, int64_t n, uint64_t* out, int64_t ldw_out, cudaStream_t s) {
    int rows_per = 0, segs = 0;
    const int64_t units = byte_units(n, &rows_per, &segs);
    u8_to_packed_kernel<<<static_cast<unsigned>(units), kUnitThreads, 0, s>>>(in, n, out, ldw_out, rows_per, segs);
}

void launch_packed_copy(const uint64_t* in, int64_t ldw_in, int64_t rows, int64_t n, uint64_t* out, int64_t ldw_out,
                        int reflexive, cudaStream_t s) {
    packed_copy_kernel<<<grid_for(rows, kRowThreads / 32), kRowThreads, 0, s>>>(in, ldw_in, rows, n, out, ldw_out,
                                                                                 reflexive);
}

void launch_packed_to_u8(const uint64_t* in, int64_t ldw, int64_t n, uint8_t* out, int reflexive, cudaStream_t s) {
    int rows_per = 0, segs = 0;
    const int64_t units = byte_units(n, &rows_per, &segs);
    packed_to_u8_kernel<<<static_cast<unsigned>(units), kUnitThreads, 0, s>>>(in, ldw, n, out, reflexive, rows_per, segs);
}

void launch_packed_or(uint64_t* out, int64_t ldw_out, const uint64_t* src, int64_t ldw_src, int64_t rows, int64_t n,
                      cudaStream_t s) {
    packed_or_kernel<<<grid_for(rows * ((n + 63) / 64), 256), 256, 0, s>>>(out, ldw_out, src, ldw_src, rows, n);
}

void launch_identity_packed(uint64_t* out, int64_t ldw, int64_t n, cudaStream_t s) {
    identity_packed_kernel<<<grid_for(n * ldw, 256), 256, 0, s>>>(out, ldw, n);
}

void launch_packed_negate(const uint64_t* in, int64_t ldw_in, int64_t n, const uint64_t* rows, const uint64_t* cols,
                          uint64_t* out, int64_t ldw_out, cudaStream_t s) {
    negate_restrict_kernel<<<grid_for(n, kRowThreads / 32), kRowThreads, 0, s>>>(in, ldw_in, n, rows, cols, out,
                                                                                  ldw_out);
}

void launch_packed_union(const uint64_t* A, const uint64_t* B, int64_t n, uint64_t* out, cudaStream_t s) {
    packed_union_kernel<<<grid_for(n, kRowThreads / 32), kRowThreads, 0, s>>>(A, B, n, out);
}

void launch_u8_union(const uint8_t* A, const uint8_t* B, int64_t n, uint8_t* out, cudaStream_t s) {
    const bool vec = ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B) | reinterpret_cast<uintptr_t>(out)) &
                      15) == 0;
    const int64_t bytes = n * n;
    u8_union_kernel<<<grid_for(vec ? bytes / 16 + 1 : bytes, 256), 256, 0, s>>>(A, B, bytes, out, vec);
}

void launch_u8_negate(const uint8_t* in, int64_t n, const uint64_t* rows, const uint64_t* cols, uint8_t* out,
                      cudaStream_t s) {
    int rows_per = 0, segs = 0;
    const int64_t units = byte_units(n, &rows_per, &segs);
    u8_negate_kernel<<<static_cast<unsigned>(units), kUnitThreads, 0, s>>>(in, n, rows, cols, out, rows_per, segs);
}

void launch_set_diag_e4m3(uint8_t* R, int64_t ld, int64_t n, cudaStream_t s) {
    set_diag_kernel<<<grid_for(n, 256), 256, 0, s>>>(R, ld, n);
}

void launch_set_diag_e2m1(uint8_t* Q, int64_t ld4, int64_t n, cudaStream_t s) {
    set_diag_e2m1_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(Q, ld4, n);
}

void launch_block_flags(const uint8_t* A, int64_t ld, int64_t rows_pad, int64_t n_pad, uint8_t* flags,
                        cudaStream_t s, int64_t flags_ld) {
    dim3 grid(static_cast<unsigned>(n_pad / 128), static_cast<unsigned>(rows_pad / 128));
    block_flags_kernel<<<grid, 256, 0, s>>>(A, ld, flags_ld > 0 ? flags_ld : n_pad / 128, flags);
}

namespace {
__global__ void e4m3_to_01_kernel(uint8_t* __restrict__ p, int64_t bytes) {
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < bytes;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        p[i] = (p[i] & 0x7Fu) != 0 ? 1 : 0;
}
__global__ void to_e4m3_bytes_kernel(uint8_t* __restrict__ p, int64_t bytes) {
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < bytes;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        p[i] = p[i] != 0 ? static_cast<uint8_t>(BMLP_E4M3_ONE) : 0;
}
int byte_grid(int64_t bytes) {
    int64_t g = (bytes + 255) / 256;
    if (g > 152 * 16) g = 152 * 16;
    return static_cast<int>(g < 1 ? 1 : g);
}
}  // namespace

void launch_e4m3_bytes_to_01(uint8_t* p, int64_t bytes, cudaStream_t s) {
    e4m3_to_01_kernel<<<byte_grid(bytes), 256, 0, s>>>(p, bytes);
}

void launch_01_to_e4m3_bytes(uint8_t* p, int64_t bytes, cudaStream_t s) {
    to_e4m3_bytes_kernel<<<byte_grid(bytes), 256, 0, s>>>(p, bytes);
}

}  // namespace bmlp
