// Library-internal declarations shared by the C ABI and the kernel files.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/bmlp.h"

// e4m3 encoding of 1.0 (sign 0, exponent 0111, mantissa 000) used for the
// 0/1 tensor-core operands.
#define BMLP_E4M3_ONE 0x38

namespace bmlp {

// Tile shape of the tensor-core product: BM x BN output tile, BK bytes
// (= E4M3 elements) of the reduction dimension per pipeline stage.
constexpr int TC_BM = 128;
constexpr int TC_BN = 256;
constexpr int TC_BK = 128;
constexpr int TC_STAGES = 4;
constexpr int TC_THREADS = 192;   // warp 0 TMA, warp 1 MMA, warps 2..5 epilogue
constexpr int TC_PAD = 256;       // matrices are padded to a multiple of this

// Epilogue modes of the tensor-core product kernel.
enum TcMode : int {
    TC_MODE_RMS = 0,    // out = old | (C > 0), also writes out^T; changed flag
    TC_MODE_SMP = 1,    // N = (C > 0) & ~V ; V |= N ; next = N; block flags
    TC_MODE_PLAIN = 2   // out = (C > 0)
};

struct TcParams {
    int32_t m_tiles, n_tiles, k_blocks;
    int32_t mode;
    int64_t ld;                 // row stride (bytes) of every 8-bit matrix
    const uint8_t* old_r;       // RMS: R of this iteration (row-major)
    uint8_t* out_r;             // RMS: new R; SMP: next frontier; PLAIN: output
    uint8_t* out_rt;            // RMS: new R^T
    uint8_t* visited;           // SMP: V (row-major, 0 / 1 bytes)
    const uint8_t* kflags;      // SMP: nonzero flag per (M block, K block) of A, or null
    uint8_t* kflags_next;       // SMP: flags for the next frontier
    int* changed;               // set to 1 when any output bit changed / is new
    int* error;                 // set to a nonzero code when a wait timed out
    long long wait_cycles;      // bound of each in-kernel wait
    // RMS block maps (only when k_blocks <= 256): fmap[rb * fm_ld + cb] = 1 iff the 128 x 128 block (rb, cb)
    // of R is nonzero, fmapT the transpose (fmapT[cb * fm_ld + rb]); rows padded with zeros to fm_ld, a
    // multiple of 16. The epilogue fills the maps of the new R (cleared by the caller).
    const uint8_t* fmap;
    const uint8_t* fmapT;
    uint8_t* fmap_next;
    uint8_t* fmapT_next;
    int32_t fm_ld;
    unsigned long long* issued; // multiply-adds issued in units of 128 x 32 x 128 (rows x columns x K), or null
    const int* guard;           // 4-bit squaring kernel: if not null and *guard == 0 the launch does nothing (a step
                                // of a device-side loop that a decision kernel switched off)
    // squaring kernels on packed operands: if not null, the epilogue also writes R' and R'^T as bit rows of ldb
    // 32-bit words (bit j of word u = column 32 u + j), n_pad rows each
    uint32_t* out_bits;
    uint32_t* out_bits_t;
    int64_t ldb;
    // if not null, R of this iteration as such bit rows, instead of old_r (may be out_bits). out_r may be null with out_bits
    // set: R' leaves as bit rows only; without old_r and old_bits R' is the product alone
    const uint32_t* old_bits;
    int32_t k_first;            // squaring kernels on packed operands: first of the k_blocks blocks of K
};

// One problem of a grouped batch (device copy; built on the host).
struct GroupProblem {  // aligned as CUtensorMap (TMA descriptors must be 64-byte aligned)
    CUtensorMap mapA[2];   // A operand: M[parity] (row-major R)
    CUtensorMap mapB[2];   // B operand: T[parity] (R^T)
    CUtensorMap mapBF;     // composition: B of the final product = R1^T
    uint8_t* M[2];         // E4M3 R ping-pong (tensor-core engine)
    uint8_t* T[2];         // E4M3 R^T ping-pong
    uint8_t* X;            // composition: final product
    uint8_t* R1T;          // composition: E4M3 R1^T
    uint64_t* P[2];        // packed ping-pong (packed engine, and the tensor-core engine's bit-row start)
    uint64_t* PR1;         // composition: packed R1
    const void* in1;       // caller's R1 (closure input, or composition r1)
    const void* in2;       // caller's R2 (composition r2)
    void* out;             // caller's output
    int64_t n;
    int64_t ld;            // n_pad (tensor-core engine)
    int64_t ldw;           // words per packed row
    int32_t m_tiles, n_tiles, k_blocks;
    int32_t kind;          // 0 closure, 1 composition
    int32_t engine;        // 0 tensor cores, 1 packed
    int32_t fmt;           // caller's format
    int32_t reflexive;
    int32_t cap;           // iteration cap
};

// Per-problem loop state of a grouped batch (device memory).
struct GroupState {
    unsigned long long* ones;  // ones of the current R while on bit rows
    int* top;        // and the most of one row
    int* phase;      // 0: on bit rows, 1: handed over to the tensor cores
    int* ppar;       // packed buffer that held R when the bit-row squarings ended
    int* parity;     // buffer holding the current R
    int* active;     // still iterating
    int* iters;      // products issued
    int* changed;    // set by the last product
    int* notconv;    // stopped at the cap while still changing
    int* tc_offs;    // exclusive prefix of active tensor-core tiles (nprob + 1)
    int* tc_total;
    int* pk_offs;    // exclusive prefix of active packed rows (nprob + 1)
    int* pk_total;
};

// Optional time budget of a long kernel: the first warp to look records the
// start (%globaltimer) in *t0; any warp that finds more than budget_ns
// elapsed raises *hit and stops taking work. budget_ns = 0: no budget.
struct Deadline {
    unsigned long long budget_ns;
    unsigned long long* t0;
    int* hit;
#ifdef __CUDACC__
    __device__ __forceinline__ bool past() const {
        if (budget_ns == 0) return false;
        unsigned long long now;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
        unsigned long long s = *reinterpret_cast<volatile unsigned long long*>(t0);
        if (s == 0) {
            atomicCAS(t0, 0ull, now);
            s = *reinterpret_cast<volatile unsigned long long*>(t0);
        }
        if (now > s && now - s > budget_ns) {
            *reinterpret_cast<volatile int*>(hit) = 1;
            return true;
        }
        return false;
    }
#endif
};

// A kernel's limit of dynamic shared memory belongs to the kernel on the device, not to a context or a thread: set to what
// one launch needs, it could be lowered by another thread's smaller launch between this one's setting and its launch, which
// is then refused. So every setting of a kernel raises the limit to the same value, the most that any of its launches needs.
template <class K>
inline cudaError_t allow_smem(K* kernel, size_t most) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(most));
}

// Grow-only device buffer owned by a context.
struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
};

}  // namespace bmlp

struct bmlp_ctx {
    int device = 0;
    int sm_count = 0;
    int clock_khz = 0;           // SM clock rate, read once (the query takes hundreds of microseconds)
    char err[512] = {0};
    bmlp::DevBuf ws[48];
    void* batch = nullptr;       // cached grouped-batch graph (batch.cu)
    int tune[32];                // autotuned engine per size bucket (-1 = unknown)
    int* d_ctl = nullptr;        // device control words (see CTL_* below)
    int* h_ctl = nullptr;        // pinned host mirror
    cudaEvent_t ev[2] = {nullptr, nullptr};
    cudaEvent_t ev_insert = nullptr;  // after the last insertion's use of its workspaces, whatever its stream
    bmlp_stats stats{};
    void* encode_fn = nullptr;   // cuTensorMapEncodeTiled from the driver
    double t_call = 0.0;         // host time at the start of the current call (s)
    uint64_t budget_ns = 0;      // time budget of the current call (0 = none)
    void* dispatch = nullptr;    // learned dispatcher state (dispatch.cu)
};

namespace bmlp {

// CTL_QCOUNT, CTL_T0, CTL_ISSUED and CTL_BITS are 64-bit words, CTL_COST and CTL_PSTAT (the ones and nonzero words
// a bit-row squaring wrote) two of them and CTL_THIN eight (two ints each, 8-byte aligned); CTL_STEP the changed flags of up to eight
// squarings issued together; CTL_SAMPLE the ones of sampled rows. A read of the control words ends before CTL_SAMPLE
// unless the sample is wanted.
constexpr int kThinSampleRows = 256;
enum CtlWord : int {
    CTL_CHANGED = 0, CTL_ERROR = 1, CTL_OPEN = 2, CTL_LEVELS = 3, CTL_QCOUNT = 4, CTL_T0 = 6, CTL_BUDGET = 8,
    CTL_ISSUED = 10, CTL_COST = 12, CTL_THIN = 16, CTL_BITS = 34, CTL_PSTAT = 36, CTL_STEP = 40,
    CTL_SAMPLE = 48, CTL_WORDS = 48 + kThinSampleRows
};
// The pinned host mirror has two more ints: CTL_HOST_I64 is a 64-bit slot for values read from elsewhere.
constexpr int CTL_HOST_I64 = CTL_WORDS;
constexpr int CTL_HOST_WORDS = CTL_WORDS + 2;

// Degrees, roots and rows of the tiled frontiers (frontier.cu).
constexpr int WS_TILE_PREP = 41;
// Bit rows and the barrier of the one-launch closures (small.cu).
constexpr int WS_SMALL = 40;
// Workspace slots of the grouped batch and of its device-driven large problems (the others are private to api.cu).
constexpr int WS_BATCH = 15;
constexpr int WS_SOLO = 25;

// ---- grouped batch (batch.cu)
// Problems with n >= solo_n (0: none) that may use the tensor cores run as device-driven single-problem pipelines
// (bit-row squarings, then 4-bit tensor-core squarings) inside the same graph; the rest are grouped.
bmlp_status batch_run_impl(bmlp_ctx* ctx, const bmlp_problem* probs, int64_t count, int variant, long long wait_cycles,
                           int32_t* iters_out, cudaStream_t s, int64_t solo_n = 0);
// The step-cost model of the bit-row squarings (api.cu): seconds of a step from its word ORs, and of a dense 4-bit
// tensor-core product of n_pad.
double bitrow_s_per_word();
double bitrow_row_s_per_word();
double bitrow_step_s();
double tc4_product_s(int64_t n_pad);
// Synchronise s on behalf of the current call (counted in bmlp_stats.host_syncs).
cudaError_t host_sync(bmlp_ctx* ctx, cudaStream_t s);
void batch_cache_free(bmlp_ctx* ctx);

// ---- learned dispatcher (dispatch.cu)
bmlp_status dispatch_features_packed(bmlp_ctx* ctx, const uint64_t* P, int64_t n, int64_t ldw, float* feat_host,
                                     cudaStream_t s);
// features and prediction on the device, one host wait: *choice = the predicted fastest bmlp_variant
bmlp_status dispatch_choose_many_packed(bmlp_ctx* ctx, const uint64_t* const* P, const int64_t* n, const int64_t* ldw,
                                        int64_t m, float* feat_host, int32_t* choice, cudaStream_t s);
bmlp_status dispatch_choose_packed(bmlp_ctx* ctx, const uint64_t* P, int64_t n, int64_t ldw, int32_t* choice,
                                   cudaStream_t s);
bool dispatch_trained(const bmlp_ctx* ctx);
bmlp_status dispatch_predict(bmlp_ctx* ctx, const float* feats, int64_t m, float* pred, int32_t* choice,
                             cudaStream_t s);
bmlp_status dispatch_set_params(bmlp_ctx* ctx, const float* params, const float* mu, const float* sig);
bmlp_status dispatch_get_params(bmlp_ctx* ctx, float* params, float* mu, float* sig);
bmlp_status dispatch_loss_grad(bmlp_ctx* ctx, const float* X, const float* Y, const uint8_t* C, int64_t m, float* loss,
                               float* grad);
bmlp_status dispatch_train(bmlp_ctx* ctx, const float* X, const float* Y, const uint8_t* C, int64_t m,
                           const bmlp_train_cfg* cfg, float* final_loss);
bmlp_status dispatch_save(bmlp_ctx* ctx, const char* path);
bmlp_status dispatch_load(bmlp_ctx* ctx, const char* path);
void dispatch_free(bmlp_ctx* ctx);

// ---- workspace / error helpers (api.cu)
bmlp_status set_err(bmlp_ctx* ctx, bmlp_status st, const char* fmt, ...);
bmlp_status cuda_err(bmlp_ctx* ctx, cudaError_t e, const char* what);
bmlp_status ws_get(bmlp_ctx* ctx, int slot, size_t bytes, void** out);

// ---- encoders / decoders (encode.cu). All launched on `s`.
// u8 (any nonzero = 1) n x n, ld = n  ->  E4M3 0/1 R and R^T, n_pad x n_pad
void launch_u8_to_e4m3(const uint8_t* in, int64_t n, uint8_t* R, uint8_t* RT, int64_t n_pad, cudaStream_t s);
// packed rows (ldw_in words) -> E4M3 R and R^T (RT may be null)
void launch_packed_to_e4m3(const uint64_t* in, int64_t ldw_in, int64_t rows, int64_t n, uint8_t* R, uint8_t* RT,
                           int64_t n_pad, int64_t rows_pad, cudaStream_t s);
// E4M3 / 0-1 bytes (ld) -> u8 n x n (diagonal forced to 1 when reflexive)
void launch_bytes_to_u8(const uint8_t* R, int64_t ld, int64_t n, uint8_t* out, int reflexive, cudaStream_t s);
// E4M3 / 0-1 bytes (ld) -> packed rows (ldw_out words), rows x n
void launch_bytes_to_packed(const uint8_t* R, int64_t ld, int64_t rows, int64_t n, uint64_t* out, int64_t ldw_out,
                            int reflexive, cudaStream_t s);
// u8 n x n -> packed rows
void launch_u8_to_packed(const uint8_t* in, int64_t n, uint64_t* out, int64_t ldw_out, cudaStream_t s);
// packed (ldw_in) -> packed (ldw_out), masking bits >= n, optional diagonal
void launch_packed_copy(const uint64_t* in, int64_t ldw_in, int64_t rows, int64_t n, uint64_t* out, int64_t ldw_out,
                        int reflexive, cudaStream_t s);
// packed -> u8 n x n
void launch_packed_to_u8(const uint64_t* in, int64_t ldw, int64_t n, uint8_t* out, int reflexive, cudaStream_t s);
// out rows |= src rows (bits < n)
void launch_packed_or(uint64_t* out, int64_t ldw_out, const uint64_t* src, int64_t ldw_src, int64_t rows, int64_t n,
                      cudaStream_t s);
// identity as packed rows: row i has only bit i
void launch_identity_packed(uint64_t* out, int64_t ldw, int64_t n, cudaStream_t s);
// caller matrix (u8 n x n or packed n x ceil(n/64)) -> packed E2M1 R and R^T (n_pad x n_pad / 2 bytes)
void launch_u8_to_e2m1(const uint8_t* in, int64_t n, uint8_t* R, uint8_t* RT, int64_t n_pad, cudaStream_t s);
void launch_packed_to_e2m1(const uint64_t* in, int64_t ldw_in, int64_t n, uint8_t* R, uint8_t* RT, int64_t n_pad,
                           cudaStream_t s);
// packed E2M1 rows (ld4 bytes) -> u8 n x n / packed rows of ldw_out words (+ I if reflexive)
void launch_e2m1_to_packed(const uint8_t* Q, int64_t ld4, int64_t n, uint64_t* out, int64_t ldw_out, int reflexive,
                           cudaStream_t s);
// 1 per nonzero 128 x 128 block of an n x n matrix (fmt u8 with rows of n bytes, or packed with rows of
// ldw_in words), n_pad / 128 blocks a side
void launch_input_block_flags(const void* in, int32_t fmt, int64_t ldw_in, int64_t n, int64_t n_pad, uint8_t* flags,
                              int64_t flags_ld, cudaStream_t s);
// out = rows x cols AND NOT in over n x n packed rows (null vector = all constants)
void launch_packed_negate(const uint64_t* in, int64_t ldw_in, int64_t n, const uint64_t* rows, const uint64_t* cols,
                          uint64_t* out, int64_t ldw_out, cudaStream_t s);
// the union of two n x n matrices (packed rows of ceil(n / 64) words, or bytes) into out, and NEG on bytes (as
// launch_packed_negate); out may be an input
void launch_packed_union(const uint64_t* A, const uint64_t* B, int64_t n, uint64_t* out, cudaStream_t s);
void launch_u8_union(const uint8_t* A, const uint8_t* B, int64_t n, uint8_t* out, cudaStream_t s);
void launch_u8_negate(const uint8_t* in, int64_t n, const uint64_t* rows, const uint64_t* cols, uint8_t* out,
                      cudaStream_t s);
// E4M3 bytes -> 0 / 1 in place (0x00 and 0x80 are zero, any other byte one), and 0 / 1 -> E4M3 0x00 / 0x38
void launch_e4m3_bytes_to_01(uint8_t* p, int64_t bytes, cudaStream_t s);
void launch_01_to_e4m3_bytes(uint8_t* p, int64_t bytes, cudaStream_t s);
// set the diagonal of an n x n byte matrix (ld) to E4M3 one
void launch_set_diag_e4m3(uint8_t* R, int64_t ld, int64_t n, cudaStream_t s);
void launch_set_diag_e2m1(uint8_t* Q, int64_t ld4, int64_t n, cudaStream_t s);
// per (M block, K block) nonzero flags of a byte matrix rows_pad x n_pad
// (row stride of flags: flags_ld, default n_pad / 128)
void launch_block_flags(const uint8_t* A, int64_t ld, int64_t rows_pad, int64_t n_pad, uint8_t* flags,
                        cudaStream_t s, int64_t flags_ld = 0);

// ---- tensor-core product (tc_product.cu)
// Set up tensor maps for A (rows x K) and B^T (cols x K) byte matrices.
bmlp_status make_tmap(bmlp_ctx* ctx, CUtensorMap* map, const void* base, int64_t rows, int64_t cols_bytes,
                      int64_t ld, int box_rows);
int tc_smem_bytes();
cudaError_t launch_tc_product(const CUtensorMap& a, const CUtensorMap& b, const TcParams& p, int grid,
                              cudaStream_t s);
// squaring step (RMS mode only) on packed E2M1 operands (n_pad x n_pad / 2 bytes, p.ld = n_pad / 2,
// p.k_blocks = n_pad / 256) as M = 256 MMAs per CTA pair (tcgen05 .cta_group::2, 2-CTA clusters) on pair tiles
// of 256 rows x 480 columns, or 256 columns for small n_pad (p.n_tiles = tc4_tiles(n_pad, sms)); maps over R (A, box 128 rows)
// and R^T (b0: box 128 rows; b1: box tc4_b1_rows() rows), 128 bytes wide. p.issued counts 128 x 32 x 128
// multiply-add units.
int tc4_tiles(int64_t n_pad, int sms);
int tc4_b1_rows();
// the same squaring step on E4M3 operands (n_pad x n_pad bytes, p.ld = n_pad, p.k_blocks = n_pad / 128) as
// kind::f8f6f4 M = 256 MMAs per CTA pair on pair tiles of 256 x tc8_tile_n() (p.n_tiles = ceil(n_pad / that));
// no block maps (p.fmap must be null): A box 128 rows, b_half box 128 rows of R^T
int tc8_tile_n();
cudaError_t launch_tc8_product_duo(const CUtensorMap& a, const CUtensorMap& b_half, const TcParams& p, int sms,
                                   cudaStream_t s);
cudaError_t launch_tc4_product_duo(const CUtensorMap& a, const CUtensorMap& b0, const CUtensorMap& b1,
                                   const TcParams& p, int sms, cudaStream_t s);
// E4M3 bytes <-> packed E2M1 nibbles (sizes multiples of 16 bytes)
void launch_e4m3_to_e2m1(const uint8_t* in, uint8_t* out, int64_t bytes_in, cudaStream_t s);
void launch_e2m1_to_e4m3(const uint8_t* in, uint8_t* out, int64_t bytes_out, cudaStream_t s);
// grouped form: tc_group_kernel(const GroupProblem*, const GroupState*, int nprob, int phase, int* error,
// long long wait_cycles); phase 0 = squaring step of every active problem, 1 = final products of compositions
void* tc_group_kernel_ptr();
cudaError_t prepare_tc_group();

// ---- packed kernels (packed.cu)
// dst_i = (or_a ? A_i : 0) | OR_{k : A_ik = 1} B_k over n packed rows of ldw
// words (ldw even, matrices 16-byte aligned: rows move as 128-bit words; bits
// of A at columns >= n zero); raises *changed when dst_i != A_i. With A = B and or_a = 1 this is
// one squaring step R <- R + R R. tables: the Four Russians form (shared-memory
// tables of 4-row ORs; its time does not depend on the bits per word), else one
// warp per row gathering the named rows of B (time in proportion to the ones
// of A). pstat (or nullptr): the ones and the nonzero words of dst are added
// into pstat[0] and pstat[1].
cudaError_t launch_product_packed(const uint64_t* A, const uint64_t* B, uint64_t* dst, int64_t n, int64_t ldw,
                                  int or_a, int* changed, int sms, cudaStream_t s,
                                  Deadline dl = Deadline{0, nullptr, nullptr}, unsigned long long* pstat = nullptr,
                                  bool tables = true);
// Word index of n packed rows: row i's nonzero words are entries ptr[2 i] .. ptr[2 i + 1] - 1 (word index and value, in
// increasing order; the rows' ranges lie in any order), ptr[2 n] = the entries in all, ptr[2 n + 1] = the
// largest row's. ptr holds 2 n + 2 words (16-byte aligned), idx and val n * ldw entries (the dense worst case).
struct WordIndex {
    int64_t* ptr;
    int32_t* idx;
    uint64_t* val;
};
cudaError_t launch_wcsr_build(const uint64_t* P, int64_t n, int64_t ldw, const WordIndex& x, cudaStream_t s);
// Query rows that another form has begun (launch_smp_rows): of row r, words + 3 r ceil(n / 64) holds its frontier, the
// constants it has reached and its source, ceil(n / 64) words each; levels[r] the levels done, or 0 when it is finished.
struct RowState {
    uint64_t* words;
    int* levels;
};
cudaError_t launch_smp_packed(const WordIndex& x, const WordIndex& T, int64_t n, int64_t ldw, const uint64_t* src,
                              int64_t ldw_src, int64_t q, uint64_t* out, int64_t ldw_out, int* levels, int* qcounter,
                              int reflexive, int sms, cudaStream_t s, Deadline dl, RowState from = RowState{nullptr, nullptr});
// C = P | A B on packed rows through the word indexes of A and B (A = B = P: a squaring step); *changed (or null) is
// raised when C != P
cudaError_t launch_indexed_rows(const WordIndex& A, const WordIndex& B, const uint64_t* P, int64_t n, int64_t ldw,
                                uint64_t* C, int sms, cudaStream_t s, int* changed = nullptr);
// Full closure rows by 64-source bit-sliced frontier expansion over the word index of R^T (rows 0 .. n-1 of out,
// ldw_out words each). scratch: smp_sliced_grid(n, sms) x 3 n words; *bcounter = 0 and *levels = 0 beforehand.
int64_t smp_sliced_grid(int64_t n, int sms);
cudaError_t launch_smp_sliced(const WordIndex& T, int64_t n, uint64_t* scratch, uint64_t* out, int64_t ldw_out, unsigned long long* bcounter,
                              int* levels, int max_levels, int sms, cudaStream_t s, Deadline dl);
// The same expansion with the whole frontier of a batch in one SM's shared memory (frontier.cu; n <= 65,536): the rows
// of src (ld_src words each), or of every constant when src is null, into out (ld_out words each), OR-ed with the source
// row when reflexive. x: the word index of R, ones: its ones. In two parts, between which the host reads the counts:
// launch_smp_tile_prep (prep: smp_tile_prep_bytes) counts the constants that something reaches (counts[0] = n1) and the
// rows to expand (counts[1]; with `derive` those that do not follow from another row, else n). launch_smp_tiles expands
// `rows` rows (q, or counts[1]), smp_tile_width(n1, rows) of them in a batch (0: n1 is too large; scratch:
// smp_tile_bytes), and forms the derived ones. *counter = 0 and *levels = 0 beforehand; *levels receives the largest level
// count. If counts[2] is then larger than *levels, a second call with `again` (same arguments) makes *levels exact.
// counts[3] is the largest in-degree.
size_t smp_tile_prep_bytes(int64_t n);
cudaError_t launch_smp_tile_prep(const WordIndex& x, int64_t n, void* prep, int* counts, bool derive, int sms, cudaStream_t s);
int smp_tile_width(int64_t n1, int64_t rows, int sms);
size_t smp_tile_bytes(int64_t n, int64_t n1, int64_t ones, int width, int sms);
cudaError_t launch_smp_tiles(const WordIndex& x, int64_t n, int64_t n1, int64_t ones, const uint64_t* src, int64_t ld_src,
                             int64_t rows, uint64_t* out, int64_t ld_out, int reflexive, int width, void* prep, void* scratch,
                             bool derive, bool again, int* counts, unsigned long long* counter, int* levels, int max_levels,
                             int sms, cudaStream_t s, Deadline dl);
// The expansion of a few query rows straight from R's packed rows (ld_r words, bits at columns >= n ignored), one cluster
// of plan.ctas CTAs per row: 16, 8, 4 or 2, or 0 when q rows do not fit the GPU at once (or are more than kRowsMaxQueries) or
// n is too large. Results and levels as launch_smp_tiles, but for rows that stop (only with plan.may_stop and a `state`, and
// *stopped is raised then): launch_smp_packed finishes those from the state, or a second launch from their sources in it
// (src = words + 2 ceil(n / 64), ld_src = 3 ceil(n / 64), state {null, levels}), which leaves the others' results as they are.
constexpr int64_t kRowsMaxQueries = 63;
struct RowQueryPlan {
    int ctas;
    bool may_stop;
    int most;         // constants that a row reaches before it stops because reading their rows costs too much
    int first_level;  // levels after which it may stop because more of them would
    // what a level and a constant's row cost more than over word indexes, and what a row that stops has to gain (seconds)
    float level_gain, row_gain, need;
#ifdef __CUDACC__
    // Whether a row that has reached `visited` of n constants after lv levels, `found` of them in the last one, has too many
    // levels before it. Two kinds are told from the rows that end soon or fill up (visited ~ levels^alpha so far): a front that
    // goes on widening like a grid's (alpha about 2), and after 96 levels a thin one that does not widen, a path, which is
    // taken to go on for up to twice as long again. Either is taken to reach all constants, whose rows are cheap here.
    __device__ __forceinline__ bool too_deep(int64_t n, int lv, int found, int visited) const {
        if (lv < first_level || found == 0) return false;
        const float l = static_cast<float>(lv), v = static_cast<float>(visited), left = static_cast<float>(n) / v;
        const float alpha = fmaxf(1.0f, static_cast<float>(found) * l / v);
        float more;
        if (alpha >= 1.5f) {
            if (alpha > 4.5f || 2 * found < lv) return false;
            more = l * (exp2f(log2f(left) / alpha) - 1.0f);
        } else {
            if (lv < 96 || found > 8) return false;
            more = l * fminf(2.0f, left - 1.0f);
        }
        return more * level_gain + (static_cast<float>(n) - v) * row_gain >= need;
    }
#endif
};
RowQueryPlan smp_rows_plan(int64_t n, int64_t q);
cudaError_t launch_smp_rows(const uint64_t* R, int64_t ld_r, int64_t n, const uint64_t* src, int64_t ld_src, int64_t q,
                            uint64_t* out, int64_t ld_out, int reflexive, int* levels, int max_levels, const RowQueryPlan& plan,
                            RowState state, int* stopped, cudaStream_t s, Deadline dl);
// ---- a squaring restricted to the rows and columns that still hold zeros (thin.cu)
// P, PT: bit rows (n_pad rows of ldw = n_pad / 64 words) of a matrix S with R <= S <= R' = R + R R and of S^T; Src, SrcT:
// those of R and R^T (the same arrays when S = R). All are written by the squaring kernel's epilogue.
// launch_thin_sample: over `rows` rows of P spread over its n rows, stat[0] = the most ones of one with
// at least n / 2, stat[1] = the most zeros of such a row (both zero beforehand), ones (or null) = the ones of each.
// launch_thin_stats: B = the columns with fewer than n / 2 ones in S, or with at most kThinCap in R and a zero in S (Bmask,
// blist), Rb = the rows with a zero outside B (rlist), Smask the rows of Rb with at most kThinCap ones in R; stat[0..5] = |B|, |Rb|, and, with at most kThinCap counted
// of each, the ones of R in B's columns and in Rb's rows, the most of one column of B and of one row of Rb.
// launch_thin_squaring: R' on those columns and rows; the new ones are ORed into P, PT and, where Q is not null, into S
// and S^T as E2M1 (Q, QT), *changed raised when there are any. An entry with more than kThinCap ones stops once the zeros
// that it is there for are filled, at the latest after kThinCap named rows, and raises *incomplete when it stops with
// some open: S then holds some of R' only, or, with all_or_none, is as it was. The counts are read on the device;
// `entries` (their sum, or a bound) sizes the grids, T: that many rows of ldw words of scratch.
constexpr int kThinCap = 512;
struct ThinLists {
    uint64_t* Bmask;   // ldw words
    uint64_t* Smask;   // ldw words
    int32_t* colcnt;   // n
    int32_t* srccnt;   // n
    int32_t* blist;    // n
    int32_t* rlist;    // n
};
size_t thin_aux_bytes(int64_t n, int64_t ldw);
ThinLists thin_lists(void* aux, int64_t n, int64_t ldw);
cudaError_t launch_thin_sample(const uint64_t* P, int64_t ldw, int64_t n, int rows, unsigned long long* stat, int* ones,
                               cudaStream_t s);
cudaError_t launch_thin_stats(int64_t n, const uint64_t* P, const uint64_t* PT, const uint64_t* Src, const uint64_t* SrcT,
                              int64_t ldw, const ThinLists& t, unsigned long long* stat, int sms, cudaStream_t s);
cudaError_t launch_thin_squaring(int64_t n, uint64_t* P, uint64_t* PT, const uint64_t* Src, const uint64_t* SrcT,
                                 int64_t ldw, const ThinLists& t, const unsigned long long* stat, int64_t entries,
                                 uint64_t* T, uint8_t* Q, uint8_t* QT, int64_t ld4, int* changed, int* incomplete,
                                 bool all_or_none, int sms, cudaStream_t s);
// Seconds of the row ORs of such a squaring (api.cu): per word in all, and per one of its largest entry.
double thin_word_s();
double thin_one_s();
double thin_fixed_seconds(int64_t n_pad);
bool thin_is_enabled();
int thin_sample_rows();
double thin_row_spread();
// nonzero words of R + R R (out[0] += their total) and the word ORs of that squaring (out[1] += their total), from
// the word index of R (ldw words per row, at most 49,152), without forming R + R R; bits_out (if not null) += the
// ones of R
cudaError_t launch_square_growth(const WordIndex& x, int64_t n, int64_t ldw, unsigned long long* out, int sms, cudaStream_t s,
                                 unsigned long long* bits_out = nullptr);
// R^T's bit rows (n x ldw words) from R's word index: cleared, then every set bit (i, j) of R sets bit i of row j
// by a 64-bit atomic OR. Work in proportion to the ones of R, against n x ldw words read and written by
// launch_bit_transpose.
cudaError_t launch_scatter_transpose(const WordIndex& x, int64_t n, int64_t ldw, uint64_t* out, int sms, cudaStream_t s);
// word ORs of launch_indexed_rows (sum over the set bits k of a row of A of the nonzero words of row k of B):
// cost[0] += their total over all rows, cost[1] = max(cost[1], the largest row's)
cudaError_t launch_indexed_cost(const WordIndex& A, const WordIndex& B, int64_t n, unsigned long long* cost, int sms,
                                cudaStream_t s);
// (R+ + {(u, v)})+ in place on a transitive R+ (n packed rows of ldw words)
cudaError_t launch_insert_fact(uint64_t* P, int64_t n, int64_t ldw, int64_t u, int64_t v, int sms, cudaStream_t s);
// The same for m <= kInsertChunk facts at once (pairs: m x 2 constants in device memory, checked by the caller) through
// insert_chunk_words(ldw) words of scratch.
constexpr int kInsertChunk = 1024;
int64_t insert_chunk_words(int64_t ldw);
cudaError_t launch_insert_chunk(uint64_t* P, int64_t n, int64_t ldw, const int32_t* pairs, int m, uint64_t* scratch,
                                int sms, cudaStream_t s);
// out = in^T on n x n packed rows of ldw words (every word of out written, padding words with zeros)
// ---- small relations (small.cu): closure of `in`, or with r1 the composition (I + in+) r1, in one cooperative launch.
// *arrived must be zero; result[0] = products, result[1] = 1 if the last of max_iters still changed R (a composition is then not written).
constexpr int64_t kSmallN = 1024;
size_t small_closure_bytes(int64_t n);
cudaError_t launch_small_closure(const void* in, const void* r1, void* out, int64_t n, bool bytes, int reflexive,
                                 int max_iters, void* scratch, unsigned* arrived, int* result, int* error,
                                 long long wait_cycles, int sms, cudaStream_t s);
// *ones += the ones of `words` 64-bit words (16-byte aligned, an even number).
cudaError_t launch_packed_ones(const uint64_t* P, int64_t words, unsigned long long* ones, int sms, cudaStream_t s);
cudaError_t launch_bit_transpose(const uint64_t* in, uint64_t* out, int64_t n, int64_t ldw, cudaStream_t s);
int smp_packed_max_words();
// One closure by frontier expansion inside a grouped batch (device copy): every row of R1+ as one query row.
struct FrontierJob {
    const uint64_t* P;     // R as packed rows (n x ldw words, padding bits and words zero)
    uint64_t* PT;          // R^T, written by the launch
    int64_t* wptr;         // word index of R (as WordIndex)
    int32_t* widx;
    uint64_t* wval;
    int64_t* wptrT;        // word index of R^T
    int32_t* widxT;
    uint64_t* wvalT;
    uint64_t* out;         // the closure rows (n x ldw words)
    int64_t n, ldw;        // ldw even
    int64_t first;         // first row of this job in the launch's row numbering (jobs in increasing order)
    int* levels;           // receives the deepest level + 1 (atomicMax; cleared by the caller)
};
// Transposes, word indexes and the frontier expansion of every row of every job (device array `jobs`,
// `total` rows in all; max_n / max_ldw over the jobs; *counter is cleared by the launch).
cudaError_t launch_frontier_group(const FrontierJob* jobs, int njobs, int64_t max_n, int64_t max_ldw, int64_t total,
                                  unsigned long long* counter, int sms, cudaStream_t s);

}  // namespace bmlp
