// Internal declarations shared by the host API and the kernels of the codec library.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <utility>
#include <vector>

#include "tc.h"

constexpr int TC_TILE_PIXELS = 128;   // pixels per tile = threads per epilogue group
constexpr int TC_MAX_C = 1024;
constexpr int TC_MAX_CODE_LEN = 12;
constexpr int kMaxRoundtripChunks = 64;   // longest code the decode lookup table covers

constexpr int kManyStreams = 8;               // streams that a list of tensors is spread over
constexpr int kCanonWords = 12;               // words per table of a canonical code's bounds (6) and bases (6)

// Device status word: first error wins.
__device__ __forceinline__ void tc_dev_set_status(unsigned int *status, unsigned int code)
{
    atomicCAS(status, 0u, code);
}

struct tc_ctx {
    int device = 0;
    int sm_count = 0;
    int max_smem_optin = 0;
    unsigned int *d_status = nullptr;     // device status word
    void *scratch = nullptr;              // look-back state, ticket counter
    // Look-back state of the resident-basis encoder: two arrays in turn, each call clearing what the call before left in the other.
    unsigned long long *lookback[2] = {};
    long long lookback_words[2] = {};     // of each, from its start, that may not be zero
    int lookback_next = 0;
    bool lookback_ready = false;          // both have been zeroed once
    size_t scratch_bytes = 0;
    void *host_arena = nullptr;           // device staging of tc_roundtrip_host (grown on demand)
    size_t host_arena_bytes = 0;
    // tc_roundtrip_host works through the batch in chunks, two in flight: copy-in and copy-out
    // streams beside the caller's, events that hand a chunk from one to the next, and a small
    // pinned array for the chunks' stream lengths (created at first use)
    cudaStream_t copy_in = nullptr, copy_out = nullptr;
    cudaEvent_t ev_in[2] = {nullptr, nullptr}, ev_done[2] = {nullptr, nullptr}, ev_out[2] = {nullptr, nullptr};
    unsigned long long *chunk_bits = nullptr;   // pinned HOST [kMaxRoundtripChunks]
    // tc_encode_many / tc_decode_many spread their items over these streams (created at first use)
    cudaStream_t many_streams[kManyStreams] = {};
    cudaEvent_t many_fork = nullptr, many_join[kManyStreams] = {};
    int force_exact = 0;                  // 1: route every tensor through the fp64 kernels; 2: skip the resident-basis kernels; 3: skip the run-skipping decoder
    bool no_workspace = false;            // calls run as if no memory could be had for their workspaces
    bool force_jacobi = false;            // the eigensolver for devices that cannot hold the clusters
    int last_encode_path = 0;             // 0 = fp64 kernels, 1 = tensor-core kernels (resident basis), 2 = fp32 kernels, 3 = tensor-core kernels (streamed basis)
    int last_decode_path = 0;
    bool last_decode_runs = false;        // path 1 by the run-skipping decoder
    tc_codebook *stats_cb[9] = {};        // tc_stats: fixed-length code tables (one per bit width) for streams coded without a codebook
};

struct tc_model {
    int c = 0, k = 0, bits = 0, basis_dtype = 0;
    double lo = 0, step = 0;
    double basis_scale = 1.0;               // 8-bit basis: entries are integers times this; 1 otherwise
    int center = 0;                         // symbol whose level is nearest to y = 0
    // host copies; a model fitted on the device holds its basis there only, and `basis` is filled
    // from d_basis64 the first time the host needs it (export, folding)
    mutable std::vector<double> basis;      // [c][c], or empty
    std::vector<double> mean, eig;          // [c]
    std::vector<float> blk_bits, blk_odd;   // [(k + 15) / 16]  see finish_model
    float max_bias = 0.f;                   // no |d_enc_bias| is larger, as a fraction of the quantiser's range
    int device = 0;
    // device copies, all but the first two (of a fitted model: owns64) inside one allocation
    void *d_block = nullptr;
    bool owns64 = true;
    double *d_basis64 = nullptr;            // [c][c] exact values of the (rounded) basis
    double *d_mean64 = nullptr;             // [c]
    __nv_bfloat16 *d_basis_bf16 = nullptr;  // [k][c]   bf16 basis, or the integers of an 8-bit basis (exact in bf16)
    __nv_bfloat16 *d_basis_core = nullptr;  // the same in the MMA's shared-memory order (8 x 8 core matrices); layers of up to 256 channels
    __nv_bfloat16 *d_basis_t_bf16 = nullptr;// [c][k]   transpose, for the inverse projection
    float *d_enc_bias = nullptr;            // [k]  -(T mu + lo)_j / step
    float *d_dec_bias = nullptr;            // [c]  mu_c + (lo + center*step) * sum_j T[j][c]
    float *d_tmu32 = nullptr;               // [k]  (T mu)_j
    CUtensorMap basis_map;                  // d_basis_bf16 as a [k][c] tensor, boxes of 256 rows x 32 channels, 64-byte swizzle
    bool has_basis_map = false;
    CUtensorMap basis_t_map;                // d_basis_t_bf16 as a [c][k] tensor, boxes of 128 channel rows x 64 coefficients, 128-byte swizzle
    bool has_basis_t_map = false;
};

struct tc_codebook {
    int bits = 0, groups = 0, max_len = 0, lut_bits = 0;
    int modal = -1;                         // per-layer table: the symbol coded by the single bit 0 (-1: none)
    float mean_bits = 0.f;                  // bits per symbol: of the counts it was built from, else for symbols of probability 2^-length
                                            // (from 2.5 bits on within 10 % of the coded layers' rate)
    std::vector<uint8_t> lengths;           // host [groups][2^bits]
    int device = 0;
    void *d_block = nullptr;                // one allocation that holds the arrays below
    uint32_t *d_enc = nullptr;              // [groups][2^bits]  (code << 8) | length
    uint16_t *d_lut = nullptr;              // [groups][2^lut_bits]  (symbol << 8) | length
    uint32_t *d_lut32 = nullptr;            // [groups][2^lut_bits]  bf16(symbol) << 16 | symbol << 8 | length
    uint32_t *d_canon = nullptr;            // [groups][kCanonWords]  bounds and bases of the canonical code (tcdev::canon_length)
    uint8_t *d_sorted = nullptr;            // [groups][2^bits]  symbols in the order of their codes
};

// ---- kernel argument blocks -------------------------------------------------------------

struct EncodeArgs {
    const void *x;
    int n, c, hw, k, bits, groups;
    long long pixels;
    long long n_tiles;
    int chunk_pixels;
    int splits;                 // chunks per pixel (1, 2 or 4; more than 1 only with chunk_pixels == 1)
    const double *basis64;      // [c][c]
    const double *mean64;       // [c]
    const __nv_bfloat16 *basis_bf16;   // [k][c]  (tensor-core path)
    const __nv_bfloat16 *basis_core;   // basis_bf16 in 8 x 8 core matrices, or null
    const CUtensorMap *basis_map;      // HOST pointer to the model's tensor map of basis_bf16, or null
    const float *enc_bias;      // [k]  -(T mu + lo)_j / step
    const float *tmu32;         // [k]  (T mu)_j
    double lo, step;
    double basis_scale;         // basis_bf16 holds basis / basis_scale (8-bit basis: integers); 1 otherwise
    const uint32_t *enc;        // [groups][2^bits]
    uint32_t *stream;           // output words
    unsigned long long capacity_bits;
    uint16_t *chunk_len;        // bits of every chunk
    unsigned long long *tile_off;
    float *dbg_coef;            // nullable
    uint8_t *dbg_sym;           // nullable
    unsigned long long *tile_state;   // look-back state, zeroed before launch
    unsigned int *ticket;             // zeroed before launch; the look-back words follow it
    bool alone;                       // no other stream of this call (see launch_chained)
    int epilogue_groups;              // resident-basis encoder: 2 or 4 a block, as a list has it; 0: by the tensor's tiles
    int sms;                          // SMs that a persistent kernel of its own takes at most in a list
    long long clear_words;            // 64-bit words from `ticket` on that the first of several kernels zeroes (0: they are zero)
    unsigned long long *other_state;  // resident-basis encoder: look-back state that no tile of this call uses,
    long long other_words;            // and how many words of it to zero for the next
    unsigned int *status;
    unsigned long long *clamped;      // nullable: counts coefficients outside the range
    int emit;                         // 0: symbols only (statistics mode)
    const uint8_t *sym_in;            // exact kernels: non-null = the symbols [P][K] are given, skip the projection
    unsigned long long *hist;         // tensor-core encoder, statistics: non-null = per-coefficient counts [kHistCopies][K][2^bits] of every symbol but hist_modal are added here
    int hist_modal;                   // the symbol of the zero level, which most coefficients hold: statistics mode counts all the others
    int modal;                        // per-layer table: the symbol whose code is the single bit 0, or -1 if no code has one bit
    float max_bias;                   // see tc_model
    const float *blk_bits, *blk_odd;  // HOST, per block of 16 coefficients: expected code bits, expected number of symbols that are not the zero level
};

struct DecodeArgs {
    const uint32_t *stream;
    unsigned long long stream_bits;
    const uint16_t *chunk_len;          // bits of every chunk
    int splits;                         // chunks per pixel (1, 2 or 4)
    const unsigned long long *tile_off;
    const uint8_t *symbols;     // non-null: take symbols from here instead of the stream
    uint8_t *sym_out;           // exact kernels: non-null = write the decoded symbols [P][K] there and stop
    int n, c, hw, k, bits, groups;
    long long pixels;
    long long n_tiles, n_chunks;
    int chunk_pixels;
    int lut_bits;
    const uint16_t *lut;
    const uint32_t *lut32;              // tensor-core path
    const uint32_t *canon;              // [groups][kCanonWords], see tc_codebook
    const uint8_t *sorted;              // [groups][2^bits]
    const __nv_bfloat16 *basis_t_bf16;  // [c][k]
    bool alone;                         // no other stream of this call (see launch_chained)
    int sms;                            // SMs that a persistent kernel of its own takes at most in a list
    const CUtensorMap *basis_t_map;     // HOST pointer to the model's tensor map of basis_t_bf16, or null
    const float *dec_bias;              // [c]
    int center;                         // subtracted from every symbol before the MMA
    int modal;                          // per-layer table: the symbol whose code is the single bit 0, or -1 if no code has one bit
    float code_bits;                    // bits per symbol to expect (tc_codebook::mean_bits)
    int mean_tile_bytes;                // caller's hint: mean size of a tile's stream segment, 0 = not known
    int dense_head;                     // run-skipping decoder: leading coefficients that are too often non-modal for run skipping to pay
    int relu;                           // x_hat = max(x_hat, 0) before it is rounded to the tensor type
    int smem_budget;                    // shared memory the tensor-core kernel may lay out (set by its launcher)
    int item_pixels;                    // streaming decoder: pixels per work item chosen by its launcher (0: the layout's default)
    const double *basis64;
    const double *mean64;
    double lo, step;
    double basis_scale;                 // basis_t_bf16 holds basis / basis_scale
    void *xhat;
    unsigned int *status;
};

// ---- encode dispatch shared by tc_encode and tc_encode_noalloc (tc_api.cu) --------------------
// Launch of a kernel that may be set up while the one before it in the stream still runs (`early`; it calls chain_wait): as it is for the second and
// later kernels of a call, behind kernels of this library, and by launch_first for a call's first kernel, behind anyone's.  Not with
// other streams of the call at work (`early` false): a product's blocks that wait hold shared memory their kernels could
// use (decode of a network's 16 layers 274 us, 250 without).
template <typename... P, typename... A>
inline cudaError_t launch_chained(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cfg.attrs = &attr; cfg.numAttrs = early ? 1 : 0;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
    if (err != cudaSuccess) cudaGetLastError();
    return err;
}

// The first kernel of a call, early as well: launches that wait for one another's end start at multiples of 2.05 us here, and 4.1 apart at
// least (a kernel that spins for 1 to 10 us, queued 300 times), which is a quarter of a small call's time.  The kernels ahead of it
// in the stream may be anyone's: until it has called chain_wait such a kernel reads nothing but models and codebooks, which are
// complete when the functions that make them return, and writes nothing; afterwards it reads what
// others wrote (maps, streams) not through the read-only path, whose lines may be older than the wait.  Captured calls start after all that the graph
// holds before them.  Small blocks that arrive early all pile onto the first SMs that have room (decode of 384x8x8 x 241, 121 blocks:
// 25 -> 56 us), so they ask for as much shared memory as keeps them apart (spread_bytes; more than eight an SM start in their
// turn: 64x56x56 x 64 with a table per channel, 1 568 blocks, 45 -> 56 us).
constexpr size_t kSmBytes = 228 * 1024, kBlockBytes = 1024, kSpreadMost = 118 * 1024;       // of an SM; what the system keeps of a block's
// Dynamic shared memory with which as many blocks fit an SM as it would get of `blocks` and no more, `own` bytes being static variables (0: no
// spreading).  (The static ones left out of it, seven fitted an SM that was to take eight: decode of 16x16x16 x 592 with a table per channel 28.8 ->
// 40.2 us, 64x16x16 x 592 33.4 -> 37.3.)
inline size_t spread_bytes(long long blocks, int sm_count, size_t own)
{
    const long long per_sm = (blocks + sm_count - 1) / sm_count;
    if (per_sm <= 1) return kSpreadMost;
    return per_sm <= 8 ? (kSmBytes / (size_t)(per_sm + 1) / 1024 + 1) * 1024 - kBlockBytes - own : 0;
}
// Static shared memory of a kernel that is kept apart, asked for at its first launch (`known`, of that kernel): a byte or two of another variant's let
// one block more onto an SM.
inline size_t static_bytes(std::atomic<size_t> &known, const void *kernel)
{
    size_t bytes = known.load(std::memory_order_relaxed);
    cudaFuncAttributes at;
    if (bytes == 0 && cudaFuncGetAttributes(&at, kernel) == cudaSuccess) known.store(bytes = at.sharedSizeBytes, std::memory_order_relaxed);
    else if (bytes == 0) cudaGetLastError();
    return bytes;
}
template <typename... P, typename... A>
inline cudaError_t launch_first(bool alone, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (alone && cudaStreamIsCapturing(s, &capture) != cudaSuccess) { cudaGetLastError(); alone = false; }
    return launch_chained(alone && capture == cudaStreamCaptureStatusNone, kernel, grid, block, smem, s, std::forward<A>(args)...);
}

// launch_chained, always early, in clusters of `blocks` along the grid's second dimension.
template <typename... P, typename... A>
inline cudaError_t launch_chained_cluster(int blocks, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args)
{
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = (unsigned int)blocks; attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cfg.attrs = attr; cfg.numAttrs = 2;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
    if (err != cudaSuccess) cudaGetLastError();
    return err;
}

// ---- several tensors in one launch of a persistent kernel ------------------------------------
constexpr int kListItems = 32;                // tensors of a launch (their arguments are kernel parameters)
struct ListWork {
    long long tiles;
    double tile_us;                           // what a tile takes a block, after its first
    int blocks;
};
// Deals `sms` blocks (at least one for each tensor; `sms` are no fewer) so that the slowest block is done as early as possible.
void deal_blocks(std::vector<ListWork> &work, int sms);
// Launches that `tensors` of one kernel take on `sms` SMs: tensors r, r + launches, ... go together.
int list_launches(size_t tensors, int sms);
// Deals the device to the kernels of a list that run at the same time: classes[j] share launches (tensors in descending order of
// work), `others` tensors of `others_us` us of one SM have kernels of their own.  sms[j] = SMs of a class; returns those of the others.
int deal_list(const std::vector<std::vector<ListWork>> &classes, double others_us, int others, int sm_count, std::vector<int> &sms);
extern "C" double tc_list_own_us(long long tiles, int c, int k, double bits, bool per_channel, bool tensor_cores, bool exact, bool encode);

// Tiles that a context's two look-back arrays serve: 128 KB (half a megabyte made tc_create 0.25 ms longer; a larger call's memset is
// 1 % of it).
constexpr long long kLookbackTiles = 8192;
constexpr size_t kEncodeScratchHeader = 64;   // ticket counter, padded; the per-tile look-back words follow
tc_status tc_encode_with_scratch(tc_ctx *ctx, const tc_model *m, const tc_codebook *cb, const tc_tensor *x, int chunk_pixels,
                                 int splits, void *stream_out, size_t capacity, uint16_t *chunk_len, uint64_t *tile_off,
                                 const tc_debug_out *debug, void *scratch, void *work, cudaStream_t s,
                                 unsigned long long *hist = nullptr, unsigned long long *clamped = nullptr, int list_sms = 0);
// Copies of the counts that the encoder's blocks share in statistics mode: the atomics of a leading coefficient all meet in one line of L2,
// which takes one at a time (256x14x14 x 256: 96 us with one copy, 48 with eight).
constexpr int kHistCopies = 8;
// tensors of fewer tiles than this many per SM take the one-thread-per-value exact kernels
constexpr int kExactParallelTilesPerSm = 2;

// ---- launchers (defined in the .cu files) ----------------------------------------------
tc_status tc_launch_encode_simt(const tc_ctx *ctx, const EncodeArgs &a, int dtype, cudaStream_t s);
tc_status tc_launch_decode_simt(const tc_ctx *ctx, const DecodeArgs &a, int dtype, cudaStream_t s);
tc_status tc_launch_encode_simt_fp32(const tc_ctx *ctx, const EncodeArgs &a, cudaStream_t s);
tc_status tc_launch_decode_simt_fp32(const tc_ctx *ctx, const DecodeArgs &a, cudaStream_t s);
tc_status tc_launch_project_quantise(const EncodeArgs &a, int dtype, uint8_t *sym, cudaStream_t s);
int tc_pack_symbols_parts(const EncodeArgs &a);
tc_status tc_launch_unpack_symbols(const tc_ctx *ctx, const DecodeArgs &a, uint8_t *sym, cudaStream_t s);
tc_status tc_launch_pack_symbols(const tc_ctx *ctx, const EncodeArgs &a, const uint8_t *sym, long long first_tile, long long end_tile, cudaStream_t s);
tc_status tc_launch_unpack_operand(const tc_ctx *ctx, const DecodeArgs &a, void *operand, long long first_tile, long long end_tile, cudaStream_t s);

// Wide layers with workspace (wide_gemm.cu).  The workspace of one tensor is at most about kWideWorkspace:
// larger tensors are worked through in passes.
constexpr size_t kWideWorkspace = 64ull << 20;
size_t tc_encode_wide_workspace(int c, int k, long long n_tiles);
size_t tc_decode_wide_workspace(int k, long long n_tiles);
tc_status tc_launch_encode_wide_gemm(const tc_ctx *ctx, const EncodeArgs &a, void *workspace, cudaStream_t s);
tc_status tc_launch_decode_wide_gemm(const tc_ctx *ctx, const DecodeArgs &a, void *workspace, cudaStream_t s);
// Tensor map of a bf16 matrix [rows][cols] (cols a multiple of 8): boxes of 64 columns x box_rows rows, 128-byte swizzle.
bool tc_tensor_map_sw128(CUtensorMap *map, const void *base, long long rows, int cols, int box_rows);
tc_status tc_launch_reconstruct(const DecodeArgs &a, int dtype, const uint8_t *sym, cudaStream_t s);
bool tc_encode_tc_supported(const tc_ctx *ctx, const EncodeArgs &a);
tc_status tc_launch_encode_tc(const tc_ctx *ctx, const EncodeArgs &a, cudaStream_t s);
// Kernels of a list's tensors, those with kind[i] >= 0 on entry, which tc_encode_tc_supported takes.
void tc_encode_tc_list_classes(const tc_ctx *ctx, std::vector<EncodeArgs> &args, std::vector<int> &kind);
constexpr int kEncodeClasses = 16, kEncodeFourGroups = 8;     // classes; the bit of those with four epilogue groups a block
double tc_encode_tc_tile_us(const EncodeArgs &a, int which);
tc_status tc_launch_encode_tc_list(const tc_ctx *ctx, const std::vector<EncodeArgs> &tensors, int sms, cudaStream_t s);
bool tc_decode_tc_supported(const tc_ctx *ctx, const DecodeArgs &a);
tc_status tc_launch_decode_tc(const tc_ctx *ctx, const DecodeArgs &a, cudaStream_t s);
bool tc_decode_runs_supported(const tc_ctx *ctx, const DecodeArgs &a);
tc_status tc_launch_decode_runs(const tc_ctx *ctx, const DecodeArgs &a, cudaStream_t s);
double tc_decode_runs_tile_us(const DecodeArgs &a);
tc_status tc_launch_decode_runs_list(const tc_ctx *ctx, const std::vector<DecodeArgs> &tensors, int sms, cudaStream_t s);
bool tc_encode_wide_supported(const tc_ctx *ctx, const EncodeArgs &a);
tc_status tc_launch_encode_wide(const tc_ctx *ctx, const EncodeArgs &a, cudaStream_t s);
bool tc_decode_wide_supported(const tc_ctx *ctx, const DecodeArgs &a);
tc_status tc_launch_decode_wide(const tc_ctx *ctx, const DecodeArgs &a, cudaStream_t s);
size_t tc_decode_tc_staging_bytes(const tc_ctx *ctx, const DecodeArgs &a);     // per tile
size_t tc_decode_wide_staging_bytes(const tc_ctx *ctx, const DecodeArgs &a);   // per tile

tc_status tc_launch_channel_sums(const void *x, int dtype, int n, int c, int hw, double *sums, int sm_count,
                                 cudaStream_t s);
tc_status tc_launch_mean(double *sums, int c, long long pixels, cudaStream_t s);      // in place
tc_status tc_launch_covariance(const void *x, int dtype, int n, int c, int hw, const double *mean,
                               double *cov, int sm_count, cudaStream_t s);
tc_status tc_launch_range0(const void *x, int dtype, int n, int c, int hw, const double *mean,
                           const double *row0, double *block_minmax, int *n_blocks_out,
                           cudaStream_t s);
int tc_range0_max_blocks(long long pixels);
tc_status tc_launch_fold_counts(unsigned long long *counts, int copies, int n, cudaStream_t s);
tc_status tc_launch_histogram(const uint8_t *sym, long long pixels, int k, int groups, int bits,
                              unsigned long long *hist, cudaStream_t s);
tc_status tc_launch_sqerr(const void *x, const void *xhat, int dtype, long long count,
                          double *sum_sq, unsigned long long *zeros, int sm_count, cudaStream_t s);

// ---- host algorithms (host_algos.cpp) ---------------------------------------------------
int tc_huffman_lengths_host(const uint64_t *counts, int nsym, int lmax, uint8_t *len);
void tc_canonical_codes_host(const uint8_t *len, int nsym, uint32_t *code);
int tc_eigh_host(double *a, int n, double *evals, double *evecs);

// ---- fit on the device (eigh_device.cu) ---------------------------------------------------
tc_status tc_launch_moments_to_cov(const double *sum, const double *outer, long long count, int c, double *mean, double *cov,
                                   cudaStream_t s);
tc_status tc_launch_scale_mirror(double *cov, int c, double denom, cudaStream_t s);
size_t tc_eigh_device_workspace_bytes(int c);
tc_status tc_eigh_device(const double *a, int c, double *evals, double *evecs, void *work, bool jacobi, cudaStream_t s);
tc_status tc_eigh_outcome(double outcome);
size_t tc_eigh_cluster_workspace_bytes(int n);   // eigh_cluster.cu
tc_status tc_launch_eigh_cluster(const double *a, int n, void *work, double **vt, double **lambda, int **state, cudaStream_t s);
tc_status tc_launch_round_basis(double *basis, int c, int dtype, double *scale_slot, cudaStream_t s);
tc_status tc_launch_model_consts(const double *basis, const double *mean, int c, int k, double lo, double step, double center,
                                 float *enc_bias, float *tmu32, float *dec_bias, cudaStream_t s);
tc_status tc_launch_basis_bf16(const double *basis, int c, int k, double basis_scale, bool int8, void *b, void *bt, void *bc, cudaStream_t s);
