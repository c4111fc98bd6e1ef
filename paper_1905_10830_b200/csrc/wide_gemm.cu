// Layers the resident-basis kernels do not take (more than 256 channels, or rows of H*W that are no
// multiple of four elements), with workspace: the projection (Section 3, "Linear transform") and its
// inverse as tiled matrix products of their own, the entropy coder in kernels before and after them.
//
//   encode:  pixels to rows ([P][C])  ->  Y = X T^T, quantised to symbols ([P][K] bytes)  ->  pack_symbols
//   decode:  unpack_symbols, centred bf16 ([P][K])  ->  X_hat = T^T Q + bias, NCHW
//
// A fused kernel gives a tile of 128 pixels to an SM, which then streams the whole basis (0.66 MB at
// 576 channels, 1.8 MB at 960) past it, decodes its symbols with eight warps, and has every SM
// wait for the slowest of a few tiles.  Here a work unit of the product is one block of at most 256
// coefficients (channels) of a tile, the units are dealt over all SMs, both operands arrive by
// tiled TMA copies with 128-byte swizzle, and the coder's chunks run side by side over the chip.
// The workspace traffic (2 bytes per value written and read) stays in the 126 MB L2 for the most part.
// 576x14x14 x 128: encode 132 -> 60 us, decode 108 -> 56;
// 960x7x7 x 128: encode 140 -> 48, decode 140 -> 45; 512x7x7 x 64: encode 52 -> 25, decode 46 -> 21.
// The product itself is bound by the operands' way from L2 (48 KB per 64 of the depth, at about 32 bytes a cycle
// and SM); one copy per operand and stage, since a producer thread issues one in about 100 cycles.
//
// Arithmetic as in the streaming kernels: bf16 products, fp32 accumulation over steps of 16 channels
// (coefficients) in ascending order, the same quantiser and dequantiser expressions.
#include "device_utils.cuh"
#include "sm100_ptx.cuh"

namespace {

using namespace tcdev;
using namespace sm100;

constexpr int kPanelK = 64;                                   // reduction depth of a ring stage
constexpr int kStageA = 128 * kPanelK * 2;                    // 16 KB: 128 rows of the first operand
constexpr int kMaxN = 256;                                    // columns of an accumulator
constexpr int kStageBytes = kStageA + kMaxN * kPanelK * 2;    // 48 KB
constexpr int kStages = 4;
// four epilogue warps per quarter of TMEM's lanes: with two, layers of few channels (little to multiply) took longer
// (80x27x19 x 37 decode 25.2 against 23.3 us, 16x112x112 x 128 206 against 182)
constexpr int kEpiWarps = 16, kProducerWarp = kEpiWarps, kMmaWarp = kEpiWarps + 1;
constexpr int kThreads = (kEpiWarps + 2) * 32;
constexpr int kTrWarpBytes = 2048;                            // decode: transpose block of a warp, 32 channel rows x 32 pixels
constexpr int kTmemCols = 512;
constexpr float kMagic = 12582912.0f;                         // 1.5 * 2^23: adding it rounds to the nearest integer, ties to even

struct GemmArgs {
    int n_panels, k_depth;      // reduction: panels of 64, its length
    int n_cols;                 // columns of a unit (a multiple of 32, at most 256)
    int blocks;                 // units that share the pixels of a tile
    long long units;
    long long p_first, p_end;   // pixels of this launch (row 0 of the workspace is p_first)
    // encode
    int k;
    float inv_step, vmax;
    const float *bias;          // [k] / [c]
    uint8_t *sym;               // [pixels][k]
    // decode
    int c, hw, relu;
    float step;
    __nv_bfloat16 *xhat;
    unsigned int *status;
};

// kEncode: rows of a unit = 128 pixels, columns = coefficients; else rows = 128 channels, columns = pixels.
template <bool kEncode>
__global__ void __launch_bounds__(kThreads, 1) wide_gemm_kernel(GemmArgs a, const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_full[kStages], s_empty[kStages], s_tfull[2], s_tempty[2];
    __shared__ uint32_t s_tmem_base;
    // (taken from lane 0: the compiler knows that the branches between the roles are the same for a whole warp)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t ring = smem_u32(smem);
    chain_next();
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(smem_u32(&s_full[s]), 1); mbar_init(smem_u32(&s_empty[s]), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&s_tfull[b]), 1); mbar_init(smem_u32(&s_tempty[b]), kEpiWarps); }
        mbar_fence_init();
    }
    if (warp == kMmaWarp) { tmem_alloc(smem_u32(&s_tmem_base), kTmemCols); tmem_relinquish(); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, s_tmem_base, 0);
    chain_wait();                                             // the workspace operand; earlier readers of what this kernel writes
    // rows of both operands of unit u: (tile of pixels, block)
    auto tile_of = [&](long long u) { return (int)(u / a.blocks); };
    auto block_of = [&](long long u, int tile) { return (int)(u - (long long)tile * a.blocks); };

    if (warp == kProducerWarp) {
        if (lane == 0) {
            int s = 0;
            uint32_t phase = 1;
            bool alive = true;
            for (long long u = blockIdx.x; u < a.units && alive; u += gridDim.x) {
                const int tile = tile_of(u), block = block_of(u, tile);
                const int row_a = kEncode ? tile * 128 : block * 128, row_b = kEncode ? block * a.n_cols : tile * a.n_cols;
                for (int kp = 0; kp < a.n_panels; ++kp) {
                    if (!mbar_wait(smem_u32(&s_empty[s]), phase)) { alive = false; break; }
                    const uint32_t bar = smem_u32(&s_full[s]), dst = ring + (uint32_t)s * kStageBytes;
                    mbar_arrive_expect_tx(bar, (uint32_t)(kStageA + a.n_cols * kPanelK * 2));
                    tma_load_2d(dst, &map_a, kp * kPanelK, row_a, bar);
                    tma_load_2d(dst + kStageA, &map_b, kp * kPanelK, row_b, bar);
                    if (++s == kStages) { s = 0; phase ^= 1u; }
                }
            }
            if (!alive) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
        }
    } else if (warp == kMmaWarp) {
        const uint32_t issuer = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(128, a.n_cols, false, false);
        const uint64_t desc = make_smem_desc_sw128(ring, 1024);
        const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32);
        int s = 0, n = 0;
        uint32_t phase = 0;
        bool alive = true;
        for (long long u = blockIdx.x; u < a.units && alive; u += gridDim.x, ++n) {
            const int acc = n & 1;
            if (!mbar_wait(smem_u32(&s_tempty[acc]), (uint32_t)(((n >> 1) & 1) ^ 1))) { alive = false; break; }
            tc_fence_after_sync();
            for (int kp = 0; kp < a.n_panels; ++kp) {
                if (!mbar_wait(smem_u32(&s_full[s]), phase)) { alive = false; break; }
                tc_fence_after_sync();
                const uint32_t a_lo = desc_lo + (uint32_t)s * (kStageBytes >> 4), b_lo = a_lo + (kStageA >> 4);
                const int steps = min(kPanelK, a.k_depth - kp * kPanelK) >> 4;
                auto step = [&](int q) {
                    mma_bf16_ss_guarded(tmem_base + acc * kMaxN, a_lo + 2 * q, desc_hi, b_lo + 2 * q, desc_hi, idesc, (kp | q) ? 1u : 0u, issuer);
                };
                if (steps == kPanelK / 16) {
#pragma unroll
                    for (int q = 0; q < kPanelK / 16; ++q) step(q);
                } else
                    for (int q = 0; q < steps; ++q) step(q);
                mma_commit_guarded(smem_u32(&s_empty[s]), issuer);
                if (++s == kStages) { s = 0; phase ^= 1u; }
            }
            if (alive) mma_commit_guarded(smem_u32(&s_tfull[acc]), issuer);
        }
        if (!alive && issuer) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
    } else {
        const int set = warp >> 2, wq = warp & 3;              // which part of the columns; TMEM lane quarter
        constexpr int kSets = kEpiWarps / 4, kStep = kEncode ? 16 : 32;
        const int part = (a.n_cols / kStep + kSets - 1) / kSets * kStep;
        const int col_first = set * part, cols = min(part, a.n_cols - col_first);     // none for the last sets of a narrow unit
        bool alive = true;
        int n = 0;
        for (long long u = blockIdx.x; u < a.units; u += gridDim.x, ++n) {
            const int acc = n & 1;
            if (!mbar_wait(smem_u32(&s_tfull[acc]), (uint32_t)((n >> 1) & 1))) { alive = false; break; }
            tc_fence_after_sync();
            const int tile = tile_of(u), block = block_of(u, tile);
            const uint32_t trow = tmem_base + acc * kMaxN + ((uint32_t)(wq * 32) << 16) + col_first;
            if constexpr (kEncode) {
                const long long p = a.p_first + (long long)tile * 128 + wq * 32 + lane;
                const int j_first = block * a.n_cols + col_first, j_end = min(j_first + cols, a.k);
                uint8_t *dst = a.sym + (p - a.p_first) * a.k;
#pragma unroll 1
                for (int j0 = j_first; j0 < j_end; j0 += 16) {
                    uint32_t r[16];
                    tmem_ld_32x32b_x16(trow + (j0 - j_first), r);
                    float4 b4[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) b4[i] = __ldg(reinterpret_cast<const float4 *>(a.bias + j0) + i);
                    const float *bias = reinterpret_cast<const float *>(b4);
                    tmem_ld_wait(r);
                    // level rounded to nearest even and clamped while a float (see the streaming kernel)
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        r[i] = __float_as_uint(fminf(fmaxf(fmaf(__uint_as_float(r[i]), a.inv_step, bias[i]) + kMagic, kMagic), a.vmax));
                    uint32_t w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        w[i] = __byte_perm(__byte_perm(r[4 * i], r[4 * i + 1], 0x0040), __byte_perm(r[4 * i + 2], r[4 * i + 3], 0x0040), 0x5410);
                    if (p < a.p_end) *reinterpret_cast<uint4 *>(dst + j0) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            } else {
                const int ch = block * 128 + wq * 32 + lane;
                const float bias = ch < a.c ? __ldg(a.bias + ch) : 0.f;
                const float floor_v = a.relu ? 0.f : __int_as_float((int)0xff800000u);
                const int rows = min(32, a.c - (block * 128 + wq * 32));          // channel rows of this warp that exist
                const uint32_t tb = ring + kStages * kStageBytes + (uint32_t)warp * kTrWarpBytes;
                const long long p_unit = a.p_first + (long long)tile * a.n_cols + col_first;
                const bool vec = (a.hw & 3) == 0 && ((uintptr_t)a.xhat & 7u) == 0;
                // This lane's pixels in a pass of 32: four of them with 8-byte stores (eight lanes a row, four
                // rows an instruction), else one (a row an instruction).
                const int px_lane = vec ? 4 * (lane & 7) : lane;
                long long p = p_unit + px_lane;
                long long img = p / a.hw;
                int sp = (int)(p - img * a.hw);
                const long long img_stride = (long long)a.c * a.hw;
                for (int c0 = 0; c0 < cols && rows > 0; c0 += 32, p += 32) {
                    uint32_t r[32];
                    tmem_ld_32x32b_x32(trow + c0, r);
                    tmem_ld_wait(r);
                    // row = channel, 64 bytes; 16-byte pieces exchanged by XOR with (row / 2) % 4
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t h[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const __nv_bfloat162 v = __floats2bfloat162_rn(fmaxf(fmaf(__uint_as_float(r[8 * q + 2 * i]), a.step, bias), floor_v),
                                                                           fmaxf(fmaf(__uint_as_float(r[8 * q + 2 * i + 1]), a.step, bias), floor_v));
                            h[i] = *reinterpret_cast<const uint32_t *>(&v);
                        }
                        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(tb + lane * 64u + ((uint32_t)(q ^ ((lane >> 1) & 3)) << 4)), "r"(h[0]),
                                     "r"(h[1]), "r"(h[2]), "r"(h[3]) : "memory");
                    }
                    __syncwarp();
                    const bool ok = p < a.p_end;
                    __nv_bfloat16 *dst = a.xhat + img * img_stride + (long long)(block * 128 + wq * 32) * a.hw + sp;
                    if (vec) {
                        const int r0 = lane >> 3;
                        dst += (long long)r0 * a.hw;
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const int row = r0 + 4 * k;
                            uint32_t lo, hi;
                            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(lo), "=r"(hi)
                                         : "r"(tb + row * 64u + ((uint32_t)((px_lane >> 3) ^ ((row >> 1) & 3)) << 4) + (uint32_t)(px_lane & 7) * 2u));
                            if (ok && row < rows) *reinterpret_cast<uint2 *>(dst) = make_uint2(lo, hi);
                            dst += 4 * (long long)a.hw;
                        }
                    } else {
#pragma unroll 8
                        for (int row = 0; row < 32; ++row) {
                            unsigned short v;
                            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v)
                                         : "r"(tb + row * 64u + ((uint32_t)((px_lane >> 3) ^ ((row >> 1) & 3)) << 4) + (uint32_t)(px_lane & 7) * 2u));
                            if (ok && row < rows) *reinterpret_cast<unsigned short *>(dst) = v;
                            dst += a.hw;
                        }
                    }
                    sp += 32;
                    while (sp >= a.hw) { sp -= a.hw; ++img; }
                    __syncwarp();                             // the block may be overwritten
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_tempty[acc]));
        }
        if (!alive && lane == 0) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// Pixels [p_first, p_end) of an NCHW tensor as rows of C channels.  A block turns 64 pixels x 64 channels
// through shared memory; bound by the memory it moves (L2 for the rows).
constexpr int kTurn = 64;
__global__ void __launch_bounds__(256) pixel_rows_kernel(const __nv_bfloat16 *x, int c, int hw, long long p_first, long long p_end, __nv_bfloat16 *rows,
                                                         unsigned long long *clear, long long clear_words)
{
    chain_next();
    chain_wait();
    for (long long i = (blockIdx.y * (long long)gridDim.x + blockIdx.x) * 256 + threadIdx.x; i < clear_words; i += (long long)gridDim.x * gridDim.y * 256)
        clear[i] = 0ull;                                      // the coder's look-back state
    __shared__ __nv_bfloat16 s[kTurn][kTurn + 2];             // [channel][pixel]; the padding keeps the column reads apart
    const int c0 = blockIdx.y * kTurn, t = threadIdx.x;
    const long long p0 = p_first + (long long)blockIdx.x * kTurn;
    if ((hw & 3) == 0 && ((uintptr_t)x & 7u) == 0) {          // four pixels a load
        const int px = (t & 15) * 4, cr = t >> 4;
        const long long p = p0 + px;
        if (p < p_end) {
            const long long img = p / hw;
            const __nv_bfloat16 *src = x + img * c * (long long)hw + (p - img * hw);
            uint2 v[kTurn / 16];
#pragma unroll
            for (int i = 0; i < kTurn / 16; ++i)
                if (c0 + cr + 16 * i < c) v[i] = *reinterpret_cast<const uint2 *>(src + (long long)(c0 + cr + 16 * i) * hw);
#pragma unroll
            for (int i = 0; i < kTurn / 16; ++i) {
                uint32_t *d = reinterpret_cast<uint32_t *>(&s[cr + 16 * i][px]);
                d[0] = v[i].x;
                d[1] = v[i].y;
            }
        }
    } else {
        const int px = t & 63, cr = t >> 6;
        const long long p = p0 + px;
        if (p < p_end) {
            const long long img = p / hw;
            const __nv_bfloat16 *src = x + img * c * (long long)hw + (p - img * hw);
            __nv_bfloat16 v[kTurn / 4];
#pragma unroll
            for (int i = 0; i < kTurn / 4; ++i)
                if (c0 + cr + 4 * i < c) v[i] = src[(long long)(c0 + cr + 4 * i) * hw];
#pragma unroll
            for (int i = 0; i < kTurn / 4; ++i) s[cr + 4 * i][px] = v[i];
        }
    }
    __syncthreads();
    // a thread writes 8 channels of a pixel (16 bytes); C is a multiple of 16
    for (int i = t; i < kTurn * kTurn / 8; i += 256) {
        const int pp = i >> 3, c8 = (i & 7) * 8;
        if (p0 + pp >= p_end || c0 + c8 >= c) continue;
        __align__(16) __nv_bfloat16 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = s[c8 + k][pp];
        *reinterpret_cast<uint4 *>(rows + (p0 + pp - p_first) * c + c0 + c8) = *reinterpret_cast<const uint4 *>(v);
    }
}

// Columns per unit: at least K / 256 blocks; more of them while the rounds of the grid get cheaper (a
// unit costs its columns plus about 64 for the shared operand and the hand-over).
int best_columns(long long tiles, int k, int sm_count)
{
    int best = 0;
    double best_cost = 0.0;
    for (int blocks = (k + kMaxN - 1) / kMaxN; blocks <= (k + 63) / 64; ++blocks) {
        const int cols = ((k + blocks - 1) / blocks + 31) / 32 * 32;
        const long long units = tiles * ((k + cols - 1) / cols);
        const double cost = (double)((units + sm_count - 1) / sm_count) * (cols + 64);
        if (best == 0 || cost < best_cost) { best = cols; best_cost = cost; }
    }
    return best;
}

// Pixels per unit of the inverse: 64 to 256 in steps of a transposed pass, where the rounds of the grid are cheapest.  A unit
// costs what its operands bring from L2, its pixels and 128 channels.  Against 256, or 128 or 64 while that left SMs
// idle: 512x7x7 x 64 (one round of 96 instead of two of 64) 23.2 -> 21.1 us, 960x7x7 x 128 46.9 -> 45.2, 576x14x14 x 128
// 56.5 -> 56.0, 128x28x28 x 64 per channel 29.3 -> 27.4.
int best_pixels(long long pixels, int blocks, int sm_count)
{
    int best = 0;
    long long best_cost = 0;
    for (int n = kMaxN; n >= 64; n -= 32) {
        const long long units = (pixels + n - 1) / n * blocks, cost = (units + sm_count - 1) / sm_count * (n + 128);
        if (best == 0 || cost < best_cost) { best = n; best_cost = cost; }
    }
    return best;
}

template <bool kEncode>
tc_status launch_gemm(int sms, bool early, const GemmArgs &g, const CUtensorMap &map_a, const CUtensorMap &map_b, cudaStream_t s)
{
    const size_t smem = (size_t)kStages * kStageBytes + (kEncode ? 0 : kEpiWarps * kTrWarpBytes);
    if (cudaFuncSetAttribute(wide_gemm_kernel<kEncode>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return TC_ERR_CUDA;
    const unsigned int grid = (unsigned int)(g.units < sms ? g.units : sms);
    return launch_chained(early, wide_gemm_kernel<kEncode>, grid, kThreads, smem, s, g, map_a, map_b) == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

// Tiles of a pass over a tensor whose workspace would exceed the cap.
long long tiles_per_pass(long long n_tiles, size_t tile_bytes)
{
    const long long most = (long long)(kWideWorkspace / tile_bytes);
    if (n_tiles <= most) return n_tiles;
    const long long passes = (n_tiles + most - 1) / most;
    return (n_tiles + passes - 1) / passes;
}

size_t up(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

size_t tc_encode_wide_workspace(int c, int k, long long n_tiles)
{
    const size_t px = (size_t)tiles_per_pass(n_tiles, (size_t)TC_TILE_PIXELS * (2 * c + k)) * TC_TILE_PIXELS;
    return up(px * c * 2) + up(px * k);
}

size_t tc_decode_wide_workspace(int k, long long n_tiles)
{
    return up((size_t)tiles_per_pass(n_tiles, (size_t)TC_TILE_PIXELS * 2 * k) * TC_TILE_PIXELS * k * 2);
}

tc_status tc_launch_encode_wide_gemm(const tc_ctx *ctx, const EncodeArgs &a, void *workspace, cudaStream_t s)
{
    const long long per_pass = tiles_per_pass(a.n_tiles, (size_t)TC_TILE_PIXELS * (2 * a.c + a.k));
    __nv_bfloat16 *rows = (__nv_bfloat16 *)workspace;
    uint8_t *sym = (uint8_t *)workspace + up((size_t)per_pass * TC_TILE_PIXELS * a.c * 2);
    for (long long t0 = 0; t0 < a.n_tiles; t0 += per_pass) {
        const long long t1 = t0 + per_pass < a.n_tiles ? t0 + per_pass : a.n_tiles;
        const long long p0 = t0 * TC_TILE_PIXELS, p1 = t1 * TC_TILE_PIXELS < a.pixels ? t1 * TC_TILE_PIXELS : a.pixels;
        const dim3 grid((unsigned int)((p1 - p0 + kTurn - 1) / kTurn), (unsigned int)((a.c + kTurn - 1) / kTurn));
        // Early for a tensor of one pass (400x7x7 x 3243, three of them, 296 -> 300 us); kept apart up to five blocks an SM (us in turn, early on the first SMs
        // that are free, and so: 128x1x1 x 18688, 4.0 an SM, 26.1, 32.2, 24.1; 64x7x7 x 404, 2.1, 20.9, 22.6, 20.4; 160x1x1 x 16512, 5.2, 24.6, 24.8, 28.4).
        const long long blocks = (long long)grid.x * grid.y;
        static std::atomic<size_t> own;
        const size_t spread = a.alone && blocks <= 5ll * a.sms ? spread_bytes(blocks, a.sms, static_bytes(own, (const void *)pixel_rows_kernel)) : 0;
        if (spread > 0 && cudaFuncSetAttribute(pixel_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpreadMost) != cudaSuccess) return TC_ERR_CUDA;
        if (launch_first(a.alone && per_pass >= a.n_tiles, pixel_rows_kernel, grid, 256, spread, s, (const __nv_bfloat16 *)a.x, a.c, a.hw, p0, p1, rows,
                         (unsigned long long *)a.ticket, t0 == 0 ? a.clear_words : 0ll) != cudaSuccess) return TC_ERR_CUDA;
        GemmArgs g{};
        g.n_panels = (a.c + kPanelK - 1) / kPanelK;
        g.k_depth = a.c;
        g.n_cols = best_columns(t1 - t0, a.k, a.sms);
        g.blocks = (a.k + g.n_cols - 1) / g.n_cols;
        CUtensorMap map_x, map_t;
        if (!tc_tensor_map_sw128(&map_x, rows, p1 - p0, a.c, 128) || !tc_tensor_map_sw128(&map_t, a.basis_bf16, a.k, a.c, g.n_cols)) return TC_ERR_CUDA;
        g.units = (t1 - t0) * g.blocks;
        g.p_first = p0; g.p_end = p1;
        g.k = a.k;
        g.inv_step = (float)(a.basis_scale / a.step);          // the operand holds basis / basis_scale
        g.vmax = kMagic + (float)((1 << a.bits) - 1);
        g.bias = a.enc_bias;
        g.sym = sym;
        g.status = a.status;
        tc_status st = launch_gemm<true>(a.sms, a.alone, g, map_x, map_t, s);
        if (st != TC_OK) return st;
        if ((st = tc_launch_pack_symbols(ctx, a, sym, t0, t1, s)) != TC_OK) return st;
    }
    return TC_OK;
}

tc_status tc_launch_decode_wide_gemm(const tc_ctx *ctx, const DecodeArgs &a, void *workspace, cudaStream_t s)
{
    const long long per_pass = tiles_per_pass(a.n_tiles, (size_t)TC_TILE_PIXELS * 2 * a.k);
    __nv_bfloat16 *q = (__nv_bfloat16 *)workspace;
    for (long long t0 = 0; t0 < a.n_tiles; t0 += per_pass) {
        const long long t1 = t0 + per_pass < a.n_tiles ? t0 + per_pass : a.n_tiles;
        const long long p0 = t0 * TC_TILE_PIXELS, p1 = t1 * TC_TILE_PIXELS < a.pixels ? t1 * TC_TILE_PIXELS : a.pixels;
        tc_status st = tc_launch_unpack_operand(ctx, a, q, t0, t1, s);
        if (st != TC_OK) return st;
        GemmArgs g{};
        g.n_panels = (a.k + kPanelK - 1) / kPanelK;
        g.k_depth = a.k;
        g.blocks = (a.c + 127) / 128;
        g.n_cols = best_pixels(p1 - p0, g.blocks, a.sms);
        g.units = ((p1 - p0 + g.n_cols - 1) / g.n_cols) * g.blocks;
        CUtensorMap map_q;
        if (!tc_tensor_map_sw128(&map_q, q, p1 - p0, a.k, g.n_cols)) return TC_ERR_CUDA;
        g.p_first = p0; g.p_end = p1;
        g.c = a.c; g.hw = a.hw; g.relu = a.relu;
        g.step = (float)(a.step * a.basis_scale);              // the operand holds basis / basis_scale
        g.bias = a.dec_bias;
        g.xhat = (__nv_bfloat16 *)a.xhat;
        g.status = a.status;
        if ((st = launch_gemm<false>(a.sms, a.alone, g, *a.basis_t_map, map_q, s)) != TC_OK) return st;
    }
    return TC_OK;
}
