// Fused tensor-core encode for bf16 tensors (Section 3: transform, quantiser, VLC).
//
// One persistent block per SM walks tiles of 128 consecutive pixels.  Warp roles:
//   warps 0-15       epilogue groups on tiles in turn: four of four warps up to 128 coefficients, a thread
//                    per pixel, else two of eight.  Of these warps 0-3 own the
//                    leading coefficients of the tile's 128 pixels and warps 4-7 the others, split
//                    where the expected work of both is the same: TMEM -> registers, quantise, code.  A
//                    thread packs its codes into a run of its own in shared memory, in one pass, and the
//                    runs are joined once the tile's bit offsets are known (scan); tiles whose runs
//                    would not fit take two passes over the accumulator, lengths first.
//   warps 21, 22     store warps, every other tile each: resolve the tile's stream offset by
//                    look-back and copy the group's staging buffer out, while the group
//                    already works on its next tile
//   warps 16-19      loaders: 16- and 8-byte cp.async NCHW -> shared memory in the MMA's MN-major layout (128-byte swizzle)
//   warp 20          one thread issues tcgen05.mma:  D[pixel][coef] = X_tile[pixel][c] * T[coef][c]
// The basis T (bf16, K x C) stays resident in shared memory; the X tile streams through a ring
// of 32-channel panels; every group has an fp32 accumulator in tensor memory, so that the
// epilogue of one tile overlaps the loads and MMAs of the next.  The time of a tile in a group is that of its chain (wait, codes,
// scan, join, with barriers between), so the groups in flight set the rate where the accumulators leave room for four: us with two
// groups of eight warps and with four of four, 96x112x112 x 128 203 -> 155, 64x56x56 x 512 at 4 and 8 bits 151 -> 122 and 173 -> 138,
// 128x38x38 x 656 135 -> 110, 80x8x7 x 30965 169 -> 133, 32x44x44 x 2384 at 8 bits 373 -> 313.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <type_traits>

#include "device_utils.cuh"
#include "sm100_ptx.cuh"

namespace {

using namespace tcdev;
using namespace sm100;

constexpr int kPanelCh = 32;                      // channels per ring stage
constexpr int kMaxStages = 8;                     // ring stages (six where the staging buffers need the room)
constexpr int kStageBytes = kPanelCh * TC_TILE_PIXELS * 2;   // 8 KB
constexpr int kStaticSmem = 1024;                 // the static shared variables, up to the ring's alignment
constexpr int kSlots = 4;                         // packed tiles of a group that may wait in its staging buffer
constexpr int kMaxStagingBytes = 49152;           // a tile of 256 coefficients of 12 bits
constexpr int kEpiWarps = 16;                     // 2 groups x (2 column halves x 4 lane quarters), or 4 x 4 quarters
constexpr int kLoaderWarp0 = kEpiWarps, kMmaWarp = kEpiWarps + 4;
constexpr int kStoreWarp0 = kMmaWarp + 1;         // two store warps follow
constexpr int kThreads = (kEpiWarps + 7) * 32;
constexpr int kTmemCols = 512;
constexpr int kMaxGroups = 4;                     // epilogue groups (tiles in flight behind the MMAs)
constexpr int kSetupBar = kMaxGroups + 1;         // named barrier of all warps but the loaders (1 ...: the epilogue groups)
constexpr int kPairMaxBits = 6;                   // symbols of up to 6 bits can be coded two at a time (tables of up to 4096 entries)
constexpr int kRunStep = 512;                     // bytes between a thread's words in the private runs (128 threads of a half)

// How a launch uses the block: chosen on the host.
struct Plan {
    int groups;                // epilogue groups: two of eight warps, two threads a pixel, or four of four, a thread a pixel
    int stages;                // ring stages
    uint32_t staging_bytes;    // per epilogue group, a multiple of 16; 0: does not fit
    int run_words[2];          // words of a thread's private run, first and second half's threads; 0: two passes
    int split_blk;             // blocks of 16 coefficients of the first half's threads
    int skip_blk;              // blocks from here on are tested for holding nothing but the modal symbol
    float skip_dist;           // a position nearer to the modal level than this (as a fraction of the quantiser's range) rounds to it
    int entries;               // of the code table in shared memory
};

struct SmemLayout {
    uint32_t basis, ring, staging, run_bytes, enc, len8, bias, bias_mid, xch, total;
};

__host__ __device__ inline SmemLayout smem_layout(int c, int k, const Plan &pl)
{
    SmemLayout l;
    l.basis = 0;
    l.ring = (uint32_t)(((size_t)k * c * 2 + 1023) & ~(size_t)1023);
    l.run_bytes = (uint32_t)(pl.run_words[0] + pl.run_words[1]) * kRunStep;      // per group
    l.staging = l.ring + (uint32_t)pl.stages * kStageBytes;                     // per group: the buffer, then the runs
    l.enc = l.staging + (uint32_t)pl.groups * (pl.staging_bytes + l.run_bytes);
    l.len8 = l.enc + (uint32_t)pl.entries * 8;           // code lengths as bytes
    l.bias = (l.len8 + (uint32_t)pl.entries + 15u) & ~15u;
    l.bias_mid = l.bias + (uint32_t)k * 4;
    l.xch = l.bias_mid + (uint32_t)k * 4;               // per group: [2 halves][128] prefix and bits of every pixel, [3][128] chunk boundaries
    l.total = l.xch + (uint32_t)pl.groups * (2u * 128u * 4u + 3u * 128u * 2u);
    return l;
}

// Quantiser in fp32.  The level is rounded to the nearest integer (ties to even) by adding
// 1.5 * 2^23 -- the integer then sits in the low mantissa bits.  (A float -> int conversion
// instruction would do the same but issues at a quarter of the rate.)
constexpr float kMagic = 12582912.0f;
constexpr uint32_t kMagicBits = 0x4B400000u;

// Sinks of a thread's codes that are not written to shared memory: only counted, or packed into global memory.
struct CountSink {
    unsigned int bits;
};
struct GlobalSink {
    BitWriter w;
    bool on;
    __device__ __forceinline__ void put(uint32_t code, int len) { if (on) w.put(code, len); }
    __device__ __forceinline__ void put_word(uint32_t bits) { put(bits >> 16, 16); put(bits & 0xffffu, 16); }
};

// Two coefficients at once.  The position on the quantiser's grid is computed as a fraction of
// its range, t = (y - lo) / (step (2^b - 1)), with a saturating multiply-add: the clamp to the
// first and last level costs nothing.  A second multiply-add (packed: two fp32 lanes per
// instruction, each rounded exactly as the scalar instruction rounds) scales t back to levels and
// adds the magic constant, which leaves the level, rounded to nearest even, in the mantissa.
__device__ __forceinline__ void quantise_bits2(uint32_t acc0, uint32_t acc1, float inv_range, float bias0, float bias1, float top,
                                               uint32_t &q0, uint32_t &q1)
{
    float t0, t1;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(t0) : "f"(__uint_as_float(acc0)), "f"(inv_range), "f"(bias0));
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(t1) : "f"(__uint_as_float(acc1)), "f"(inv_range), "f"(bias1));
    asm("{\n\t.reg .b64 v, s, m;\n\t"
        "mov.b64 v, {%2, %3};\n\t"
        "mov.b64 s, {%4, %4};\n\t"
        "mov.b64 m, {%5, %5};\n\t"
        "fma.rn.f32x2 v, v, s, m;\n\t"
        "mov.b64 {%0, %1}, v;\n\t}"
        : "=r"(q0), "=r"(q1) : "f"(t0), "f"(t1), "f"(top), "f"(kMagic));
}

// Raises `far` to the larger distance of two coefficients from the modal symbol's level, as fractions of
// the quantiser's range (`mid`: the bias seen from that level): one packed multiply-add, one
// three-input maximum.
__device__ __forceinline__ void farthest2(float &far, uint32_t acc0, uint32_t acc1, float inv_range, float mid0, float mid1)
{
    asm("{\n\t.reg .b64 v, s, m;\n\t.reg .f32 u0, u1;\n\t"
        "mov.b64 v, {%1, %2};\n\t"
        "mov.b64 s, {%3, %3};\n\t"
        "mov.b64 m, {%4, %5};\n\t"
        "fma.rn.f32x2 v, v, s, m;\n\t"
        "mov.b64 {u0, u1}, v;\n\t"
        "max.NaN.abs.f32 %0, %0, u0, u1;\n\t}"
        : "+f"(far) : "r"(acc0), "r"(acc1), "f"(inv_range), "f"(mid0), "f"(mid1));
}

// The codes of a block's sixteen symbols, two a piece: (1 << length, code), at most 24 bits.
template <bool kPerChannel, bool kPair>
__device__ __forceinline__ void block_pieces(const uint32_t (&qv)[16], uint32_t enc_addr, const uint32_t *enc, int j0, int bits,
                                             uint32_t (&mul)[8], uint32_t (&code)[8])
{
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if constexpr (kPair) {
            const uint32_t idx = (qv[2 * i] - kMagicBits) + ((qv[2 * i + 1] - kMagicBits) << bits);
            asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(mul[i]), "=r"(code[i]) : "r"(enc_addr + idx * 8u));
        } else {
            uint32_t m0, c0, m1, c1;
            if constexpr (kPerChannel) {
                const int j = j0 + 2 * i;
                const uint32_t e0 = __ldg(enc + (j << bits) + (qv[2 * i] & 0xffu)), e1 = __ldg(enc + ((j + 1) << bits) + (qv[2 * i + 1] & 0xffu));
                m0 = 1u << (e0 & 0xffu); c0 = e0 >> 8; m1 = 1u << (e1 & 0xffu); c1 = e1 >> 8;
            } else {
                asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(m0), "=r"(c0) : "r"(enc_addr + (qv[2 * i] - kMagicBits) * 8u));
                asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(m1), "=r"(c1) : "r"(enc_addr + (qv[2 * i + 1] - kMagicBits) * 8u));
            }
            mul[i] = m0 * m1;
            code[i] = c0 * m1 + c1;
        }
    }
}

// Appends them.  How many symbols are joined before they are appended is chosen for the whole warp (lanes
// that go different ways run one after the other): sixteen or eight where every lane's
// codes of them fit 31 bits -- a product of powers of two that reaches 2^32 is zero --
// else four, else two.  Joining is a multiply-add, appending costs ten instructions.
template <typename Sink>
__device__ __forceinline__ void append_block(Sink &sink, const uint32_t (&mul)[8], const uint32_t (&code)[8])
{
    uint32_t m4[4], c4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { m4[i] = mul[2 * i] * mul[2 * i + 1]; c4[i] = code[2 * i] * mul[2 * i + 1] + code[2 * i + 1]; }
    const uint32_t m8a = m4[0] * m4[1], m8b = m4[2] * m4[3];
    if (__all_sync(0xffffffffu, m8a != 0u && m8b != 0u)) {
        const uint32_t c8a = c4[0] * m4[1] + c4[1], c8b = c4[2] * m4[3] + c4[3], m16 = m8a * m8b;
        if (__all_sync(0xffffffffu, m16 != 0u)) sink.put(c8a * m8b + c8b, 31 - __clz((int)m16));
        else { sink.put(c8a, 31 - __clz((int)m8a)); sink.put(c8b, 31 - __clz((int)m8b)); }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (__all_sync(0xffffffffu, m4[i] != 0u)) sink.put(c4[i], 31 - __clz((int)m4[i]));
            else { sink.put(code[2 * i], 31 - __clz((int)mul[2 * i])); sink.put(code[2 * i + 1], 31 - __clz((int)mul[2 * i + 1])); }
        }
    }
}

// A thread's blocks quantised and coded from the accumulator once more, for tiles that the plan does not fit.  A
// function of its own, so that what it keeps in registers does not weigh on the loop that every tile goes through (inlined, it
// cost that loop up to 7 %: 64x56x56 x 256 at 8 bits 103 -> 110 us).  All lanes of the warp call it together.
template <bool kPerChannel, bool kPair, typename Sink>
__device__ __noinline__ Sink code_again(Sink sink, uint32_t trow, int blk0, int blk1, float inv_range, float top, const float *s_bias,
                                        uint32_t enc_addr, const uint32_t *enc, int bits)
{
#pragma unroll 1
    for (int blk = blk0; blk < blk1; ++blk) {
        uint32_t r[16], qv[16], mul[8], code[8];
        tmem_ld_32x32b_x16(trow + blk * 16, r);
        tmem_ld_wait(r);
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
            const float4 b4 = *reinterpret_cast<const float4 *>(s_bias + blk * 16 + i);
            quantise_bits2(r[i], r[i + 1], inv_range, b4.x, b4.y, top, qv[i], qv[i + 1]);
            quantise_bits2(r[i + 2], r[i + 3], inv_range, b4.z, b4.w, top, qv[i + 2], qv[i + 3]);
        }
        block_pieces<kPerChannel, kPair>(qv, enc_addr, enc, blk * 16, bits, mul, code);
        append_block(sink, mul, code);
    }
    return sink;
}

// The issuing warp's way through the tiles of a block: the accumulators in turn, the panels of a tile through the ring of stages.  Once a wait has run
// out it issues nothing more -- what has not landed is not multiplied, and its stage not handed back to be loaded while it is read -- and
// it leaves only when what it has issued is done: the block frees tensor memory next.  (Not by leaving the inner loop at the wait, which keeps it from being unrolled.)
#pragma nv_exec_check_disable
template <int kGroups, int kUnroll, typename Basis, typename Accumulator, typename Landed, typename Panel, typename Done, typename Drain>
__host__ __device__ __forceinline__ bool issue_tiles(long long tiles, int panels, int stages, Basis basis, Accumulator accumulator, Landed landed, Panel panel,
                                                     Done done, Drain drain)
{
    if (!basis()) return false;
    bool alive = true;
    int s = 0;
    uint32_t phase = 0;
    for (long long tl = 0; tl < tiles && alive; ++tl) {
        const int acc = (int)(tl % kGroups);
        if (!accumulator(acc, (uint32_t)(((tl / kGroups) & 1) ^ 1))) { alive = false; break; }
#pragma unroll kUnroll
        for (int kp = 0; kp < panels; ++kp) {
            if (alive) alive = landed(s, phase);
            panel(kp, s, alive);
            if (++s == stages) { s = 0; phase ^= 1u; }
        }
        if (alive) done(acc);
    }
    drain();
    return alive;
}

// The epilogue's two ways (kRuns):
//   one pass: every thread packs the codes of its coefficients, as they are quantised, into a private
//     run of words in shared memory (word w of all threads side by side: no bank conflicts); when
//     the tile's bit offsets are known the few words are shifted to their place in the staging buffer.
//     Nothing but the packed bits is kept, so the loop over the coefficients stays rolled.
//   two passes, where runs and staging do not both fit (near-lossless codes of wide layers): code
//     lengths first, then the coefficients are quantised again and packed straight to their place; the
//     accumulator is held until then.
// What bounded the epilogue before (symbols in registers between a length pass and a pack pass, both
// unrolled over 128 coefficients): 117 KB of straight-line code per tile -- instruction fetch -- and a
// second table lookup per symbol.
// Blocks of 16 coefficients from skip_blk on are first tested, by the whole warp, for holding nothing
// but the modal symbol (the single bit 0): sixteen zero bits then.
// kPair (per-layer tables, b <= 6): the code tables are indexed by two neighbouring symbols at once
// (q0 | q1 << b), which halves the lookups.
// kGroups: epilogue groups, two (a pixel's coefficients split between two threads) or four.
// kHist (statistics, Section 3.1 "Variable length coding": the entropy needs the distribution of
// the symbols): every symbol but the zero level is also counted, per coefficient channel, into one of the copies of a.hist, one
// atomic each.
// `block` of `blocks` that share the tensor's tiles.
template <bool kPerChannel, bool kDebug, bool kPair, bool kHist, bool kRuns, int kGroups>
__device__ __forceinline__ void encode_tiles(const EncodeArgs &a, const Plan &pl, unsigned int block, unsigned int blocks)
{
    extern __shared__ __align__(1024) unsigned char smem[];      // swizzled ring stages: aligned to their 1 KB atoms
    __shared__ __align__(8) unsigned long long s_full[kMaxStages], s_empty[kMaxStages], s_tfull[kGroups], s_tempty[kGroups];
    __shared__ __align__(8) unsigned long long s_basis_ready;
    __shared__ uint32_t s_tmem_base;
    __shared__ unsigned int s_warp_sums[kGroups][2][4], s_overflow[kGroups];
    __shared__ int s_go[kGroups];                    // per group: its polling warp's waits for the tile have succeeded
    __shared__ unsigned long long s_base[kGroups];
    __shared__ int s_write_ok[kGroups];
    // staging hand-over to the store warp: slot n % kSlots for a group's n-th tile
    __shared__ __align__(8) unsigned long long s_stg_full[kGroups][kSlots], s_stg_free[kGroups][kSlots];
    __shared__ unsigned int s_padded[kGroups][kSlots], s_stg_at[kGroups][kSlots];   // bits of the tile, its place in the staging buffer
    __shared__ int s_store_cmd[kGroups][kSlots];     // 1: copy the staged tile out, 2: nothing to copy, 3: stop

    // (taken from lane 0: the compiler knows that the branches between the roles are the same for a whole warp)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int nsym = 1 << a.bits;
    constexpr int kGroupWarps = kEpiWarps / kGroups, kGroupThreads = 32 * kGroupWarps, kAccCols = kTmemCols / kGroups;
    constexpr bool kHalves = kGroupWarps == 8;                   // two threads a pixel
    constexpr bool enc_in_smem = !kPerChannel;
    constexpr bool kCanSkip = !kPerChannel && !kDebug && !kHist;     // blocks of modal symbols are passed over
    const int enc_entries = pl.entries;
    const SmemLayout L = smem_layout(a.c, a.k, pl);
    const int n_stages = pl.stages;
    unsigned char *s_basis = smem + L.basis;
    uint32_t *s_enc = reinterpret_cast<uint32_t *>(smem + L.enc);
    float *s_bias = reinterpret_cast<float *>(smem + L.bias), *s_bias_mid = reinterpret_cast<float *>(smem + L.bias_mid);
    const uint32_t ring_addr = smem_u32(smem + L.ring);
    const uint32_t basis_addr = smem_u32(s_basis);
    const int n_panels = (a.c + kPanelCh - 1) / kPanelCh;

    // ---- set-up ---------------------------------------------------------------------
    chain_next();                                             // (a decoder that follows is set up meanwhile)
    if (tid < kGroups) s_overflow[tid] = 0;
    if (tid == 0) {
        for (int s = 0; s < n_stages; ++s) { mbar_init(smem_u32(&s_full[s]), 128); mbar_init(smem_u32(&s_empty[s]), 1); }
        for (int b = 0; b < kGroups; ++b) {
            mbar_init(smem_u32(&s_tfull[b]), 1);
            mbar_init(smem_u32(&s_tempty[b]), kGroupWarps);                 // one arrival per warp of the group
            for (int i = 0; i < kSlots; ++i) { mbar_init(smem_u32(&s_stg_full[b][i]), kGroupWarps); mbar_init(smem_u32(&s_stg_free[b][i]), 1); }
        }
        mbar_init(smem_u32(&s_basis_ready), 1);
        mbar_fence_init();
        // the basis, in the order the MMA reads it (K-major core matrices: element (j, ch) at
        // (j/8)*sbo + (ch/8)*128 + (j%8)*16 + (ch%8)*2), by the copy engine: no thread moves a byte of it,
        // and only the MMA warp waits for it.  (Copied by 600 threads, 128 KB in 8192 pieces, it stood in
        // front of the first tile's loads: 23.3 us for 98 tiles of 256 channels, 17.4 like this.)
        const uint32_t bytes = (uint32_t)a.k * (uint32_t)a.c * 2u;
        mbar_arrive_expect_tx(smem_u32(&s_basis_ready), bytes);
        for (uint32_t at = 0; at < bytes; at += 16384u)
            bulk_load(smem_u32(smem + L.basis) + at, reinterpret_cast<const char *>(a.basis_core) + at, min(16384u, bytes - at), smem_u32(&s_basis_ready));
    }
    const long long my_tiles = (a.n_tiles > block) ? (a.n_tiles - block + blocks - 1) / blocks : 0;
    __syncthreads();
    // the loaders start with the first tile at once, the others lay out the basis and the tables meanwhile
    const bool loader = warp >= kLoaderWarp0 && warp < kMmaWarp;
    const int setup_tid = warp < kLoaderWarp0 ? tid : tid - 128;
    constexpr int kSetupThreads = kThreads - 128;
    if (warp == kMmaWarp) { tmem_alloc(smem_u32(&s_tmem_base), kTmemCols); tmem_relinquish(); }
    if (!loader) {
        for (int i = setup_tid; i < a.k; i += kSetupThreads) {
            const float b = a.enc_bias[i] / (float)(nsym - 1);   // as a fraction of the range
            s_bias[i] = b;
            s_bias_mid[i] = b - (float)(a.modal < 0 ? 0 : a.modal) / (float)(nsym - 1);   // the same, seen from the modal symbol's level
        }
        if (enc_in_smem)
            for (int i = setup_tid; i < enc_entries; i += kSetupThreads) {
                // per-layer table: (1 << length, code) pairs, so that appending a code to a register is
                // one multiply-add, and the lengths once more as bytes.  In pair mode entry
                // q0 | q1 << b holds the two codes joined (q0's first), at most 24 bits.
                uint32_t len, code;
                if constexpr (kPair) {
                    const uint32_t e0 = a.enc[i & (nsym - 1)], e1 = a.enc[i >> a.bits];
                    len = (e0 & 0xffu) + (e1 & 0xffu);
                    code = ((e0 >> 8) << (e1 & 0xffu)) | (e1 >> 8);
                } else {
                    const uint32_t e = a.enc[i];
                    len = e & 0xffu;
                    code = e >> 8;
                }
                s_enc[2 * i] = 1u << len;
                s_enc[2 * i + 1] = code;
                (smem + L.len8)[i] = (unsigned char)len;
            }
        for (long long i = (long long)block * kSetupThreads + setup_tid; i < a.other_words; i += (long long)blocks * kSetupThreads) a.other_state[i] = 0ull;
        tc_fence_before_sync();
        named_bar_sync(kSetupBar, kSetupThreads);
        tc_fence_after_sync();
    }
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, s_tmem_base, 0);

    if (warp >= kLoaderWarp0 && warp < kMmaWarp) {
        // ================= loaders =================
        // A lane moves groups of 8 pixels of every eighth channel: one copy of 16 bytes where the group starts
        // on a 16-byte boundary of global memory and lies in one image, else two of 8.  With H*W an odd
        // multiple of 4 the groups of the channels of one parity are aligned (the parity changes from image
        // to image), so a warp takes channels of one parity only: its lanes agree up to an image
        // boundary.  What bounds the loads is the copy unit, by lanes rather than bytes: 8-byte copies
        // alone reach 3.3 TB/s of input (123 us for 256x14x14 x 4096 and nothing else), this mix
        // 4.6 TB/s, 16-byte copies 6.4 TB/s.  (Eight channels x 32 bytes per instruction, which the
        // unswizzled operand layout asks for, reached 1.85 TB/s.)  In the swizzled layout 64 pixels of a
        // channel are 128 contiguous bytes, the 16-byte pieces exchanged by XOR with the channel modulo 8.
        const int lw = warp - kLoaderWarp0;
        const int px = 8 * (lane & 15);                            // first pixel of this lane's group in the tile
        const int ch0 = (lw & 1) + 2 * (lane >> 4) + 4 * (lw >> 1);  // channels ch0, ch0 + 8, ... of a panel
        const uint32_t dst0 = (uint32_t)((px >> 6) * (kStageBytes / 2) + ch0 * 128 + ((((px & 63) >> 3) ^ ch0) << 4));
        const __nv_bfloat16 *xin = reinterpret_cast<const __nv_bfloat16 *>(a.x);
        const size_t row8 = 16 * (size_t)a.hw;        // bytes from a channel to the eighth after it; a panel (four of them) passes 4 GB at 2^26 pixels a map
        static_assert(kPanelCh == 32, "a lane copies four channels of a panel");
        int s = 0;                                 // ring stage of the next panel
        uint32_t phase = 1;
        bool alive = true;
        for (long long tl = 0; tl < my_tiles && alive; ++tl) {
            const long long p0 = (block + tl * blocks) * TC_TILE_PIXELS + px;
            const long long img = p0 < a.pixels ? p0 / a.hw : 0;
            const int sp = p0 < a.pixels ? (int)(p0 - img * a.hw) : 0;
            const bool split = sp + 4 >= a.hw;                 // the second four pixels start the next image
            const char *src = reinterpret_cast<const char *>(xin + (img * a.c + ch0) * (long long)a.hw + sp);
            const uint32_t n1 = p0 < a.pixels ? 8u : 0u, n2 = p0 + 4 < a.pixels ? 8u : 0u;
            const char *src2 = n2 == 0u ? src : src + (split ? ((long long)a.c * a.hw - a.hw + 4) * 2 : 8);    // the second four pixels
            const bool whole = !split && n2 != 0u && ((uintptr_t)src & 15u) == 0;
            for (int kp = 0; kp < n_panels; ++kp) {
                if (!mbar_wait(smem_u32(&s_empty[s]), phase, 200u)) { alive = false; break; }
                const uint32_t dst = ring_addr + s * kStageBytes + dst0;
                const bool full = (kp + 1) * kPanelCh <= a.c;              // else half a panel (C is a multiple of 16)
                if (whole) {
                    cp_async_16(dst, src, 16u);
                    cp_async_16(dst + 1024u, src + row8, 16u);
                    if (full) {
                        cp_async_16(dst + 2048u, src + 2 * row8, 16u);
                        cp_async_16(dst + 3072u, src + 3 * row8, 16u);
                    }
                } else {
                    cp_async_8(dst, src, n1);
                    cp_async_8(dst + 8u, src2, n2);
                    cp_async_8(dst + 1024u, src + row8, n1);
                    cp_async_8(dst + 1032u, src2 + row8, n2);
                    if (full) {
                        cp_async_8(dst + 2048u, src + 2 * row8, n1);
                        cp_async_8(dst + 2056u, src2 + 2 * row8, n2);
                        cp_async_8(dst + 3072u, src + 3 * row8, n1);
                        cp_async_8(dst + 3080u, src2 + 3 * row8, n2);
                    }
                }
                src += 4 * row8;
                src2 += 4 * row8;
                // the stage's barrier gets this thread's arrival when its copies have landed: the thread goes
                // on to the next stage, so that all free stages are in flight (with a wait for the panel
                // before the last the loads were bound by their latency, two panels at a time)
                cp_async_arrive_noinc(smem_u32(&s_full[s]));
                if (++s == n_stages) { s = 0; phase ^= 1u; }
            }
        }
        cp_async_wait_all();                       // (of a block whose other waits ran out, too)
        if (!alive) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
    } else if (warp == kMmaWarp) {
        // ================= MMA issuer =================
        // The whole warp walks the loop (issue_tiles) and waits on the barriers; lane 0 issues, through instructions
        // that carry their own guard (a branch taken by one lane around every MMA costs about 90
        // cycles per instruction).
        const uint32_t issuer = lane == 0 ? 1u : 0u;
        const uint32_t idesc = make_idesc_bf16(TC_TILE_PIXELS, a.k, /*A MN-major*/ true, /*B K-major*/ false);
        const uint64_t a_desc = make_smem_desc_mn_sw128(ring_addr, kStageBytes / 2, 1024);
        const uint64_t b_desc = make_smem_desc(basis_addr, 128, (uint32_t)(a.c / 8) * 128u);
        const uint32_t a_desc_lo = (uint32_t)a_desc, a_desc_hi = (uint32_t)(a_desc >> 32), b_desc_hi = (uint32_t)(b_desc >> 32);
        uint32_t d_tmem = 0, b_lo = 0;
        // (rolled with a table per channel and four groups, whose coder the unrolled loop cost seven registers in local memory: 64x14x14 x 1000 29.6 -> 31.2 us)
        const bool alive = issue_tiles<kGroups, kPerChannel && kGroups == 4 ? 1 : 4>(
            my_tiles, n_panels, n_stages,
            [&] { return mbar_wait(smem_u32(&s_basis_ready), 0u); },
            [&](int acc, uint32_t parity) {
                if (!mbar_wait(smem_u32(&s_tempty[acc]), parity)) return false;
                tc_fence_after_sync();
                d_tmem = tmem_base + acc * kAccCols;
                b_lo = (uint32_t)b_desc;
                return true;
            },
            [&](int s, uint32_t parity) { return mbar_wait(smem_u32(&s_full[s]), parity); },
            [&](int kp, int s, bool issue) {
                const uint32_t on = issue ? issuer : 0u;
                fence_proxy_async_smem();            // the loaders' copies, made visible to the tensor core
                tc_fence_after_sync();
                const uint32_t a_lo = a_desc_lo + (uint32_t)s * (kStageBytes >> 4);
                mma_bf16_ss_guarded(d_tmem, a_lo, a_desc_hi, b_lo, b_desc_hi, idesc, kp ? 1u : 0u, on);
                if ((kp + 1) * kPanelCh <= a.c)          // else half a panel
                    mma_bf16_ss_guarded(d_tmem, a_lo + (2048u >> 4), a_desc_hi, b_lo + (256u >> 4), b_desc_hi, idesc, 1u, on);
                b_lo += (kPanelCh / 8) * (128u >> 4);
                mma_commit_guarded(smem_u32(&s_empty[s]), on);
            },
            [&](int acc) { mma_commit_guarded(smem_u32(&s_tfull[acc]), issuer); },
            // (the basis has come: its barrier is in its second phase)
            [&] { mma_commit_guarded(smem_u32(&s_basis_ready), issuer); mbar_wait(smem_u32(&s_basis_ready), 1u); });
        if (!alive && issuer) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
    } else if (warp >= kStoreWarp0) {
        // ================= store warps =================
        unsigned int stopped = 0;                                // groups that hand over nothing more
        for (long long tl = warp - kStoreWarp0; tl < my_tiles; tl += 2) {
            const int grp = (int)(tl % kGroups);
            const long long n = tl / kGroups;
            const uint32_t stg_addr = smem_u32(smem + L.staging + (uint32_t)grp * (pl.staging_bytes + L.run_bytes));
            const long long tile = block + tl * blocks;
            const int slot = (int)(n % kSlots);
            if (stopped >> grp & 1u) continue;
            if (!mbar_wait(smem_u32(&s_stg_full[grp][slot]), (uint32_t)((n / kSlots) & 1), 400u)) { if (lane == 0) tc_dev_set_status(a.status, TC_ERR_TIMEOUT); break; }
            const int cmd = s_store_cmd[grp][slot];
            if (cmd == 3) { stopped |= 1u << grp; continue; }
            if (cmd == 1) {
                const unsigned long long padded = s_padded[grp][slot];
                const uint32_t src = stg_addr + s_stg_at[grp][slot];
                bool ok;
                const unsigned long long base = lookback_resolve(a.tile_state, tile, padded, a.status, ok);
                const bool fits = base + padded <= a.capacity_bits;
                if (ok && !fits && lane == 0) tc_dev_set_status(a.status, TC_ERR_BUFFER_TOO_SMALL);
                if (ok && fits) {
                    uint4 *dst = reinterpret_cast<uint4 *>(a.stream + (base >> 5));
                    for (unsigned int i = lane; i < (unsigned int)(padded >> 7); i += 32) {
                        uint4 v;
                        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(src + i * 16u));
                        dst[i] = v;
                    }
                }
                if (lane == 0) {
                    a.tile_off[tile] = base;
                    if (tile == a.n_tiles - 1) a.tile_off[a.n_tiles] = base + padded;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_stg_free[grp][slot]));
        }
    } else {
        // ================= epilogue groups =================
        const int grp = warp / kGroupWarps;
        const int wg = warp % kGroupWarps;
        const int half = kHalves ? wg >> 2 : 0;    // which part of the coefficients
        const int wq = wg & 3;                     // TMEM lane quarter
        const int m = wq * 32 + lane;              // pixel within the tile = TMEM lane
        const int tg = tid % kGroupThreads;        // thread within the group
        const int n_blk = a.k >> 4;                // blocks of 16 coefficients: the first split_blk belong to the first half's threads
        const int blk0 = half ? pl.split_blk : 0, blk1 = half ? n_blk : pl.split_blk;
        const int chunk_blks = a.splits > 1 ? n_blk / a.splits : n_blk;    // blocks per chunk of a pixel
        const int bound0 = max(1, (blk0 + chunk_blks - 1) / chunk_blks);   // the first chunk boundary that lies before one of this thread's blocks
        const uint32_t stg_addr = smem_u32(smem + L.staging + (uint32_t)grp * (pl.staging_bytes + L.run_bytes));
        const uint32_t enc_addr = smem_u32(s_enc);
        const uint32_t len8_addr = smem_u32(smem + L.len8);
        const uint32_t run_addr = stg_addr + pl.staging_bytes + (half ? (uint32_t)pl.run_words[0] * kRunStep : 0u) + (uint32_t)m * 4u;
        const uint32_t run_end = run_addr + (uint32_t)pl.run_words[half] * kRunStep;
        uint32_t *xch = reinterpret_cast<uint32_t *>(smem + L.xch + grp * (2 * 128 * 4 + 3 * 128 * 2));   // [2][128]: prefix in the warp << 12 | bits
        unsigned short *bound = reinterpret_cast<unsigned short *>(xch + 256);                            // [3][128]: bits before chunk boundary 1 ..., from its thread's start
        // The staging buffer is a ring; the place [prev_at, prev_end) of the newest tile handed to the store
        // warp may still be in use, those before it are free (the polling warp has waited for that).
        unsigned int prev_at = 0, prev_end = 0;
        unsigned int n_done = 0;                   // tiles this group has handed to its store warp
        const float inv_range = (float)(a.basis_scale / (a.step * (double)(nsym - 1)));   // the operand holds basis / basis_scale
        const float top = (float)(nsym - 1);
        const float coef_scale = (float)a.basis_scale;
        const int bar_id = 1 + grp;
        bool alive = true;
        [[maybe_unused]] const int skip_blk = pl.skip_blk;
        const uint32_t trow = tmem_base + grp * kAccCols + ((uint32_t)(wq * 32) << 16);

        auto resolve_base = [&](long long tile, unsigned long long padded) {
            if (wg == 0) {
                bool ok;
                const unsigned long long base = lookback_resolve(a.tile_state, tile, padded, a.status, ok);
                if (lane == 0) {
                    const bool fits = base + padded <= a.capacity_bits;
                    if (ok && !fits) tc_dev_set_status(a.status, TC_ERR_BUFFER_TOO_SMALL);
                    s_base[grp] = base;
                    s_write_ok[grp] = (ok && fits) ? 1 : 0;
                }
            }
        };

        for (long long tl = grp; tl < my_tiles && alive; tl += kGroups) {
            const long long tile = block + tl * blocks;
            const long long p = tile * TC_TILE_PIXELS + m;
            const bool valid = p < a.pixels;
            // One warp of the group waits -- for the accumulator, and for the store warp to be done with the
            // tile before the last -- and lets the others in through a hardware barrier: a parked warp
            // issues nothing, whereas polling warps took two thirds of the SM's instructions.
            if (wg == 0) {
                bool go = mbar_wait(smem_u32(&s_tfull[grp]), (uint32_t)((tl / kGroups) & 1), 200u);
                const unsigned int back = prev_end > pl.staging_bytes ? 1u : 2u;      // (the tile before lies in the runs, too)
                if (n_done >= back) go = go && mbar_wait(smem_u32(&s_stg_free[grp][(n_done - back) % kSlots]), ((n_done - back) / kSlots) & 1u);
                if (lane == 0) s_go[grp] = go;
                tc_fence_before_sync();
            }
            named_bar_sync(bar_id, kGroupThreads);
            tc_fence_after_sync();
            if (!s_go[grp]) { alive = false; break; }
            [[maybe_unused]] unsigned int n_clamped = 0;       // statistics mode: coefficients outside the quantiser's range

            // Quantises and codes block `blk` of 16 coefficients, which are on their way into r; `first`: the
            // tile's first pass (counts for the statistics, debug outputs).  The next block's load is
            // issued as soon as r has been read: a load waited for at once took 700 cycles beside the MMAs'
            // traffic, more than the coding.  All lanes of the warp call it together.
            auto code_block = [&](int blk, uint32_t (&r)[16], auto &sink, auto first) {
                constexpr bool kCount = std::is_same<std::decay_t<decltype(sink)>, CountSink>::value;
                constexpr bool kKeep = decltype(first)::value && (kHist || kDebug);        // r is needed once more
                tmem_ld_wait(r);
                const uint32_t next = trow + min(blk + 1, blk1 - 1) * 16;
                uint32_t qv[16];
#pragma unroll
                for (int i = 0; i < 16; i += 4) {
                    const float4 b4 = *reinterpret_cast<const float4 *>(s_bias + blk * 16 + i);
                    quantise_bits2(r[i], r[i + 1], inv_range, b4.x, b4.y, top, qv[i], qv[i + 1]);
                    quantise_bits2(r[i + 2], r[i + 3], inv_range, b4.z, b4.w, top, qv[i + 2], qv[i + 3]);
                }
                if constexpr (!kKeep) tmem_ld_32x32b_x16(next, r);
                if constexpr (kKeep) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int j = blk * 16 + i;
                        if constexpr (kHist) {
                            // every symbol other than the zero level is counted; the zero level's count is what
                            // is left of the pixels, which the caller works out
                            if (valid && qv[i] != kMagicBits + (uint32_t)a.hist_modal) atomicAdd(a.hist + ((size_t)(block % kHistCopies) * a.k + j) * nsym + (qv[i] & 0xffu), 1ull);
                            // outside the quantiser's range [lo, lo + (2^b - 1) step]
                            const float t = fmaf(__uint_as_float(r[i]), inv_range, s_bias[j]);
                            n_clamped += (valid && (t < 0.f || t > 1.f)) ? 1u : 0u;
                        }
                        if constexpr (kDebug) {
                            if (valid && a.dbg_coef) a.dbg_coef[p * a.k + j] = fmaf(__uint_as_float(r[i]), coef_scale, -a.tmu32[j]);
                            if (valid && a.dbg_sym) a.dbg_sym[p * a.k + j] = (uint8_t)(qv[i] & 0xffu);
                        }
                    }
                }
                if constexpr (kKeep) tmem_ld_32x32b_x16(next, r);
                if constexpr (kCount) {
#pragma unroll
                    for (int i = 0; i < 16; i += kPair ? 2 : 1) {
                        uint32_t l;
                        if constexpr (kPerChannel) l = __ldg(a.enc + (blk * 16 + i) * nsym + (qv[i] & 0xffu)) & 0xffu;
                        else {
                            // (the magic constant is zero in the low bits; its upper bits fall out of the address)
                            uint32_t idx = qv[i] - kMagicBits;
                            if constexpr (kPair) idx += (qv[i + 1] - kMagicBits) << a.bits;
                            asm("ld.shared.u8 %0, [%1];" : "=r"(l) : "r"(len8_addr + idx));
                        }
                        sink.bits += l;
                    }
                } else {
                    uint32_t mul[8], code[8];
                    block_pieces<kPerChannel, kPair>(qv, enc_addr, a.enc, blk * 16, a.bits, mul, code);
                    append_block(sink, mul, code);
                }
            };

            // The thread's blocks in order; `mark(i)` is called where the i-th chunk boundary of the pixel
            // (1 ...) lies before a block.  From skip_blk on two blocks at a time are tested for holding nothing
            // but the modal symbol.
            auto code_blocks = [&](auto &sink, auto first, auto &&mark) {
                constexpr bool kCount = std::is_same<std::decay_t<decltype(sink)>, CountSink>::value;
                if (blk0 >= blk1) return;
                int blk = blk0, bound_i = bound0, bound_blk = bound0 * chunk_blks;
                auto at = [&] {
                    if (blk == bound_blk) { mark(bound_i); ++bound_i; bound_blk += chunk_blks; }
                };
                // blocks up to `end` one by one
                auto one_by_one = [&](int end) {
                    if (blk >= end) return;
                    uint32_t r[16];
                    tmem_ld_32x32b_x16(trow + blk * 16, r);
#pragma unroll 1
                    do {
                        at();
                        code_block(blk, r, sink, first);
                    } while (++blk < end);
                    tmem_ld_wait(r);
                };
                if constexpr (!kCanSkip) one_by_one(blk1);
                else {
                    int plain = min(max(skip_blk, blk), blk1);               // this far without the test
#pragma unroll 1
                    while (true) {
                        if (plain + 2 > blk1) plain = blk1;
                        one_by_one(plain);
                        if (blk >= blk1) break;
#pragma unroll 1
                        while (blk + 2 <= blk1 && bound_blk != blk + 1) {
                            uint32_t r0[16], r1[16];
                            tmem_ld_32x32b_x16(trow + blk * 16, r0);
                            tmem_ld_32x32b_x16(trow + blk * 16 + 16, r1);
                            float4 mid[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) mid[i] = *reinterpret_cast<const float4 *>(s_bias_mid + blk * 16 + 4 * i);
                            tmem_ld_wait(r0);
                            tmem_ld_wait(r1);
                            // farthest of the 32 positions from the modal level (not a number: stays one, fails the test)
                            float far[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                farthest2(far[0], r0[4 * i], r0[4 * i + 1], inv_range, mid[i].x, mid[i].y);
                                farthest2(far[1], r0[4 * i + 2], r0[4 * i + 3], inv_range, mid[i].z, mid[i].w);
                                farthest2(far[2], r1[4 * i], r1[4 * i + 1], inv_range, mid[4 + i].x, mid[4 + i].y);
                                farthest2(far[3], r1[4 * i + 2], r1[4 * i + 3], inv_range, mid[4 + i].z, mid[4 + i].w);
                            }
                            if (!__all_sync(0xffffffffu, (far[0] < pl.skip_dist) & (far[1] < pl.skip_dist) & (far[2] < pl.skip_dist) & (far[3] < pl.skip_dist))) break;
                            at();
                            if constexpr (kCount) sink.bits += 32;             // 32 times the code 0 (one bit)
                            else sink.put_word(0u);
                            blk += 2;
                        }
                        plain = min(blk + 2, blk1);
                    }
                }
            };

            // first pass: code lengths, and with private runs the codes
            unsigned int my_bits;
            [[maybe_unused]] SmemBitWriter<kRunStep> run;
            if constexpr (kRuns) {
                run.init(run_addr, run_end, 0u);
                auto bits_so_far = [&] { return (run.addr - run_addr) / (kRunStep / 32) + (unsigned int)run.pending; };
                code_blocks(run, std::true_type{}, [&](int i) { bound[(i - 1) * 128 + m] = (unsigned short)bits_so_far(); });
                my_bits = bits_so_far();
                if (__any_sync(0xffffffffu, run.addr > run_end) && lane == 0) s_overflow[grp] = n_done + 1;
            } else {
                CountSink count{0u};
                code_blocks(count, std::true_type{}, [&](int i) { bound[(i - 1) * 128 + m] = (unsigned short)count.bits; });
                my_bits = count.bits;
            }
            if constexpr (kHist) {
                if (a.clamped) {
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) n_clamped += __shfl_xor_sync(0xffffffffu, n_clamped, d);
                    if (lane == 0 && n_clamped) atomicAdd(a.clamped, (unsigned long long)n_clamped);
                }
            }
            if (!valid) my_bits = 0;

            // bit offsets: pixel-major, first half before second half.  Each warp scans its own half's bits of
            // its 32 pixels; a pixel's offset is the sum of both halves' prefixes.
            unsigned int inc = my_bits;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned int up = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += up;
            }
            if constexpr (kHalves) xch[half * 128 + m] = ((inc - my_bits) << 12) | my_bits;       // at most 31 * 256 * 12 bits before, 256 * 12 own
            if (lane == 31) s_warp_sums[grp][half][wq] = inc;
            named_bar_sync(bar_id, kGroupThreads);
            const uint32_t theirs = kHalves ? xch[(half ^ 1) * 128 + m] : 0u;
            const unsigned int other = theirs & 0xfffu, pixel_bits = my_bits + other;
            unsigned int before = 0, tile_bits = 0, warp_bits = 0;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const unsigned int sw = s_warp_sums[grp][0][w] + (kHalves ? s_warp_sums[grp][1][w] : 0u);
                if (w < wq) before += sw;
                if (w == wq) warp_bits = sw;
                tile_bits += sw;
            }
            const unsigned int pixel_off = before + (inc - my_bits) + (theirs >> 12);
            const unsigned int my_off = pixel_off + (half ? other : 0u);
            // chunk lengths.  Chunks of several pixels: a chunk ends at the offset of the pixel chunk_pixels
            // further on, which sits in this warp, or is a sum of warp totals.  Several chunks per pixel:
            // from the bits before their boundaries.
            if (a.chunk_pixels > 1) {
                const int cpx = a.chunk_pixels;
                unsigned int chunk_end = 0;
                if (cpx < 32) {
                    const unsigned int further = __shfl_down_sync(0xffffffffu, pixel_off, cpx);
                    chunk_end = (lane + cpx < 32) ? further : before + warp_bits;
                } else {
#pragma unroll
                    for (int w = 0; w < 4; ++w)
                        if (w < wq + (cpx >> 5)) chunk_end += s_warp_sums[grp][0][w] + (kHalves ? s_warp_sums[grp][1][w] : 0u);
                }
                if (valid && half == 0 && (m & (cpx - 1)) == 0) a.chunk_len[p >> (__ffs(cpx) - 1)] = (uint16_t)(chunk_end - pixel_off);
            } else if (valid && half == 0) {
                if (a.splits == 1) a.chunk_len[p] = (uint16_t)pixel_bits;
                else {
                    // start of chunk s in the pixel: a boundary among the second half's blocks counts from my_bits on
                    auto starts = [&](int sc) { return bound[(sc - 1) * 128 + m] + (sc * chunk_blks >= pl.split_blk ? my_bits : 0u); };
                    uint32_t *dst = reinterpret_cast<uint32_t *>(a.chunk_len + a.splits * p);
                    const unsigned int s1 = starts(1);
                    if (a.splits == 2) dst[0] = s1 | ((pixel_bits - s1) << 16);
                    else {
                        const unsigned int s2 = starts(2), s3 = starts(3);
                        dst[0] = s1 | ((s2 - s1) << 16);
                        dst[1] = (s3 - s2) | ((pixel_bits - s3) << 16);
                    }
                }
            }
            const unsigned long long padded = ((unsigned long long)tile_bits + 127ull) & ~127ull;
            if (tg == 0) lookback_publish(a.tile_state, tile, padded);
            const bool staged = padded <= (unsigned long long)pl.staging_bytes * 8ull && !(kRuns && s_overflow[grp] == n_done + 1);
            const bool fits = staged || (kRuns && padded <= (unsigned long long)(pl.staging_bytes + L.run_bytes) * 8ull);    // coded again, where the runs are in the way
            if (kRuns && staged) {                 // the accumulator is free for the tile after next
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_tempty[grp]));
            }
            // place in the staging ring: behind the newest tile, or at the buffer's start if it would not
            // fit before the end
            const unsigned int tile_bytes = fits ? (unsigned int)(padded >> 3) : 0u;
            const unsigned int stg_at = prev_end + tile_bytes > pl.staging_bytes ? 0u : prev_end;
            if (n_done >= 1 && stg_at < prev_end && prev_at < stg_at + tile_bytes) {
                // one warp waits for all (the condition is the same in every thread): warps whose waits end
                // differently would leave the others at the group's barriers
                if (wg == 0) {
                    const bool go = mbar_wait(smem_u32(&s_stg_free[grp][(n_done - 1) % kSlots]), ((n_done - 1) / kSlots) & 1u);
                    if (lane == 0) s_go[grp] = go;
                }
                named_bar_sync(bar_id, kGroupThreads);
                if (!s_go[grp]) { alive = false; break; }
            }
            prev_at = stg_at;
            prev_end = stg_at + tile_bytes;
            const uint32_t tile_addr = stg_addr + stg_at;

            if (staged) {
                // every word below tile_bits / 32 is stored by the writer of its last bit; the last
                // partial word and the padding up to the 128-bit boundary start as zero
                const unsigned int first_open = tile_bits >> 5, end_word = (unsigned int)(padded >> 5);
                if ((unsigned int)tg < end_word - first_open)
                    asm volatile("st.shared.u32 [%0], %1;" ::"r"(tile_addr + (first_open + tg) * 4u), "r"(0u) : "memory");
                if constexpr (kRuns) {
                    // the run's words, shifted to the thread's offset
                    const int sh = (int)(my_off & 31u);
                    const unsigned int n_words = my_bits >> 5;
                    uint32_t dst = tile_addr + (my_off >> 5) * 4u, src = run_addr, prev = 0;
                    const unsigned int most = __reduce_max_sync(0xffffffffu, n_words);
#pragma unroll 2
                    for (unsigned int i = 0; i < most; ++i) {
                        if (i < n_words) {
                            uint32_t w;
                            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w) : "r"(src));
                            asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst), "r"(__funnelshift_r(w, prev, sh)) : "memory");
                            prev = w;
                            src += kRunStep;
                            dst += 4;
                        }
                    }
                    const int rest = valid ? run.pending : 0;
                    const uint32_t last = rest ? run.lo << (32 - rest) : 0u;
                    uint32_t tail = __funnelshift_r(last, prev, sh);
                    if (sh + rest >= 32) {
                        asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst), "r"(tail) : "memory");
                        dst += 4;
                        tail = last << (32 - sh);
                    }
                    named_bar_sync(bar_id, kGroupThreads);      // all full words stored
                    if (tail && valid) asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(dst), "r"(tail) : "memory");
                } else {
                    SmemBitWriter<4> w;
                    w.init(valid ? tile_addr : 0u, valid ? tile_addr + tile_bytes : 0u, valid ? my_off : 0u);
                    code_blocks(w, std::false_type{}, [](int) {});
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&s_tempty[grp]));
                    named_bar_sync(bar_id, kGroupThreads);
                    w.finish();
                }
                if (tg == 0) { s_padded[grp][n_done % kSlots] = (unsigned int)padded; s_stg_at[grp][n_done % kSlots] = stg_at; s_store_cmd[grp][n_done % kSlots] = 1; }
            } else if (kRuns && fits) {
                // a run is longer than the plan allows for, or the tile than the staging buffer
                const unsigned int first_open = tile_bits >> 5, end_word = (unsigned int)(padded >> 5);
                if ((unsigned int)tg < end_word - first_open)
                    asm volatile("st.shared.u32 [%0], %1;" ::"r"(tile_addr + (first_open + tg) * 4u), "r"(0u) : "memory");
                SmemBitWriter<4> w;
                w.init(valid ? tile_addr : 0u, valid ? tile_addr + tile_bytes : 0u, valid ? my_off : 0u);
                w = code_again<kPerChannel, kPair>(w, trow, blk0, blk1, inv_range, top, s_bias, enc_addr, a.enc, a.bits);
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_tempty[grp]));
                named_bar_sync(bar_id, kGroupThreads);
                w.finish();
                if (tg == 0) { s_padded[grp][n_done % kSlots] = (unsigned int)padded; s_stg_at[grp][n_done % kSlots] = stg_at; s_store_cmd[grp][n_done % kSlots] = 1; }
            } else {
                // rare: the tile does not fit -> resolve its position first and pack straight into (zeroed) global memory
                resolve_base(tile, padded);
                named_bar_sync(bar_id, kGroupThreads);
                if (s_write_ok[grp]) {
                    uint4 *z = reinterpret_cast<uint4 *>(a.stream + (s_base[grp] >> 5));
                    for (unsigned int i = tg; i < (unsigned int)(padded >> 7); i += kGroupThreads) z[i] = make_uint4(0u, 0u, 0u, 0u);
                }
                named_bar_sync(bar_id, kGroupThreads);
                GlobalSink g;
                g.on = valid && s_write_ok[grp];
                g.w.init(a.stream, s_base[grp] + my_off);
                code_blocks(g, std::false_type{}, [](int) {});
                if (g.on) g.w.finish();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_tempty[grp]));
                if (tg == 0) {
                    const unsigned long long base = s_base[grp];
                    a.tile_off[tile] = base;
                    if (tile == a.n_tiles - 1) a.tile_off[a.n_tiles] = base + padded;
                    s_store_cmd[grp][n_done % kSlots] = 2;
                }
            }
            // hand the tile to the store warp (a warp's arrival releases its lanes' writes)
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_stg_full[grp][n_done % kSlots]));
            ++n_done;
        }
        if (!alive) {
            if (tg == 0) { tc_dev_set_status(a.status, TC_ERR_TIMEOUT); s_store_cmd[grp][n_done % kSlots] = 3; }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_stg_full[grp][n_done % kSlots]));   // lets the store warp leave
        }
    }

    // ---- teardown ---------------------------------------------------------------------
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

template <bool kPerChannel, bool kDebug, bool kPair, bool kHist, bool kRuns, int kGroups>
__global__ void __launch_bounds__(kThreads, 1) encode_tc_kernel(EncodeArgs a, Plan pl)
{
    encode_tiles<kPerChannel, kDebug, kPair, kHist, kRuns, kGroups>(a, pl, blockIdx.x, gridDim.x);
}

// Several tensors in one launch, each with blocks of its own.  A block's set-up and first tile take 13 us and a launch on a stream
// beside others 3 us of host time, so that a list of small tensors was bound by launches and one of large ones paid the set-up of
// a quarter of the SMs for each: nine tensors of up to 50 000 values 72 -> 33 us, ten 76 -> 34, the 13 narrower layers of a residual
// network at batch 64 143 -> 122, all 16 164 -> 148.
struct EncodeList {
    unsigned int first[kListItems + 1];        // block that each item starts at; past the last item 2^32 - 1
    struct { EncodeArgs a; Plan pl; } item[kListItems];
};
template <bool kPerChannel, bool kPair, bool kRuns, int kGroups>
__global__ void __launch_bounds__(kThreads, 1) encode_tc_list_kernel(const __grid_constant__ EncodeList list)
{
    int i = 0;
    while (blockIdx.x >= list.first[i + 1]) ++i;
    encode_tiles<kPerChannel, false, kPair, false, kRuns, kGroups>(list.item[i].a, list.item[i].pl, blockIdx.x - list.first[i],
                                                          min(list.first[i + 1], gridDim.x) - list.first[i]);
}

}  // namespace

// For the tests: what the issuing warp does when its wait number `fails` (0 ...; none if negative) runs out, one event an entry: 100 + stage (a panel's
// products and its stage handed back), 200 + accumulator (handed on), 300 (the wait for all of it), -1 (the wait that ran out).  The number of events.
extern "C" int tc_issue_events(int groups, long long tiles, int panels, int stages, int fails, int32_t *events, int room)
{
    int n = 0;
    auto put = [&](int32_t e) { if (n < room) events[n] = e; ++n; };
    auto wait = [&] { if (fails-- != 0) return true; put(-1); return false; };
    auto on_barrier = [&](int, uint32_t) { return wait(); };
    auto panel = [&](int, int s, bool issue) { if (issue) put(100 + s); };
    auto done = [&](int acc) { put(200 + acc); };
    auto drain = [&] { put(300); };
    if (groups == 4) issue_tiles<4, 1>(tiles, panels, stages, wait, on_barrier, on_barrier, panel, done, drain);
    else issue_tiles<2, 1>(tiles, panels, stages, wait, on_barrier, on_barrier, panel, done, drain);
    return n;
}

// Four groups: up to as many coefficients as let their accumulators fit tensor memory, and where a block has more tiles than two, one below 64
// coefficients, since few tiles are coded sooner by eight warps each than by four; 16 coefficients are not split between warps and take four always
// (us with two and with four groups, a tile a block: 128x16x16 at 96 coefficients 10.6 and 12.4, 80x28x28 x 3 10.4 and 12.4, 96x7x8 x 6 at 16 10.3 and 9.3;
// two: 128x16x16 x 124 16.5 and 18.2; three: 16x12x7 x 528 12.3 and 11.8; five: 128x14x14 x 432 23.2 and 21.4.  Four's time over two's, 300 drawn
// layers: 80 coefficients and more 1.06, 1.05, 0.98 at one, two and three tiles; 64 1.04, 1.01, 1.01; 32 and 48 1.01, 0.99, 0.98; 16 0.99, 0.97, 0.97).
// Also where their buffers leave no room for private runs, which two would have: dense codes of 128 coefficients of wide layers (256x14x14 x 1500 at
// 6 bits 73.4 and 74.0, at 8 bits 80.0 and 77.3, 240x14x14 x 1500 at 5 bits 72.6 and 69.1; four tiles a block 240x14x14 x 300 23.2 and 24.9).
constexpr int kFourGroupsCoefs = 128;

// What a launch does with the shared memory that the basis leaves, from the code lengths to expect of
// the model's coefficients (a code without a one-bit symbol: b bits for each).  A tile's size varies
// by a few per cent about its mean, a thread's run by its symbols that are not the zero level.  A tile
// that breaks the estimate is coded once more, over the staging buffer and the runs behind it (256x14x14 x 4096, 4 bits, maps of
// twice the calibration's spread: 243 us; 348 when such tiles went straight into global memory, as those still do that
// fit neither).
// Preferred, in this order: symbol pairs before single symbols, private runs before two passes, eight
// ring stages before six.
static Plan make_plan(const tc_ctx *ctx, const EncodeArgs &a)
{
    const int n_blk = a.k / 16;
    const bool few = a.n_tiles <= (long long)std::min(2, a.k / 32) * ctx->sm_count;
    const bool four_groups = a.k <= kFourGroupsCoefs && !a.hist && !a.dbg_coef && !a.dbg_sym && (a.epilogue_groups ? a.epilogue_groups == 4 : !few);
    const bool modal = a.groups == 1 && a.modal >= 0;
    auto blk_bits = [&](int b) { return modal || a.groups != 1 ? a.blk_bits[b] : std::max(a.blk_bits[b], 16.f * a.bits); };
    Plan best{};
    // The test for modal blocks adds the bias up differently from the quantiser: the two positions differ by the rounding of s_bias_mid and
    // of the two results, together at most 2^-24 of the largest bias plus three.  Four times that is kept clear, besides
    // 0.001 of a level.  (At 8 bits and a mean of a thousand ranges that is 0.06 of a level; the 0.001 alone let symbols
    // next to a rounding boundary pass for the modal one there.  Here and not from s_bias in the kernel, which cost the coder
    // 2 to 3 %: 64x56x56 x 256 at 8 bits 107 -> 110 us.)
    best.skip_dist = 0.499f / (float)((1 << a.bits) - 1) - (a.max_bias + 1.f) * 2.4e-7f;
    // A test of 32 coefficients x 32 pixels pays from a success in three on: fewer than about one other
    // symbol expected in it.
    best.skip_blk = n_blk;
    while (modal && best.skip_blk > 0 && 64.f * a.blk_odd[best.skip_blk - 1] < 1.2f) --best.skip_blk;
    // blocks of the two threads of a pixel: equal work, a coded block counted as three passed over
    auto cost = [&](int b0, int b1) { return 3 * std::max(0, std::min(b1, best.skip_blk) - b0) + (b1 - std::max(b0, std::min(b1, best.skip_blk))); };
    best.groups = four_groups ? 4 : 2;
    best.split_blk = best.groups == 4 ? n_blk : 1;
    for (int x = 2; x <= n_blk && best.groups == 2; ++x)
        if (std::max(cost(0, x), cost(x, n_blk)) < std::max(cost(0, best.split_blk), cost(best.split_blk, n_blk))) best.split_blk = x;
    double tile_bits = 0.0;
    int want_words[2];
    for (int h = 0; h < 2; ++h) {
        double bits = 0.0, odd = 0.0;
        const int b0 = h ? best.split_blk : 0, b1 = h ? n_blk : best.split_blk;
        for (int b = b0; b < b1; ++b) { bits += blk_bits(b); odd += a.blk_odd[b]; }
        tile_bits += TC_TILE_PIXELS * bits;
        // (the largest of 10^5 threads' runs: about 10 standard deviations' worth of other symbols)
        want_words[h] = b1 > b0 ? std::min((int)((bits + 11.0 * std::sqrt(odd)) / 32.0) + 2, (b1 - b0) * 6) : 0;
    }
    const uint32_t want_staging = (uint32_t)(1.08 * tile_bits / 8.0) + 128u;
    const int budget = ctx->max_smem_optin - kStaticSmem;
    for (int t = 0; t < 8; ++t) {
        Plan pl = best;
        const bool pair = !(t & 4), runs = !(t & 2);
        if (pair && (a.groups != 1 || a.bits > kPairMaxBits)) continue;
        pl.stages = (t & 1) ? 6 : 8;
        pl.entries = a.groups != 1 ? 0 : pair ? 1 << (2 * a.bits) : 1 << a.bits;
        for (int h = 0; h < 2; ++h) pl.run_words[h] = runs ? want_words[h] : 0;
        pl.staging_bytes = 0;
        const long long left = (long long)budget - smem_layout(a.c, a.k, pl).total;
        const long long per_group = (left / pl.groups) & ~15ll;
        if (per_group < 4096 || (per_group < (long long)want_staging && t != 7)) continue;
        pl.staging_bytes = (uint32_t)std::min<long long>(per_group, kMaxStagingBytes);
        return pl;
    }
    best.staging_bytes = 0;
    return best;
}

static bool coded_in_pairs(const EncodeArgs &a, const Plan &pl) { return a.groups == 1 && pl.entries > (1 << a.bits); }

bool tc_encode_tc_supported(const tc_ctx *ctx, const EncodeArgs &a)
{
    // K <= C leading components (PCA truncation): K is the N dimension of the MMA
    if (a.c % 16 != 0 || a.k % 16 != 0 || a.k < 16 || a.k > a.c || a.c > 256 || a.hw % 4 != 0) return false;
    // the loaders copy groups of four pixels with 8-byte cp.async: the tensor must start on an 8-byte boundary
    if (((uintptr_t)a.x & 7u) != 0) return false;
    // chunks are whole blocks of 16 coefficients
    if (a.splits != 1 && !(a.splits == 2 && a.k % 32 == 0) && !(a.splits == 4 && a.k % 64 == 0 && a.chunk_pixels == 1)) return false;
    if (a.groups != 1 && a.groups != a.k) return false;
    if (!a.basis_core) return false;
    return make_plan(ctx, a).staging_bytes > 0;
}

template <bool kPerChannel, bool kPair, bool kRuns>
static void (*pick_kernel(bool debug, bool hist, int groups))(EncodeArgs, Plan)
{
    if constexpr (!kPerChannel)
        if (hist) return encode_tc_kernel<false, false, kPair, true, kRuns, 2>;
    if (debug) return encode_tc_kernel<kPerChannel, true, kPair, false, kRuns, 2>;
    return groups == 4 ? encode_tc_kernel<kPerChannel, false, kPair, false, kRuns, 4> : encode_tc_kernel<kPerChannel, false, kPair, false, kRuns, 2>;
}

// Which kernel codes the tensor: bit 0 a table per channel, bit 1 symbol pairs, bit 2 private runs, bit 3 four groups.
static int kernel_class(const EncodeArgs &a, const Plan &pl)
{
    const bool per_channel = a.groups != 1;
    return (per_channel ? 1 : 0) | (coded_in_pairs(a, pl) ? 2 : 0) | (pl.run_words[0] > 0 ? 4 : 0) | (pl.groups == 4 ? kEncodeFourGroups : 0);
}
template <int kGroups>
static const void *list_kernel(int which)
{
    switch (which & 7) {
    case 1: return (const void *)encode_tc_list_kernel<true, false, false, kGroups>;
    case 5: return (const void *)encode_tc_list_kernel<true, false, true, kGroups>;
    case 2: return (const void *)encode_tc_list_kernel<false, true, false, kGroups>;
    case 6: return (const void *)encode_tc_list_kernel<false, true, true, kGroups>;
    case 4: return (const void *)encode_tc_list_kernel<false, false, true, kGroups>;
    default: return (const void *)encode_tc_list_kernel<false, false, false, kGroups>;
    }
}

constexpr double kShortListUs = 18.0, kSharedListUs = 40.0;       // see tc_encode_tc_list_classes

// us that a tile takes a block: 1.35 with 64 coefficients at 1.1 bits each, 2.0 with 128 at 1.9, 1.75 with 96 at 2.8 (four groups), 3.95
// with 256 at 1.1, 6.9 at 4.1 (8 to 130 tiles a block, after the first)
double tc_encode_tc_tile_us(const EncodeArgs &a, int which)
{
    double bits = 0.0;
    for (int b = 0; b < a.k / 16; ++b) bits += a.blk_bits[b];
    return which & kEncodeFourGroups ? 0.8 + 0.0075 * a.k + 0.0022 * bits : std::max(1.2, 0.011 * a.k) + 0.004 * bits;
}

// Narrow tensors code faster with four groups a block, but in a short list a block gets a tile or two (fifteen small tensors
// of 16 to 144 channels, 25 us of work), and where wider ones take a launch anyway theirs as well costs more than that
// (47.6 -> 54.5 us in two launches; eleven of 16 to 144, 8 us of work, 25.4 -> 38.8; 16 layers, 100 us of work: 130.6 -> 124.3).
void tc_encode_tc_list_classes(const tc_ctx *ctx, std::vector<EncodeArgs> &args, std::vector<int> &kind)
{
    double all_us = 0.0, class_us[kEncodeClasses] = {};
    for (size_t i = 0; i < args.size(); ++i) {
        if (kind[i] < 0) continue;
        args[i].epilogue_groups = 4;
        kind[i] = kernel_class(args[i], make_plan(ctx, args[i]));
        const double us = (double)args[i].n_tiles * tc_encode_tc_tile_us(args[i], kind[i]) / ctx->sm_count;
        class_us[kind[i]] += us;
        all_us += us;
    }
    for (size_t i = 0; i < args.size(); ++i) {
        if (kind[i] < 0 || !(kind[i] & kEncodeFourGroups) || (all_us > kShortListUs && class_us[kind[i]] > kSharedListUs)) continue;
        args[i].epilogue_groups = 2;
        const int two = kernel_class(args[i], make_plan(ctx, args[i]));        // (not the same one less a bit: there is more room)
        if (all_us <= kShortListUs || (class_us[two] > 0.0 && class_us[two] + class_us[kind[i]] <= kSharedListUs)) kind[i] = two;
        else args[i].epilogue_groups = 4;
    }
}

// For the tests: the classes of a list of `n` tensors (1: a call with one tensor), each of `tiles` tiles and with `coef_bits` expected of each coefficient,
// on a device of `sm_count` SMs and `smem` bytes of shared memory a block.
extern "C" void tc_encode_classes(int n, const int *c, const int *k, const int *bits, const int *tables, const long long *tiles, const float *coef_bits, int sm_count,
                                  int smem, int *out)
{
    tc_ctx ctx;
    ctx.sm_count = sm_count;
    ctx.max_smem_optin = smem;
    std::vector<EncodeArgs> args(n);
    std::vector<std::vector<float>> blk_bits(n), blk_odd(n);
    std::vector<int> kind(n, 0);
    for (int i = 0; i < n; ++i) {
        EncodeArgs &a = args[i];
        a.c = c[i]; a.k = k[i]; a.bits = bits[i]; a.groups = tables[i]; a.n_tiles = tiles[i]; a.modal = 0;
        blk_bits[i].assign(k[i] / 16, 16.f * coef_bits[i]);
        blk_odd[i].assign(k[i] / 16, 16.f * std::min(1.f, coef_bits[i] - 1.f));
        a.blk_bits = blk_bits[i].data(); a.blk_odd = blk_odd[i].data();
    }
    if (n > 1) tc_encode_tc_list_classes(&ctx, args, kind);
    else kind[0] = kernel_class(args[0], make_plan(&ctx, args[0]));
    std::copy(kind.begin(), kind.end(), out);
}

// Encodes tensors of one class (tc_encode_tc_list_classes) on `sms` SMs, in list_launches launches (40 of 128x14x14 x 32 in
// two of 20 each: 57 us, in one of 32 and one of 8: 62).
tc_status tc_launch_encode_tc_list(const tc_ctx *ctx, const std::vector<EncodeArgs> &tensors, int sms, cudaStream_t s)
{
    const size_t launches = list_launches(tensors.size(), sms);
    for (size_t r = 0; r < launches; ++r) {
        const int n = (int)((tensors.size() - r + launches - 1) / launches);
        EncodeList list;
        std::vector<ListWork> work(n);
        uint32_t smem = 0;
        int which = 0;
        for (int i = 0; i < n; ++i) {
            const EncodeArgs &a = tensors[r + i * launches];
            list.item[i].a = a;
            list.item[i].pl = make_plan(ctx, a);
            which = kernel_class(a, list.item[i].pl);
            smem = std::max(smem, smem_layout(a.c, a.k, list.item[i].pl).total);
            work[i] = {a.n_tiles, tc_encode_tc_tile_us(a, which), 1};
        }
        deal_blocks(work, sms);
        unsigned int blocks = 0;
        for (int i = 0; i <= kListItems; ++i) {
            list.first[i] = i <= n ? blocks : ~0u;
            if (i < n) blocks += (unsigned int)work[i].blocks;
        }
        list.first[n] = ~0u;
        const void *kernel = which & kEncodeFourGroups ? list_kernel<4>(which) : list_kernel<2>(which);
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) { cudaGetLastError(); return TC_ERR_CUDA; }
        void *params[] = {&list};
        // cooperative, as for one tensor: the blocks of a tensor look back at one another
        if (cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(kThreads), params, smem, s) != cudaSuccess) { cudaGetLastError(); return TC_ERR_CUDA; }
    }
    return TC_OK;
}

tc_status tc_launch_encode_tc(const tc_ctx *ctx, const EncodeArgs &a, cudaStream_t s)
{
    if (a.n_tiles <= 0) return TC_OK;
    const bool per_channel = a.groups != 1, debug = a.dbg_coef || a.dbg_sym;
    if (a.hist && (per_channel || debug)) return TC_ERR_UNSUPPORTED;      // statistics run with a per-layer table
    Plan pl = make_plan(ctx, a);
    if (pl.staging_bytes == 0) return TC_ERR_UNSUPPORTED;
    const bool pair = coded_in_pairs(a, pl), runs = pl.run_words[0] > 0;
    const SmemLayout l = smem_layout(a.c, a.k, pl);
    void (*kernel)(EncodeArgs, Plan) = per_channel ? (runs ? pick_kernel<true, false, true>(debug, false, pl.groups) : pick_kernel<true, false, false>(debug, false, pl.groups))
                                     : pair        ? (runs ? pick_kernel<false, true, true>(debug, a.hist, pl.groups) : pick_kernel<false, true, false>(debug, a.hist, pl.groups))
                                                   : (runs ? pick_kernel<false, false, true>(debug, a.hist, pl.groups) : pick_kernel<false, false, false>(debug, a.hist, pl.groups));
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.total) != cudaSuccess)
        return TC_ERR_CUDA;
    const unsigned int grid = (unsigned int)((a.n_tiles < ctx->sm_count) ? a.n_tiles : ctx->sm_count);
    EncodeArgs args = a;
    void *params[] = {&args, &pl};
    // cooperative launch: the grid must be co-resident, which is what makes the look-back safe (launched early as well it
    // started no sooner)
    const cudaError_t err = cudaLaunchCooperativeKernel((void *)kernel, dim3(grid), dim3(kThreads), params, l.total, s);
    if (err != cudaSuccess) {
        if (getenv("TC_VERBOSE")) fprintf(stderr, "tc: encode launch failed: %s\n", cudaGetErrorString(err));
        cudaGetLastError();
        return TC_ERR_CUDA;
    }
    return TC_OK;
}
