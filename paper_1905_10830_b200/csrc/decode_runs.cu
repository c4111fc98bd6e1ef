// Fused tensor-core decode for bf16 tensors with a per-layer code table (Section 3: VLD, inverse
// quantiser, inverse transform) whose work follows the information in the stream.
//
// After the PCA most coefficients of a pixel quantise to one symbol -- the level nearest zero --
// and the Huffman code gives that symbol the one-bit code 0 (Section 3.1, "Variable length
// coding"; Appendix E: the tail channels collapse to a single value).  A run of such symbols is
// a run of zero bits, so a decoder thread counts leading zeros and jumps over the whole run at
// once; only the other symbols cost a table lookup and a store.  The operand of the inverse
// projection is therefore filled first with the value of the modal symbol (16-byte stores) and
// the decoded symbols are then written into it one by one.
//
// One persistent block per SM.  Warp roles:
//   warps 0-15         VLD groups of as many warps as a tile has chunks for -- eight with two chunks per
//                      pixel, four with one, two with a chunk of two pixels -- on tiles of 128 pixels in
//                      turn, each group with its own operand buffer (all K coefficients of the tile,
//                      K-major).  One or two threads per pixel walk the pixel's chunks.  A group's time
//                      per tile is the latency of its chunks' symbols, so the groups in flight set the
//                      rate: with two groups whatever their size 64x56x56 x 64 took 62 us, with eight 24.
//   warps 16-23        epilogue, four warps on each accumulator: TMEM -> registers,
//                      x_hat = step * acc + bias, round to bf16, NCHW stores (the accumulator is held
//                      transposed: lane = channel)
//   warp 24            one thread issues the tcgen05.mma of the work items, a tile's blocks of 128 channels:
//                      D[c][pixel] = T[j][c] * (Q[pixel][j] - center)
// The transposed basis is the A operand and lives in TENSOR memory, not in shared memory: each
// block of 128 channels takes K / 2 columns (two bf16 per column), 256 columns at C = K = 256,
// loaded once per block with tcgen05.st.  That leaves shared memory to the symbols -- two whole
// tiles in flight, 128 KB at K = 256 -- and takes the basis off the MMA's shared-memory reads.
// The other 256 columns hold two accumulators of 128 pixels, so that the epilogue of one item overlaps the
// MMAs of the next.
// The operand is handed back in panels of 128 coefficients: the MMA thread commits a barrier per
// panel, and a VLD thread of the group's next tile waits only for the panels that it writes.
//
// What bounds it is the VLD groups' instructions and their chains (256x14x14 x 4096 at 4 bits: 139 us with the products and the stores
// left out, 160 in all; 219 before the items, stores and registers took their present form).  Every warp takes its turn at the issue
// slots, an instruction in about twelve cycles, so that the MMA warp's loop is unrolled; and what does not fit the registers goes to local
// memory and comes back from L2 (shared memory leaves the L1 no room): hence the split of the registers below.
//
// A tile whose stream is dense (more than kDenseBits128 / 128 bits per symbol) gains nothing
// from run skipping; its threads then decode symbol by symbol, eight symbols per 16-byte store.
#include <algorithm>

#include "device_utils.cuh"
#include "sm100_ptx.cuh"

namespace {

using namespace tcdev;
using namespace sm100;

constexpr int kVldWarps = 16, kMaxGroups = 8, kEpiWarp0 = kVldWarps, kMmaWarp = kEpiWarp0 + 8;
constexpr int kThreads = (kMmaWarp + 4) * 32;                  // the MMA warp is one of a warpgroup of four, which leave registers to the VLD groups
constexpr int kTmemCols = 512;
constexpr int kAccBase = 256, kAccCols = 128;                 // two accumulators behind the basis columns
// Coefficients per hand-over panel.  A commit keeps the issuing warp for some 400 cycles: with eight panels of 32 (and
// a commit an item) VLD threads waited no less, and the commits held up the MMAs.
constexpr int kPanelK = 128;
constexpr int kMaxPanels = 2;                                 // K <= 256
constexpr uint32_t kRunGuard = 0x800u;                        // bit 11 set: at most 20 zero bits are skipped per step (20 + 12 <= 32: one refill per step)
constexpr int kDenseBits128 = 224;                            // tiles above 1.75 bits per symbol are decoded symbol by symbol
// A chunk that starts inside a staged segment is read for at most (symbols of the chunk) x 12
// bits, whatever the bits say; the slack after the last buffer keeps those reads inside the
// block's shared memory even for a corrupt stream (the buffers lie back to back).
constexpr int kStreamSlack = 1024;
constexpr int kStaticSmem = 1536;                             // room for the kernel's static shared variables
constexpr int kTrWarpBytes = 4096;                            // epilogue block of one warp: 16 channel rows x 128 pixels
// Named barriers.  Hand-overs between warps that both run ordinary instructions use them instead
// of mbarriers: the waiting side is parked by the hardware, whereas a warp polling an mbarrier
// keeps issuing and takes issue slots from the warps that work.  (mbarriers remain where the
// tensor core signals: accumulator ready, operand panel consumed.)
constexpr int kBarGroup = 1;                                  // + group: the VLD threads of a group, once per tile
constexpr int kBarAccFree = kBarGroup + kMaxGroups;           // + accumulator: drained, epilogue warps -> MMA warp
constexpr int kBarBasis = kBarAccFree + 2;                    // basis in tensor memory, epilogue warps -> MMA warp, once
constexpr int kBarEpi = kBarAccFree + 3;                      // + accumulator: ready, polling epilogue warp -> its other three

struct SmemLayout {
    uint32_t lut, opnd, tbuf, sbuf, total;
    uint32_t opnd_bytes;                                      // one operand buffer (one per VLD group)
    uint32_t stream_buf;                                      // bytes per staged stream buffer (two per group; 0: does not fit)
    int groups;                                               // VLD groups
    int mode;                                                 // how the tensor's values leave (see store_mode)
};
enum { kRows16, kRows8, kRowsAny, kMaps };

// group_warps: warps of a VLD group.  As many groups as warps and shared memory allow beside stream
// buffers of `want_bytes`, what a tile's segment is expected to take (two groups: for what is left, at least 4 KB).  A segment
// that does not fit its buffer is read from global memory word by word, which costs more than a group less: with room
// for 2.5 bits per symbol whatever the rate, 512 maps of 28x28 at 8 bits (4.8 to 4.3 bits per value) took 115 us at
// 128 channels, 186 at 176 and 200 at 192; sized by the rate 95, 153 and 163, and 256 maps of 64x56x56 121 -> 101.
inline SmemLayout smem_layout(int k, int lut_entries, int group_warps, uint32_t want_bytes, int mode, int budget)
{
    SmemLayout l;
    l.lut = 0;                                                // 32-bit entries: bf16(symbol - center) << 16 | length
    l.opnd = ((uint32_t)lut_entries * 4u + 1023u) & ~1023u;
    l.opnd_bytes = (uint32_t)k * TC_TILE_PIXELS * 2;
    const int most = kVldWarps / group_warps < kMaxGroups ? kVldWarps / group_warps : kMaxGroups;
    l.mode = mode;
    l.stream_buf = 0;
    l.total = 0;
    for (l.groups = most; l.groups >= 2; --l.groups) {
        l.tbuf = l.opnd + (uint32_t)l.groups * l.opnd_bytes;
        l.sbuf = l.tbuf + (mode != kRows16 ? 8u * kTrWarpBytes : 0u);
        const long long left = (long long)budget - l.sbuf - kStreamSlack;
        const long long room = (left / (2ll * l.groups)) & ~127ll;
        if (room < 4096 || (room < (long long)want_bytes && l.groups > 2)) continue;
        l.stream_buf = (uint32_t)std::min(room, std::max(16384ll, ((long long)want_bytes + 127) & ~127ll));
        l.total = l.sbuf + 2u * (uint32_t)l.groups * l.stream_buf + kStreamSlack;
        break;
    }
    if (l.groups < 2) l.groups = 2;
    return l;
}

// Threads of a VLD group: one per chunk, or two per pixel with more than one chunk per pixel.
__host__ __device__ inline int group_work(int splits, int chunk_pixels)
{
    return chunk_pixels > 1 ? TC_TILE_PIXELS / chunk_pixels : TC_TILE_PIXELS * (splits >= 2 ? 2 : 1);
}

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_u16(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// MSB-first reader with a 64-bit window hi:lo (left-aligned) and one word of look-ahead.  `used`
// counts, in its low byte, the bits taken since the window was last moved on by a word; table
// entries (symbol << 8 | length) are added to it and fed to the funnel shifts as they are (the
// shifts take their amount modulo 32, lengths are at most 12).  refill() moves the window on by
// one word when 32 bits or more have been taken; a caller that takes at most 32 bits between two
// refills always sees at least 32 valid bits after one.
// kShared: the words lie in shared memory (a staged segment, with readable slack behind it);
// otherwise in global memory, where words at or past `end` read as zero.
template <bool kShared>
struct BitReader {
    uint32_t hi, lo, ahead, used;
    uint32_t next_addr;               // shared: address of the word after `ahead`
    const uint32_t *next, *end;       // global
    uint32_t origin;                  // shared: bit address (shared address * 8) init() was given; global: that position modulo 32
    uint32_t words;                   // global: words the window has moved on by

    __device__ __forceinline__ uint32_t fetch()
    {
        uint32_t w;
        if constexpr (kShared) { w = lds_u32(next_addr); next_addr += 4; }
        else { w = stream_word(next, end); ++next; }
        return w;
    }
    // kShared: `base_addr` is the shared address of the segment; else `base` / `end_word` delimit it
    __device__ __forceinline__ void init(uint32_t base_addr, const uint32_t *base, const uint32_t *end_word, uint32_t bitpos)
    {
        if constexpr (kShared) { next_addr = base_addr + (bitpos >> 5) * 4u; origin = next_addr * 8u + (bitpos & 31u); }
        else { next = base + (bitpos >> 5); end = end_word; origin = bitpos & 31u; }
        const uint32_t w0 = fetch(), w1 = fetch();
        ahead = fetch();
        const uint32_t sh = bitpos & 31u;
        hi = __funnelshift_l(w1, w0, sh);
        lo = w1 << sh;
        used = sh;
        words = 0;
    }
    __device__ __forceinline__ void idle()
    {
        hi = lo = ahead = used = origin = words = 0;
        next_addr = 0; next = end = nullptr;
    }
    // `entry`: a bit count below 32, or a table entry with the count in its low byte (what lies
    // above only reaches bits of `used` that nothing reads)
    __device__ __forceinline__ void take(uint32_t entry)
    {
        hi = __funnelshift_l(lo, hi, entry);
        lo = __funnelshift_l(0u, lo, entry);
        used += entry;
    }
    __device__ __forceinline__ void refill()
    {
        // with c = used - 32 bits of the next word's span already taken, the window gains `ahead`
        // behind its 64 - used valid bits: hi |= ahead >> (32 - c), lo |= ahead << c (the shifts take
        // their amount modulo 32)
        if constexpr (kShared) {
            asm volatile(
                "{\n\t.reg .pred p;\n\t.reg .b32 t, u;\n\t"
                "and.b32 t, %3, 32;\n\t"
                "setp.ne.u32 p, t, 0;\n\t"
                "shf.l.wrap.b32 t, %2, 0, %3;\n\t"
                "shf.l.wrap.b32 u, 0, %2, %3;\n\t"
                "@p or.b32 %0, %0, t;\n\t"
                "@p or.b32 %1, %1, u;\n\t"
                "@p add.u32 %3, %3, -32;\n\t"
                "@p ld.shared.u32 %2, [%4];\n\t"
                "@p add.u32 %4, %4, 4;\n\t}"
                : "+r"(hi), "+r"(lo), "+r"(ahead), "+r"(used), "+r"(next_addr));
        } else if (used & 32u) {
            hi |= __funnelshift_l(ahead, 0u, used);
            lo |= __funnelshift_l(0u, ahead, used);
            used -= 32u;
            ahead = fetch();
            ++words;
        }
    }
    // bits taken since init()
    __device__ __forceinline__ uint32_t consumed() const
    {
        if constexpr (kShared) return (next_addr - 12u) * 8u + (used & 0xffu) - origin;   // the window starts three words behind next_addr
        else return words * 32u + (used & 0xffu) - origin;
    }
};

// How channel rows leave.  What a store costs is the lines of 128 bytes that it touches, 6.5 cycles each an SM, unless the store right
// before it touched them too: 256x14x14 x 4096 written as 64 bytes of four rows an instruction takes 188 us and nothing else (what the
// decoder did), 256 bytes of one row 109; 64x56x56 x 1024 as 64 bytes of eight rows 150, the same with the four pieces of a row one
// after the other 73.  So a warp stores all 128 pixels of its 16 channels at a time:
//   kRows16: every group of eight pixels is 16-byte aligned and inside one image: straight from the registers, 16 bytes a thread and
//            64 of eight rows an instruction, a row's four pieces in succession;
//   kRows8:  the same of groups of four: through a block of the warp in shared memory, a row an instruction, 8 bytes a thread;
//   kRowsAny: rows that start anywhere (H*W no multiple of 4, an unaligned tensor): through the block, a pixel a thread, a row in four
//            instructions in succession;
//   kMaps:   maps of up to four pixels: their rows are all over memory, but 32 channels of a map lie in a line or two: a channel a thread (two where
//            a map is a pixel), a map or a pixel an instruction.  As rows they took several times as long (us as rows and so: 208x1x1 x 229248, 96
//            coefficients, 444 and 50; 112x1x2 x 54144 65 and 23; 256x1x3 x 32720 129 and 40; 160x2x2 x 40800 67 and 46).  Five pixels leave faster
//            as rows, as do 16 channels, of which a line holds several maps (16x1x2 x 46848: rows 21, so 23).
constexpr int kSmallMap = 4;
inline int store_mode(const DecodeArgs &a)
{
    if (a.hw <= kSmallMap && a.c > 16) return kMaps;
    if ((a.hw & 3) != 0 || ((uintptr_t)a.xhat & 7u) != 0) return kRowsAny;
    return (a.hw & 7) == 0 && ((uintptr_t)a.xhat & 15u) == 0 ? kRows16 : kRows8;
}
// The accumulator is read as matrix fragments: of 32 columns thread q of four gets 8 g + 2 q + {0, 1}, g = 0 ... 3.  Which pixel a column
// stands for is free (the order of the operand's rows); so that a thread's columns are consecutive pixels, they are
// pixels 8 q + 2 g + {0, 1}.
__device__ __forceinline__ uint32_t column_of(uint32_t p) { return (p & ~31u) | ((p & 6u) << 2) | ((p >> 2) & 6u) | (p & 1u); }
__device__ __forceinline__ uint32_t pixel_of(uint32_t n) { return (n & ~31u) | ((n & 6u) << 2) | ((n >> 2) & 6u) | (n & 1u); }

// two accumulator values -> two bf16: x_hat = step * acc + bias (one packed fused multiply-add)
template <bool kRelu>
__device__ __forceinline__ uint32_t decoded_pair(uint32_t x0, uint32_t x1, float step, float bias)
{
    float f0, f1;
    asm("{\n\t.reg .b64 v, s, b;\n\t"
        "mov.b64 v, {%2, %3};\n\t"
        "mov.b64 s, {%4, %4};\n\t"
        "mov.b64 b, {%5, %5};\n\t"
        "fma.rn.f32x2 v, v, s, b;\n\t"
        "mov.b64 {%0, %1}, v;\n\t}"
        : "=f"(f0), "=f"(f1) : "r"(x0), "r"(x1), "f"(step), "f"(bias));
    if constexpr (kRelu) { f0 = fmaxf(f0, 0.f); f1 = fmaxf(f1, 0.f); }   // the layer's non-linearity, when it follows the decoder
    const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// The thread's index, read anew: what a role derives from its own reading is not worked out ahead of the other roles and kept through them (with
// registers as short as here such values went to local memory, that is to L2: L1 is what shared memory leaves of it).
__device__ __forceinline__ int own_tid()
{
    int t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
}

// `block` of `blocks` that share the tensor's tiles.
template <bool kRelu>
__device__ __forceinline__ void decode_tiles(const DecodeArgs &a, const SmemLayout &L, unsigned int block, unsigned int blocks)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_empty[kMaxGroups][kMaxPanels], s_bfull[kMaxGroups], s_tfull[2], s_drained;
    __shared__ uint32_t s_tmem_base;
    // [group][tile parity][thread set][warp]: bits per warp, for the start positions.  Two copies: a warp
    // that is done with its tile early writes the next tile's sum while a slower warp may still
    // be reading this tile's; the group's barrier (one per tile) only orders the write after next.
    __shared__ unsigned int s_wsum[kMaxGroups][2][2][4];

    // (taken from lane 0: the compiler knows that the branches between the roles are the same for a whole warp)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int lut_size = 1 << a.lut_bits;
    const int S = a.splits, cp = a.chunk_pixels;
    const int tpp = S >= 2 ? 2 : 1;                            // threads per pixel
    const int chunks_per_thread = S / tpp;                     // 1, or 2 with four chunks per pixel
    const int n_work = group_work(S, cp);                      // threads of a group that own chunks
    const int group_warps = (n_work + 31) / 32, n_thr = group_warps * 32;     // whole warps take part in the group's barriers
    const int G = L.groups;
    const uint32_t lut_addr = smem_u32(smem + L.lut);
    const uint32_t opnd_addr = smem_u32(smem + L.opnd);
    const int n_blocks = (a.c + 127) / 128;                    // blocks of 128 channels
    const int items = n_blocks;                                // work items per tile: its channel blocks

    // ---- set-up ---------------------------------------------------------------------
    chain_next();
    if (tid < G * (kMaxPanels + 1)) {
        const int g = tid / (kMaxPanels + 1), p = tid - g * (kMaxPanels + 1);
        if (p < kMaxPanels) mbar_init(smem_u32(&s_empty[g][p]), 1);                     // the commit of the tile's last item
        else mbar_init(smem_u32(&s_bfull[g]), (uint32_t)group_warps);                   // operand complete: one arrival per warp
        if (tid < 2) mbar_init(smem_u32(&s_tfull[tid]), 1);
        if (tid == 2) mbar_init(smem_u32(&s_drained), 1);
        mbar_fence_init();
    }
    if (warp == kMmaWarp) { tmem_alloc(smem_u32(&s_tmem_base), kTmemCols); tmem_relinquish(); }
    {
        // per-layer table: bf16(symbol - center) << 16 | code length
        uint32_t *s_lut = reinterpret_cast<uint32_t *>(smem + L.lut);
#pragma unroll 5
        for (int i = tid; i < lut_size; i += kThreads) {
            const uint32_t e = __ldg(a.lut32 + i);
            const float f = (float)((int)((e >> 8) & 0xffu) - a.center);
            s_lut[i] = (__float_as_uint(f) & 0xffff0000u) | (e & 0xffu);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, s_tmem_base, 0);
    if (warp >= kEpiWarp0 && warp < kMmaWarp) {
        // Transposed basis -> tensor memory: row c of block b (channel 128 b + c) goes to lane c,
        // its K coefficients, two per 32-bit column in memory order, to columns b K/2 ... of the A
        // operand.  A warp reaches the 32 lanes of its quarter; rows past C are zero (their outputs
        // are never stored).
        const int wq = warp & 3;
        const uint32_t *src = reinterpret_cast<const uint32_t *>(a.basis_t_bf16);
        for (int blk = (warp - kEpiWarp0) >> 2; blk < n_blocks; blk += 2) {
            const int ch = blk * 128 + wq * 32 + lane;
            const uint32_t *row = src + (size_t)(ch < a.c ? ch : 0) * (a.k / 2);
            const uint32_t trow = tmem_base + ((uint32_t)(wq * 32) << 16) + (uint32_t)(blk * (a.k / 2));
#pragma unroll 2
            for (int j = 0; j < a.k / 2; j += 16) {
                if (a.k / 2 - j >= 16) {
                    uint32_t r[16];
#pragma unroll
                    for (int i = 0; i < 16; i += 4) {
                        const uint4 v = ch < a.c ? __ldg(reinterpret_cast<const uint4 *>(row + j + i)) : make_uint4(0u, 0u, 0u, 0u);
                        r[i] = v.x; r[i + 1] = v.y; r[i + 2] = v.z; r[i + 3] = v.w;
                    }
                    tmem_st_32x32b_x16(trow + j, r);
                } else {                                         // K % 32 == 16: eight columns left
                    uint32_t r[8];
#pragma unroll
                    for (int i = 0; i < 8; i += 4) {
                        const uint4 v = ch < a.c ? __ldg(reinterpret_cast<const uint4 *>(row + j + i)) : make_uint4(0u, 0u, 0u, 0u);
                        r[i] = v.x; r[i + 1] = v.y; r[i + 2] = v.z; r[i + 3] = v.w;
                    }
                    tmem_st_32x32b_x8(trow + j, r);
                }
            }
        }
        tmem_st_wait();
        // (only the MMA warp waits for the basis; the VLD groups are on their first tiles meanwhile)
        tc_fence_before_sync();
        named_bar_arrive(kBarBasis, 256 + 32);
    }

    const int my_tiles = (a.n_tiles > block) ? (int)((a.n_tiles - block + blocks - 1) / blocks) : 0;

    if (warp < kEpiWarp0) {
        // ================= VLD groups =================
        // 28 warps of 72 registers are launched: 16 of 80, 8 of 72 and 4 of 40 take as many
        asm volatile("setmaxnreg.inc.sync.aligned.u32 80;");
        const int tid = own_tid(), warp = tid >> 5, lane = tid & 31;
        const int grp = warp / group_warps;
        const int tg = tid - grp * n_thr;        // thread within the group
        if (grp < G) {
            const int set = cp > 1 ? 0 : tg >> 7;    // which thread of the pixel (warp-uniform)
            const int t = cp > 1 ? tg : (tg & 127);  // pixel within the tile, or chunk within the tile (cp > 1)
            const int wq = (t >> 5) & 3;
            const bool owner = tg < n_work;          // this thread has chunks to decode
            const int k_sub = a.k / S;               // coefficients per chunk of one pixel
            const int k_first = set * chunks_per_thread * k_sub;           // this thread's coefficients of a pixel
            const int k_last = cp > 1 ? a.k : k_first + chunks_per_thread * k_sub;
            const int p_first = k_first / kPanelK, p_last = (k_last + kPanelK - 1) / kPanelK;     // panels it touches
            const int chunks_per_tile = S * TC_TILE_PIXELS / cp;
            const uint32_t opnd_g = opnd_addr + (uint32_t)grp * L.opnd_bytes;
            const uint32_t sbuf_bytes = L.stream_buf;
            const uint32_t sbuf_g = smem_u32(smem + L.sbuf) + (uint32_t)grp * 2u * sbuf_bytes;
            const int bar_id = kBarGroup + grp;
            const int lb = a.lut_bits;
            const int dense_head = (a.dense_head + 7) & ~7;    // leading coefficients decoded symbol by symbol
            const uint32_t modal2 = (__float_as_uint((float)((a.modal < 0 ? a.center : a.modal) - a.center)) >> 16) * 0x00010001u;   // two bf16 copies of the modal symbol's value
            // The chunk that the thread decodes is not the one whose length it adds up: with one or two pixels a chunk the
            // threads of a warp write neighbouring columns of the operand, free of bank conflicts.
            const int src_lane = cp == 1 ? (int)pixel_of((uint32_t)lane) : cp == 2 ? (int)(pixel_of(2u * lane) >> 1) : lane;
            const int tc = (t & ~31) | src_lane;
            bool alive = true;

            // Offsets of a tile and the chunk lengths of this thread's pixel (up to four) or of its chunk, as they
            // lie in memory: read two tiles ahead and looked at (tile_info) a tile later.  Looked at at once, the
            // offsets' way from memory stood in every tile's time: 6 000 of the 19 000 cycles that a tile of 256
            // coefficients took a group.
            // (even lanes hold a tile's start, odd lanes its end)
            struct RawTile { unsigned long long at; unsigned int l01, l23; };
            auto load_tile = [&](int tl) {
                RawTile rt{1, 0, 0};                             // (no tile: not valid)
                if (tl >= my_tiles) return rt;
                const long long tile = block + (long long)tl * blocks;
                rt.at = a.tile_off[tile + (lane & 1)];
                if (owner) {
                    const long long ch = tile * chunks_per_tile + (long long)t * (cp > 1 ? 1 : S);
                    if (cp > 1 || S == 1) { if (ch < a.n_chunks) rt.l01 = a.chunk_len[ch]; }
                    else if (ch < a.n_chunks) {      // S chunks of one pixel: an aligned word holds two lengths
                        rt.l01 = *reinterpret_cast<const unsigned int *>(a.chunk_len + ch);
                        if (S == 4) rt.l23 = *reinterpret_cast<const unsigned int *>(a.chunk_len + ch + 2);
                    }
                }
                return rt;
            };
            // validated; a tile that cannot be valid decodes nothing
            // (room: buffers that the segment takes, 0 if it is read from global memory; landed: its copy was started a tile ahead)
            struct TileInfo { unsigned int bits; bool ok, landed; int room; unsigned int l01, l23; };
            auto tile_info = [&](const RawTile &rt, unsigned long long &base) {
                TileInfo ti{0, false, false, 0, 0, 0};
                base = __shfl_sync(0xffffffffu, rt.at, 0);
                const unsigned long long end = __shfl_sync(0xffffffffu, rt.at, 1);
                ti.ok = (base & 127ull) == 0 && (end & 127ull) == 0 && base <= end && end <= a.stream_bits;
                if (!ti.ok) return ti;
                ti.bits = (unsigned int)min(end - base, 0x7fffff80ull);           // (no tile's chunks take more)
                if ((cp * (k_last - k_first) * TC_MAX_CODE_LEN) / 8 + 16 <= kStreamSlack) ti.room = ti.bits <= sbuf_bytes * 8u ? 1 : ti.bits <= sbuf_bytes * 16u ? 2 : 0;
                ti.l01 = rt.l01;
                ti.l23 = rt.l23;
                return ti;
            };
            // Starts the copy of a tile's segment into stream buffer `which` (16 bytes per cp.async): while the tile before
            // is decoded, or, where one of the two takes both buffers, at the tile's own turn (encode and decode of 256x14x14 x 1024 at 8 bits 203 -> 171 us
            // against reading such segments word by word from global memory).
            auto stage_tile = [&](const TileInfo &ti, unsigned long long base, int which) {
                if (ti.room) {
                    const uint32_t dst = sbuf_g + (uint32_t)which * sbuf_bytes;
                    const unsigned char *src = reinterpret_cast<const unsigned char *>(a.stream) + (base >> 3);
                    const uint32_t n16 = ti.bits >> 7;
                    for (uint32_t i = tg; i < n16; i += n_thr) cp_async_16(dst + i * 16u, src + (size_t)i * 16u, 16u);
                }
                cp_async_commit();
            };

            chain_wait();                                        // the stream
            const RawTile first = load_tile(grp);
            RawTile ahead = load_tile(grp + G);
            unsigned long long tile_base;
            TileInfo cur = tile_info(first, tile_base);
            stage_tile(cur, tile_base, 0);
            cur.landed = true;
            int li = 0;
            // (a thread whose wait ran out keeps walking the tiles without decoding: the group's
            // barriers and the hand-over to the MMA thread need every thread's arrival)
            for (int tl = grp; tl < my_tiles; tl += G, ++li) {
                const long long tile = block + (long long)tl * blocks;
                // start of every chunk = sum of the lengths before it in the tile (chunk order: pixel,
                // then part of the pixel): scan over the pixels' totals
                const unsigned int len0 = cur.l01 & 0xffffu, len1 = cur.l01 >> 16, len2 = cur.l23 & 0xffffu, len3 = cur.l23 >> 16;
                const unsigned int tot = len0 + len1 + len2 + len3;
                unsigned int inc = tot;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned int up = __shfl_up_sync(0xffffffffu, inc, d);
                    if (lane >= d) inc += up;
                }
                if (lane == 31) s_wsum[grp][li & 1][set][wq] = inc;
                cp_async_wait<0>();
                // every thread's part of this tile's segment has landed, and every thread is done
                // with the tile before: its stream buffer may take the next tile's segment
                named_bar_sync(bar_id, n_thr);
                if (!cur.landed) {
                    if (cur.ok) stage_tile(cur, a.tile_off[tile], cur.room == 2 ? 0 : li & 1);
                    cp_async_wait<0>();
                    named_bar_sync(bar_id, n_thr);
                }
                TileInfo nxt = tile_info(ahead, tile_base);
                nxt.landed = cur.room + nxt.room <= 2;
                if (nxt.landed) stage_tile(nxt, tile_base, nxt.room == 2 ? 0 : (li + 1) & 1);
                ahead = load_tile(tl + 2 * G);
                unsigned int before = 0, tile_total = 0;
                const int n_wq = (n_work / tpp + 31) / 32;          // warps of one thread set
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const unsigned int sw = w < n_wq ? s_wsum[grp][li & 1][set][w] : 0u;
                    if (w < wq) before += sw;
                    tile_total += sw;
                }
                // this thread's first chunk: after the pixels before it and the chunks of the pixel before its own
                unsigned int chunk_start = before + inc - tot;
                unsigned int my_len0 = len0, my_len1 = len1;
                if (cp == 1 && set == 1) {
                    if (S == 2) { chunk_start += len0; my_len0 = len1; }
                    else { chunk_start += len0 + len1; my_len0 = len2; my_len1 = len3; }
                }
                chunk_start = __shfl_sync(0xffffffffu, chunk_start, src_lane);
                my_len0 = __shfl_sync(0xffffffffu, my_len0, src_lane);
                if (S == 4) my_len1 = __shfl_sync(0xffffffffu, my_len1, src_lane);

                const long long ch = tile * chunks_per_tile + (long long)tc * (cp > 1 ? 1 : S);
                bool active = cur.ok && owner && ch < a.n_chunks;
                bool bad = !cur.ok || tile_total > cur.bits;
                if (bad) active = false;
                const long long px0 = tile * TC_TILE_PIXELS + (long long)tc * cp;
                const int n_pix = active ? (int)min((long long)cp, a.pixels - px0) : 0;
                const uint32_t seg_addr = sbuf_g + (cur.room == 2 ? 0u : (uint32_t)(li & 1) * sbuf_bytes);
                // dense tiles are decoded symbol by symbol
                const bool runs = a.modal >= 0 &&
                                  cur.bits <= (unsigned int)(kDenseBits128 * TC_TILE_PIXELS / 128) * (unsigned int)a.k;
                const uint32_t wait_parity = (uint32_t)((li & 1) ^ 1);   // the buffer's hand-back by the tile before this one

                // Walks this thread's chunks.  Control flow is kept uniform across the warp: the lanes
                // of a warp step together (a lane that has finished its chunk idles until all have),
                // the panels of a chunk are waited for and filled by all lanes at once, before its first
                // symbol, and a wait that runs out is seen by every lane -- lanes that wander off on
                // their own would run the rest of the tile one after the other.
                auto decode_tile = [&](auto &r) {
                    uint32_t expect = 0;               // bits the chunks decoded so far should have taken
                    for (int pp = 0; pp < cp; ++pp) {
                        const bool decode = pp < n_pix;
                        const uint32_t row = column_of((uint32_t)(tc * cp + pp));
                        const uint32_t row_addr = opnd_g + (row >> 3) * 128u + (row & 7u) * 16u;
                        int ready = p_first;           // panels [p_first, ready) of the warp's rows are handed back and filled
                        // waits for panel p to be handed back by the MMAs of the tile before, then fills this
                        // thread's coefficients of it from coefficient `from` on with the modal symbol
                        auto prepare = [&](int p, int from) {
                            if (pp == 0 && alive) alive = mbar_wait(smem_u32(&s_empty[grp][p]), wait_parity, 200u);
                            if (owner) {
                                const int g0 = max(p * (kPanelK / 8), max(k_first, from) >> 3), g1 = min((p + 1) * (kPanelK / 8), k_last >> 3);
                                for (int g = g0; g < g1; ++g) sts_v4(row_addr + (uint32_t)g * 2048u, modal2, modal2, modal2, modal2);
                            }
                        };
                        for (int ci = 0; ci < (cp > 1 ? 1 : chunks_per_thread); ++ci) {
                            const int kf = cp > 1 ? 0 : k_first + ci * k_sub, ke = cp > 1 ? a.k : kf + k_sub;
                            // the leading coefficients (and every coefficient of a dense tile) symbol by symbol,
                            // eight symbols per 16-byte store; the rest run by run
                            const int kd = runs ? min(max(dense_head, kf), ke) : ke;
                            for (int k0 = kf; k0 < kd; k0 += 8) {
                                while (ready * kPanelK <= k0) prepare(ready++, kd);
                                uint32_t pk[4];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    r.refill();
                                    const uint32_t e0 = lds_u32(lut_addr + (r.hi >> (32 - lb)) * 4u);
                                    r.take(decode ? e0 : 0u);
                                    const uint32_t e1 = lds_u32(lut_addr + (r.hi >> (32 - lb)) * 4u);
                                    r.take(decode ? e1 : 0u);
                                    pk[i] = __byte_perm(e0, e1, 0x7632);
                                }
                                if (decode) sts_v4(row_addr + (uint32_t)(k0 >> 3) * 2048u, pk[0], pk[1], pk[2], pk[3]);
                            }
                            while (ready * kPanelK < ke) prepare(ready++, kd);
                            uint32_t pos = (uint32_t)kd, rem = decode ? (uint32_t)(ke - kd) : 0u;
                            while (__any_sync(0xffffffffu, rem != 0u)) {
                                r.refill();
                                // a run of the modal symbol is a run of zero bits: at most 20 per step
                                const uint32_t n = min((uint32_t)__clz((int)(r.hi | kRunGuard)), rem);
                                r.take(n);
                                pos += n;
                                rem -= n;
                                const bool sym = rem != 0u;            // a symbol follows the run
                                const uint32_t e = lds_u32(lut_addr + (r.hi >> (32 - lb)) * 4u);
                                r.take(sym ? e : 0u);
                                // coefficient pos of the row: core-matrix column pos / 8 (2048 bytes apart), 2 bytes per coefficient inside
                                if (sym) sts_u16(row_addr + pos * 2u + (pos >> 3) * 2032u, e >> 16);
                                pos += sym ? 1u : 0u;
                                rem -= sym ? 1u : 0u;
                            }
                            // a chunk of one pixel (or part of it) must end exactly where its length says
                            if (cp == 1) {
                                expect += ci == 0 ? my_len0 : my_len1;
                                if (active && r.consumed() != expect) bad = true;
                            }
                        }
                        while (ready < p_last) prepare(ready++, 0);
                    }
                    if (cp > 1 && active && r.consumed() != my_len0) bad = true;
                };
                if (cur.room) {
                    BitReader<true> r;
                    if (active) r.init(seg_addr, nullptr, nullptr, chunk_start);
                    else r.idle();
                    decode_tile(r);
                } else {
                    BitReader<false> r;
                    if (active) {
                        const uint32_t *seg = a.stream + (a.tile_off[tile] >> 5);
                        r.init(0u, seg, seg + (cur.bits >> 5), chunk_start);
                    } else r.idle();
                    decode_tile(r);
                }
                // (the issuing thread makes the operand visible to the tensor core's proxy)
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_bfull[grp]));
                if (bad) tc_dev_set_status(a.status, TC_ERR_CORRUPT_STREAM);
                cur = nxt;
            }
            cp_async_wait<0>();
            if (!alive) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
        }
    } else if (warp < kMmaWarp && L.mode == kMaps) {
        // ================= epilogue, maps of up to kSmallMap pixels =================
        // As below, but for a thread's 16 columns of its own channel at a time.
        const int warp = own_tid() >> 5, lane = own_tid() & 31;
        const int set = (warp - kEpiWarp0) >> 2, wq = warp & 3;
        const int n_items = my_tiles * items;
        const bool shared = n_items == 1;                         // one item only: half of the pixels each
        const int acc = shared ? 0 : set;
        const int hw = (int)a.hw, map = a.c * hw;
        const int ch = (items == 2 ? set * 128 : 0) + wq * 32 + lane;
        const bool ch_ok = ch < a.c;
        const float step = (float)(a.step * a.basis_scale), bias = ch_ok ? __ldg(a.dec_bias + ch) : 0.f;
        // bytes that leave at a time: a map's row of the channel, or one pixel of two channels (the neighbouring lane's), or of one
        const bool fours = hw == 4 && ((uintptr_t)a.xhat & 7u) == 0, twos = hw == 2 && ((uintptr_t)a.xhat & 3u) == 0;
        const bool pairs = hw == 1 && ((uintptr_t)a.xhat & 3u) == 0;
        const int odd = lane & 1;
        const uint32_t places = smem_u32(smem + L.tbuf) + (uint32_t)(warp - kEpiWarp0) * kTrWarpBytes;       // of a tile's pixels in the tensor, where neither holds
        const uint32_t trow = tmem_base + kAccBase + acc * kAccCols + ((uint32_t)(wq * 32) << 16);
        bool alive = true;
        chain_wait();                                            // earlier readers of the tensor
        for (int it = acc; it < n_items; it += 2) {
            const long long tile = block + (long long)(items == 2 ? it >> 1 : it) * blocks, img = tile * TC_TILE_PIXELS / hw;
            const int sp = (int)(tile * TC_TILE_PIXELS - img * hw);
            const int n_valid = ch_ok ? (int)min((long long)TC_TILE_PIXELS, a.pixels - tile * TC_TILE_PIXELS) : 0;
            __nv_bfloat16 *const out = reinterpret_cast<__nv_bfloat16 *>(a.xhat) + img * map + (long long)ch * hw;
            if (wq == 0) {
                if (alive) alive = mbar_wait(smem_u32(&s_tfull[acc]), (uint32_t)((it >> 1) & 1), 50u);
                tc_fence_before_sync();
            }
            named_bar_sync(kBarEpi + set, 128);
            tc_fence_after_sync();
            if (!pairs && !fours && !twos) {
                int to[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int x = sp + 4 * lane + i, m = hw == 3 ? (x * 171) >> 9 : x >> (hw >> 1);          // x / hw
                    to[i] = m * map + (x - m * hw);
                }
                sts_v4(places + 16u * lane, to[0], to[1], to[2], to[3]);
                __syncwarp();
            }
#pragma unroll 1
            for (int c0 = shared ? 64 * set : 0; c0 < (shared ? 64 * set + 64 : TC_TILE_PIXELS); c0 += 16) {
                uint32_t r[16];
                tmem_ld_32x32b_x16(trow + c0, r);
                tmem_ld_wait(r);
                const int px0 = (int)pixel_of((uint32_t)c0);      // column c0 + 8 g + 2 q + {0, 1}: pixel px0 + 8 q + 2 g + {0, 1}
                int at = (pairs ? px0 + odd : fours ? px0 >> 2 : px0 >> 1) * map - (pairs ? odd : 0);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t w[2];
#pragma unroll
                    for (int g = 0; g < 2; ++g) w[g] = decoded_pair<kRelu>(r[8 * g + 2 * q], r[8 * g + 2 * q + 1], step, bias);
                    const int px = px0 + 8 * q;
                    if (pairs) {
#pragma unroll
                        for (int g = 0; g < 2; ++g) {
                            const uint32_t theirs = __shfl_xor_sync(0xffffffffu, w[g], 1);
                            const uint32_t v = __byte_perm(w[g], theirs, odd ? 0x3276 : 0x5410);
                            if (px + 2 * g + odd < n_valid) *reinterpret_cast<uint32_t *>(out + (at + 2 * g * map)) = v;
                        }
                        at += 8 * map;
                    } else if (fours) {
                        if (px < n_valid) *reinterpret_cast<uint2 *>(out + at) = make_uint2(w[0], w[1]);
                        at += 2 * map;
                    } else if (twos) {
#pragma unroll
                        for (int g = 0; g < 2; ++g)
                            if (px + 2 * g < n_valid) *reinterpret_cast<uint32_t *>(out + (at + g * map)) = w[g];
                        at += 4 * map;
                    } else {
                        int to[4];
                        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(to[0]), "=r"(to[1]), "=r"(to[2]), "=r"(to[3]) : "r"(places + 4u * px));
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (px + i < n_valid) *reinterpret_cast<unsigned short *>(out + to[i]) = (unsigned short)(w[i >> 1] >> (16 * (i & 1)));
                    }
                }
            }
            tc_fence_before_sync();
            if (!shared) named_bar_arrive(kBarAccFree + acc, 128 + 32);
        }
        if (!alive && lane == 0) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
    } else if (warp < kMmaWarp) {
        // ================= epilogue =================
        // An item is a tile's 128 pixels of one block of 128 channels.  Four warps serve each accumulator, so that the waits of one
        // item run beside the work of another; a warp stores the 32 channels of its quarter of TMEM, 16 at a time.
        const int warp = own_tid() >> 5, lane = own_tid() & 31;
        const int mode = L.mode;
        const int set = (warp - kEpiWarp0) >> 2, wq = warp & 3;
        const int n_items = my_tiles * items;
        const bool shared = n_items == 1;                         // one item only: half of the channels each
        const int acc = shared ? 0 : set;
        const float step = (float)(a.step * a.basis_scale);        // the operand holds basis / basis_scale
        __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(a.xhat);
        auto convert = [&](uint32_t x0, uint32_t x1, float bias) { return decoded_pair<kRelu>(x0, x1, step, bias); };
        // Position of this lane's first pixel of a tile: image and offset inside it of the block's first tile, moved on from
        // tile to tile by a constant number of pixels (a division of 64-bit numbers per item was a fifth of
        // the epilogue's instructions).
        const int px_lane = mode == kRows16 ? 8 * (lane & 3) : mode == kRows8 ? 4 * lane : lane;
        const unsigned int hw = (unsigned int)a.hw;
        const long long px_step = (long long)blocks * TC_TILE_PIXELS * (items == 2 ? 1 : 2);
        const unsigned int img_step = (unsigned int)(px_step / a.hw), sp_step = (unsigned int)(px_step - (long long)img_step * a.hw);
        const long long first_px = ((long long)block + (items == 2 ? 0 : (long long)acc * blocks)) * TC_TILE_PIXELS + px_lane;
        unsigned int tile_img = (unsigned int)(first_px / a.hw), tile_sp = (unsigned int)(first_px - (long long)tile_img * a.hw);
        const int ch_base = (items == 2 ? set * 128 : 0) + wq * 32;         // first channel of this warp
        const int h_first = shared ? set : 0, halves = min(shared ? set + 1 : 2, (a.c - ch_base) / 16);      // of 16 channels (C is a multiple of 16)
        float bias[4];                                                      // of this thread's channels, eight apart
#pragma unroll
        for (int i = 0; i < 4; ++i) bias[i] = i < 2 * halves ? __ldg(a.dec_bias + ch_base + 8 * i + (lane >> 2)) : 0.f;
        // The warp's block: row = channel (256 bytes); the halves of every 128 bytes of an odd row are exchanged, so that
        // neither the row writes (two rows x 64 bytes a phase) nor the reads collide.
        const uint32_t tb = smem_u32(smem + L.tbuf) + (uint32_t)(warp - kEpiWarp0) * kTrWarpBytes;
        const uint32_t tb_wr = tb + (uint32_t)(lane >> 2) * 256u + (uint32_t)(lane & 3) * 16u, swap = (uint32_t)(lane & 4) << 4;
        bool alive = true;
        const uint32_t trow = tmem_base + kAccBase + acc * kAccCols + ((uint32_t)(wq * 32) << 16);
        chain_wait();                                            // earlier readers of the tensor
        // (after a wait that ran out the warps keep walking the items: the MMA warp waits for their arrivals)
        for (int it = acc; it < n_items; it += 2) {
            const unsigned int tile = block + (unsigned int)(items == 2 ? it >> 1 : it) * blocks;
            const int n_valid = tile == (unsigned int)a.n_tiles - 1u ? (int)(a.pixels - (a.n_tiles - 1) * TC_TILE_PIXELS) : TC_TILE_PIXELS;
            // one warp waits for the accumulator and lets the others in
            if (wq == 0) {
                if (alive) alive = mbar_wait(smem_u32(&s_tfull[acc]), (uint32_t)((it >> 1) & 1), 50u);
                tc_fence_before_sync();
            }
            named_bar_sync(kBarEpi + set, 128);
            tc_fence_after_sync();
            uint32_t r[16];                                       // 32 pixels
            if (h_first < halves) tmem_ld_16x256b_x4(trow + ((uint32_t)(16 * h_first) << 16), r);
            auto hand_back = [&] {
                tc_fence_before_sync();
                if (!shared) named_bar_arrive(kBarAccFree + acc, 128 + 32);
            };
            if (h_first >= halves) hand_back();
#pragma unroll 1
            for (int h = h_first; h < halves; ++h) {
                const float bias0 = h ? bias[2] : bias[0], bias1 = h ? bias[3] : bias[1];
                unsigned int img = tile_img, sp = tile_sp;
                // this lane's place of the tensor in the first of the 16 channels, `pixels` further on each time
                auto place = [&](unsigned int pixels) {
                    __nv_bfloat16 *at = out + ((long long)img * a.c + (ch_base + 16 * h)) * a.hw + sp;
                    sp += pixels;
                    while (sp >= hw) { sp -= hw; ++img; }
                    return at;
                };
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    tmem_ld_wait(r);
                    uint32_t w[2][4];                             // [row, eight apart][two pixels of eight]
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        w[0][g] = convert(r[4 * g], r[4 * g + 1], bias0);
                        w[1][g] = convert(r[4 * g + 2], r[4 * g + 3], bias1);
                    }
                    // the next columns are on their way, or the accumulator handed back, while these are stored
                    if (b < 3) tmem_ld_16x256b_x4(trow + ((uint32_t)(16 * h) << 16) + 32 * (b + 1), r);
                    else if (h + 1 < halves) tmem_ld_16x256b_x4(trow + (16u << 16), r);
                    else hand_back();
                    if (mode == kRows16) {
                        const bool ok = 32 * b + px_lane < n_valid;
                        uint4 *at = reinterpret_cast<uint4 *>(place(32) + (long long)(lane >> 2) * a.hw);
                        if (ok) *at = make_uint4(w[0][0], w[0][1], w[0][2], w[0][3]);
                        if (ok) at[a.hw] = make_uint4(w[1][0], w[1][1], w[1][2], w[1][3]);          // eight rows on
                    } else {
                        const uint32_t at = tb_wr + 128u * (b >> 1) + ((64u * (b & 1)) ^ swap);
                        sts_v4(at, w[0][0], w[0][1], w[0][2], w[0][3]);
                        sts_v4(at + 2048u, w[1][0], w[1][1], w[1][2], w[1][3]);
                    }
                }
                if (mode == kRows8) {
                    __syncwarp();
                    __nv_bfloat16 *at = place(0);
                    const bool ok = px_lane < n_valid;
#pragma unroll 4
                    for (int k = 0; k < 16; ++k) {
                        uint32_t lo, hi;
                        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(lo), "=r"(hi) : "r"(tb + k * 256u + (((uint32_t)lane * 8u) ^ ((k & 1u) << 6))));
                        if (ok) *reinterpret_cast<uint2 *>(at) = make_uint2(lo, hi);
                        at += a.hw;
                    }
                    __syncwarp();                               // the block may be overwritten
                } else if (mode == kRowsAny) {
                    __syncwarp();
                    __nv_bfloat16 *at[4];
#pragma unroll
                    for (int b = 0; b < 4; ++b) at[b] = place(32);
#pragma unroll 1
                    for (int k = 0; k < 16; ++k) {
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            unsigned short v;
                            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(tb + k * 256u + (((uint32_t)lane * 2u + 64u * b) ^ ((k & 1u) << 6))));
                            if (32 * b + lane < n_valid) *reinterpret_cast<unsigned short *>(at[b]) = v;
                            at[b] += a.hw;
                        }
                    }
                    __syncwarp();
                }
            }
            tile_img += img_step;
            tile_sp += sp_step;
            if (tile_sp >= hw) { tile_sp -= hw; ++tile_img; }
        }
        if (!alive && lane == 0) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == kMmaWarp) {
            // ================= MMA issuer =================
            // The items in order, on the two accumulators in turn.  The whole warp walks the loop
            // and waits on the barriers; lane 0 issues, through instructions that carry their own guard
            // (no branch around an MMA).  An MMA leaves its issuing thread every 64 cycles at best, with 64 columns as
            // with 128: items of 64 pixels of both blocks took twice as many instructions (125 us for the products of
            // 256x14x14 x 4096 alone) and a warp per accumulator.
            // A = transposed basis in tensor memory (128 channels per instruction), B = the decoded
            // symbols of the tile (the group's operand buffer).
            named_bar_sync(kBarBasis, 256 + 32);
            tc_fence_after_sync();
            chain_wait();                                            // its waits run out two seconds from here, not from the launch
            const uint32_t issuer = (own_tid() & 31) == 0 ? 1u : 0u;
            const uint32_t idesc = make_idesc_bf16(128, TC_TILE_PIXELS, /*A K-major*/ false, /*B K-major*/ false);
            const int n_k16 = a.k >> 4;
            int buf = 0;                                              // operand buffer (VLD group) of the tile, and the parity of its turn
            uint32_t turn = 0;
            int it = 0;
            bool alive = true;
            for (int tl = 0; tl < my_tiles; ++tl) {
                // (after a wait that ran out the warp keeps walking the items: the epilogue waits for its commits)
                if (alive) alive = mbar_wait(smem_u32(&s_bfull[buf]), turn);     // the group's VLD threads have arrived
                __syncwarp();
                // the operand was written with ordinary stores by threads that have arrived on the
                // barrier: one proxy fence here, between that synchronisation and the MMA's
                // operand reads, orders them for all writers
                fence_proxy_async_smem();
                const uint64_t b_base = make_smem_desc(opnd_addr + (uint32_t)buf * L.opnd_bytes, 2048, 128);
                const uint32_t b_hi = (uint32_t)(b_base >> 32);
                for (int blk = 0; blk < items; ++blk, ++it) {
                    const int acc = it & 1;
                    const uint32_t d_tmem = tmem_base + kAccBase + acc * kAccCols;
                    if (it >= 2) named_bar_sync(kBarAccFree + acc, 128 + 32);     // the epilogue has drained the accumulator
                    __syncwarp();
                    tc_fence_after_sync();
                    // eight-row groups are 128 bytes apart; a step of 16 coefficients moves the start address on by two
                    // core-matrix columns of 2048 bytes
                    uint32_t b_lo = (uint32_t)b_base;
                    uint32_t a_col = tmem_base + (uint32_t)(blk * (a.k / 2));
                    int q = 0;
                    auto step = [&] {
                        mma_bf16_ts_guarded(d_tmem, a_col, b_lo, b_hi, idesc, q ? 1u : 0u, issuer);
                        b_lo += 4096u >> 4;
                        a_col += 8;
                        ++q;
                    };
                    // a panel that the last item has read goes back to the VLD threads
                    auto panel_read = [&] {
                        if (blk == items - 1) mma_commit_guarded(smem_u32(&s_empty[buf][(q - 1) / (kPanelK / 16)]), issuer);
                    };
                    // (eight at a time: an instruction of this warp waits its turn among the others', and a turn of a rolled loop around one
                    // MMA took 140 cycles)
                    while (q + 8 <= n_k16) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) step();
                        panel_read();
                    }
                    if (q + 4 <= n_k16) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) step();
                    }
                    while (q < n_k16) step();
                    if (n_k16 % 8 != 0) panel_read();
                    mma_commit_guarded(smem_u32(&s_tfull[acc]), issuer);
                }
                if (++buf == G) { buf = 0; turn ^= 1u; }
            }
            // the block frees tensor memory next: not ahead of MMAs that nobody waits for (an epilogue whose own wait ran out)
            mma_commit_guarded(smem_u32(&s_drained), issuer);
            mbar_wait(smem_u32(&s_drained), 0u);
            if (!alive && issuer) tc_dev_set_status(a.status, TC_ERR_TIMEOUT);
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

template <bool kRelu>
__global__ void __launch_bounds__(kThreads, 1) decode_runs_kernel(DecodeArgs a, SmemLayout L)
{
    decode_tiles<kRelu>(a, L, blockIdx.x, gridDim.x);
}

// Several tensors in one launch, each with blocks of its own (see encode_tc_list_kernel): 16 layers of a residual network at
// batch 64 199 -> 155 us, nine tensors of up to 50 000 values 62 -> 31.
struct DecodeList {
    unsigned int first[kListItems + 1];        // block that each item starts at; past the last item 2^32 - 1
    struct { DecodeArgs a; SmemLayout l; } item[kListItems];
};
template <bool kRelu>
__global__ void __launch_bounds__(kThreads, 1) decode_runs_list_kernel(const __grid_constant__ DecodeList list)
{
    int i = 0;
    while (blockIdx.x >= list.first[i + 1]) ++i;
    decode_tiles<kRelu>(list.item[i].a, list.item[i].l, blockIdx.x - list.first[i], min(list.first[i + 1], gridDim.x) - list.first[i]);
}

}  // namespace

static SmemLayout runs_layout(const tc_ctx *ctx, const DecodeArgs &a)
{
    // (a dense tile's segment is at most 3 % longer than the mean)
    const double tile_bytes = a.mean_tile_bytes > 0 ? a.mean_tile_bytes : std::max(2.5, (double)a.code_bits) * a.k * TC_TILE_PIXELS / 8;
    const uint32_t want = (uint32_t)std::min(1.03 * tile_bytes, 1e6);
    return smem_layout(a.k, 1 << a.lut_bits, (group_work(a.splits, a.chunk_pixels) + 31) / 32, want, store_mode(a), ctx->max_smem_optin - kStaticSmem);
}

// The roles' registers are dealt from what a block is launched with: with fewer a thread than this the VLD warps would wait for theirs
// for good, so a build whose kernels came out smaller does not run them.
constexpr int kLaunchRegisters = 72;
static_assert(16 * 80 + 8 * 72 + 4 * 40 <= 28 * kLaunchRegisters && kThreads == 28 * 32, "VLD, epilogue and MMA warpgroups");
static bool registers_suffice()
{
    static const bool ok = [] {
        for (const void *kernel : {(const void *)decode_runs_kernel<false>, (const void *)decode_runs_kernel<true>, (const void *)decode_runs_list_kernel<false>,
                                   (const void *)decode_runs_list_kernel<true>}) {
            cudaFuncAttributes at;
            if (cudaFuncGetAttributes(&at, kernel) != cudaSuccess) { cudaGetLastError(); return false; }
            if (at.numRegs < kLaunchRegisters) return false;
        }
        return true;
    }();
    return ok;
}

bool tc_decode_runs_supported(const tc_ctx *ctx, const DecodeArgs &a)
{
    // K <= C leading components (PCA truncation): K is the reduction dimension of the MMA
    if (a.c % 16 != 0 || a.k % 16 != 0 || a.k < 16 || a.k > a.c || a.c > 256) return false;
    if (a.groups != 1) return false;                           // per-channel tables do not fit shared memory
    if (a.lut_bits > TC_MAX_CODE_LEN) return false;
    if (a.chunk_pixels > 1 ? a.splits != 1 : (a.splits != 1 && a.splits != 2 && a.splits != 4)) return false;
    if (a.splits > 1 && (a.k % a.splits != 0 || (a.k / a.splits) % 8 != 0)) return false;
    return runs_layout(ctx, a).stream_buf > 0 && registers_suffice();
}

tc_status tc_launch_decode_runs(const tc_ctx *ctx, const DecodeArgs &a, cudaStream_t s)
{
    if (a.n_tiles <= 0) return TC_OK;
    const SmemLayout l = runs_layout(ctx, a);
    if (l.stream_buf == 0) return TC_ERR_UNSUPPORTED;
    void (*kernel)(DecodeArgs, SmemLayout) = a.relu ? decode_runs_kernel<true> : decode_runs_kernel<false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.total) != cudaSuccess)
        return TC_ERR_CUDA;
    const unsigned int grid = (unsigned int)((a.n_tiles < ctx->sm_count) ? a.n_tiles : ctx->sm_count);
    return launch_first(a.alone, kernel, grid, kThreads, l.total, s, a, l) == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

// us that a tile takes a block: 1.6 with 64 coefficients at 1.1 bits each, 1.8 with 128, 2.7 with 160 (two items a tile), 3.5 with 256; 2.9
// with 128 at 4.1 bits, 5.8 with 256; 0.9 more for every 128 channels where rows start anywhere, 0.5 of small maps (40 tiles a block, less the first)
double tc_decode_runs_tile_us(const DecodeArgs &a)
{
    const double bits = a.mean_tile_bytes > 0 ? a.mean_tile_bytes * 8.0 / TC_TILE_PIXELS : (double)a.code_bits * a.k;
    return 1.25 + (a.c > 128 ? 0.9 : 0.0) + 0.0035 * std::max(0, a.k - 128) + 0.003 * bits + (store_mode(a) == kRowsAny ? 0.9 : store_mode(a) == kMaps ? 0.5 : 0.0) * ((a.c + 127) / 128);
}

// Decodes tensors that tc_decode_runs_supported takes, all with the same `relu`, on `sms` SMs, in list_launches launches.
tc_status tc_launch_decode_runs_list(const tc_ctx *ctx, const std::vector<DecodeArgs> &tensors, int sms, cudaStream_t s)
{
    const size_t launches = list_launches(tensors.size(), sms);
    for (size_t r = 0; r < launches; ++r) {
        const int n = (int)((tensors.size() - r + launches - 1) / launches);
        DecodeList list;
        std::vector<ListWork> work(n);
        uint32_t smem = 0;
        for (int i = 0; i < n; ++i) {
            const DecodeArgs &a = tensors[r + i * launches];
            list.item[i].a = a;
            list.item[i].l = runs_layout(ctx, a);
            smem = std::max(smem, list.item[i].l.total);
            work[i] = {a.n_tiles, tc_decode_runs_tile_us(a), 1};
        }
        deal_blocks(work, sms);
        unsigned int blocks = 0;
        for (int i = 0; i <= kListItems; ++i) {
            list.first[i] = i <= n ? blocks : ~0u;
            if (i < n) blocks += (unsigned int)work[i].blocks;
        }
        list.first[n] = ~0u;
        const void *kernel = tensors[r].relu ? (const void *)decode_runs_list_kernel<true> : (const void *)decode_runs_list_kernel<false>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) { cudaGetLastError(); return TC_ERR_CUDA; }
        void *params[] = {&list};
        if (cudaLaunchKernel(kernel, dim3(blocks), dim3(kThreads), params, smem, s) != cudaSuccess) { cudaGetLastError(); return TC_ERR_CUDA; }
    }
    return TC_OK;
}
