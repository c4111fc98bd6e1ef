// Device helpers shared by the codec kernels: block scan of bit lengths, the cross-tile
// look-back that turns tile sizes into stream offsets, and the MSB-first bit writer/reader.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "tc_internal.h"

namespace tcdev {

constexpr unsigned long long kFlagAggregate = 1ull << 62;
constexpr unsigned long long kFlagPrefix = 2ull << 62;
constexpr unsigned long long kValueMask = (1ull << 62) - 1;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // bounded look-back wait: 2 s

__device__ __forceinline__ unsigned long long ld_volatile_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_volatile_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long global_timer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Kernels that follow each other (launch_chained, launch_first): a kernel lets the next one start setting up once all its own blocks run
// (chain_next), and every thread that touches what others wrote or read waits for the kernel before it, and so for everything before that, ahead of the
// first access to it (chain_wait).  What it reads of theirs does not go through the read-only path.
// chain_next is a kernel's first act, also of the persistent decoder, encoder and tiled product where they end a call: whoever starts then waits in
// its turn.  Only the exact inverse and the entropy coder of stored symbols, which end a call, do so behind their wait: with the kernels of four calls'
// halves set up behind one another a round trip of 256x14x14 f32 took 48 us instead of 43.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A word of a stream, 0 at or past `end`.  Not through the read-only path (see launch_first), and free to be scheduled among
// stores as such a load is: its address comes from offsets that were read after the wait.
__device__ __forceinline__ uint32_t stream_word(const uint32_t *next, const uint32_t *end)
{
    uint32_t w;
    asm("{\n\t.reg .pred p;\n\tsetp.lt.u64 p, %1, %2;\n\tmov.u32 %0, 0;\n\t@p ld.global.u32 %0, [%1];\n\t}" : "=&r"(w) : "l"(next), "l"(end));
    return w;
}

__device__ __forceinline__ double load_as_double(const float *p) { return (double)__ldg(p); }
__device__ __forceinline__ double load_as_double(const __nv_bfloat16 *p)
{
    const unsigned short raw = __ldg(reinterpret_cast<const unsigned short *>(p));
    return (double)__uint_as_float((unsigned int)raw << 16);
}

// Round a double to the output type with a single rounding (ties to even).
__device__ __forceinline__ void store_rounded(float *p, double v) { *p = __double2float_rn(v); }
__device__ __forceinline__ void store_rounded(__nv_bfloat16 *p, double v)
{
    // double -> float with round-to-odd keeps enough information for the final RNE to bf16.
    float f = __double2float_rz(v);
    if ((double)f != v) f = __uint_as_float(__float_as_uint(f) | 1u);
    *p = __float2bfloat16_rn(f);
}

// Exclusive scan of one unsigned value per thread over a 128-thread group (4 warps).
// `warp_sums` is 4 words of shared memory; `bar_id`/`bar_threads` name the barrier to use
// (named barrier, so that other warps of the block are not involved).
__device__ __forceinline__ unsigned int group_exclusive_scan_128(unsigned int v, unsigned int *warp_sums,
                                                                int tid128, int bar_id, unsigned int &total)
{
    const int lane = tid128 & 31, warp = tid128 >> 5;
    unsigned int inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned int up = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += up;
    }
    if (lane == 31) warp_sums[warp] = inc;
    asm volatile("bar.sync %0, 128;" ::"r"(bar_id) : "memory");
    unsigned int before = 0, all = 0;
#pragma unroll
    for (int wv = 0; wv < 4; ++wv) {
        const unsigned int s = warp_sums[wv];
        if (wv < warp) before += s;
        all += s;
    }
    total = all;
    return before + inc - v;
}

// Decoupled look-back over per-tile sizes.  A tile first publishes its own padded size
// (lookback_publish, one thread), later one full warp resolves the sum of the sizes of all
// earlier tiles (lookback_resolve) and publishes the inclusive prefix.  Every earlier tile is
// owned by a block that is resident (tickets or a co-resident persistent grid), so the waits
// end; they are bounded all the same, and a wait that runs out clears `ok` and records a
// timeout in the status word.
__device__ __forceinline__ void lookback_publish(unsigned long long *state, long long tile, unsigned long long own)
{
    st_volatile_u64(state + tile, (tile == 0 ? kFlagPrefix : kFlagAggregate) | own);
}

__device__ __forceinline__ unsigned long long lookback_resolve(unsigned long long *state, long long tile,
                                                               unsigned long long own, unsigned int *status, bool &ok)
{
    const int lane = threadIdx.x & 31;
    ok = true;
    if (tile == 0) return 0;
    unsigned long long exclusive = 0;
    long long idx = tile - 1;
    const unsigned long long t0 = global_timer_ns();
    while (true) {
        const long long mine = idx - lane;
        unsigned long long s = kFlagPrefix;   // tiles before the first one: prefix 0
        if (mine >= 0) {
            s = ld_volatile_u64(state + mine);
            while ((s >> 62) == 0) {
                if (global_timer_ns() - t0 > kWaitLimitNs) break;
                __nanosleep(200);          // (a polling warp takes issue slots from the block's working warps)
                s = ld_volatile_u64(state + mine);
            }
        }
        const bool timed_out = (s >> 62) == 0;
        if (__any_sync(0xffffffffu, timed_out)) { ok = false; break; }
        const unsigned int prefix_lanes = __ballot_sync(0xffffffffu, (s >> 62) == 2);
        const int first_prefix = prefix_lanes ? (__ffs(prefix_lanes) - 1) : 32;
        unsigned long long contrib = (lane <= first_prefix) ? (s & kValueMask) : 0ull;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) contrib += __shfl_xor_sync(0xffffffffu, contrib, d);
        exclusive += contrib;
        if (prefix_lanes) break;
        idx -= 32;
    }
    if (!ok && lane == 0) tc_dev_set_status(status, TC_ERR_TIMEOUT);
    // publish the inclusive prefix even after a timeout so that later tiles are released
    if (lane == 0) st_volatile_u64(state + tile, kFlagPrefix | ((exclusive + own) & kValueMask));
    return exclusive;
}

__device__ __forceinline__ unsigned long long tile_lookback(unsigned long long *state, long long tile,
                                                            unsigned long long own, unsigned int *status, bool &ok)
{
    if ((threadIdx.x & 31) == 0) lookback_publish(state, tile, own);
    __syncwarp();
    return lookback_resolve(state, tile, own, status, ok);
}

// MSB-first bit writer into a zero-initialised word array.  The first and the last word a
// writer touches may be shared with its neighbours and are merged with atomicOr; words in
// between belong to this writer alone.
struct BitWriter {
    uint32_t *words;           // the (shared or global) word holding the writer's first bit
    unsigned long long acc;    // pending bits, right-aligned
    int pending;               // number of pending bits incl. the lead-in of the first word
    unsigned int word;         // index of the word being filled, relative to `words`
    bool first;

    __device__ __forceinline__ void init(uint32_t *base, unsigned long long bitpos)
    {
        words = base + (bitpos >> 5);
        word = 0;
        pending = (int)(bitpos & 31);
        acc = 0;
        first = true;
    }
    __device__ __forceinline__ void put(uint32_t code, int len)
    {
        acc = (acc << len) | code;
        pending += len;
        if (pending >= 32) {
            const uint32_t out = (uint32_t)(acc >> (pending - 32));
            if (first) { atomicOr(words + word, out); first = false; }
            else words[word] = out;
            ++word;
            pending -= 32;
            acc &= (1ull << pending) - 1ull;
        }
    }
    __device__ __forceinline__ void finish()
    {
        if (pending > 0) {
            const uint32_t out = (uint32_t)(acc << (32 - pending));
            if (out) atomicOr(words + word, out);
        }
    }
};

// Bit writer into shared memory, words kStep bytes apart.  A word is stored (plain, predicated store)
// by the writer that supplies its last bit, nothing at or past `limit`; bits that other writers own
// in that word are zero in the stored value.  What is left after the last full word -- a
// writer's tail -- is merged afterwards with one shared-memory OR per writer (finish()), behind a
// barrier, so that it cannot be overwritten by the store of the word's last writer.  A put adds fewer
// than 32 bits (the pending count stays below 32 between puts).
template <int kStep>
struct SmemBitWriter {
    uint32_t addr, limit;      // shared addresses: of the word being filled, past the last word
    uint32_t lo, hi;           // pending bits, right-aligned in hi:lo (bits above `pending` are stale)
    int pending;
    __device__ __forceinline__ void init(uint32_t base_addr, uint32_t end_addr, unsigned int bitpos)
    {
        addr = base_addr + (bitpos >> 5) * (uint32_t)kStep;
        limit = end_addr;
        pending = (int)(bitpos & 31u);
        lo = hi = 0;
    }
    __device__ __forceinline__ void put(uint32_t code, int len)
    {
        // hi:lo <<= len; lo |= code; pending += len; if (pending >= 32) { store bits
        // [pending-32, pending) of hi:lo; addr += step; pending -= 32; }  (the funnel shift takes
        // its amount modulo 32, so `pending` itself serves as pending - 32)
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t.reg .b32 t, o;\n\t"
            "shf.l.wrap.b32 %1, %0, %1, %5;\n\t"
            "shl.b32 t, %0, %5;\n\t"
            "or.b32 %0, t, %4;\n\t"
            "add.s32 %2, %2, %5;\n\t"
            "setp.ge.s32 p, %2, 32;\n\t"
            "setp.lt.and.u32 q, %3, %6, p;\n\t"
            "shf.r.wrap.b32 o, %0, %1, %2;\n\t"
            "@q st.shared.u32 [%3], o;\n\t"
            "@p add.s32 %3, %3, %7;\n\t"
            "@p add.s32 %2, %2, -32;\n\t}"
            : "+r"(lo), "+r"(hi), "+r"(pending), "+r"(addr)
            : "r"(code), "r"(len), "r"(limit), "n"(kStep));
    }
    // 32 bits at once: the pending count stays
    __device__ __forceinline__ void put_word(uint32_t bits)
    {
        const uint32_t out = __funnelshift_r(bits, lo, pending);       // the pending bits, then the first of the new ones
        if (addr < limit) asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(out) : "memory");
        addr += kStep;
        lo = bits;
        hi = 0;
    }
    // call after a barrier that follows every writer's puts
    __device__ __forceinline__ void finish()
    {
        const uint32_t out = pending > 0 ? (lo << (32 - pending)) : 0u;
        if (out && addr < limit) asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(addr), "r"(out) : "memory");
    }
};

// Decoding with the bounds of a canonical code instead of a table of all bit patterns, for per-channel
// codes.  A table of 2^12 entries per channel lives in global memory (2 MB at 256 channels), and the
// length of a symbol -- which the next symbol waits for -- took a load from L2 each time.  The bounds
// are 24 bytes per channel at an address that does not depend on the stream, so they are loaded
// ahead; the length follows from eleven comparisons, two per packed add; the symbol itself
// (canon_symbol) is off the critical path.
struct CanonBounds {
    uint4 a;
    uint2 b;
};
__device__ __forceinline__ CanonBounds canon_bounds(const uint32_t *table)      // global memory, 16-byte aligned
{
    return {__ldg(reinterpret_cast<const uint4 *>(table)), __ldg(reinterpret_cast<const uint2 *>(table + 4))};
}
// length of the code that `window` starts with (left-aligned, at least 12 valid bits)
__device__ __forceinline__ uint32_t canon_length(uint32_t window, const CanonBounds &c)
{
    // a half-word's sum reaches bit 15 when the pattern lies past the codes of up to l bits
    const uint32_t v = (window >> 17) * 0x00010001u, m = 0x80008000u;
    const uint32_t s = ((v + c.a.x) & m) | (((v + c.a.y) & m) >> 1) | (((v + c.a.z) & m) >> 2) | (((v + c.a.w) & m) >> 3) |
                       (((v + c.b.x) & m) >> 4) | (((v + c.b.y) & m) >> 5);
    return 1u + (uint32_t)__popc(s);
}
// its symbol: `bases` = the code's half-words of bases, `sorted` = its symbols in code order
__device__ __forceinline__ uint32_t canon_place(uint32_t window, uint32_t len, const uint16_t *bases)
{
    return ((uint32_t)bases[len - 1] + (window >> (32 - len))) & 0xffffu;
}
__device__ __forceinline__ uint32_t canon_symbol(uint32_t window, uint32_t len, const uint16_t *bases, const uint8_t *sorted)
{
    return __ldg(sorted + canon_place(window, len, bases));
}

// MSB-first reader over 32-bit words with a 64-bit window held in two registers.  Words at or
// past `end` read as zero, so a corrupt offset can never cause an out-of-bounds load.
// kShared: the words lie in shared memory (a staged segment) instead of global memory.
template <bool kShared>
struct WindowReaderT {
    const uint32_t *words;
    unsigned long long next, end;     // word indices
    uint32_t hi, lo;                  // upcoming bits, left-aligned in hi:lo
    int avail;                        // valid bits in the window

    __device__ __forceinline__ uint32_t fetch()
    {
        uint32_t w = 0u;
        if (next < end) {
            if constexpr (kShared) w = words[next];
            else w = __ldg(words + next);
        }
        ++next;
        return w;
    }
    __device__ __forceinline__ void init(const uint32_t *base, unsigned long long bitpos, unsigned long long end_bits)
    {
        words = base;
        next = bitpos >> 5;
        end = end_bits >> 5;
        const uint32_t w0 = fetch(), w1 = fetch();
        const int sh = (int)(bitpos & 31);
        hi = __funnelshift_l(w1, w0, sh);
        lo = w1 << sh;
        avail = 64 - sh;
    }
    __device__ __forceinline__ uint32_t peek(int nbits) const { return hi >> (32 - nbits); }
    // nbits < 32
    __device__ __forceinline__ void skip(int nbits)
    {
        hi = __funnelshift_l(lo, hi, nbits);
        lo <<= nbits;
        avail -= nbits;
    }
    // keeps more than 32 valid bits in the window
    __device__ __forceinline__ void refill()
    {
        if (avail <= 32) {
            const uint32_t w = fetch();
            const int s = 32 - avail;                 // 0..31
            hi |= __funnelshift_l(w, 0u, s);
            lo |= w << s;
            avail += 32;
        }
    }
};
using WindowReader = WindowReaderT<false>;

// c[8 x 8] += a[8 x 4] b[4 x 8]: a lane holds a[lane / 4][lane % 4], b[lane % 4][lane / 4] and c[lane / 4][2 (lane % 4) + 0, 1]
__device__ __forceinline__ void mma_f64(double2 &c, double a, double b)
{
    asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c.x), "+d"(c.y) : "d"(a), "d"(b));
}


// every thread of the cluster has come; what they wrote (shared memory of any block, global memory) is visible
__device__ __forceinline__ void cluster_sync()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t peer_address(const void *p, uint32_t rank)
{
    uint32_t out;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return out;
}

}  // namespace tcdev
