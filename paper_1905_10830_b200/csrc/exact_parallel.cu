// Exact (fp64) projection and reconstruction with one thread per output value, for tensors of
// few pixels (the fp32 maps of one image: Section 4's ResNet-18 layers at batch 1).
//
// The exact encode / decode kernels give a pixel to a thread, which then walks C x K products
// alone: a 512 x 7 x 7 map keeps 49 threads busy for milliseconds.  Here every (pixel,
// coefficient) pair of the projection y_j = sum_c T[j][c] (x_c - mu_c) (Section 3, first
// equation) and every (pixel, channel) pair of the inverse x_hat_c = sum_j T[j][c] y_hat_j + mu_c
// is a thread of its own.  Each thread adds its products in the same order and with the same
// unfused double operations as the per-pixel kernels, so the results are bit-identical to theirs
// (and to the definition evaluated in fp64); the entropy coder then runs in the per-pixel kernels
// on the symbols these kernels leave in memory.
#include <algorithm>

#include "device_utils.cuh"

namespace {

using namespace tcdev;

constexpr int kPx = 32;        // pixels per block (one warp row: loads along the pixels coalesce)
constexpr int kOut = 16;       // coefficients (encode) or channels (decode) per block
constexpr int kPer = 4;        // of these, per thread
constexpr int kRows = kOut / kPer;
constexpr int kRed = 32;       // terms of the sums staged per step (channels in the projection, coefficients in the inverse)

// What bounds these two: shared-memory reads and, with few blocks, the chain of additions.  A thread adds
// up four outputs of a pixel, so that a term costs it one 8-byte read of its own and two broadcast reads of 16
// bytes, four wavefronts for four products, and four chains of additions are in flight (one output a thread took three
// wavefronts a product).  64x56x56 projection 9.7 -> 7.9 us, 256x14x14 reconstruction 11.9 -> 10.1.
template <typename TIn>
__global__ void __launch_bounds__(kPx * kRows) project_quantise_kernel(EncodeArgs a, uint8_t *sym)
{
    __shared__ __align__(16) uint8_t s_q[kPx][kOut];
    __shared__ float s_y[kPx][kOut + 1];
    // the operands of kRed terms of every sum of the block: centred pixels and basis entries
    __shared__ double s_d[kRed][kPx];
    __shared__ __align__(16) double s_t[kRed][kOut + 2];
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * kPx + tx;
    chain_next();
    chain_wait();
    const long long block = blockIdx.y * (long long)gridDim.x + blockIdx.x;
    for (long long i = block * (kPx * kRows) + t; i < a.clear_words; i += (long long)gridDim.x * gridDim.y * (kPx * kRows))
        reinterpret_cast<unsigned long long *>(a.ticket)[i] = 0ull;              // the coder's look-back state
    const long long p = (long long)blockIdx.x * kPx + tx;
    const int j0 = blockIdx.y * kOut;
    const int nsym = 1 << a.bits;
    const double top = (double)(nsym - 1);
    const bool p_ok = p < a.pixels;
    const long long img = p_ok ? p / a.hw : 0;
    const TIn *xp = reinterpret_cast<const TIn *>(a.x) + img * a.c * (long long)a.hw + (p_ok ? p - img * a.hw : 0);
    // staging roles: thread (tx, ty) fetches channels ty, ty + 4, ... of pixel tx, and channel tx of
    // coefficients ty, ty + 4, ...
    double d[kRed / kRows], mu[kRed / kRows], tv[kPer];
    auto fetch = [&](int c0) {
#pragma unroll
        for (int i = 0; i < kRed / kRows; ++i) {
            const int ch = c0 + ty + kRows * i;
            const bool ok = p_ok && ch < a.c;
            d[i] = ok ? (double)(float)xp[(long long)ch * a.hw] : 0.0;
            mu[i] = ok ? __ldg(a.mean64 + ch) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int j = j0 + ty + kRows * i;
            tv[i] = (j < a.k && c0 + tx < a.c) ? __ldg(a.basis64 + (long long)j * a.c + c0 + tx) : 0.0;
        }
    };
    double acc[kPer] = {};
    fetch(0);
    for (int c0 = 0; c0 < a.c; c0 += kRed) {
        __syncthreads();                               // the previous step's operands have been used
#pragma unroll
        for (int i = 0; i < kRed / kRows; ++i) s_d[ty + kRows * i][tx] = __dsub_rn(d[i], mu[i]);
#pragma unroll
        for (int i = 0; i < kPer; ++i) s_t[tx][ty + kRows * i] = tv[i];
        __syncthreads();
        if (c0 + kRed < a.c) fetch(c0 + kRed);         // in flight while this step is added up
        const int n = min(kRed, a.c - c0);
        // every sum takes its terms in channel order, one unfused multiply and add each
#pragma unroll 8
        for (int cc = 0; cc < n; ++cc) {
            const double x = s_d[cc][tx];
            const double2 u = *reinterpret_cast<const double2 *>(&s_t[cc][ty * kPer]), v = *reinterpret_cast<const double2 *>(&s_t[cc][ty * kPer + 2]);
            acc[0] = __dadd_rn(acc[0], __dmul_rn(u.x, x));
            acc[1] = __dadd_rn(acc[1], __dmul_rn(u.y, x));
            acc[2] = __dadd_rn(acc[2], __dmul_rn(v.x, x));
            acc[3] = __dadd_rn(acc[3], __dmul_rn(v.y, x));
        }
    }
    unsigned int clamped = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const double u = __ddiv_rn(__dsub_rn(acc[i], a.lo), a.step);
        double r = rint(u);
        if (p_ok && j0 + ty * kPer + i < a.k && (u < 0.0 || u > top)) ++clamped;
        r = fmin(fmax(r, 0.0), top);
        s_q[tx][ty * kPer + i] = (uint8_t)(unsigned int)r;
        s_y[tx][ty * kPer + i] = (float)acc[i];
    }
    if (a.clamped) {
        const unsigned int n = __reduce_add_sync(0xffffffffu, clamped);
        if (tx == 0 && n) atomicAdd(a.clamped, (unsigned long long)n);
    }
    __syncthreads();
    // a pixel's kOut symbols are contiguous in [P][K]
    if (a.k % kOut == 0 && ((uintptr_t)sym & 15u) == 0 && !a.dbg_sym && !a.dbg_coef) {
        const long long pp = (long long)blockIdx.x * kPx + t;
        if (t < kPx && pp < a.pixels) *reinterpret_cast<uint4 *>(sym + pp * a.k + j0) = *reinterpret_cast<const uint4 *>(s_q[t]);
        return;
    }
    for (int i = t; i < kPx * kOut; i += kPx * kRows) {
        const int px = i / kOut, jj = i - px * kOut;
        const long long pp = (long long)blockIdx.x * kPx + px;
        if (pp < a.pixels && j0 + jj < a.k) {
            const uint8_t q = s_q[px][jj];
            sym[pp * a.k + j0 + jj] = q;
            if (a.dbg_sym) a.dbg_sym[pp * a.k + j0 + jj] = q;
            if (a.dbg_coef) a.dbg_coef[pp * a.k + j0 + jj] = s_y[px][jj];
        }
    }
}

template <typename TOut>
__global__ void __launch_bounds__(kPx * kRows) reconstruct_kernel(DecodeArgs a, const uint8_t *sym)
{
    // operands of kRed terms of every sum of the block: dequantised coefficients and basis entries, each
    // computed or fetched once
    __shared__ double s_yh[kRed][kPx + 1];
    __shared__ __align__(16) double s_t[kRed][kOut];
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * kPx + tx;
    const long long p0 = (long long)blockIdx.x * kPx;
    const int n_px = (int)min((long long)kPx, a.pixels - p0);
    const long long p = p0 + tx;
    const int c0 = blockIdx.y * kOut;
    // staging roles: thread t fetches eight symbols of pixel t / 4, and the basis entries
    // (coef, ch) = (t / 16 + 8 i, t % 16) of a step
    constexpr int kQ = kPx * kRed / (kPx * kRows);
    const int q_px = t / (kRed / kQ), q_j = t % (kRed / kQ) * kQ, t_j = t / kOut, t_c = t % kOut;
    const uint8_t *src = sym + (p0 + q_px) * a.k;
    const bool by8 = a.k % 8 == 0 && ((uintptr_t)sym & 7u) == 0;
    uint32_t q[2];
    double tv[kRed / (kPx * kRows / kOut)];
    auto fetch = [&](int j0) {
        const int j = j0 + q_j;
        q[0] = q[1] = 0u;
        if (q_px < n_px) {
            if (by8) {
                if (j < a.k) {
                    const uint2 v = *reinterpret_cast<const uint2 *>(src + j);
                    q[0] = v.x; q[1] = v.y;
                }
            } else
                for (int i = 0; i < kQ; ++i)
                    if (j + i < a.k) q[i >> 2] |= (uint32_t)src[j + i] << (8 * (i & 3));
        }
#pragma unroll
        for (int i = 0; i < kRed / (kPx * kRows / kOut); ++i) {
            const int jt = j0 + t_j + kPx * kRows / kOut * i;
            tv[i] = (jt < a.k && c0 + t_c < a.c) ? __ldg(a.basis64 + (long long)jt * a.c + c0 + t_c) : 0.0;
        }
    };
    double acc[kPer] = {};
    chain_wait();                                      // the symbols
    chain_next();
    fetch(0);
    for (int j0 = 0; j0 < a.k; j0 += kRed) {
        __syncthreads();                               // the previous step's operands have been used
#pragma unroll
        for (int i = 0; i < kRed / (kPx * kRows / kOut); ++i) s_t[t_j + kPx * kRows / kOut * i][t_c] = tv[i];
#pragma unroll
        for (int i = 0; i < kQ; ++i) s_yh[q_j + i][q_px] = __dadd_rn(a.lo, __dmul_rn((double)(q[i >> 2] >> (8 * (i & 3)) & 0xffu), a.step));
        __syncthreads();
        if (j0 + kRed < a.k) fetch(j0 + kRed);         // in flight while this step is added up
        const int n = min(kRed, a.k - j0);
#pragma unroll 8
        for (int jj = 0; jj < n; ++jj) {
            const double y = s_yh[jj][tx];
            const double2 u = *reinterpret_cast<const double2 *>(&s_t[jj][ty * kPer]), v = *reinterpret_cast<const double2 *>(&s_t[jj][ty * kPer + 2]);
            acc[0] = __dadd_rn(acc[0], __dmul_rn(u.x, y));
            acc[1] = __dadd_rn(acc[1], __dmul_rn(u.y, y));
            acc[2] = __dadd_rn(acc[2], __dmul_rn(v.x, y));
            acc[3] = __dadd_rn(acc[3], __dmul_rn(v.y, y));
        }
    }
    if (tx >= n_px) return;
    const long long img = p / a.hw;
    TOut *out = reinterpret_cast<TOut *>(a.xhat) + img * a.c * (long long)a.hw + (p - img * a.hw);
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int c = c0 + ty * kPer + i;
        if (c >= a.c) break;
        double v = __dadd_rn(acc[i], __ldg(a.mean64 + c));
        if (a.relu && v < 0.0) v = 0.0;
        store_rounded(out + (long long)c * a.hw, v);
    }
}

// Entropy coder on symbols that already sit in memory ([P][K] bytes, row 0 = the first pixel of tile
// `first_tile`): one block per tile of 128 pixels, `parts` threads per pixel, each coding a run of
// K / parts consecutive coefficients (a multiple of 8, so that a thread fetches its symbols in 8-byte
// pieces and a chunk -- one of 1, 2 or 4 runs of a pixel -- is a whole number of thread runs).
// Code lengths first (the lookups of a run are independent loads), then the bit offsets -- runs
// inside a pixel, pixels inside the tile -- then every thread packs its run into words in
// shared memory (whole words by plain stores, its tail by an atomic OR), then the tile's place in the
// stream is found by look-back and the words leave 16 bytes at a time.  A tile that does not fit the
// staging buffer is packed into zeroed global memory.  Same stream, chunk lengths and tile offsets as the
// one-thread-per-pixel coder.
// What bounds it: instructions, about ten per symbol, and for few tiles the one block's latency -- hence
// up to eight threads a pixel, a per-layer table in shared memory and two codes a piece (960x7x7 x 128
// from a cold cache: 45 us with four threads, tables and packed words in global memory, 42 staged with an
// atomic OR a word, 22 like this).
// kCluster: a tile is dealt to the gridDim.y blocks of a cluster, each with the pixels of its own, where the tiles would leave most SMs
// idle.  The first block takes the ticket and finds the tile's place in the stream; the blocks exchange their bits through
// distributed shared memory, and a block hands the word that it shares with the block before to that one.
// 960x7x7 x 128 47.1 -> 41.0 us with the kernels before, 512x14x14 f32 56 -> 44, 768x7x7 x 16 26.7 -> 21.6.
constexpr int kMaxParts = 8, kMaxTileBlocks = 4;

template <bool kPerLayer, bool kCluster>
__global__ void __launch_bounds__(TC_TILE_PIXELS * kMaxParts) pack_symbols_kernel(EncodeArgs a, const uint8_t *sym, int parts, long long first_tile,
                                                                                  unsigned int staging_bytes)
{
    __shared__ long long s_tile;
    __shared__ unsigned int s_run_bits[TC_TILE_PIXELS * kMaxParts];
    __shared__ unsigned int s_warp_sums[4];
    __shared__ unsigned int s_pixel_off[TC_TILE_PIXELS + 1];
    __shared__ unsigned long long s_base;
    __shared__ int s_write_ok;
    __shared__ uint32_t s_enc[256];
    __shared__ unsigned int s_totals[kMaxTileBlocks], s_head;  // bits of every block of the cluster; the word shared with the next block
    extern __shared__ __align__(16) uint32_t s_words[];
    const int t = threadIdx.x;
    const int nsym = 1 << a.bits;
    const int blocks = kCluster ? (int)gridDim.y : 1, rank = kCluster ? (int)blockIdx.y : 0, block_px = TC_TILE_PIXELS / blocks;
    if constexpr (kCluster) { cluster_sync(); }               // the others run: their shared memory may be written
    if constexpr (kPerLayer)
        for (int i = t; i < nsym; i += blockDim.x) s_enc[i] = __ldg(a.enc + i);
    chain_wait();                                             // the symbols and the cleared look-back state
    chain_next();
    if (t == 0 && rank == 0) {
        s_tile = (long long)atomicAdd(a.ticket, 1u);
        if constexpr (kCluster) {
            for (int r = 1; r < blocks; ++r)
                asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(peer_address(&s_tile, r)), "l"(s_tile) : "memory");
        }
    }
    if constexpr (kCluster) { cluster_sync(); }
    else { __syncthreads(); }
    const long long tile = s_tile;
    const int px = t / parts, part = t - px * parts;          // of the block's pixels; the threads of a pixel are neighbours
    const long long p = tile * TC_TILE_PIXELS + rank * block_px + px;
    const bool valid = p < a.pixels;
    const int run = a.k / parts, j0 = part * run;
    const uint8_t *src = sym + (p - first_tile * TC_TILE_PIXELS) * a.k + j0;
    // code << 8 | length of the symbol in byte b of w, coefficient j
    auto entry = [&](uint32_t w, int b, int j) {
        const uint32_t q = (w >> (8 * b)) & 0xffu;
        if constexpr (kPerLayer) return s_enc[q];
        else return __ldg(a.enc + j * nsym + q);
    };

    unsigned int my_bits = 0;
    if (valid)
#pragma unroll 4
        for (int i = 0; i < run; i += 8) {
            const uint2 v = *reinterpret_cast<const uint2 *>(src + i);
#pragma unroll
            for (int b = 0; b < 8; ++b) my_bits += entry(b < 4 ? v.x : v.y, b & 3, j0 + i + b) & 0xffu;
        }
    s_run_bits[t] = my_bits;
    __syncthreads();
    // pixel totals, scanned by the first 128 threads
    if (t < TC_TILE_PIXELS) {
        unsigned int pixel_bits = 0, total = 0;
        for (int r = 0; r < parts && t < block_px; ++r) pixel_bits += s_run_bits[t * parts + r];
        const unsigned int off = group_exclusive_scan_128(pixel_bits, s_warp_sums, t, 1, total);
        s_pixel_off[t] = off;
        if (t == 0) s_pixel_off[TC_TILE_PIXELS] = total;
        if constexpr (kCluster) {
            if (t < blocks) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_address(s_totals + rank, t)), "r"(total) : "memory");
        } else if (t == 0) lookback_publish(a.tile_state, tile, ((unsigned long long)total + 127ull) & ~127ull);
    }
    unsigned int tile_bits, block_off = 0;                    // bits of the tile, and of its blocks before this one
    if constexpr (kCluster) {
        cluster_sync();
        tile_bits = 0;
        for (int r = 0; r < blocks; ++r) {
            if (r < rank) block_off += s_totals[r];
            tile_bits += s_totals[r];
        }
        if (t == 0 && rank == 0) lookback_publish(a.tile_state, tile, ((unsigned long long)tile_bits + 127ull) & ~127ull);
    } else {
        __syncthreads();
        tile_bits = s_pixel_off[TC_TILE_PIXELS];
    }
    const unsigned long long padded = ((unsigned long long)tile_bits + 127ull) & ~127ull;
    const bool staged = padded <= (unsigned long long)staging_bytes * 8ull;
    unsigned int my_off = block_off + s_pixel_off[px];
    for (int r = 0; r < part; ++r) my_off += s_run_bits[px * parts + r];
    // chunk lengths: a chunk is chunk_pixels pixels, or one of `splits` runs of one pixel
    if (valid) {
        if (a.splits > 1) {
            const int per_chunk = parts / a.splits;
            if (part % per_chunk == 0) {
                unsigned int bits = 0;
                for (int r = 0; r < per_chunk; ++r) bits += s_run_bits[t + r];
                a.chunk_len[p * a.splits + part / per_chunk] = (uint16_t)bits;
            }
        } else if (part == 0 && (p % a.chunk_pixels) == 0) {
            const int last = min(px + a.chunk_pixels, block_px);
            a.chunk_len[p / a.chunk_pixels] = (uint16_t)(s_pixel_off[last] - s_pixel_off[px]);
        }
    }
    // the tile's place in the stream (one warp; without staging everyone needs it first)
    auto resolve = [&] {
        if (t < 32) {
            bool ok;
            const unsigned long long base = lookback_resolve(a.tile_state, tile, padded, a.status, ok);
            if (t == 0) {
                const bool fits = base + padded <= a.capacity_bits;
                if (ok && !fits) tc_dev_set_status(a.status, TC_ERR_BUFFER_TOO_SMALL);
                s_base = base;
                s_write_ok = (ok && fits) ? 1 : 0;
                a.tile_off[tile] = base;
                if (tile == a.n_tiles - 1) a.tile_off[a.n_tiles] = base + padded;
            }
        }
    };
    auto pack = [&](auto &w) {
        uint2 next = *reinterpret_cast<const uint2 *>(src);
#pragma unroll 1
        for (int i = 0; i < run; i += 8) {
            const uint2 v = next;
            if (i + 8 < run) next = *reinterpret_cast<const uint2 *>(src + i + 8);
#pragma unroll
            for (int b = 0; b < 8; b += 2) {                  // two codes a piece, at most 24 bits
                const uint32_t x = b < 4 ? v.x : v.y;
                const uint32_t e0 = entry(x, b & 3, j0 + i + b), e1 = entry(x, (b & 3) + 1, j0 + i + b + 1);
                w.put(((e0 >> 8) << (e1 & 0xffu)) | (e1 >> 8), (int)((e0 & 0xffu) + (e1 & 0xffu)));
            }
        }
    };
    const unsigned int n16 = (unsigned int)(padded >> 7);
    // the place that the first block found, for all of its cluster
    auto resolve_for_all = [&] {
        if (rank != 0) return;
        resolve();
        if (t == 0) {
            for (int r = 1; r < blocks; ++r) {
                asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(peer_address(&s_base, r)), "l"(s_base) : "memory");
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_address(&s_write_ok, r)), "r"(s_write_ok) : "memory");
            }
        }
    };
    if constexpr (kCluster) {
        const unsigned int my_bits_all = s_totals[rank], next_off = block_off + my_bits_all, end_word = n16 * 4;
        if (staged) {
            // This block's words: from the first that starts in its bits to the first that starts in the next block's (the last block: to
            // the tile's end).  Word w lies at s_words[w - from].
            const unsigned int from = (block_off >> 5) & ~3u, w_lo = (block_off + 31) >> 5, w_hi = rank == blocks - 1 ? end_word : (next_off + 31) >> 5;
            const uint32_t words = (uint32_t)__cvta_generic_to_shared(s_words) - from * 4u;
            const unsigned int first_open = next_off >> 5;
            if (first_open + t < w_hi) s_words[first_open + t - from] = 0u;
            SmemBitWriter<4> w;
            w.init(words, words + w_hi * 4u, my_off);
            if (valid) pack(w);
            __syncthreads();
            if (valid) w.finish();
            __syncthreads();
            if (t == 0 && my_bits_all && (block_off & 31u) != 0)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_address(&s_head, rank - 1)), "r"(s_words[(block_off >> 5) - from]) : "memory");
            resolve_for_all();
            cluster_sync();
            if (!s_write_ok) return;
            if (rank < blocks - 1 && (next_off & 31u) != 0 && s_totals[rank + 1]) {
                if (t == 0) s_words[first_open - from] |= s_head;
                __syncthreads();
            }
            uint32_t *dst = a.stream + (s_base >> 5);
            for (unsigned int i = (w_lo & ~3u) + 4 * t; i < w_hi; i += 4 * blockDim.x) {
                if (i >= w_lo && i + 4 <= w_hi) *reinterpret_cast<uint4 *>(dst + i) = *reinterpret_cast<const uint4 *>(s_words + (i - from));
                else
                    for (unsigned int k = max(i, w_lo); k < min(i + 4, w_hi); ++k) dst[k] = s_words[k - from];
            }
        } else {
            resolve_for_all();
            cluster_sync();
            uint4 *dst = reinterpret_cast<uint4 *>(a.stream + (s_base >> 5));
            for (unsigned int i = rank * blockDim.x + t; s_write_ok && i < n16; i += blocks * blockDim.x) dst[i] = make_uint4(0u, 0u, 0u, 0u);
            cluster_sync();
            if (s_write_ok && valid) {
                BitWriter w;
                w.init(a.stream, s_base + my_off);
                pack(w);
                w.finish();
            }
        }
    } else if (staged) {
        // every word below tile_bits / 32 is stored by the writer of its last bit; the rest starts as zero
        const unsigned int first_open = tile_bits >> 5, end_word = n16 * 4;
        const uint32_t words = (uint32_t)__cvta_generic_to_shared(s_words);
        if (t < end_word - first_open) s_words[first_open + t] = 0u;
        SmemBitWriter<4> w;
        w.init(words, words + end_word * 4u, my_off);
        if (valid) pack(w);
        __syncthreads();
        if (valid) w.finish();
        resolve();
        __syncthreads();
        if (!s_write_ok) return;
        uint4 *dst = reinterpret_cast<uint4 *>(a.stream + (s_base >> 5));
        for (unsigned int i = t; i < n16; i += blockDim.x) dst[i] = reinterpret_cast<const uint4 *>(s_words)[i];
    } else {
        resolve();
        __syncthreads();
        if (!s_write_ok) return;
        uint4 *dst = reinterpret_cast<uint4 *>(a.stream + (s_base >> 5));
        for (unsigned int i = t; i < n16; i += blockDim.x) dst[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        if (valid) {
            BitWriter w;
            w.init(a.stream, s_base + my_off);
            pack(w);
            w.finish();
        }
    }
}

// Entropy decoder that leaves the symbols in memory, row 0 = the first pixel of tile `first_tile`: as bytes
// ([P][K], for the fp64 inverse of tensors of few pixels), or centred and as bf16 (kOperand: the
// operand of the tensor cores' inverse transform):
// one thread per chunk (up to 512 per tile), so that every chunk of the tile is
// walked at the same time; the inverse transform then runs in reconstruct_kernel.  A tile's chunks may be dealt to
// gridDim.y blocks, each with the pixels of its own.  Same checks as
// the per-pixel decoder: tile offsets aligned, ordered and inside the stream, every chunk inside
// its tile and consumed to exactly its recorded length.
constexpr int kUnpackThreads = 512;
constexpr int kFirstBits = 6;                                  // of a per-layer code: lengths that the first table resolves
constexpr uint32_t kRowBytes = 80;                            // 32 symbols of a row, padded: the lanes' 16-byte pieces fall into all banks
constexpr uint32_t kRowsWarpBytes = 32 * kRowBytes;

// MSB-first reader with a 64-bit window hi:lo (left-aligned) and the word behind it already loaded: a
// refill never waits for memory.  Words at or past `end` read as zero.  kEarly: of a kernel that was launched early, for which the stream is
// no read-only memory (64x56x56 x 64 with a table per channel 45.6 us through the read-only path, 46.8 past it).
template <bool kEarly>
struct AheadReader {
    const uint32_t *next, *end;
    uint32_t hi, lo, ahead;
    int avail;                   // valid bits in the window

    __device__ __forceinline__ uint32_t fetch()
    {
        const uint32_t v = kEarly ? stream_word(next, end) : next < end ? __ldg(next) : 0u;
        ++next;
        return v;
    }
    __device__ __forceinline__ void init(const uint32_t *base, unsigned long long bitpos, unsigned long long end_bits)
    {
        next = base + (bitpos >> 5);
        end = base + (end_bits >> 5);
        const uint32_t w0 = fetch(), w1 = fetch();
        ahead = fetch();
        const int sh = (int)(bitpos & 31);
        hi = __funnelshift_l(w1, w0, sh);
        lo = w1 << sh;
        avail = 64 - sh;
    }
    __device__ __forceinline__ void skip(uint32_t nbits)         // below 32
    {
        hi = __funnelshift_l(lo, hi, nbits);
        lo <<= nbits;
        avail -= (int)nbits;
    }
    // more than 32 valid bits: enough for two codes
    __device__ __forceinline__ void refill()
    {
        if (avail <= 32) {
            const int s = 32 - avail;                 // 0..31
            hi |= __funnelshift_l(ahead, 0u, s);
            lo |= ahead << s;
            avail += 32;
            ahead = fetch();
        }
    }
};

// The same over a segment staged in shared memory, without a branch: `used` counts the bits taken since the
// window last moved on by a word.
struct StagedReader {
    uint32_t next, end;          // shared addresses
    uint32_t hi, lo, ahead, used;

    __device__ __forceinline__ uint32_t fetch()
    {
        uint32_t v = 0;
        if (next < end) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(next));
        next += 4;
        return v;
    }
    __device__ __forceinline__ void init(uint32_t base, unsigned int bitpos, uint32_t end_addr)
    {
        next = base + (bitpos >> 5) * 4u;
        end = end_addr;
        const uint32_t w0 = fetch(), w1 = fetch();
        ahead = fetch();
        used = bitpos & 31u;
        hi = __funnelshift_l(w1, w0, used);
        lo = w1 << used;
    }
    __device__ __forceinline__ void skip(uint32_t nbits)
    {
        hi = __funnelshift_l(lo, hi, nbits);
        lo = __funnelshift_l(0u, lo, nbits);
        used += nbits;
    }
    __device__ __forceinline__ void refill()
    {
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t.reg .b32 t, u;\n\t"
            "setp.ge.u32 p, %3, 32;\n\t"
            "setp.lt.and.u32 q, %4, %5, p;\n\t"
            "shf.l.wrap.b32 t, %2, 0, %3;\n\t"      // ahead >> (32 - (used - 32)); the shifts take their amount modulo 32
            "shf.l.wrap.b32 u, 0, %2, %3;\n\t"
            "@p or.b32 %0, %0, t;\n\t"
            "@p or.b32 %1, %1, u;\n\t"
            "@p add.u32 %3, %3, -32;\n\t"
            "@p mov.b32 %2, 0;\n\t"
            "@q ld.shared.u32 %2, [%4];\n\t"
            "@p add.u32 %4, %4, 4;\n\t}"
            : "+r"(hi), "+r"(lo), "+r"(ahead), "+r"(used), "+r"(next) : "r"(end));
    }
};

// The zero level in n coefficients from j on of the pixels px0, px0 + step, ... below px1 (a function of its own: nothing of it
// in the registers of the tiles that decode).
template <bool kOperand>
__device__ __noinline__ void clear_rows(void *out, long long row0, int px0, int px1, int step, int k, int j, int n, int center)
{
    for (int px = px0; px < px1; px += step)
        for (int i = j; i < j + n; ++i) {
            if constexpr (kOperand) ((uint16_t *)out)[(row0 + px) * k + i] = 0;
            else ((uint8_t *)out)[(row0 + px) * k + i] = (uint8_t)center;
        }
}

// What bounds it: the chain length -> shift -> length of a chunk's symbols, with a handful of warps on
// the chip (a 256x14x14 map has two tiles).  Per-layer tables are staged in shared memory; of
// per-channel codes the bounds are (K x 48 bytes, read ahead of the symbol), and the symbols in code
// order while they are few.  These are looked up eight at a time behind the chain: one lookup after each
// symbol made every step wait for a load from L2, which shares its scoreboard with the chain's
// shared-memory loads.  The tile's segment is staged too: read from global memory, a word
// ahead or not, any lane's refill waits for the last lane's load, which is in the same register.  The
// threads of a warp walk the same run of coefficients of neighbouring pixels, and symbols leave
// eight at a time.  256x14x14 f32 at 6 bits, with the inverse transform and the launches: 64.5 us with a
// 2^12-entry table per channel in global memory and a byte stored per symbol, 40 with bounds, 35 with the
// staged segment, 27 with the symbols looked up behind the chain and per-channel codes in an
// instantiation of their own (the choice inside the loop kept the bounds from being read ahead).
// kFull: with many warps on an SM the shared-memory pipe bounds it instead, eleven wavefronts a step of a warp:
// bank conflicts of the 2^12-entry table (seven), and the stores, a row each per lane (four).  Codes of up to six bits then
// come from a table that every lane has in a bank of its own, and rows leave 64 bytes at a time.  576x14x14 x 1024
// decode 376 -> 341 us, x 128 (21 warps an SM) 60.5 -> 57.1; 384x14x14 x 128 (5 warps) would lose, 39.1 -> 41.5, to the
// second lookup in the chain, 512x7x7 x 64 (25 tiles) 23.3 -> 27.3.
// Two or four blocks a tile where that leaves no SM with two: the eight or sixteen warps of a tile share an SM's issue slots while others
// idle (256x14x14 f32, per-channel codes, with the inverse 23.8 -> 21.5 us, 512x14x14 f32 45 -> 37, 768x7x7 x 16 26.7 -> 22.6).
template <bool kOperand, bool kPerLayer, bool kFull, bool kEarly>
__global__ void __launch_bounds__(kUnpackThreads) unpack_symbols_kernel(DecodeArgs a, void *out, long long first_tile, unsigned int table_bytes,
                                                                         unsigned int segment_bytes)
{
    __shared__ uint32_t s_first[kFull ? (32 << kFirstBits) : 1];
    __shared__ unsigned int s_warp_sums[kUnpackThreads / 32], s_before[kUnpackThreads / 32];
    __shared__ unsigned int s_start[kUnpackThreads];
    extern __shared__ __align__(16) unsigned char s_tables[];   // the per-layer table, or the bounds and bases of every channel's code
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    chain_next();
    const int lut_size = 1 << a.lut_bits, nsym = 1 << a.bits;
    // per-layer table: value << 16 | length, the value being the symbol or its centred bf16
    uint32_t *s_lut = reinterpret_cast<uint32_t *>(s_tables), *s_canon = s_lut;
    auto value = [&](uint32_t q) { return kOperand ? __float_as_uint((float)((int)q - a.center)) >> 16 : q; };
    const uint32_t tables = (uint32_t)__cvta_generic_to_shared(s_tables);
    const uint32_t s_sorted = tables + (uint32_t)a.k * kCanonWords * 4u;          // of per-channel codes, when there is room
    const bool sorted_staged = !kPerLayer && table_bytes > (unsigned int)a.k * kCanonWords * 4u;
    auto stage = [&](uint32_t dst, const void *src, unsigned int n16) {           // pieces of 16 bytes
        for (unsigned int i = t; i < n16; i += blockDim.x)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * 16u), "l"(reinterpret_cast<const uint4 *>(src) + i) : "memory");
    };
    if constexpr (kPerLayer) {
        for (int i = t; i < lut_size; i += blockDim.x) {
            const uint32_t e = __ldg(a.lut + i);
            s_lut[i] = (value(e >> 8) << 16) | (e & 0xffu);
        }
        // the codes of up to kFirstBits bits, every lane's copy in a bank of its own; longer ones: 0
        if constexpr (kFull)
            for (int i = warp; i < (1 << kFirstBits); i += blockDim.x / 32) {
                const uint32_t e = __ldg(a.lut + (a.lut_bits >= kFirstBits ? i << (a.lut_bits - kFirstBits) : i >> (kFirstBits - a.lut_bits)));
                s_first[i * 32 + lane] = (e & 0xffu) <= kFirstBits ? (value(e >> 8) << 16) | (e & 0xffu) : 0u;
            }
    } else {
        stage(tables, a.canon, (unsigned int)a.k * kCanonWords / 4u);
        if (sorted_staged) stage(s_sorted, a.sorted, (unsigned int)(a.k * nsym) / 16u);
    }
    chain_wait();                                               // the stream; earlier readers of the workspace
    const long long tile = first_tile + blockIdx.x;
    const unsigned long long base = a.tile_off[tile], end = a.tile_off[tile + 1];
    const bool tile_ok = (base & 127ull) == 0 && (end & 127ull) == 0 && base <= end && end <= a.stream_bits;
    // Rows that are not decoded hold the zero level (centred: 0; with kFull, whose lanes keep step, what zero bits
    // decode to), not what the workspace held before.
    auto clear = [&](int px0, int px1, int step, int j, int n) {       // n coefficients from j on of pixels of the tile
        const int n_px = (int)min((long long)TC_TILE_PIXELS, a.pixels - tile * TC_TILE_PIXELS);
        clear_rows<kOperand>(out, (tile - first_tile) * TC_TILE_PIXELS, px0, min(px1, n_px), step, a.k, j, n, a.center);
    };
    // this block's chunks of the tile, and their pixels
    const int chunks_per_tile = a.splits * TC_TILE_PIXELS / a.chunk_pixels;      // at most 512
    const int per = chunks_per_tile / (int)gridDim.y, c_first = (int)blockIdx.y * per;
    const int block_px = TC_TILE_PIXELS / (int)gridDim.y, px_first = (int)blockIdx.y * block_px;
    if (!tile_ok) {
        clear(px_first + t, px_first + block_px, blockDim.x, 0, a.k);
        if (t == 0) tc_dev_set_status(a.status, TC_ERR_CORRUPT_STREAM);
        return;
    }
    const bool staged = end - base <= (unsigned long long)segment_bytes * 8ull;
    const uint32_t seg = tables + table_bytes;
    if (staged) stage(seg, a.stream + (base >> 5), (unsigned int)((end - base) >> 7));
    // where every chunk of the block starts: the lengths of its tile's earlier chunks
    const long long tile_ch = tile * chunks_per_tile;
    const unsigned int len_t = (t < per && tile_ch + c_first + t < a.n_chunks) ? a.chunk_len[tile_ch + c_first + t] : 0u;
    unsigned int inc = len_t, before = 0;
    for (int i = t; i < c_first; i += blockDim.x) before += tile_ch + i < a.n_chunks ? a.chunk_len[tile_ch + i] : 0u;
    before = __reduce_add_sync(0xffffffffu, before);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned int up = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += up;
    }
    if (lane == 31) { s_warp_sums[warp] = inc; s_before[warp] = before; }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    unsigned int off_t = inc - len_t;
    for (int w = 0; w < warp; ++w) off_t += s_warp_sums[w];
    if (c_first)
        for (int w = 0; w < (int)blockDim.x / 32; ++w) off_t += s_before[w];
    s_start[t] = off_t;
    __syncthreads();
    // this thread's chunk: chunk_pixels whole pixels, or one of `splits` runs of one pixel (the threads of a warp take the same run)
    const int part = a.splits > 1 ? t / block_px : 0, my_px = a.splits > 1 ? px_first + t % block_px : px_first + t * a.chunk_pixels;
    const int in_block = a.splits > 1 ? (t % block_px) * a.splits + part : t;
    const long long ch = tile_ch + c_first + in_block;
    if (warp * 32 >= per) return;
    // a lane without a chunk walks zeros beside its warp where the warp's rows leave together
    const bool mine = t < per && ch < a.n_chunks;
    if (!kFull && !mine) return;
    const unsigned int want = mine ? a.chunk_len[ch] : 0u, off = mine ? s_start[in_block] : 0u;
    bool bad = base + off + want > end;
    auto walk = [&](auto &r) {
        unsigned int used = 0;
        const int run = a.k / a.splits, j_first = part * run;
        const int first_px = my_px;
        // decodes kN symbols from coefficient j on into v (one per element)
        auto decode = [&](int j, auto &v) {
            constexpr int kN = sizeof(v) / sizeof(v[0]);
#pragma unroll
            for (int i = 0; i < kN; ++i) {
                if ((i & 1) == 0) r.refill();
                uint32_t len;
                if constexpr (kPerLayer) {
                    uint32_t e;
                    if constexpr (kFull) {
                        e = s_first[(r.hi >> (32 - kFirstBits)) * 32 + lane];
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %0, 0;\n\t@p ld.shared.u32 %0, [%1];\n\t}"
                                     : "+r"(e) : "r"(tables + (r.hi >> (32 - a.lut_bits)) * 4u));
                    } else
                        e = s_lut[r.hi >> (32 - a.lut_bits)];
                    len = e & 0xffu;
                    v[i] = e >> 16;
                } else {
                    const uint32_t *c = s_canon + (j + i) * kCanonWords;
                    const CanonBounds cb{*reinterpret_cast<const uint4 *>(c), *reinterpret_cast<const uint2 *>(c + 4)};
                    len = canon_length(r.hi, cb);
                    v[i] = canon_place(r.hi, len, reinterpret_cast<const uint16_t *>(c + 6));
                }
                r.skip(len);
                used += len;
            }
            if constexpr (!kPerLayer) {
                if (sorted_staged) {
#pragma unroll
                    for (int i = 0; i < kN; ++i)
                        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v[i]) : "r"(s_sorted + (uint32_t)((j + i) * nsym) + v[i]));
                } else {
#pragma unroll
                    for (int i = 0; i < kN; ++i) v[i] = __ldg(a.sorted + (size_t)(j + i) * nsym + v[i]);
                }
#pragma unroll
                for (int i = 0; i < kN; ++i) v[i] = value(v[i]);
            }
        };
        if constexpr (kFull) {
            // runs are multiples of 8; 32 symbols of the warp's 32 rows are turned through shared memory, so that a
            // store covers 64 bytes of a row
            const uint32_t rows = tables + table_bytes + segment_bytes + (uint32_t)warp * kRowsWarpBytes;
            const int per_lane = a.splits > 1 ? 1 : a.chunk_pixels, px0 = px_first + (a.splits > 1 ? (warp * 32) % block_px : warp * 32 * per_lane);
            for (int lp = 0; lp < per_lane; ++lp) {
                const unsigned int used_before = used;
#pragma unroll 1
                for (int j = j_first; j < j_first + run; j += 32) {
                    const int n8 = min(4, (j_first + run - j) >> 3);
#pragma unroll 1
                    for (int g = 0; g < n8; ++g) {
                        uint32_t v[8];
                        decode(j + 8 * g, v);
                        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(rows + lane * kRowBytes + g * 16u), "r"(v[0] | (v[1] << 16)),
                                     "r"(v[2] | (v[3] << 16)), "r"(v[4] | (v[5] << 16)), "r"(v[6] | (v[7] << 16)) : "memory");
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int row = (lane >> 2) + 8 * i, px = px0 + row * per_lane + lp;
                        const long long p = tile * TC_TILE_PIXELS + px;
                        uint4 q;
                        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                                     : "r"(rows + row * kRowBytes + (lane & 3) * 16u));
                        if ((lane & 3) < n8 && px < TC_TILE_PIXELS && p < a.pixels)
                            *reinterpret_cast<uint4 *>((uint16_t *)out + (p - first_tile * TC_TILE_PIXELS) * a.k + j + (lane & 3) * 8) = q;
                    }
                    __syncwarp();
                }
                if (tile * TC_TILE_PIXELS + first_px + lp >= a.pixels) used = used_before;        // a pixel that does not exist
            }
        } else {
            const bool by8 = a.k % 8 == 0 && run % 8 == 0;
            for (int lp = first_px; lp < first_px + (a.splits > 1 ? 1 : a.chunk_pixels); ++lp) {
                const long long p = tile * TC_TILE_PIXELS + lp;
                if (p >= a.pixels) break;
                const long long row = (p - first_tile * TC_TILE_PIXELS) * a.k;
                if (by8) {
#pragma unroll 1
                    for (int j = j_first; j < j_first + run; j += 8) {
                        uint32_t v[8];
                        decode(j, v);
                        if constexpr (kOperand)
                            *reinterpret_cast<uint4 *>((uint16_t *)out + row + j) =
                                make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
                        else
                            *reinterpret_cast<uint2 *>((uint8_t *)out + row + j) =
                                make_uint2(v[0] | (v[1] << 8) | (v[2] << 16) | (v[3] << 24), v[4] | (v[5] << 8) | (v[6] << 16) | (v[7] << 24));
                    }
                } else {
#pragma unroll 1
                    for (int j = j_first; j < j_first + run; ++j) {
                        uint32_t v[1];
                        decode(j, v);
                        if constexpr (kOperand) ((uint16_t *)out)[row + j] = (uint16_t)v[0];
                        else ((uint8_t *)out)[row + j] = (uint8_t)v[0];
                    }
                }
            }
        }
        if (mine && used != want) bad = true;
    };
    const bool walks = mine && !bad;
    if (!kFull && !walks) {
        clear(my_px, my_px + a.chunk_pixels, 1, part * (a.k / a.splits), a.k / a.splits);
    } else if (staged) {
        StagedReader r;
        r.init(seg, walks ? off : 0u, walks ? seg + (uint32_t)((end - base) >> 3) : seg);
        walk(r);
    } else {
        AheadReader<kEarly> r;
        r.init(a.stream, base + (walks ? off : 0u), walks ? end : base);
        walk(r);
    }
    if (bad) tc_dev_set_status(a.status, TC_ERR_CORRUPT_STREAM);
}

}  // namespace

// For the tests.
extern "C" size_t tc_spread_bytes(long long blocks, int sm_count, size_t own) { return spread_bytes(blocks, sm_count, own); }

tc_status tc_launch_project_quantise(const EncodeArgs &a, int dtype, uint8_t *sym, cudaStream_t s)
{
    if (a.pixels <= 0) return TC_OK;
    const dim3 block(kPx, kRows), grid((unsigned int)((a.pixels + kPx - 1) / kPx), (unsigned int)((a.k + kOut - 1) / kOut));
    void (*kernel)(EncodeArgs, uint8_t *) = dtype == TC_F32 ? project_quantise_kernel<float> : project_quantise_kernel<__nv_bfloat16>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpreadMost) != cudaSuccess) return TC_ERR_CUDA;
    // Early where that leaves the basis in L1: with several blocks an SM kept apart by shared memory wide layers lose (512x14x14 f32, 224
    // blocks, 39.0 -> 43.6 us, 176x34x33 22.6 -> 24.3; 32x56x56 10.2 -> 8.3, 96x45x45 15.8 -> 15.3, 256x7x7 20.5 -> 18.8).
    const long long blocks = (long long)grid.x * grid.y;
    static std::atomic<size_t> own[2];
    const size_t spread = a.alone && (blocks <= a.sms || a.c <= 128) ? spread_bytes(blocks, a.sms, static_bytes(own[dtype != TC_F32], (const void *)kernel)) : 0;
    return launch_first(spread > 0, kernel, grid, block, spread, s, a, sym) == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_reconstruct(const DecodeArgs &a, int dtype, const uint8_t *sym, cudaStream_t s)
{
    if (a.pixels <= 0) return TC_OK;
    const dim3 block(kPx, kRows), grid((unsigned int)((a.pixels + kPx - 1) / kPx), (unsigned int)((a.c + kOut - 1) / kOut));
    void (*kernel)(DecodeArgs, const uint8_t *) = dtype == TC_F32 ? reconstruct_kernel<float> : reconstruct_kernel<__nv_bfloat16>;
    // Its blocks are there before the entropy decoder's are done, whose shared memory keeps them off the SMs with one, and pile onto others: kept apart where
    // an SM gets several (f32, us without and with: 256x8x16 x 10 47.0 and 31.6, 128x8x16 x 20 27.7 and 20.0, 64x8x16 x 36 18.1 and 15.1; fewer or
    // lighter ones lose by it, 32x8x16 x 17 13.4 and 14.2, 64x8x16 x 26 13.3 and 13.9; so do those that would fill all places, of which the decoder's blocks still have
    // some, 337x8x16 x 13, 7.7 blocks an SM, 111 and 117, 480x8x16 x 9, 7.3, 84.4 and 77.5; more than eight are even).
    const long long blocks = (long long)grid.x * grid.y;
    static std::atomic<size_t> own[2];
    const size_t spread = a.alone && blocks > (a.k >= 128 ? 2 : 3) * (long long)a.sms && 2 * blocks <= 15ll * a.sms ? spread_bytes(blocks, a.sms, static_bytes(own[dtype != TC_F32], (const void *)kernel)) : 0;
    if (spread > 0 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpreadMost) != cudaSuccess) return TC_ERR_CUDA;
    return launch_chained(a.alone, kernel, grid, block, spread, s, a, sym) == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

// How many threads per pixel the parallel coder would use for K coefficients and `splits` chunks
// per pixel: the largest of 8, 4, 2, 1 that gives every thread a multiple of 8 coefficients and
// every chunk a whole number of threads (0: none, use the one-thread-per-pixel coder).
int tc_pack_symbols_parts(const EncodeArgs &a)
{
    if (((uintptr_t)a.stream & 15u) != 0) return 0;
    for (int parts = kMaxParts; parts >= 1; parts >>= 1)
        if (a.k % (8 * parts) == 0 && parts % a.splits == 0) return parts;
    return 0;
}

// Coefficients from which a tile is worth a cluster: its barriers cost 2 us (64x56x56 f32 14.3 -> 15.8 us, 128 to 256 coefficients
// even, 384x7x7 x 64 20.5 -> 18.5).
constexpr int kClusterCoefs = 384;

tc_status tc_launch_pack_symbols(const tc_ctx *ctx, const EncodeArgs &a, const uint8_t *sym, long long first_tile, long long end_tile, cudaStream_t s)
{
    if (end_tile <= first_tile) return TC_OK;
    const int parts = tc_pack_symbols_parts(a);
    if (parts == 0 || ((uintptr_t)sym & 7u) != 0) return TC_ERR_UNSUPPORTED;
    // staging for four bits per symbol, at most 96 KB: two blocks of 1024 threads still fit an SM
    const unsigned int staging = (unsigned int)std::min<long long>((long long)a.k * TC_TILE_PIXELS / 2, 96 * 1024);
    const long long tiles = end_tile - first_tile;
    // Blocks of a tile: two or four while all of them fit the SMs side by side, each has the threads for the scan and no chunk reaches
    // over a block's end.
    int tile_blocks = 1;
    while (tile_blocks < kMaxTileBlocks && a.alone && a.k >= kClusterCoefs && tiles * tile_blocks * 2 <= ctx->sm_count &&
           TC_TILE_PIXELS / (2 * tile_blocks) * parts >= 128 && a.chunk_pixels <= TC_TILE_PIXELS / (2 * tile_blocks))
        tile_blocks *= 2;
    void (*kernel)(EncodeArgs, const uint8_t *, int, long long, unsigned int) =
        tile_blocks > 1 ? (a.groups == 1 ? pack_symbols_kernel<true, true> : pack_symbols_kernel<false, true>)
                        : (a.groups == 1 ? pack_symbols_kernel<true, false> : pack_symbols_kernel<false, false>);
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpreadMost) != cudaSuccess) return TC_ERR_CUDA;
    const dim3 grid((unsigned int)tiles, (unsigned int)tile_blocks), block(TC_TILE_PIXELS / tile_blocks * parts);
    // Set up while the kernel before is still at work, kept apart by shared memory: small blocks that arrive early all pile onto the
    // first SMs that have room (960x7x7 x 128, 49 blocks: 49 us unchained, 65 chained, 48 chained and spread; 64x56x56 f32 17.2
    // unchained, 14.9 chained and spread; 400x7x7 x 800, 307 blocks, 87.8 -> 66.9; 80x27x27 x 64, 365 blocks of 256 threads, 25.2 ->
    // 22.7).  Not large blocks of which some SMs get two: the first SMs that are free take two each (576x14x14 x 128, 196 blocks of 1 024
    // threads: 55.4 -> 57.4).  Nor so many that little L1 is left, with tables per channel, which are looked up through it, from four an SM on (us in
    // turn and early: 784x14x14, 185 blocks a pass, at 7 bits 766 and 583, 400x14x14, 299, 285 and 227; 240x1x1 x 124928, 488 blocks, at 8 bits 211 and
    // 231, 144x1x1 x 109568, 856, 81 and 111; with one table from six on above
    // 128 coefficients: 192x7x7, 456 blocks, 80.1 and 77.2, 208x7x7 x 2100, 804, 74.8 and 82.0, 32x27x19 x 282, 1131, 37.4 and 35.0).
    if (tile_blocks > 1)
        return launch_chained_cluster(tile_blocks, kernel, grid, block, std::max<size_t>(staging, kSpreadMost), s, a, sym, parts, first_tile, staging) == cudaSuccess ? TC_OK : TC_ERR_CUDA;
    const bool apart = tiles <= ctx->sm_count || tiles > 2ll * ctx->sm_count || block.x <= 512;
    static std::atomic<size_t> own[2];
    const size_t spread = a.alone && apart && tiles <= (a.groups != 1 ? 3ll : a.k <= 128 ? 8ll : 5ll) * ctx->sm_count ? spread_bytes(tiles, ctx->sm_count, static_bytes(own[a.groups != 1], (const void *)kernel)) : 0;
    if (spread > 0)
        return launch_chained(true, kernel, grid, block, std::max<size_t>(staging, spread), s, a, sym, parts, first_tile, staging) == cudaSuccess ? TC_OK : TC_ERR_CUDA;
    kernel<<<grid, block, staging, s>>>(a, sym, parts, first_tile, staging);
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

// Symbols of per-channel codes up to this size are staged with every tile; more of them cost a tile longer than
// the lookups in L2 that they save.
constexpr unsigned int kSortedStaged = 16 * 1024;

template <bool kOperand, bool kEarly>
static void (*pick_unpack(bool per_channel, bool full))(DecodeArgs, void *, long long, unsigned int, unsigned int)
{
    return per_channel ? unpack_symbols_kernel<kOperand, false, false, kEarly> : full ? unpack_symbols_kernel<kOperand, true, kOperand, kEarly> : unpack_symbols_kernel<kOperand, true, false, kEarly>;
}

template <bool kOperand>
static tc_status launch_unpack(const DecodeArgs &a, void *out, long long first_tile, long long end_tile, int sm_count, cudaStream_t s)
{
    if (end_tile <= first_tile) return TC_OK;
    const int chunks = a.splits * TC_TILE_PIXELS / a.chunk_pixels;
    if (chunks > kUnpackThreads) return TC_ERR_UNSUPPORTED;
    // beside the tables (at most 48 KB and the symbols) room for a segment of three bits per symbol, at most 48 KB
    unsigned int tables = (unsigned int)(a.groups == 1 ? std::max<size_t>((size_t)4 << a.lut_bits, 16) : (size_t)a.k * kCanonWords * 4);
    bool tables_staged = true;
    if (a.groups != 1) {
        const unsigned int sorted = (unsigned int)a.k << a.bits;                   // bytes
        tables_staged = sorted % 16 == 0 && ((uintptr_t)a.sorted & 15u) == 0 && sorted <= kSortedStaged;
        if (tables_staged) tables += sorted;
    }
    const unsigned int segment = (unsigned int)std::min<long long>((long long)a.k * TC_TILE_PIXELS * 3 / 8, 48 * 1024);
    // Two or four blocks a tile of 256 chunks and more, as long as every block has an SM (320x7x7 x 180, 69 tiles in four blocks each:
    // 20.5 -> 22.6 us; 128x28x28 f32, two blocks of 64 chunks: 18.1 -> 18.5).
    const long long tiles = end_tile - first_tile;
    int parts = 1;
    while (parts < 4 && chunks >= 256 && tiles * parts * 2 <= sm_count && chunks % (128 * parts) == 0) parts *= 2;
    // a block of few chunks has more threads for staging while all blocks are resident at once
    const int threads = (chunks / parts + 31) / 32 * 32, least = tiles * parts < 4 * sm_count ? 256 : 32;
    // from 16 warps an SM on the shared-memory pipe is what bounds a per-layer decoder (see the kernel)
    const bool full = kOperand && a.groups == 1 && tiles * ((chunks + 31) / 32) >= 16 * (long long)sm_count;
    static std::atomic<size_t> own[3];
    auto own_bytes = [&] { return static_bytes(own[a.groups != 1 ? 2 : full], (const void *)pick_unpack<kOperand, true>(a.groups != 1, full)); };
    // In its turn where the symbols are looked up through L1, which spreading would take from them (us in turn and early: 240x13x13 x 183 at 8 bits 45.4
    // and 48.8, 176x7x7 x 352 31.5 and 33.2, 848x16x16 x 526 at 5 bits 579 and 612; staged: 144x12x12 x 97 20.6 and 18.4, 512x56x56 19.6 and 18.3).
    // And with long chunks of codes per channel (768x1x1 x 3072 in chunks of 3072 220 and 230, 192x28x28 of 6144 377 and 401).
    const bool long_chunks = a.k / a.splits * a.chunk_pixels > 512;
    const size_t spread = a.alone && tables_staged && (a.groups == 1 || !long_chunks) ? spread_bytes(tiles * parts, sm_count, own_bytes()) : 0;
    // In its turn as well where an operand's segments are expected not to fit their buffer and are read through L1, of which a product ahead leaves
    // little to blocks that start under it, and that takes longer than the launch saves: long chunks, or several blocks an SM (us in turn and early:
    // 384x14x14 x 651 at 7.5 bits a value 206 and 259, 944x34x5 x 44 at 7.3 bits, chunks of 944 symbols, 102.6 and 107.6; 704x28x28 at 4.4 bits, chunks of 176,
    // 26.8 and 23.1, 400x14x14 x 10 at 3.9 bits, chunks of 400, 39.1 and 36.1).
    const double tile_bytes = a.mean_tile_bytes > 0 ? (double)a.mean_tile_bytes : (double)a.code_bits * a.k * TC_TILE_PIXELS / 8;
    const bool through_l1 = kOperand && a.groups == 1 && tile_bytes > 1.05 * segment;
    const bool early = spread > 0 && !(through_l1 && (tiles * parts > sm_count || long_chunks));
    void (*kernel)(DecodeArgs, void *, long long, unsigned int, unsigned int) = spread > 0 ? pick_unpack<kOperand, true>(a.groups != 1, full) : pick_unpack<kOperand, false>(a.groups != 1, full);
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024) != cudaSuccess) return TC_ERR_CUDA;
    const size_t rows = full ? (size_t)(threads / 32) * kRowsWarpBytes : 0;
    const size_t smem = std::max<size_t>(tables + segment + rows, spread);
    return launch_first(early, kernel, dim3((unsigned int)tiles, (unsigned int)parts), std::max(threads, least), smem, s, a, out, first_tile, tables,
                        segment) == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_unpack_symbols(const tc_ctx *ctx, const DecodeArgs &a, uint8_t *sym, cudaStream_t s)
{
    return launch_unpack<false>(a, sym, 0, a.n_tiles, ctx->sm_count, s);
}

tc_status tc_launch_unpack_operand(const tc_ctx *ctx, const DecodeArgs &a, void *operand, long long first_tile, long long end_tile, cudaStream_t s)
{
    return launch_unpack<true>(a, operand, first_tile, end_tile, ctx->sm_count, s);
}
