// Calibration and statistics kernels (off the timed path): channel sums, centred covariance
// and the range of coefficient 0 for the fit (Section 3; Section 3.1 "Linear transform" and
// "Quantization"), symbol histograms for the entropy and the codebook (Section 3.1 "Variable
// length coding"), and the squared error of a round trip (Section 3, MSE distortion).
#include "device_utils.cuh"

#include <algorithm>

namespace {

using namespace tcdev;

// of a value in a register (load_as_double reads global memory)
__device__ __forceinline__ double as_double(float v) { return (double)v; }
__device__ __forceinline__ double as_double(__nv_bfloat16 v) { return (double)__bfloat162float(v); }

// V elements that one load brings (V sizeof(TIn) is 2 to 16 bytes, and the address a multiple of it)
template <typename TIn, int V>
struct alignas(V * sizeof(TIn)) Vector { TIn v[V]; };

// sums[c] += sum over pixels of x[n][c][:].  A warp takes one channel of every gridDim.y-th image, four rows in flight, and adds
// to the sum once: one block and one atomic per row left 256x14x14 x 256 at 39 us, this takes 11.5 us.
constexpr int kSumWarps = 8, kSumRows = 4;

template <typename TIn, int V>
__global__ void __launch_bounds__(32 * kSumWarps) channel_sums_kernel(const TIn *x, int n, int c, int hw, double *sums)
{
    const int ch = blockIdx.x * kSumWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31, pieces = hw / V;
    if (ch >= c) return;
    double s[2] = {};
    for (long long img = (long long)blockIdx.y * kSumRows; img < n; img += (long long)gridDim.y * kSumRows) {
        const int rows = (int)min((long long)kSumRows, n - img);
        for (int i = lane; i < pieces; i += 32) {
            Vector<TIn, V> got[kSumRows];
#pragma unroll
            for (int r = 0; r < kSumRows; ++r)
                if (r < rows) got[r] = reinterpret_cast<const Vector<TIn, V> *>(x + ((img + r) * c + ch) * (long long)hw)[i];
#pragma unroll
            for (int r = 0; r < kSumRows; ++r)
                if (r < rows) {
#pragma unroll
                    for (int e = 0; e < V; ++e) s[e & 1] += as_double(got[r].v[e]);
                }
        }
    }
    double sum = s[0] + s[1];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    if (lane == 0) atomicAdd(sums + ch, sum);
}

__global__ void mean_kernel(double *sums, int c, double pixels)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < c) sums[i] = __ddiv_rn(sums[i], pixels);
}

// cov[a][b] += sum over a block's slabs of pixels of (x_a - mu_a)(x_b - mu_b) for a 64 x 64 block of channel
// pairs; grid = (pixel slabs, channel-block pairs with b-block >= a-block).
// On the fp64 tensor cores (m8n8k4: the rate of the multiply-add pipe, 64 a cycle and SM, for an eighth of the operand
// reads): a warp holds 32 x 32 sums, so that eight reads of 8 bytes feed sixteen instructions.  Multiply-adds outside the tensor
// cores, sixteen sums a thread, were bound by those reads.  The next slab's values are on their way while a slab is added up;
// on the diagonal one operand serves both sides and the warp below it has nothing to do.  256x14x14 x 256: 318 -> 188 us
// (multiply-adds alone 113).
constexpr int kCovTile = 64, kCovSlab = 32, kCovPitch = kCovSlab + 4, kCovThreads = 128;

template <typename TIn>
__global__ void __launch_bounds__(kCovThreads, 4) covariance_kernel(const TIn *x, int n, int c, int hw, const double *mean,
                                                                    double *cov, int blocks_per_dim)
{
    __shared__ double sa[kCovTile][kCovPitch], sb[kCovTile][kCovPitch];
    __shared__ double s_mean[2][kCovTile];
    // decode the (ablk <= bblk) pair from blockIdx.y
    int pair = blockIdx.y, ablk = 0;
    while (pair >= blocks_per_dim - ablk) { pair -= blocks_per_dim - ablk; ++ablk; }
    const int bblk = ablk + pair;
    const bool diagonal = pair == 0;
    const long long pixels = (long long)n * hw;
    const int t = threadIdx.x, pp = t % kCovSlab, ch0 = t / kCovSlab;      // staging: pixel pp of channels ch0, ch0 + 4, ...
    constexpr int kEvery = kCovThreads / kCovSlab, kCh = kCovTile / kEvery;
    if (t < 2 * kCovTile) {
        const int ch = (t < kCovTile ? ablk : bblk) * kCovTile + t % kCovTile;
        s_mean[t / kCovTile][t % kCovTile] = ch < c ? mean[ch] : 0.0;
    }
    __syncthreads();
    TIn va[kCh], vb[kCh];
    bool there = false;
    const TIn *const from_a = x + (long long)(ablk * kCovTile + ch0) * hw, *const from_b = x + (long long)(bblk * kCovTile + ch0) * hw;
    const int most_a = c - ablk * kCovTile - ch0, most_b = diagonal ? 0 : c - bblk * kCovTile - ch0;      // channels there are from ch0 on
    const long long stride = (long long)kEvery * hw;
    auto fetch = [&](long long p0) {
        const long long p = p0 + pp;
        there = p < pixels;
        if (!there) return;
        const long long img = p / hw, at = img * c * (long long)hw + (p - img * hw);
        const TIn *a = from_a + at, *b = from_b + at;
#pragma unroll
        for (int i = 0; i < kCh; ++i, a += stride, b += stride) {
            if (kEvery * i < most_a) va[i] = *a;
            if (kEvery * i < most_b) vb[i] = *b;
        }
    };
    const int warp = t >> 5, lane = t & 31, wr = warp >> 1, wc = warp & 1;
    const double *const rows = &sa[32 * wr + (lane >> 2)][lane & 3];
    const double *const cols = diagonal ? &sa[32 * wc + (lane >> 2)][lane & 3] : &sb[32 * wc + (lane >> 2)][lane & 3];
    double2 acc[4][4] = {};
    const long long step = (long long)gridDim.x * kCovSlab;
    long long p0 = (long long)blockIdx.x * kCovSlab;
    if (p0 < pixels) fetch(p0);
    for (; p0 < pixels; p0 += step) {
        __syncthreads();                               // the previous slab has been added up
#pragma unroll
        for (int i = 0; i < kCh; ++i) {
            const int ch = ch0 + kEvery * i;
            sa[ch][pp] = there && kEvery * i < most_a ? (double)(float)va[i] - s_mean[0][ch] : 0.0;
            if (!diagonal) sb[ch][pp] = there && kEvery * i < most_b ? (double)(float)vb[i] - s_mean[1][ch] : 0.0;
        }
        __syncthreads();
        if (p0 + step < pixels) fetch(p0 + step);
        if (diagonal && wr > wc) continue;
#pragma unroll
        for (int k = 0; k < kCovSlab; k += 4) {
            double u[4], v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                u[i] = rows[8 * i * kCovPitch + k];
                v[i] = cols[8 * i * kCovPitch + k];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_f64(acc[i][j], u[i], v[j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int ca = ablk * kCovTile + 32 * wr + 8 * i + (lane >> 2), cb = bblk * kCovTile + 32 * wc + 8 * j + 2 * (lane & 3);
            if (ca < c && cb < c && ca <= cb) atomicAdd(cov + (long long)ca * c + cb, acc[i][j].x);
            if (ca < c && cb + 1 < c && ca <= cb + 1) atomicAdd(cov + (long long)ca * c + cb + 1, acc[i][j].y);
        }
}

// Per-block min and max of coefficient 0: y0 = sum_c T[0][c] (x_c - mu_c), summed in channel
// order without contraction.  Bound by the latency of the loads, so 32 of them go ahead of the chain of additions (256x14x14 x 256:
// 37 us with four ahead, 14.9 now, 118 where the compiler put every load beside its addition).
constexpr int kRangeThreads = 128, kRangeAhead = 32;

template <typename TIn>
__global__ void __launch_bounds__(kRangeThreads) range0_kernel(const TIn *x, int n, int c, int hw, const double *mean,
                                                               const double *row0, double *block_minmax)
{
    extern __shared__ double s_rm[];      // [2][c]: row0, mean
    for (int i = threadIdx.x; i < c; i += blockDim.x) { s_rm[i] = row0[i]; s_rm[c + i] = mean[i]; }
    __syncthreads();
    const long long pixels = (long long)n * hw;
    double mn = INFINITY, mx = -INFINITY;
    for (long long first = (long long)blockIdx.x * blockDim.x; first < pixels; first += (long long)gridDim.x * blockDim.x) {
        const long long p = min(first + threadIdx.x, pixels - 1);      // threads past the end repeat the last pixel
        const long long img = p / hw, s = p - img * hw;
        const TIn *src = x + img * c * (long long)hw + s;
        double y = 0.0;
        int cc = 0;
        for (; cc + kRangeAhead <= c; cc += kRangeAhead) {             // loads ahead of the chain of additions
            TIn got[kRangeAhead];
#pragma unroll
            for (int i = 0; i < kRangeAhead; ++i) got[i] = src[(long long)(cc + i) * hw];
            __syncwarp();                                              // (else the compiler moves each load to its addition)
#pragma unroll
            for (int i = 0; i < kRangeAhead; ++i) y = __dadd_rn(y, __dmul_rn(s_rm[cc + i], __dsub_rn(as_double(got[i]), s_rm[c + cc + i])));
        }
        for (; cc < c; ++cc)
            y = __dadd_rn(y, __dmul_rn(s_rm[cc], __dsub_rn(load_as_double(src + (long long)cc * hw), s_rm[c + cc])));
        mn = fmin(mn, y);
        mx = fmax(mx, y);
    }
    __shared__ double rmin[kRangeThreads / 32], rmax[kRangeThreads / 32];
    for (int d = 16; d > 0; d >>= 1) {
        mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, d));
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, d));
    }
    if ((threadIdx.x & 31) == 0) { rmin[threadIdx.x >> 5] = mn; rmax[threadIdx.x >> 5] = mx; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kRangeThreads / 32; ++i) { mn = fmin(mn, rmin[i]); mx = fmax(mx, rmax[i]); }
        block_minmax[2 * blockIdx.x] = mn;
        block_minmax[2 * blockIdx.x + 1] = mx;
    }
}

// hist[g][s] += 1 for every symbol; g = coefficient index (groups == k) or 0.
__global__ void __launch_bounds__(256) histogram_kernel(const uint8_t *sym, long long pixels, int k, int groups,
                                                        int bits, unsigned long long *hist)
{
    __shared__ unsigned int local[256];
    const int nsym = 1 << bits;
    const long long total = pixels * k;
    if (groups == 1) {
        for (int i = threadIdx.x; i < nsym; i += blockDim.x) local[i] = 0;
        __syncthreads();
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
            atomicAdd(local + sym[i], 1u);
        __syncthreads();
        for (int i = threadIdx.x; i < nsym; i += blockDim.x)
            if (local[i]) atomicAdd(hist + i, (unsigned long long)local[i]);
    } else {
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
            atomicAdd(hist + (i % k) * nsym + sym[i], 1ull);
    }
}

// Squared error and zeros of x, in pieces of V values; one atomic per block (one per warp, 12 500 to one address, took 51 us for
// 256x14x14 x 256; 14.8 now).
constexpr int kErrThreads = 256;
template <typename TIn, int V>
__global__ void __launch_bounds__(kErrThreads) sqerr_kernel(const TIn *x, const TIn *xhat, long long count, double *sum_sq,
                                                            unsigned long long *zeros)
{
    __shared__ double s_acc[kErrThreads / 32];
    __shared__ unsigned int s_zeros[kErrThreads / 32];
    double acc = 0.0;
    unsigned int z = 0;
    auto add = [&](TIn u, TIn v) {
        const double a = as_double(u), d = a - as_double(v);
        acc += d * d;
        z += (a == 0.0);
    };
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, all = (long long)gridDim.x * blockDim.x, pieces = count / V;
    for (long long i = first; i < pieces; i += all) {
        const Vector<TIn, V> u = reinterpret_cast<const Vector<TIn, V> *>(x)[i], v = reinterpret_cast<const Vector<TIn, V> *>(xhat)[i];
#pragma unroll
        for (int e = 0; e < V; ++e) add(u.v[e], v.v[e]);
    }
    for (long long i = pieces * V + first; i < count; i += all) add(x[i], xhat[i]);
    for (int d = 16; d > 0; d >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, d);
        z += __shfl_xor_sync(0xffffffffu, z, d);
    }
    if ((threadIdx.x & 31) == 0) { s_acc[threadIdx.x >> 5] = acc; s_zeros[threadIdx.x >> 5] = z; }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long zz = z;
        for (int w = 1; w < kErrThreads / 32; ++w) { acc += s_acc[w]; zz += s_zeros[w]; }
        atomicAdd(sum_sq, acc);
        atomicAdd(zeros, zz);
    }
}

// Widest piece of up to 16 bytes that `count` elements and the pointers allow
template <typename TIn>
int piece_of(long long count, const void *a, const void *b)
{
    int v = 16 / (int)sizeof(TIn);
    while (v > 1 && (count % v || (((uintptr_t)a | (uintptr_t)b) % (v * sizeof(TIn))))) v /= 2;
    return v;
}

template <typename TIn>
void launch_channel_sums(const TIn *x, int n, int c, int hw, double *sums, int sm_count, cudaStream_t s)
{
    const unsigned channels = (unsigned)((c + kSumWarps - 1) / kSumWarps);
    long long images = std::max(1u, 8u * (unsigned)sm_count / channels);             // eight blocks an SM
    images = std::min(images, ((long long)n + kSumRows - 1) / kSumRows);
    const dim3 grid(channels, (unsigned)images);
    switch (piece_of<TIn>(hw, x, x)) {
    case 8: channel_sums_kernel<TIn, 16 / sizeof(TIn)><<<grid, 32 * kSumWarps, 0, s>>>(x, n, c, hw, sums); break;
    case 4: channel_sums_kernel<TIn, 4><<<grid, 32 * kSumWarps, 0, s>>>(x, n, c, hw, sums); break;
    case 2: channel_sums_kernel<TIn, 2><<<grid, 32 * kSumWarps, 0, s>>>(x, n, c, hw, sums); break;
    default: channel_sums_kernel<TIn, 1><<<grid, 32 * kSumWarps, 0, s>>>(x, n, c, hw, sums); break;
    }
}

template <typename TIn>
void launch_sqerr(const TIn *x, const TIn *xhat, long long count, double *sum_sq, unsigned long long *zeros, int sm_count, cudaStream_t s)
{
    constexpr int wide = 16 / sizeof(TIn);
    const bool aligned = (((uintptr_t)x | (uintptr_t)xhat) & 15u) == 0;
    long long blocks = (count + kErrThreads * wide - 1) / (kErrThreads * wide);
    blocks = std::max(1ll, std::min(blocks, 8ll * sm_count));          // eight an SM
    if (aligned) sqerr_kernel<TIn, wide><<<(unsigned)blocks, kErrThreads, 0, s>>>(x, xhat, count, sum_sq, zeros);
    else sqerr_kernel<TIn, 1><<<(unsigned)blocks, kErrThreads, 0, s>>>(x, xhat, count, sum_sq, zeros);
}

// copies[0][i] = the sum of copies[.][i]
__global__ void fold_counts_kernel(unsigned long long *counts, int copies, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long sum = 0;
    for (int k = 0; k < copies; ++k) sum += counts[(size_t)k * n + i];
    counts[i] = sum;
}

inline bool launched() { return cudaGetLastError() == cudaSuccess; }

}  // namespace

tc_status tc_launch_channel_sums(const void *x, int dtype, int n, int c, int hw, double *sums, int sm_count, cudaStream_t s)
{
    if (n == 0) return TC_OK;
    if (dtype == TC_F32) launch_channel_sums((const float *)x, n, c, hw, sums, sm_count, s);
    else launch_channel_sums((const __nv_bfloat16 *)x, n, c, hw, sums, sm_count, s);
    return launched() ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_mean(double *sums, int c, long long pixels, cudaStream_t s)
{
    mean_kernel<<<(c + 127) / 128, 128, 0, s>>>(sums, c, (double)pixels);
    return launched() ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_covariance(const void *x, int dtype, int n, int c, int hw, const double *mean, double *cov,
                               int sm_count, cudaStream_t s)
{
    const int bpd = (c + kCovTile - 1) / kCovTile;
    const int pairs = bpd * (bpd + 1) / 2;
    const long long pixels = (long long)n * hw;
    long long slabs = (pixels + kCovSlab - 1) / kCovSlab;
    const long long want = 4ll * sm_count / pairs;                      // one round of four blocks for each SM
    if (slabs > want) slabs = want;
    if (slabs < 1) slabs = 1;
    dim3 grid((unsigned int)slabs, (unsigned int)pairs);
    if (dtype == TC_F32) covariance_kernel<float><<<grid, kCovThreads, 0, s>>>((const float *)x, n, c, hw, mean, cov, bpd);
    else covariance_kernel<__nv_bfloat16><<<grid, kCovThreads, 0, s>>>((const __nv_bfloat16 *)x, n, c, hw, mean, cov, bpd);
    return launched() ? TC_OK : TC_ERR_CUDA;
}

int tc_range0_max_blocks(long long pixels)
{
    long long b = (pixels + kRangeThreads - 1) / kRangeThreads;
    if (b > 2048) b = 2048;
    if (b < 1) b = 1;
    return (int)b;
}

tc_status tc_launch_range0(const void *x, int dtype, int n, int c, int hw, const double *mean, const double *row0,
                           double *block_minmax, int *n_blocks_out, cudaStream_t s)
{
    const int blocks = tc_range0_max_blocks((long long)n * hw);
    *n_blocks_out = blocks;
    const size_t smem = sizeof(double) * 2 * (size_t)c;
    if (dtype == TC_F32)
        range0_kernel<float><<<blocks, kRangeThreads, smem, s>>>((const float *)x, n, c, hw, mean, row0, block_minmax);
    else
        range0_kernel<__nv_bfloat16><<<blocks, kRangeThreads, smem, s>>>((const __nv_bfloat16 *)x, n, c, hw, mean, row0,
                                                                         block_minmax);
    return launched() ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_histogram(const uint8_t *sym, long long pixels, int k, int groups, int bits,
                              unsigned long long *hist, cudaStream_t s)
{
    long long blocks = (pixels * k + 256 * 64 - 1) / (256 * 64);
    if (blocks > 2048) blocks = 2048;
    if (blocks < 1) blocks = 1;
    histogram_kernel<<<(unsigned int)blocks, 256, 0, s>>>(sym, pixels, k, groups, bits, hist);
    return launched() ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_sqerr(const void *x, const void *xhat, int dtype, long long count, double *sum_sq,
                          unsigned long long *zeros, int sm_count, cudaStream_t s)
{
    if (dtype == TC_F32) launch_sqerr((const float *)x, (const float *)xhat, count, sum_sq, zeros, sm_count, s);
    else launch_sqerr((const __nv_bfloat16 *)x, (const __nv_bfloat16 *)xhat, count, sum_sq, zeros, sm_count, s);
    return launched() ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_fold_counts(unsigned long long *counts, int copies, int n, cudaStream_t s)
{
    fold_counts_kernel<<<(n + 255) / 256, 256, 0, s>>>(counts, copies, n);
    return launched() ? TC_OK : TC_ERR_CUDA;
}
