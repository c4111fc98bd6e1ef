// Second half of the fit on the device (Section 3.1, "Linear transform": the PCA matrix is
// pre-computed from the covariance of calibration data, which "can be updated online"): from the
// running moments to the covariance, its eigendecomposition, the rounded basis and the constants
// the codec kernels read -- without moving a C x C matrix to the host.
//
// Eigensolver of matrices that eigh_cluster.cu does not take: one-sided Jacobi (Hestenes) on the shifted matrix G = A / |A|_F + s I.  Plane
// rotations of pairs of columns make the columns of G mutually orthogonal; then G = U S and, G
// being positive definite (s > 1), the columns of U are the eigenvectors of A.  Columns are stored
// as rows (A is symmetric).  All columns of G have norms within [s - 1, s + 1], which the method
// profits from three times: the eigenvectors are the normalised columns (no second matrix is
// rotated), inner products compare against relative bounds, and the gaps between the squared
// singular values are linear, not quadratic, in the eigenvalue gaps (a graded covariance: 13
// instead of 16 sweeps, a geometric spectrum over 12 decades 24 instead of 40).
#include "tc_internal.h"

#include <cuda_bf16.h>
#include <cfloat>

#define TC_CUDA(call)                                   \
    do {                                                \
        if ((call) != cudaSuccess) { cudaGetLastError(); return TC_ERR_CUDA; } \
    } while (0)

namespace {

constexpr int kPairThreads = 128;
// A covariance with a steeply graded spectrum takes 13 to 25 sweeps, an ordinary matrix under 10.
constexpr int kMaxSweeps = 150;
constexpr double kShift = 1.25;                        // of |A|_F: no eigenvalue of G is below 0.25
constexpr unsigned long long kBarrierLimitNs = 2000000000ull;

__device__ __forceinline__ double block_sum(double v, double *s_red)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    __syncthreads();                                   // s_red may still be read from the previous call
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < n_warps; ++w) t += s_red[w];   // same order in every thread
    return t;
}

// mean = s / M and covariance = (S - s s^T / M) / (M - 1) from the running moments (S holds the
// upper triangle), written as a full symmetric matrix
__global__ void moments_to_cov_kernel(const double *sum, const double *outer, double m, int c, double *mean, double *cov)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)c * c) return;
    const int a = (int)(i / c), b = (int)(i % c);
    const int lo = min(a, b), hi = max(a, b);
    const double prod = __dmul_rn(sum[lo], sum[hi]);
    cov[i] = __ddiv_rn(__dsub_rn(outer[(size_t)lo * c + hi], __ddiv_rn(prod, m)), __dsub_rn(m, 1.0));
    if (b == 0) mean[a] = __ddiv_rn(sum[a], m);
}

// centred sums (upper triangle) -> covariance, full symmetric
__global__ void scale_mirror_kernel(double *cov, int c, double denom)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)c * c) return;
    const int a = (int)(i / c), b = (int)(i % c);
    if (a > b) return;
    const double v = __ddiv_rn(cov[i], denom);
    cov[i] = v;
    cov[(size_t)b * c + a] = v;
}

// device bookkeeping of one decomposition, zeroed before use
struct JacobiState {
    double frob2;
    unsigned int arrived;                              // grid barrier: blocks that have come, over all barriers
    unsigned int failed;                               // a bounded wait ran out
    int outcome;                                       // sweeps if it converged, -1 if not, 0 if a wait ran out
    unsigned int rotations[kMaxSweeps];                // per sweep
};

__global__ void frobenius_kernel(const double *a, int c, JacobiState *st)
{
    __shared__ double s_red[kPairThreads / 32];
    double acc = 0.0;
    for (int j = threadIdx.x; j < c; j += blockDim.x) {
        const double v = a[(size_t)blockIdx.x * c + j];
        acc += v * v;
    }
    acc = block_sum(acc, s_red);
    if (threadIdx.x == 0) atomicAdd(&st->frob2, acc);
}

// g = a / |a|_F + s I, rows padded to `ld` with zeros; rows past c are zero (nothing rotates them)
__global__ void jacobi_init_kernel(const double *a, int c, double *g, int ld, const JacobiState *st)
{
    const int r = blockIdx.x;
    const double f2 = st->frob2, inv = f2 > 0.0 ? 1.0 / sqrt(f2) : 0.0;
    for (int j = threadIdx.x; j < ld; j += blockDim.x)
        g[(size_t)r * ld + j] = (r < c && j < c) ? a[(size_t)r * c + j] * inv + (j == r ? kShift : 0.0) : 0.0;
}

// The pair of round `round` played at table `t` (n even): player n - 1 stays, the others rotate.
__device__ __forceinline__ void round_robin_pair(int n, int round, int t, int &p, int &q)
{
    const int m = n - 1;
    if (t == 0) { p = m; q = round % m; }
    else { p = (round + t) % m; q = (round - t + m) % m; }
    if (p > q) { const int x = p; p = q; q = x; }
}

// All blocks of a cooperative launch have come `n`-th time; false if the wait ran out (or one of
// another block did): everyone leaves then.
__device__ __forceinline__ bool grid_barrier(JacobiState *st, unsigned int n)
{
    __shared__ bool s_ok;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        bool ok = true;
        const unsigned int target = n * gridDim.x;
        atomicAdd(&st->arrived, 1u);
        unsigned long long t0, t1;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
        unsigned int seen;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&st->arrived) : "memory");
            if (seen >= target) break;
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t1));
            if (t1 - t0 > kBarrierLimitNs) { ok = false; atomicExch(&st->failed, 1u); break; }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

template <int R>
__device__ __forceinline__ double norm2(const double2 (&x)[R])
{
    double a = 0.0, b = 0.0;
#pragma unroll
    for (int i = 0; i < R; ++i) { a += x[i].x * x[i].x; b += x[i].y * x[i].y; }
    return warp_sum(a + b);
}

// Makes the columns x and y (2 R elements per lane, squared norms al and be) orthogonal; false if
// they already are, to rounding: below `tol2` (squared) of the norms a rotation would only chase noise.
// The angle is computed in fp32 -- the rotations' angles steer the iteration, an error of 1e-7 of
// one leaves 1e-7 of the inner product for the next sweep -- but the matrix applied is a rotation
// to fp64: cosine and tan(angle / 2) follow from that tangent by one step of Householder's third-order
// iteration from the fp32 reciprocal (square root) -- r (1 + e / 2 + 3 e^2 / 8) with e = 1 - q r^2 for
// 1 / sqrt(q), r (1 + e + e^2) with e = 1 - k r for 1 / k; e is below 1e-6, the term left out below 1e-18 --
// and the update x -= s (y + u x), y += s (x - u y) rounds in proportion to the angle.
template <int R>
__device__ __forceinline__ bool rotate_pair(double2 (&x)[R], double2 (&y)[R], double &al, double &be, double tol2)
{
    double g0 = 0.0, g1 = 0.0;
#pragma unroll
    for (int i = 0; i < R; ++i) { g0 += x[i].x * y[i].x; g1 += x[i].y * y[i].y; }
    const double ga = warp_sum(g0 + g1);
    if (ga * ga <= tol2 * al * be) return false;
    // t = tan of the smaller angle that annuls the inner product; norms lie within [1/16, 6], and the
    // inner product is above the tolerance: no square below leaves the range of fp32
    const float d = (float)(be - al), g2 = (float)(2.0 * ga), h = sqrtf(d * d + g2 * g2);
    const double t = (double)__fdividef(g2, d + (d >= 0.f ? h : -h));
    const double q = fma(t, t, 1.0);
    const double r0 = (double)rsqrtf((float)q), re = fma(-q * r0, r0, 1.0);
    const double cs = fma(r0 * re, fma(re, 0.375, 0.5), r0);              // 1 / sqrt(q)
    const double k = 1.0 + cs, k0 = (double)__frcp_rn((float)k), ke = fma(-k, k0, 1.0);
    const double sn = cs * t, u = sn * fma(k0 * ke, 1.0 + ke, k0);         // sin / (1 + cos)
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const double2 v = x[i], w = y[i];
        x[i] = make_double2(fma(-sn, fma(u, v.x, w.x), v.x), fma(-sn, fma(u, v.y, w.y), v.y));
        y[i] = make_double2(fma(sn, fma(-u, w.x, v.x), w.x), fma(sn, fma(-u, w.y, v.y), w.y));
    }
    al = fma(-t, ga, al);
    be = fma(t, ga, be);
    return true;
}

// The columns are dealt into blocks of B.  A thread block plays the block pairs of one table of a
// round-robin tournament over the column blocks: it holds the first column block in registers
// (warp w: column w), the second in shared memory, and in B inner rounds rotates every column of
// the one against every column of the other (warp w takes column w + r).  The first round of a
// sweep also rotates the pairs inside both column blocks.  Between rounds the blocks change
// tables through global memory (L2), behind a grid barrier.
// What bounds it: the latency of an inner round -- loads, the inner product's shuffles, the angle,
// a block barrier: 960 cycles at 64 rows -- then, from about 256 rows on (1480 cycles), the shared
// memory and the fp64 pipe; a table change costs 6500 cycles.  So columns' norms are carried
// through the inner rounds instead of recomputed, and one launch does the whole decomposition:
// with a launch per round of single pairs (6.3 us each) n = 256 took 24 ms, now 3.2.  B = 16 halves
// the table changes of B = 8; from 512 rows on the registers only hold B = 8.
template <int R, int B>
__global__ void __launch_bounds__(B * 32, 1) jacobi_kernel(double *g, int n_blocks, double tol2, JacobiState *st)
{
    constexpr int ld = 64 * R;
    extern __shared__ __align__(16) double s_col[];    // [2][B][ld]; the first half only for the pairs inside a block
    __shared__ double s_norm[B];                       // squared norms of the second block's columns
    __shared__ unsigned int s_rot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *s_first = s_col, *s_second = s_col + (size_t)B * ld;
    auto column = [&](double *base, int i) { return reinterpret_cast<double2 *>(base + (size_t)i * ld) + lane; };
    double2 x[R], y[R];
    unsigned int barriers = 0;
    for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
        unsigned int rotated = 0;
        for (int round = 0; round < n_blocks - 1; ++round) {
            int bi, bj;
            round_robin_pair(n_blocks, round, blockIdx.x, bi, bj);
            const double2 *gi = column(g, bi * B + warp), *gj = column(g, bj * B + warp);
#pragma unroll
            for (int i = 0; i < R; ++i) { x[i] = __ldcg(gi + 32 * i); y[i] = __ldcg(gj + 32 * i); }
#pragma unroll
            for (int i = 0; i < R; ++i) column(s_second, warp)[32 * i] = y[i];
            if (round == 0) {
                // the pairs inside the two column blocks: warps 0 .. B/2 - 1 the first block's, the others the second's
#pragma unroll
                for (int i = 0; i < R; ++i) column(s_first, warp)[32 * i] = x[i];
                double *half = warp < B / 2 ? s_first : s_second;
#pragma unroll 1
                for (int r = 0; r < B - 1; ++r) {
                    __syncthreads();
                    int p, q;
                    round_robin_pair(B, r, warp & (B / 2 - 1), p, q);
#pragma unroll
                    for (int i = 0; i < R; ++i) { x[i] = column(half, p)[32 * i]; y[i] = column(half, q)[32 * i]; }
                    double al = norm2<R>(x), be = norm2<R>(y);
                    if (rotate_pair<R>(x, y, al, be, tol2)) {
                        ++rotated;
#pragma unroll
                        for (int i = 0; i < R; ++i) { column(half, p)[32 * i] = x[i]; column(half, q)[32 * i] = y[i]; }
                    }
                }
                __syncthreads();
#pragma unroll
                for (int i = 0; i < R; ++i) { x[i] = column(s_first, warp)[32 * i]; y[i] = column(s_second, warp)[32 * i]; }
            }
            double al = norm2<R>(x);
            const double own = norm2<R>(y);
            if (lane == 0) s_norm[warp] = own;
#pragma unroll 1
            for (int r = 0; r < B; ++r) {
                __syncthreads();
                const int qi = (warp + r) & (B - 1);
                double2 *cq = column(s_second, qi);
                double be = s_norm[qi];
#pragma unroll
                for (int i = 0; i < R; ++i) y[i] = cq[32 * i];
                if (rotate_pair<R>(x, y, al, be, tol2)) {
                    ++rotated;
                    __syncwarp();
                    if (lane == 0) s_norm[qi] = be;
#pragma unroll
                    for (int i = 0; i < R; ++i) cq[32 * i] = y[i];
                }
            }
            __syncthreads();
            double2 *oi = column(g, bi * B + warp), *oj = column(g, bj * B + warp);
#pragma unroll
            for (int i = 0; i < R; ++i) { __stcg(oi + 32 * i, x[i]); __stcg(oj + 32 * i, column(s_second, warp)[32 * i]); }
            if (round == n_blocks - 2) {
                if (threadIdx.x == 0) s_rot = 0;
                __syncthreads();
                if (lane == 0 && rotated) atomicAdd(&s_rot, rotated);
                __syncthreads();
                if (threadIdx.x == 0 && s_rot) atomicAdd(&st->rotations[sweep], s_rot);
            }
            if (!grid_barrier(st, ++barriers)) return;
        }
        if (__ldcg(&st->rotations[sweep]) == 0) {
            if (blockIdx.x == 0 && threadIdx.x == 0) st->outcome = sweep + 1;      // the last one found nothing to rotate
            return;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) st->outcome = -1;
}

// Normalises kVec columns of g into rows of vt and takes their Rayleigh quotients v^T A v against the
// untouched matrix.  A thread owns columns j of A and reads them row by row (coalesced) once for
// all kVec vectors.
constexpr int kVec = 4;
__global__ void rayleigh_kernel(const double *a, const double *g, int ld, int c, double *vt, double *lambda)
{
    __shared__ double s_red[kPairThreads / 32];
    __shared__ double s_v[kVec][TC_MAX_C];
    const int first = blockIdx.x * kVec;
    for (int k = 0; k < kVec; ++k) {
        const int i = first + k;
        double acc = 0.0;
        for (int j = threadIdx.x; j < c; j += blockDim.x) {
            const double v = i < c ? g[(size_t)i * ld + j] : 0.0;
            s_v[k][j] = v;
            acc += v * v;
        }
        const double norm = sqrt(block_sum(acc, s_red));
        for (int j = threadIdx.x; j < c && i < c; j += blockDim.x) {
            const double v = s_v[k][j] / norm;
            s_v[k][j] = v;
            vt[(size_t)i * c + j] = v;
        }
    }
    __syncthreads();
    double acc[kVec] = {};
    for (int j = threadIdx.x; j < c; j += blockDim.x) {
        double w[kVec] = {};
#pragma unroll 4
        for (int r = 0; r < c; ++r) {
            const double ar = a[(size_t)r * c + j];
#pragma unroll
            for (int k = 0; k < kVec; ++k) w[k] += ar * s_v[k][r];
        }
#pragma unroll
        for (int k = 0; k < kVec; ++k) acc[k] += w[k] * s_v[k][j];
    }
    for (int k = 0; k < kVec; ++k) {
        const double t = block_sum(acc[k], s_red);
        if (threadIdx.x == 0 && first + k < c) lambda[first + k] = t;
    }
}

// Descending eigenvalues (equal ones in their original order); each vector signed so that its
// largest-magnitude entry (the first of equal ones) is positive.  The solver's outcome goes behind the eigenvalues.
__global__ void order_sign_kernel(const double *vt, const double *lambda, int c, const int *outcome, double *evals, double *evecs)
{
    __shared__ int s_rank, s_big;
    __shared__ double s_mag[kPairThreads / 32];
    __shared__ int s_at[kPairThreads / 32];
    const int i = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double *v = vt + (size_t)i * c;
    const double li = lambda[i];
    if (threadIdx.x == 0) s_rank = 0;
    __syncthreads();
    int before = 0, at = c;
    double mag = -1.0;
    for (int j = threadIdx.x; j < c; j += blockDim.x) {
        const double lj = lambda[j], m = fabs(v[j]);
        before += (lj > li || (lj == li && j < i)) ? 1 : 0;
        if (m > mag) { mag = m; at = j; }
    }
    before = __reduce_add_sync(0xffffffffu, before);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const double om = __shfl_xor_sync(0xffffffffu, mag, d);
        const int oa = __shfl_xor_sync(0xffffffffu, at, d);
        if (om > mag || (om == mag && oa < at)) { mag = om; at = oa; }
    }
    if (lane == 0) { s_mag[warp] = mag; s_at[warp] = at; atomicAdd(&s_rank, before); }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kPairThreads / 32; ++w)
            if (s_mag[w] > mag || (s_mag[w] == mag && s_at[w] < at)) { mag = s_mag[w]; at = s_at[w]; }
        s_big = min(at, c - 1);
        evals[s_rank] = li;
        if (i == 0) evals[c] = (double)*outcome;
    }
    __syncthreads();
    const double sgn = v[s_big] < 0.0 ? -1.0 : 1.0;
    for (int j = threadIdx.x; j < c; j += blockDim.x) evecs[(size_t)s_rank * c + j] = sgn * v[j];
}

__global__ void abs_max_kernel(const double *x, long long n, double *out)
{
    __shared__ double s_red[32];
    double m = 0.0;
    for (long long i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, fabs(x[i]));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, d));
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, s_red[w]);
        *out = m;
    }
}

// nearest bfloat16 (ties to even) of a double, as a double: eight significant bits, fewer in
// the subnormal range
__device__ __forceinline__ double round_bf16(double v)
{
    if (v == 0.0 || !isfinite(v)) return v;
    int e;
    const double f = frexp(v, &e);
    int shift = 8;
    if (e - 8 < -133) shift = e + 133;
    return ldexp(rint(ldexp(f, shift)), e - shift);
}

// dtype: TC_F32 / TC_BF16 round every entry; TC_INT8: scale = *abs_max / 127, entries become
// scale * rint(v / scale), and *abs_max is replaced by the scale
__global__ void round_basis_kernel(double *basis, long long n, int dtype, double *abs_max)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double scale = 1.0;
    if (dtype == TC_INT8) scale = __ddiv_rn(*abs_max, 127.0);
    if (i < n) {
        const double v = basis[i];
        basis[i] = dtype == TC_F32 ? (double)(float)v : dtype == TC_BF16 ? round_bf16(v) : __dmul_rn(scale, rint(__ddiv_rn(v, scale)));
    }
}
__global__ void store_scale_kernel(double *abs_max) { *abs_max = __ddiv_rn(*abs_max, 127.0); }

// The constants of a model from its basis and mean, in the summation order of a plain loop
// (one thread per output, separate multiply and add):
//   tmu[j] = sum_a T[j][a] mu[a], enc_bias[j] = -(tmu[j] + lo) / step      (blockIdx.y = 0)
//   dec_bias[a] = mu[a] + (lo + center step) sum_{j<k} T[j][a]             (blockIdx.y = 1)
// 32 outputs a block: all warps bring 64 terms of each through shared memory while the first adds up the 64 before.  With one thread
// that read its own terms, the two sums one after the other: 38 us at 256 channels; 18.6 now.
constexpr int kConstTerms = 64, kConstOutputs = 32;
__global__ void __launch_bounds__(256) model_consts_kernel(const double *basis, const double *mean, int c, int k, double lo, double step, double center,
                                                           float *enc_bias, float *tmu32, float *dec_bias)
{
    __shared__ double s_terms[2][kConstTerms][kConstOutputs + 1];
    const int first = blockIdx.x * kConstOutputs, t = threadIdx.x;
    const bool rows = blockIdx.y == 0;                 // outputs are rows of the basis, terms run along them; else the columns
    const int outputs = rows ? k : c, terms = rows ? c : k;
    if (first >= outputs) return;
    // element (term, output) that this thread brings, r = 0 .. 7; consecutive threads along a row of the basis
    auto term_of = [&](int r) { return rows ? t % kConstTerms : t / kConstOutputs + 8 * r; };
    auto output_of = [&](int r) { return rows ? t / kConstTerms + 4 * r : t % kConstOutputs; };
    double got[8];
    auto fetch = [&](int at) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int term = at + term_of(r), out = first + output_of(r);
            got[r] = term < terms && out < outputs ? (rows ? basis[(size_t)out * c + term] : basis[(size_t)term * c + out]) : 0.0;
        }
    };
    fetch(0);
    double sum = 0.0;
    for (int at = 0, buffer = 0; at < terms; at += kConstTerms, buffer ^= 1) {
#pragma unroll
        for (int r = 0; r < 8; ++r) s_terms[buffer][term_of(r)][output_of(r)] = got[r];
        __syncthreads();                               // (the other buffer's sums are over: its reader has passed the barrier)
        if (at + kConstTerms < terms) fetch(at + kConstTerms);
        if (t < kConstOutputs) {
            const int count = min(kConstTerms, terms - at);
#pragma unroll 8
            for (int i = 0; i < count; ++i) {
                const double v = s_terms[buffer][i][t];
                sum = __dadd_rn(sum, rows ? __dmul_rn(v, mean[at + i]) : v);
            }
        }
    }
    const int i = first + t;
    if (t >= kConstOutputs || i >= outputs) return;
    if (rows) {
        enc_bias[i] = (float)__ddiv_rn(-__dadd_rn(sum, lo), step);
        tmu32[i] = (float)sum;
    } else dec_bias[i] = (float)__dadd_rn(mean[i], __dmul_rn(__dadd_rn(lo, __dmul_rn(center, step)), sum));
}

// bf16 operand copies: b[j][a], its transpose bt[a][j] and, unless null, bc: b in core matrices of 8 x 8
// elements (128 contiguous bytes), those of the same eight rows side by side (an 8-bit basis as its integers)
__global__ void basis_bf16_kernel(const double *basis, int c, int k, double scale_or_zero, __nv_bfloat16 *b, __nv_bfloat16 *bt,
                                  __nv_bfloat16 *bc)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)k * c) return;
    const int j = (int)(i / c), a = (int)(i % c);
    const double v = basis[i];
    const float f = scale_or_zero != 0.0 ? (float)rint(__ddiv_rn(v, scale_or_zero)) : (float)v;
    const __nv_bfloat16 h = __float2bfloat16(f);
    b[i] = h;
    bt[(size_t)a * k + j] = h;
    if (bc) bc[((size_t)(j >> 3) * (c >> 3) + (a >> 3)) * 64 + (j & 7) * 8 + (a & 7)] = h;
}

}  // namespace

tc_status tc_launch_moments_to_cov(const double *sum, const double *outer, long long count, int c, double *mean, double *cov,
                                   cudaStream_t s)
{
    const long long n = (long long)c * c;
    moments_to_cov_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(sum, outer, (double)count, c, mean, cov);
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_scale_mirror(double *cov, int c, double denom, cudaStream_t s)
{
    const long long n = (long long)c * c;
    scale_mirror_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(cov, c, denom);
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

// Column blocks and padding of the Jacobi kernel for c columns: rows of 64 R elements, blocks of B
// columns, an even number of them.
struct JacobiShape { int r, b, n_blocks, ld; };
static JacobiShape jacobi_shape(int c)
{
    JacobiShape j;
    const int need = (c + 63) / 64;
    j.r = need <= 2 ? need : need <= 4 ? 4 : need <= 6 ? 6 : need <= 8 ? 8 : need <= 12 ? 12 : 16;
    j.b = j.r <= 8 ? 16 : 8;
    j.ld = 64 * j.r;
    j.n_blocks = 2 * ((c + 2 * j.b - 1) / (2 * j.b));
    return j;
}

static size_t jacobi_workspace_bytes(int c)
{
    const JacobiShape j = jacobi_shape(c);
    return ((size_t)j.n_blocks * j.b * j.ld + (size_t)c * c + (size_t)c) * sizeof(double) + sizeof(JacobiState);
}

size_t tc_eigh_device_workspace_bytes(int c)
{
    const size_t cluster = tc_eigh_cluster_workspace_bytes(c), jacobi = jacobi_workspace_bytes(c);
    return cluster > jacobi ? cluster : jacobi;
}

// One-sided Jacobi, queued like tc_launch_eigh_cluster.
static tc_status launch_jacobi(const double *a, int c, void *work, double **vt, double **lambda, int **outcome, cudaStream_t s)
{
    const JacobiShape js = jacobi_shape(c);
    double *g = static_cast<double *>(work);
    *vt = g + (size_t)js.n_blocks * js.b * js.ld;
    *lambda = *vt + (size_t)c * c;
    JacobiState *st = reinterpret_cast<JacobiState *>(*lambda + c);
    *outcome = &st->outcome;
    TC_CUDA(cudaMemsetAsync(st, 0, sizeof(JacobiState), s));
    frobenius_kernel<<<c, kPairThreads, 0, s>>>(a, c, st);
    jacobi_init_kernel<<<js.n_blocks * js.b, kPairThreads, 0, s>>>(a, c, g, js.ld, st);
    // (the rounding of an inner product and of the columns since their rotation grows like sqrt(c);
    // a cluster of m equal eigenvalues is only resolved to m times the bound)
    const double tol = 8.0 * sqrt((double)(c < 16 ? 16 : c)) * DBL_EPSILON;
    double tol2 = tol * tol;
    int n_blocks = js.n_blocks;
    const void *kernel = js.r == 1 ? (const void *)jacobi_kernel<1, 16> : js.r == 2 ? (const void *)jacobi_kernel<2, 16>
                       : js.r == 4 ? (const void *)jacobi_kernel<4, 16> : js.r == 6 ? (const void *)jacobi_kernel<6, 16>
                       : js.r == 8 ? (const void *)jacobi_kernel<8, 16> : js.r == 12 ? (const void *)jacobi_kernel<12, 8>
                                   : (const void *)jacobi_kernel<16, 8>;
    const size_t smem = 2 * (size_t)js.b * js.ld * sizeof(double);
    TC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    void *params[] = {&g, &n_blocks, &tol2, &st};
    // cooperative: the blocks wait for one another between rounds
    TC_CUDA(cudaLaunchCooperativeKernel(kernel, dim3(js.n_blocks / 2), dim3(js.b * 32), params, smem, s));
    rayleigh_kernel<<<(c + kVec - 1) / kVec, kPairThreads, 0, s>>>(a, g, js.ld, c, *vt, *lambda);
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

// a: [c][c] symmetric, DEVICE, left untouched.  evals [c + 1], evecs [c][c] (row j = eigenvector of
// evals[j]), DEVICE; evals[c] is the outcome, for tc_eigh_outcome.  `work`: tc_eigh_device_workspace_bytes(c) bytes, DEVICE.
// Only queues work.  Reduction and division wherever the matrix fits a cluster's shared memory (576 rows), Jacobi beyond that, on
// devices that cannot hold the cluster and where `jacobi` asks for it.  tc_device_eigh on graded spectra, Jacobi against cluster: 64 rows 0.50 and 0.23 ms, 128 rows
// 1.5 and 0.42, 256 rows 5.9 and 1.3, 384 rows 12.9 and 1.8, 576 rows 20.6 and 3.8 (a third of a millisecond of it allocation);
// orthogonality 1.4e-14 to 4.4e-14 and 1.2e-15 to 2.3e-15.
tc_status tc_eigh_device(const double *a, int c, double *evals, double *evecs, void *work, bool jacobi, cudaStream_t s)
{
    if (c < 1 || c > TC_MAX_C) return TC_ERR_INVALID_ARG;
    double *vt, *lambda;
    int *outcome;
    tc_status st = jacobi ? TC_ERR_UNSUPPORTED : tc_launch_eigh_cluster(a, c, work, &vt, &lambda, &outcome, s);
    if (st == TC_ERR_UNSUPPORTED) st = launch_jacobi(a, c, work, &vt, &lambda, &outcome, s);
    if (st != TC_OK) return st;
    order_sign_kernel<<<c, kPairThreads, 0, s>>>(vt, lambda, c, outcome, evals, evecs);
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

// What tc_eigh_device left behind the eigenvalues, as a status.
tc_status tc_eigh_outcome(double outcome)
{
    return outcome > 0.0 ? TC_OK : outcome == 0.0 ? TC_ERR_TIMEOUT : TC_ERR_NOT_CONVERGED;
}

// Rounds the basis in place to `dtype`.  scale_slot (DEVICE, one double) receives the scale of an
// 8-bit basis (untouched otherwise).
tc_status tc_launch_round_basis(double *basis, int c, int dtype, double *scale_slot, cudaStream_t s)
{
    const long long n = (long long)c * c;
    if (dtype == TC_INT8) abs_max_kernel<<<1, 1024, 0, s>>>(basis, n, scale_slot);
    round_basis_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(basis, n, dtype, scale_slot);
    if (dtype == TC_INT8) store_scale_kernel<<<1, 1, 0, s>>>(scale_slot);
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_model_consts(const double *basis, const double *mean, int c, int k, double lo, double step, double center,
                                 float *enc_bias, float *tmu32, float *dec_bias, cudaStream_t s)
{
    model_consts_kernel<<<dim3((unsigned)((c + kConstOutputs - 1) / kConstOutputs), 2), 256, 0, s>>>(basis, mean, c, k, lo, step, center, enc_bias, tmu32, dec_bias);
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}

tc_status tc_launch_basis_bf16(const double *basis, int c, int k, double basis_scale, bool int8, void *b, void *bt, void *bc,
                               cudaStream_t s)
{
    const long long n = (long long)k * c;
    basis_bf16_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(basis, c, k, int8 ? basis_scale : 0.0,
                                                                 static_cast<__nv_bfloat16 *>(b), static_cast<__nv_bfloat16 *>(bt),
                                                                 static_cast<__nv_bfloat16 *>(bc));
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}
