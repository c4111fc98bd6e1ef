// Eigendecomposition of a symmetric matrix of up to 576 rows in fp64, in four kernels: Householder reduction to tridiagonal
// form by one thread-block cluster that holds the matrix on chip, divide and conquer on the tridiagonal matrix by another
// (Cuppen 1981; eigenvectors from the modified z of Gu and Eisenstat 1994), the reflectors applied to its eigenvectors, and
// Rayleigh quotients.
//
// Why this replaces the one-sided Jacobi method of eigh_device.cu wherever the matrix fits: Jacobi needs 13 to 28 sweeps
// of n - 1 dependent rounds over all of the matrix; the reduction has n dependent steps in all, each a pass over what is
// left of it, and dividing has log2(n) levels.
#include "device_utils.cuh"

#include <cfloat>

namespace {

using tcdev::cluster_sync;
using tcdev::mma_f64;
using tcdev::peer_address;

constexpr int kReduceWarps = 8, kReduceThreads = 32 * kReduceWarps;    // of a block that reduces: what every warp repeats costs issue slots
constexpr int kWarps = 16, kThreads = 32 * kWarps;                      // of one that divides, or takes Rayleigh quotients
constexpr int kMaxCluster = 16;
constexpr int kMostRows = 576;                         // what sixteen blocks' shared memory holds
constexpr int kGroup = 16;                             // eigenvectors that a block works out together: two rows of MMA tiles
constexpr int kPad = 4;                                // doubles between rows of U: rows 0 .. 3 of an operand lie 8 banks apart

struct EighArgs {
    const double *a;                                   // [n][n]
    int n;
    double *reflectors;                                // [n up to a multiple of 4][ld], row k: the vector of step k
    double *tau;                                       // [n up to a multiple of 4]
    double *gram;                                      // [groups of four reflectors][6]
    double *d, *e;                                     // [n], [n]: the tridiagonal matrix
    double *roots;                                     // [3][n up to a multiple of 16]: of a level of the division, see divide_kernel
    double *q0, *q1;                                   // [n up to a multiple of 16][ld]: row j is eigenvector j of the tridiagonal matrix
    double *vt;                                        // [n][n]: row j is eigenvector j
    double *lambda;                                    // [n]
    int *state;                                        // [0] passes over the matrix, -1: not finite, 0: a wait ran out; [1] whether q1 holds the eigenvectors
};

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %cluster_ctarank;" : "=r"(r));
    return r;
}

// 16 rows of `u` (shared memory, row pitch ld_u) times columns [col, col + 16) of `b` (global memory, row pitch ld_b),
// terms [k0, k1) with k1 - k0 a multiple of 4; rows and columns of `b` past `last` read the last ones: `u` is zero there, and
// so are its results' uses
__device__ __forceinline__ void tile_product(double2 (&acc)[2][2], const double *u, int ld_u, const double *b, int ld_b, int last, int col,
                                             int k0, int k1)
{
    const int lane = threadIdx.x & 31, lr = lane >> 2, lk = lane & 3;
    const double *left = b + min(col + lr, last), *right = b + min(col + lr + 8, last);
    constexpr int kAhead = 8;                          // steps of four terms whose operands are on their way together
#pragma unroll 1
    for (int k = k0; k < k1; k += 4 * kAhead) {
        double b0[kAhead], b1[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const size_t at = (size_t)min(k + 4 * i + lk, last) * ld_b;
            b0[i] = __ldcg(left + at); b1[i] = __ldcg(right + at);
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i) asm volatile("" : "+d"(b0[i]), "+d"(b1[i]));       // (loads are not moved to their uses)
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            if (k + 4 * i >= k1) break;
            const int row = k + 4 * i + lk;
            const double a0 = u[lr * ld_u + row], a1 = u[(lr + 8) * ld_u + row];
            mma_f64(acc[0][0], a0, b0[i]);
            mma_f64(acc[0][1], a0, b1[i]);
            mma_f64(acc[1][0], a1, b0[i]);
            mma_f64(acc[1][1], a1, b1[i]);
        }
    }
}

// Root of c + s / (a - t) + r / (b - t) inside (lo, hi), or the middle of (lo, hi) if rounding puts both outside
__device__ __forceinline__ double two_pole_root(double c, double s, double r, double a, double b, double lo, double hi)
{
    const double p = c * (a + b) + s + r, q = c * a * b + s * b + r * a;
    const double root = sqrt(fmax(p * p - 4.0 * c * q, 0.0));
    const double h = 0.5 * (p + (p >= 0.0 ? root : -root));
    const double t0 = q / h, t1 = h / c;
    if (t0 > lo && t0 < hi) return t0;
    if (t1 > lo && t1 < hi) return t1;
    return 0.5 * (lo + hi);
}

// One root of 1 + rho sum z_i^2 / (d_i - x), the j-th of m (poles ascending, strictly), as the nearer pole `origin` and the
// distance from it: the distance is what later differences need to full relative accuracy.  Each side of the root is replaced by
// a constant and one pole that match its value and slope (Bunch, Nielsen and Sorensen 1978): quadratic convergence, two to
// three steps on average; a bracket is kept and halved where a step leaves it.  The whole warp works on one root.
__device__ __forceinline__ void secular_root(const double *pole, const double *z, int m, int j, double inv_rho, double rho, int &origin, double &tau)
{
    const int lane = threadIdx.x & 31;
    const bool last = j == m - 1;
    double lo, hi, t;
    // value at the middle of the interval: which pole is nearer, and the first step with all other poles held constant
    double width;
    if (!last) width = pole[j + 1] - pole[j];
    else {
        double zz = 0.0;
        for (int i = lane; i < m; i += 32) zz += z[i] * z[i];
        width = rho * warp_sum(zz) * (1.0 + 8.0 * DBL_EPSILON);
    }
    const double mid = 0.5 * width;
    double rest = 0.0, own = 0.0;
    for (int i = lane; i < m; i += 32) {
        const double term = z[i] * z[i] / ((pole[i] - pole[j]) - mid);
        if (i == j || i == j + 1) own += term;
        else rest += term;
    }
    rest = warp_sum(rest) + inv_rho;
    const double f_mid = warp_sum(own) + rest;
    if (last) {
        origin = j;
        lo = f_mid >= 0.0 ? 0.0 : mid;
        hi = f_mid >= 0.0 ? mid : width;
        t = rest > 0.0 ? z[j] * z[j] / rest : 0.5 * (lo + hi);
        if (!(t > lo && t < hi)) t = 0.5 * (lo + hi);
    } else {
        const bool left = f_mid >= 0.0;
        origin = left ? j : j + 1;
        lo = left ? 0.0 : -mid;
        hi = left ? mid : 0.0;
        t = two_pole_root(rest, z[j] * z[j], z[j + 1] * z[j + 1], left ? 0.0 : -width, left ? width : 0.0, lo, hi);
    }
    const double base = pole[origin];
#pragma unroll 1
    for (int step = 0; step < 100; ++step) {
        double psi = 0.0, dpsi = 0.0, phi = 0.0, dphi = 0.0;
        for (int i = lane; i < m; i += 32) {
            const double r = 1.0 / ((pole[i] - base) - t), q = z[i] * z[i] * r;
            if (i <= j) { psi += q; dpsi += q * r; }
            else { phi += q; dphi += q * r; }
        }
        psi = warp_sum(psi); dpsi = warp_sum(dpsi); phi = warp_sum(phi); dphi = warp_sum(dphi);
        const double f = inv_rho + psi + phi;
        // the rounding of the sums and of t itself: nothing below that can be told from a root
        if (fabs(f) <= DBL_EPSILON * (8.0 * (phi - psi) + inv_rho + fabs(t) * (dpsi + dphi))) break;
        if (f < 0.0) lo = t; else hi = t;
        const double a = (pole[j] - base) - t;
        double next;
        if (!last) {
            const double b = (pole[j + 1] - base) - t;
            next = t + two_pole_root(f - dpsi * a - dphi * b, dpsi * a * a, dphi * b * b, a, b, lo - t, hi - t);
        } else next = t + (a + dpsi * a * a / (f - dpsi * a));
        if (!(next > lo && next < hi)) next = 0.5 * (lo + hi);
        if (next == t || next <= lo || next >= hi) break;
        t = next;
    }
    tau = t;
}

// Sums of R values per lane over a warp: lane l gets the sum of value l / (32 / P), P the power of two from R on.  Half of the
// values change lanes in each of the first rounds, so that R sums take about R + 2 shuffles instead of 5 R.
template <int R, int P = R <= 1 ? 1 : R <= 2 ? 2 : R <= 4 ? 4 : R <= 8 ? 8 : 16>
__device__ __forceinline__ double warp_sums(const double (&v)[R])
{
    static_assert(R <= 16, "at most 16 sums");
    const int lane = threadIdx.x & 31;
    double x[P];
#pragma unroll
    for (int i = 0; i < P; ++i) x[i] = i < R ? v[i < R ? i : 0] : 0.0;
    int d = 16;
#pragma unroll
    for (int m = P / 2; m > 0; m >>= 1, d >>= 1) {
        const bool upper = lane & d;
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const double keep = upper ? x[i + m] : x[i], give = upper ? x[i] : x[i + m];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, give, d);
        }
    }
#pragma unroll
    for (; d > 0; d >>= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], d);
    return x[0];
}

__device__ __forceinline__ uint32_t shared_address(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// The barrier's phase is over (two seconds at most: false).
__device__ __forceinline__ bool wait_phase(uint32_t barrier, uint32_t parity)
{
    unsigned long long t0 = 0, t1;
    for (unsigned int polls = 1;; ++polls) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(barrier), "r"(parity) : "memory");
        if (done) return true;
        if (polls % 256 == 0) {
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t1));
            if (!t0) t0 = t1;
            else if (t1 - t0 > 2000000000ull) return false;
        }
    }
}

// Reduction to tridiagonal form.  EL: elements of a row per lane (n <= 32 EL); RW: rows per warp; ON_REGISTERS: rows held in
// registers, not in shared memory.  Block `rank` of BLOCKS in the cluster holds rows rank, rank + BLOCKS, ..., its warps one or a few each.
//
// Step k annihilates column k below the first subdiagonal.  The vectors of a step lie in every block's shared memory, element j
// worked out by thread j of each block.  A warp multiplies its rows with the column's tail; the products, and row k + 1 (the next
// column) from the warp that has it, go to all blocks (bulk copies counted by the receiver's barrier).  On the way are hidden: the
// norm, the square root and the division, and the rows' update with the reflector of the step before -- the product is taken
// with the rows as they were before that update, and its two rank-one terms are put in by the receiver, from two more inner products.
//
// What bounds it: the chain of a step.  Measured alone (cycles): exchange among 4, 8, 16 blocks 925, 1090, 1460 (remote stores
// with a cluster barrier 1470, 1680, 2080; st.async 16 bytes at a time 1290, 1820, 3100; flags in L2 2800 to 3200), a sum over a
// warp 177, square root 95, division 130.  So few blocks, each with as many rows as its registers hold, and few warps: what each repeats (sums over
// the warp, of fp64 and shuffles) shares the issue slots.  256 rows: 0.70 ms with sixteen warps that share the vector work, 0.48
// with the three inner products in one pass, 0.45 with eight warps (3 400 cycles a step); 64 rows in one block 0.09.
template <int EL, int RW, int BLOCKS, bool ON_REGISTERS>
__global__ void __launch_bounds__(kReduceThreads, 1) tridiagonal_kernel(const EighArgs args)
{
    constexpr int ld = 32 * EL, slots = RW * kReduceWarps, message = slots + 32 / BLOCKS, per_thread = (ld + kReduceThreads - 1) / kReduceThreads;
    constexpr int lanes_a_sum = 32 / (RW <= 4 ? 4 : RW <= 8 ? 8 : 16);
    extern __shared__ __align__(16) double s_mem[];
    __shared__ double s_scale[kMaxCluster], s_most[kReduceWarps], s_part[3 * kReduceWarps], s_scalar[6];
    __shared__ __align__(16) double s_dot[kReduceWarps];
    __shared__ __align__(8) uint64_t s_arrived[2];
    __shared__ volatile bool s_failed;                 // a wait ran out
    const int n = args.n, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = (int)cluster_rank();
    // Column tail, last v, last w.  A block's message is the products of its rows, padded so that the lanes that read rows
    // j, j + 1, ... of different blocks meet different banks.
    double *const s_x = s_mem, *const s_pv = s_x + ld, *const s_pw = s_pv + ld;
    double *const s_sent = s_pw + ld, *const s_sent_row = s_sent + 2 * message;                            // [2][message], [2][ld]
    double *const s_got = BLOCKS > 1 ? s_sent_row + 2 * ld : s_sent;                                       // [2][BLOCKS][message]
    double *const s_got_row = BLOCKS > 1 ? s_got + 2 * BLOCKS * message : s_sent_row;                      // [2][ld]
    double *const s_rows = s_got_row + 2 * ld;
    const uint32_t arrived = shared_address(s_arrived);
    constexpr uint32_t product_bytes = slots * sizeof(double), row_bytes = ld * sizeof(double), step_bytes = BLOCKS * product_bytes + row_bytes;
    if (tid == 0) {
        s_failed = false;
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared.b64 [%0], 1;" ::"r"(arrived + 8 * i));
            asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(arrived + 8 * i), "r"(step_bytes) : "memory");
        }
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    cluster_sync();                                                    // every block runs: its shared memory may be written

    // scale: a power of two that brings the matrix to at most 1
    double most = 0.0;
    bool finite = true;
    for (int r = rank + BLOCKS * warp; r < n; r += BLOCKS * kReduceWarps)
        for (int j = lane; j < n; j += 32) { const double v = args.a[(size_t)r * n + j]; finite = finite && isfinite(v); most = fmax(most, fabs(v)); }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) most = fmax(most, __shfl_xor_sync(0xffffffffu, most, d));
    if (!__all_sync(0xffffffffu, finite)) most = INFINITY;
    if (lane == 0) s_most[warp] = most;
    __syncthreads();
    if (tid < BLOCKS) {
        for (int w = 0; w < kReduceWarps; ++w) most = fmax(most, s_most[w]);
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(peer_address(s_scale + rank, tid)), "d"(most) : "memory");
    }
    cluster_sync();
    for (int b = 0; b < BLOCKS; ++b) most = fmax(most, s_scale[b]);
    if (!(most < INFINITY)) {                                          // the same in every block
        if (rank == 0 && tid == 0) args.state[0] = -1;
        return;
    }
    if (rank == 0 && tid == 0) args.state[0] = 1;
    int exponent = 0;
    if (most > 0.0) frexp(most, &exponent);

    double a[ON_REGISTERS ? RW : 1][EL];
    // rows in shared memory, by slot; slots past the last row that a block can have do not exist there
    auto own = [&](int q) { return s_rows + (size_t)(warp + kReduceWarps * q) * ld + lane; };
    auto exists = [&](int q) { return ON_REGISTERS || warp + kReduceWarps * q < ld / BLOCKS; };
#pragma unroll
    for (int q = 0; q < RW; ++q) {
        const int r = rank + BLOCKS * (warp + kReduceWarps * q);
#pragma unroll
        for (int i = 0; i < EL; ++i) {
            const int j = lane + 32 * i;
            const double v = r < n && j < n ? ldexp(args.a[(size_t)r * n + j], -exponent) : 0.0;
            if (ON_REGISTERS) a[q][i] = v;
            else if (exists(q)) own(q)[32 * i] = v;
        }
    }
    for (int j = tid; j < ld; j += kReduceThreads) {                         // column 0 is row 0
        const double v = j < n ? ldexp(args.a[j], -exponent) : 0.0;
        s_x[j] = j > 1 ? v : 0.0;
        s_pv[j] = s_pw[j] = 0.0;
        if (j == 0 && rank == 0) args.d[0] = v;
        if (j == 1) s_scalar[0] = v;
    }
    __syncthreads();

#pragma unroll 1
    for (int k = 0; k < n - 1; ++k) {
        const int buffer = k & 1, from = (k + 1) >> 5;
        double *const sent = s_sent + buffer * message, *const sent_row = s_sent_row + buffer * ld;
        const double *const got = s_got + buffer * BLOCKS * message, *const got_row = s_got_row + buffer * ld;
        // products of the rows with the tail of the column; inner products of the tail with itself and with the last v and w
        {
            double three[3] = {}, sums[RW];
#pragma unroll
            for (int q = 0; q < RW; ++q) sums[q] = 0.0;
#pragma unroll
            for (int m = 0; m < per_thread; ++m) {
                const int j = tid + kReduceThreads * m;
                if (j >= ld) break;
                const double x = s_x[j];
                three[0] = fma(x, x, three[0]);
                three[1] = fma(x, s_pv[j], three[1]);
                three[2] = fma(x, s_pw[j], three[2]);
            }
#pragma unroll
            for (int i = 0; i < EL; ++i) {
                if (i < from) continue;
                const double x = s_x[lane + 32 * i];
#pragma unroll
                for (int q = 0; q < RW; ++q)
                    if (exists(q)) sums[q] = fma(ON_REGISTERS ? a[q][i] : own(q)[32 * i], x, sums[q]);
            }
            const double sum3 = warp_sums<3>(three), sum = warp_sums<RW>(sums);
            if (lane % 8 == 0 && lane < 24) s_part[kReduceWarps * (lane / 8) + warp] = sum3;
            if (lane % lanes_a_sum == 0 && lane / lanes_a_sum < RW) sent[warp + kReduceWarps * (lane / lanes_a_sum)] = sum;
            if ((k + 1) % BLOCKS == rank && (k + 1) / BLOCKS % kReduceWarps == warp) {
                const int mine = (k + 1) / (BLOCKS * kReduceWarps);
#pragma unroll
                for (int q = 0; q < RW; ++q)
                    if (q == mine) {
#pragma unroll
                        for (int i = 0; i < EL; ++i) sent_row[lane + 32 * i] = ON_REGISTERS ? a[q][i] : own(q)[32 * i];
                    }
            }
        }
        if (BLOCKS > 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (BLOCKS > 1 && tid < BLOCKS) {
            const uint32_t barrier = peer_address(s_arrived + buffer, tid);
            asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
                         "r"(peer_address(got + rank * message, tid)), "r"(shared_address(sent)), "r"(product_bytes), "r"(barrier) : "memory");
            if ((k + 1) % BLOCKS == rank)
                asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
                             "r"(peer_address(got_row, tid)), "r"(shared_address(sent_row)), "r"(row_bytes), "r"(barrier) : "memory");
        }
        if (warp == kReduceWarps - 1) {
            // reflector (tail, head) with the sign that adds: I - tau v v^T
            double norm2 = s_part[lane & (kReduceWarps - 1)], with_last = s_part[kReduceWarps + (lane & (2 * kReduceWarps - 1))];   // with v, with w
#pragma unroll
            for (int d = kReduceWarps / 2; d > 0; d >>= 1) {
                norm2 += __shfl_xor_sync(0xffffffffu, norm2, d);
                with_last += __shfl_xor_sync(0xffffffffu, with_last, d);
            }
            const double first = s_scalar[0];
            double tau = 0.0, alpha = first, head = 0.0;
            if (norm2 > 1e-290) {                                      // below, the column counts as reduced: off by 1e-145 at most
                alpha = sqrt(fma(first, first, norm2));
                if (first >= 0.0) alpha = -alpha;
                head = first - alpha;
                tau = -1.0 / (alpha * head);
            }
            if (lane % kReduceWarps == 0 && lane < 2 * kReduceWarps) s_scalar[1 + lane / kReduceWarps] = with_last;
            if (lane == 0) {
                s_scalar[3] = head;
                s_scalar[4] = tau;
                if (rank == 0) { args.e[k] = alpha; args.tau[k] = tau; }
            }
        }
        // rows' update with the last step's v and w
        double rv[RW], rw[RW];
#pragma unroll
        for (int q = 0; q < RW; ++q) {
            const int r = min(rank + BLOCKS * (warp + kReduceWarps * q), ld - 1);
            rv[q] = s_pv[r]; rw[q] = s_pw[r];
        }
#pragma unroll
        for (int i = 0; i < EL; ++i) {
            if (i < from) continue;
            const double pv = s_pv[lane + 32 * i], pw = s_pw[lane + 32 * i];
#pragma unroll
            for (int q = 0; q < RW; ++q) {
                if (!exists(q)) continue;
                const double x = ON_REGISTERS ? a[q][i] : own(q)[32 * i];
                const double y = fma(-rw[q], pv, fma(-rv[q], pw, x));
                if (ON_REGISTERS) a[q][i] = y; else own(q)[32 * i] = y;
            }
        }
        if (BLOCKS > 1 && !s_failed && !wait_phase(arrived + 8 * buffer, (k >> 1) & 1)) {      // then everyone walks on without waiting
            s_failed = true;
            args.state[0] = 0;
        }
        __syncthreads();
        if (BLOCKS > 1 && tid == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(arrived + 8 * buffer), "r"(step_bytes) : "memory");
        // next column c (updated with the last step), p = A v, w = tau (p - (tau v.p / 2) v), then c updated with this step
        const double v_pv = s_scalar[1], v_pw = s_scalar[2], head = s_scalar[3], tau = s_scalar[4];
        const double pv_next = s_pv[k + 1], pw_next = s_pw[k + 1];
        double v[per_thread], p[per_thread], c[per_thread], dot = 0.0;
#pragma unroll
        for (int m = 0; m < per_thread; ++m) {
            const int j = tid + kReduceThreads * m;
            v[m] = p[m] = c[m] = 0.0;
            if (j <= k || j >= n) continue;
            const double pv = s_pv[j], pw = s_pw[j];
            c[m] = fma(-pw, pv_next, fma(-pv, pw_next, got_row[j]));
            p[m] = fma(c[m], head, fma(-pw, v_pv, fma(-pv, v_pw, got[(j % BLOCKS) * message + j / BLOCKS])));
            v[m] = tau == 0.0 ? 0.0 : j == k + 1 ? head : s_x[j];
            dot = fma(v[m], p[m], dot);
            if (j == k + 1) s_scalar[5] = p[m];
        }
        dot = warp_sum(dot);
        if (lane == 0) s_dot[warp] = dot;
        __syncthreads();
        double2 half[kReduceWarps / 2];
#pragma unroll
        for (int i = 0; i < kReduceWarps / 2; ++i) half[i] = reinterpret_cast<const double2 *>(s_dot)[i];
#pragma unroll
        for (int m = kReduceWarps / 4; m > 0; m >>= 1)
#pragma unroll
            for (int i = 0; i < m; ++i) { half[i].x += half[i + m].x; half[i].y += half[i + m].y; }
        const double half_dot = 0.5 * tau * (half[0].x + half[0].y), w_next = tau * fma(-half_dot, head, s_scalar[5]);
#pragma unroll
        for (int m = 0; m < per_thread; ++m) {
            const int j = tid + kReduceThreads * m;
            if (j >= ld) break;
            const double w = tau * fma(-half_dot, v[m], p[m]), x = fma(-head, w, fma(-w_next, v[m], c[m]));
            s_pv[j] = v[m];
            s_pw[j] = w;
            s_x[j] = j > k + 2 ? x : 0.0;
            if (j == k + 2) s_scalar[0] = x;
            if (j == k + 1 && rank == 0) args.d[k + 1] = x;
            if (k % BLOCKS == rank) args.reflectors[(size_t)k * ld + j] = v[m];
        }
        __syncthreads();
    }
    if (rank == 0)
        for (int k = n - 1 + warp; k < ((n + 3) & ~3); k += kReduceWarps) {  // what a group of four reflectors lacks
            for (int j = lane; j < ld; j += 32) args.reflectors[(size_t)k * ld + j] = 0.0;
            if (lane == 0) args.tau[k] = 0.0;
        }
    cluster_sync();                                                    // no block ends while another's copies may still come
}

// What the levels of the division share, in a block's shared memory (every block has its own copy of the vectors)
struct DivideArrays {
    double *d, *e;                                     // eigenvalues of the blocks so far; the matrix's off-diagonal
    double *pole, *z, *zh, *tau, *scan;                // by position in the merged order
    int *column, *origin;
    double *u;                                         // [kGroup][ld + kPad]
};

// Division of the tridiagonal matrix: blocks of 1, 2, 4, ... rows are joined two and two, T = diag(T1 - rho u u^T, T2 - rho w w^T) +
// rho (u, +-w)(u, +-w)^T with u, w the unit vectors at the cut and rho the size of the off-diagonal element there.  A level:
// roots of the secular equations (one warp each), the z they are exact for, eigenvectors, 16 to a thread block, and their product with
// the halves' eigenvectors on the fp64 tensor cores.  Nothing is deflated: poles are set at least one unit in the last place of |T|
// apart and z kept from zero, which is backward stable and needs no branches.  What a level's roots are passes between the
// blocks through L2.  It also takes the inner products of the reflectors of each group of four.  256 rows: 0.14 ms, of which the
// roots take a third and barriers and tables' ways through L2 most of the rest.
template <int EL>
__global__ void __launch_bounds__(kThreads, 1) divide_kernel(const EighArgs args)
{
    constexpr int ld = 32 * EL;
    extern __shared__ __align__(16) double s_mem[];
    const int n = args.n, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank(), blocks = (int)gridDim.x;
    if (args.state[0] <= 0) return;
    // (1,0) (2,0) (2,1) (3,0) (3,1) (3,2)
    for (int t = rank * kWarps + warp; t < (n + 3) / 4 * 6; t += blocks * kWarps) {
        const int g = t / 6, pair = t % 6, hi = pair == 0 ? 1 : pair < 3 ? 2 : 3, lo = pair - hi * (hi - 1) / 2;
        const double *x = args.reflectors + (size_t)(4 * g + hi) * ld, *y = args.reflectors + (size_t)(4 * g + lo) * ld;
        double acc = 0.0;
#pragma unroll
        for (int i = 0; i < EL; ++i) acc = fma(x[lane + 32 * i], y[lane + 32 * i], acc);
        acc = warp_sum(acc);
        if (lane == 0) args.gram[t] = acc;
    }
    DivideArrays dv;
    dv.d = s_mem; dv.e = dv.d + ld;
    dv.pole = dv.e + ld; dv.z = dv.pole + ld; dv.zh = dv.z + ld; dv.tau = dv.zh + ld; dv.scan = dv.tau + ld;
    dv.column = reinterpret_cast<int *>(dv.scan + 32); dv.origin = dv.column + ld;
    dv.u = dv.scan + 32 + ld;
    const int n16 = (n + 15) & ~15, ld_u = ld + kPad;
    double *const root_tau = args.roots, *const root_zh = root_tau + n16;
    int *const root_origin = reinterpret_cast<int *>(root_zh + n16);
    double bound = 0.0;
    for (int i = lane; i < n; i += 32) {
        const double before = i ? fabs(args.e[i - 1]) : 0.0, behind = i + 1 < n ? fabs(args.e[i]) : 0.0;
        bound = fmax(bound, fabs(args.d[i]) + before + behind);
        if (warp == 0) { dv.d[i] = args.d[i] - before - behind; dv.e[i] = i + 1 < n ? args.e[i] : 0.0; }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) bound = fmax(bound, __shfl_xor_sync(0xffffffffu, bound, d));
    int bound_exp = 0;
    frexp(bound * (1.0 + 1e-9), &bound_exp);
    const double gap = ldexp(0.5 * DBL_EPSILON, bound_exp);            // one unit in the last place of the largest eigenvalue
    for (int g = rank; g < n16 / kGroup; g += blocks)
        for (int t = threadIdx.x; t < kGroup * kGroup; t += kThreads) {
            const int r = t / kGroup, c = t % kGroup;
            args.q0[(size_t)(g * kGroup + r) * ld + g * kGroup + c] = r == c ? 1.0 : 0.0;
        }
    cluster_sync();

    double *q_in = args.q0, *q_out = args.q1;
    int passes = 1;
#pragma unroll 1
    for (int size = 2; size < 2 * n; size *= 2) {
        const int half = size / 2;
        bool any = false;
        for (int cut = half; cut < n; cut += size) any = any || fabs(dv.e[cut - 1]) > 0.25 * gap;
        passes += any;
        // merged order of the two halves of each block, the coupling vector in that order
        for (int i = threadIdx.x; i < n; i += kThreads) {
            const int base = i / size * size, cut = base + half, end = min(base + size, n);
            const double di = dv.d[i];
            int pos = i;
            if (cut < n) {
                const bool right = i >= cut;
                int a = right ? base : cut, b = right ? cut : end;     // elements of the other half that come before
                const int other = a;
                while (a < b) {
                    const int m = (a + b) >> 1;
                    if (dv.d[m] < di || (right && dv.d[m] == di)) a = m + 1; else b = m;
                }
                pos = right ? (i - cut) + (a - other) + base : i + (a - other);
            }
            double zi = 0.0;
            if (cut < n) {
                zi = i < cut ? __ldcg(q_in + (size_t)i * ld + cut - 1) : __ldcg(q_in + (size_t)i * ld + cut);
                if (i >= cut && dv.e[cut - 1] < 0.0) zi = -zi;
                if (fabs(zi) < DBL_EPSILON) zi = zi < 0.0 ? -DBL_EPSILON : DBL_EPSILON;
            }
            dv.pole[pos] = di;
            dv.z[pos] = zi;
            dv.column[pos] = i;
        }
        __syncthreads();
        // poles at least `gap` apart (the running maximum of d_i - i gap): nothing is deflated, equal eigenvalues are told apart by
        // rounding instead.  They are multiples of `gap` before that, so that every sum here is exact: half a gap beside one, just below a
        // power of two, sums rounded to even gave neighbours the same pole, and NaN for eigenvectors (eigenvalues 1 and 2, 64 of them).
        double mine[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int pos = threadIdx.x + q * kThreads;
            if ((pos & ~31) >= n) break;
            const int at = pos & (size - 1), start = max(pos - at, pos & ~31) & 31;    // first lane of this block's in the warp
            double x = pos < n ? rint(dv.pole[pos] / gap) * gap - at * gap : -INFINITY;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const double y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane - d >= start) x = fmax(x, y);
            }
            if (lane == 31) dv.scan[pos >> 5] = x;
            mine[q] = x;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int pos = threadIdx.x + q * kThreads;
            if (pos >= n) break;
            const int base = pos & ~(size - 1), at = pos - base, cut = base + half;
            for (int c = base >> 5; c < pos >> 5; ++c) mine[q] = fmax(mine[q], dv.scan[c]);
            if (cut < n && fabs(dv.e[cut - 1]) > 0.25 * gap) dv.pole[pos] = mine[q] + at * gap;
        }
        __syncthreads();
        // roots
        for (int j = rank * kGroup + warp; j < n; j += blocks * kGroup) {
            const int base = j & ~(size - 1), cut = base + half, end = min(base + size, n);
            const double rho = cut < n ? fabs(dv.e[cut - 1]) : 0.0;
            double tau = 0.0;
            int origin = j - base;
            if (rho > 0.25 * gap) secular_root(dv.pole + base, dv.z + base, end - base, j - base, 1.0 / rho, rho, origin, tau);
            if (lane == 0) { __stcg(root_tau + j, tau); __stcg(root_origin + j, base + origin); }
        }
        cluster_sync();
        for (int i = threadIdx.x; i < n; i += kThreads) { dv.tau[i] = __ldcg(root_tau + i); dv.origin[i] = __ldcg(root_origin + i); }
        __syncthreads();
        // the z for which these are the exact roots: z_i^2 = prod (x_j - d_i) / prod (d_j - d_i), factors paired so that each lies in (0, 1]
        for (int i = rank * kGroup + warp; i < n; i += blocks * kGroup) {
            const int base = i & ~(size - 1), cut = base + half, end = min(base + size, n);
            if (!(cut < n && fabs(dv.e[cut - 1]) > 0.25 * gap)) continue;
            const double di = dv.pole[i];
            double prod = 1.0;
            for (int j = base + lane; j < end; j += 32) {
                const double num = (dv.pole[dv.origin[j]] - di) + dv.tau[j];
                prod *= j < i ? num / (dv.pole[j] - di) : j + 1 < end ? num / (dv.pole[j + 1] - di) : num;
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) prod *= __shfl_xor_sync(0xffffffffu, prod, d);
            const double zh = copysign(sqrt(fabs(prod)), dv.z[i]);
            if (lane == 0) __stcg(root_zh + i, zh);
        }
        cluster_sync();
        for (int i = threadIdx.x; i < n; i += kThreads) dv.zh[i] = __ldcg(root_zh + i);
        __syncthreads();
        // eigenvectors of the merged problem, 16 at a time, and their product with the halves' eigenvectors
        for (int g = rank; g < n16 / kGroup; g += blocks) {
            const int j = g * kGroup + warp, lo = (g * kGroup) & ~(size - 1), hi = min(max(lo + size, lo + kGroup), n16);
            double *u = dv.u + (size_t)warp * ld_u;
            for (int i = lo + lane; i < hi; i += 32) u[i] = 0.0;
            __syncwarp();
            if (j < n) {
                const int base = j & ~(size - 1), cut = base + half, end = min(base + size, n);
                if (cut < n && fabs(dv.e[cut - 1]) > 0.25 * gap) {
                    const double org = dv.pole[dv.origin[j]], tau = dv.tau[j];
                    double norm = 0.0;
                    for (int i = base + lane; i < end; i += 32) {
                        const double x = dv.zh[i] / ((dv.pole[i] - org) - tau);
                        u[dv.column[i]] = x;
                        norm = fma(x, x, norm);
                    }
                    norm = 1.0 / sqrt(warp_sum(norm));
                    __syncwarp();
                    for (int i = base + lane; i < end; i += 32) u[i] *= norm;
                } else if (lane == 0) u[dv.column[j]] = 1.0;
            }
            __syncthreads();
            for (int c = lo + 16 * warp; c < hi; c += 16 * kWarps) {
                int k0 = lo, k1 = hi;
                if (size >= 2 * kGroup) {                              // only rows of the half that holds these columns
                    if (c < lo + half) k1 = min(lo + half, hi); else k0 = lo + half;
                }
                double2 acc[2][2] = {};
                tile_product(acc, dv.u, ld_u, q_in, ld, n16 - 1, c, k0, k1);
#pragma unroll
                for (int a = 0; a < 2; ++a)
#pragma unroll
                    for (int b = 0; b < 2; ++b)
                        __stcg(reinterpret_cast<double2 *>(q_out + (size_t)(g * kGroup + 8 * a + (lane >> 2)) * ld + c + 8 * b + 2 * (lane & 3)), acc[a][b]);
            }
            __syncthreads();
        }
        for (int i = threadIdx.x; i < n; i += kThreads) dv.d[i] = dv.pole[dv.origin[i]] + dv.tau[i];
        double *const t = q_in; q_in = q_out; q_out = t;
        cluster_sync();
    }
    if (rank == 0 && threadIdx.x == 0) { args.state[0] = passes; args.state[1] = q_in == args.q1; }
}

// Rows of the tridiagonal matrix's eigenvectors -> eigenvectors of the matrix: reflectors n - 2, ..., 0 applied, four at a time
// (their inner products with one another are known, so that four sums over a warp go side by side).  One warp per vector; a
// block's warps share the reflectors, copied into shared memory two groups ahead.
constexpr int kReflectWarps = 4, kReflectStages = 3;
template <int R>
__global__ void __launch_bounds__(32 * kReflectWarps) reflect_kernel(const EighArgs args)
{
    constexpr int ld = 64 * R, group = 4 * ld + 16;    // doubles of a stage: four reflectors, their factors and inner products
    extern __shared__ __align__(16) double s_mem[];
    const int n = args.n, j = blockIdx.x * kReflectWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (args.state[0] <= 0) return;
    const int n16 = (n + 15) & ~15;
    const double *q = (args.state[1] ? args.q1 : args.q0) + (size_t)j * ld;
    double2 x[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int at = 64 * i + 2 * lane;
        x[i] = at < n16 ? *reinterpret_cast<const double2 *>(q + at) : make_double2(0.0, 0.0);
    }
    const int groups = (n + 3) / 4;
    auto fetch = [&](int g) {                          // 16-byte pieces
        if (g >= 0) {
            const uint32_t to = shared_address(s_mem + (g % kReflectStages) * group);
            const double *from = args.reflectors + (size_t)4 * g * ld;
            for (int i = threadIdx.x; i < 2 * ld; i += 32 * kReflectWarps)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * i), "l"(from + 2 * i) : "memory");
            if (threadIdx.x < 5) {
                const double *small = threadIdx.x < 2 ? args.tau + 4 * g + 2 * threadIdx.x : args.gram + 6 * g + 2 * (threadIdx.x - 2);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 32 * ld + 16 * threadIdx.x), "l"(small) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(groups - 1);
    fetch(groups - 2);
#pragma unroll 1
    for (int g = groups - 1; g >= 0; --g) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();                               // the group is there, and nobody reads the stage that is filled next
        fetch(g - 2);
        const double *stage = s_mem + (g % kReflectStages) * group, *tau = stage + 4 * ld, *gram = tau + 4;
        const double2 *v = reinterpret_cast<const double2 *>(stage) + lane;
        double dot[4] = {};
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4)
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const double2 w = v[q4 * (ld / 2) + 32 * i];
                dot[q4] = fma(w.x, x[i].x, fma(w.y, x[i].y, dot[q4]));
            }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1)
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) dot[q4] += __shfl_xor_sync(0xffffffffu, dot[q4], d);
        const double s3 = tau[3] * dot[3], s2 = tau[2] * (dot[2] - s3 * gram[5]), s1 = tau[1] * (dot[1] - s3 * gram[4] - s2 * gram[2]);
        const double s0 = tau[0] * (dot[0] - s3 * gram[3] - s2 * gram[1] - s1 * gram[0]);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const double2 w0 = v[32 * i], w1 = v[ld / 2 + 32 * i], w2 = v[ld + 32 * i], w3 = v[3 * (ld / 2) + 32 * i];
            x[i].x = fma(-s0, w0.x, fma(-s1, w1.x, fma(-s2, w2.x, fma(-s3, w3.x, x[i].x))));
            x[i].y = fma(-s0, w0.y, fma(-s1, w1.y, fma(-s2, w2.y, fma(-s3, w3.y, x[i].y))));
        }
    }
    if (j >= n) return;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int at = 64 * i + 2 * lane;
        if (at < n) args.vt[(size_t)j * n + at] = x[i].x;
        if (at + 1 < n) args.vt[(size_t)j * n + at + 1] = x[i].y;
    }
}

// lambda_j = v_j^T A v_j against the untouched matrix: an error of the vectors enters squared.  16 vectors per block.
__global__ void __launch_bounds__(kThreads) rayleigh_tiles_kernel(const EighArgs args)
{
    extern __shared__ __align__(16) double s_u[];      // [kGroup][ld_u]
    __shared__ double s_sum[kWarps][kGroup];
    const int n = args.n, n16 = (n + 15) & ~15, ld_u = n16 + kPad, first = blockIdx.x * kGroup;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (args.state[0] <= 0) return;
    for (int i = lane; i < n16; i += 32) s_u[warp * ld_u + i] = first + warp < n && i < n ? args.vt[(size_t)(first + warp) * n + i] : 0.0;
    __syncthreads();
    double sum[2] = {};
    for (int c = 16 * warp; c < n16; c += 16 * kWarps) {
        double2 acc[2][2] = {};
        tile_product(acc, s_u, ld_u, args.a, n, n - 1, c, 0, n16);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const double *u = s_u + (8 * a + (lane >> 2)) * ld_u + c + 8 * b + 2 * (lane & 3);
                sum[a] = fma(acc[a][b].x, u[0], fma(acc[a][b].y, u[1], sum[a]));
            }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        sum[a] += __shfl_xor_sync(0xffffffffu, sum[a], 1);
        sum[a] += __shfl_xor_sync(0xffffffffu, sum[a], 2);
        if ((lane & 3) == 0) s_sum[warp][8 * a + (lane >> 2)] = sum[a];
    }
    __syncthreads();
    if (threadIdx.x < kGroup && first + threadIdx.x < n) {
        double t = 0.0;
        for (int w = 0; w < kWarps; ++w) t += s_sum[w][threadIdx.x];
        args.lambda[first + threadIdx.x] = t;
    }
}

size_t round_up(size_t v, size_t to) { return (v + to - 1) / to * to; }

// How the kernels are laid out for up to 32 el rows; el = 0 where the matrix does not fit.  One block reduces up to 128 rows (no
// exchange), four up to 256, eight up to 384, sixteen beyond; from 513 on the rows no longer fit the registers.
struct Shape {
    int el, reduce_blocks, divide_blocks;
    const void *reduce, *divide, *reflect;
    size_t reduce_smem, divide_smem, reflect_smem;
};

template <int EL, int RW, int BLOCKS, bool ON_REGISTERS>
Shape shape_of(int divide_blocks)
{
    static_assert(RW * BLOCKS * kReduceWarps >= 32 * EL && (ON_REGISTERS || 32 * EL % BLOCKS == 0), "every row has a place");
    constexpr size_t ld = 32 * EL, message = RW * kReduceWarps + 32 / BLOCKS;
    Shape s{};
    s.el = EL; s.reduce_blocks = BLOCKS; s.divide_blocks = divide_blocks;
    s.reduce = (const void *)tridiagonal_kernel<EL, RW, BLOCKS, ON_REGISTERS>;
    s.divide = (const void *)divide_kernel<EL>;
    s.reflect = (const void *)reflect_kernel<EL / 2>;
    s.reduce_smem = (7 * ld + 2 * message * (BLOCKS > 1 ? BLOCKS + 1 : 1) + (ON_REGISTERS ? 0 : ld / BLOCKS * ld)) * sizeof(double);
    s.divide_smem = (7 * ld + 32 + kGroup * (ld + kPad)) * sizeof(double);
    s.reflect_smem = kReflectStages * (4 * ld + 16) * sizeof(double);
    return s;
}

Shape shape_for(int n)
{
    switch (n > kMostRows ? 0 : (n + 63) / 64) {
    case 0: return {};
    case 1: return shape_of<2, 8, 1, true>(4);
    case 2: return shape_of<4, 16, 1, true>(8);
    case 3: return shape_of<6, 6, 4, true>(kMaxCluster);
    case 4: return shape_of<8, 8, 4, true>(kMaxCluster);
    case 5: return shape_of<10, 5, 8, true>(kMaxCluster);
    case 6: return shape_of<12, 6, 8, true>(kMaxCluster);
    case 7: case 8: return shape_of<16, 4, 16, true>(kMaxCluster);
    default: return shape_of<18, 5, 16, false>(kMaxCluster);
    }
}

struct ClusterLaunch {
    cudaLaunchAttribute attr{};
    cudaLaunchConfig_t cfg{};
    ClusterLaunch(int blocks, int threads, size_t smem, cudaStream_t s)
    {
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)blocks; attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
        cfg.attrs = &attr; cfg.numAttrs = 1;
    }
};

// Sets a kernel up for such a launch; false if the device cannot hold the cluster.
bool cluster_fits(const void *kernel, const ClusterLaunch &l)
{
    int clusters = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.cfg.dynamicSmemBytes) == cudaSuccess &&
        (l.cfg.gridDim.x <= 8 || cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
        cudaOccupancyMaxActiveClusters(&clusters, kernel, &l.cfg) == cudaSuccess && clusters > 0)
        return true;
    cudaGetLastError();
    return false;
}

}  // namespace

// Workspace, 0 where the matrix does not fit: reflectors, their factors and inner products, two sets of eigenvectors of the
// tridiagonal matrix, eigenvectors, eigenvalues, the tridiagonal matrix, a level's roots, state.
size_t tc_eigh_cluster_workspace_bytes(int n)
{
    const Shape shape = shape_for(n);
    if (!shape.el) return 0;
    const size_t ld = 32 * (size_t)shape.el, n4 = round_up(n, 4), n16 = round_up(n, 16);
    return (n4 * ld + n4 + n4 / 4 * 6 + 2 + 2 * n16 * ld + round_up((size_t)n * n, 2) + 6 * n16) * sizeof(double) + 16;
}

// Queues the decomposition of a ([n][n], DEVICE, left untouched): eigenvectors (rows of *vt, in no order), eigenvalues and state
// (see EighArgs) inside `work`.  TC_ERR_UNSUPPORTED, with nothing queued, where the device cannot hold the clusters.
tc_status tc_launch_eigh_cluster(const double *a, int n, void *work, double **vt, double **lambda, int **state, cudaStream_t s)
{
    const Shape shape = shape_for(n);
    if (!shape.el) return TC_ERR_UNSUPPORTED;
    const ClusterLaunch reduce(shape.reduce_blocks, kReduceThreads, shape.reduce_smem, s), divide(shape.divide_blocks, kThreads, shape.divide_smem, s);
    if (!cluster_fits(shape.reduce, reduce) || !cluster_fits(shape.divide, divide)) return TC_ERR_UNSUPPORTED;
    const size_t ld = 32 * (size_t)shape.el, n4 = round_up(n, 4), n16 = round_up(n, 16);
    const size_t rayleigh_smem = kGroup * (n16 + kPad) * sizeof(double);
    if (cudaFuncSetAttribute(shape.reflect, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shape.reflect_smem) != cudaSuccess ||
        cudaFuncSetAttribute(rayleigh_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rayleigh_smem) != cudaSuccess) {
        cudaGetLastError();
        return TC_ERR_CUDA;
    }
    EighArgs args{};
    args.a = a; args.n = n;
    double *p = static_cast<double *>(work);
    args.reflectors = p; p += n4 * ld;
    args.q0 = p; p += n16 * ld;
    args.q1 = p; p += n16 * ld;
    args.vt = p; p += round_up((size_t)n * n, 2);
    args.tau = p; p += n4;
    args.gram = p; p += n4 / 4 * 6 + (n4 / 4 * 6) % 4;
    args.lambda = p; p += n16;
    args.d = p; p += n16;
    args.e = p; p += n16;
    args.roots = p; p += 3 * n16;
    args.state = reinterpret_cast<int *>(p);
    void *params[] = {&args};
    if (cudaLaunchKernelExC(&reduce.cfg, shape.reduce, params) != cudaSuccess || cudaLaunchKernelExC(&divide.cfg, shape.divide, params) != cudaSuccess ||
        cudaLaunchKernel(shape.reflect, dim3((unsigned)((n + kReflectWarps - 1) / kReflectWarps)), dim3(32 * kReflectWarps), params,
                         shape.reflect_smem, s) != cudaSuccess) {
        cudaGetLastError();
        return TC_ERR_CUDA;
    }
    rayleigh_tiles_kernel<<<(unsigned)(n16 / kGroup), kThreads, rayleigh_smem, s>>>(args);
    *vt = args.vt; *lambda = args.lambda; *state = args.state;
    return cudaGetLastError() == cudaSuccess ? TC_OK : TC_ERR_CUDA;
}
