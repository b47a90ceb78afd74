// Stochastic bitflip circuits (Sec. 2.5): each gate flips the bits of g_j
// with probability sin^2(theta_j) instead of acting coherently, and the
// expectation values are exact products (eq. expval_bitflip):
//   <Z_a> = prod_{j in J_a} cos(2 theta_j),  J_a = { j : g_j.a odd }.
// For L = sum_a w_a <Z_a>:
//   dL/dtheta_j = -2 tan(2 theta_j) * sum_a [g_j.a odd] w_a <Z_a>.
// Both are reductions over the bit-packed parities: a product over the set bits
// of each P_A row, and a sum over the set bits of each P_A^T row.
//
// Large problems (k_bf_sums): GB300 runs one FP64 operation per SM and clock, so
// both are sums of 64-bit integers instead. The product is the sum of the
// logarithms: -log2 |cos 2 theta_j| on a grid of 2^-F, F = 62 - ceil(log2 of the
// sum over all gates), with the cosine's sign as bit 63, whose carry-free sum is
// the product's sign; the value is 2^-(sum). The gradient's w_a <Z_a> are integers
// on a grid chosen the same way from sum |w_a <Z_a>|. The sums are exact and do
// not depend on their order. Up to a sum of 512 over all gates the grid's error is below the
// FP64 product's own rounding (2^-53 per factor); past it, or where a cosine is
// zero or not finite, k_bitflip_rows runs instead (a flag on the device decides);
// so does k_bitflip_grad where the values differ so much that the grid's error
// could pass 2^-46 of the gradient's norm.
// Four columns at a time: their 16 partial sums are one table in shared memory
// (128 bytes, each entry in its own pair of banks, so lanes that read different
// entries never collide), a lane takes a row and adds one entry per four bits of
// its words: 5 instructions per four columns whatever bits are set, against about
// 8 and an FP64 operation per set bit. 10^9 bits take 90 us (FP64: 474): bound by
// the shared-memory reads, one of 8 bytes per four columns and lane.
//
// Small problems: FP64 products and sums, one warp per row, in a fixed order
// (lane-strided, then a shuffle tree).
#include "common.cuh"

namespace iqp {

uint32_t check_word_bitflip() { return take_check_word(); }

namespace {

// c_j = cos(2 theta_j), t_j = -2 tan(2 theta_j), zero beyond m.
__global__ void k_bitflip_gates(const float *__restrict__ theta, int64_t m, int64_t mpad, double *__restrict__ c,
                                double *__restrict__ t) {
    pdl_sync();
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < mpad; j += (int64_t)gridDim.x * blockDim.x) {
        if (j < m) {
            const double x = 2.0 * (double)theta[j];
            double sn, cs;
            sincos(x, &sn, &cs);
            c[j] = cs;
            t[j] = -2.0 * sn / cs;
        } else {
            c[j] = 1.0;
            t[j] = 0.0;
        }
    }
}

constexpr int kBfThreads = 512;
constexpr int kBfCols = 2048;                  // columns per CTA: 512 tables of 16 sums, 64 KB
constexpr int kBfSmem = kBfCols / 4 * 16 * 8;
constexpr int kBfBlocks = 304;                 // blocks of the values' pass, one FP64 sum each
constexpr double kBfMaxLog = 512.0;            // sum of the logarithms up to which the integer sums are used

// FP64 sum over the block, on thread 0 (fixed order).
__device__ __forceinline__ double block_sum_f64(double v) {
    __shared__ double red[kBfThreads / 32];
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, w);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < (int)blockDim.x / 32; ++w) v += red[w];
    return v;
}

// t_j = -2 tan(2 theta_j) and x_j = -log2 |cos(2 theta_j)|, with the cosine's sign as x_j's (-0 included); c_j for the
// kernel that multiplies. bsum[b] = the block's sum of |x|.
__global__ void __launch_bounds__(256) k_bf_logs(const float *__restrict__ theta, int64_t m, int64_t mpad,
                                                 double *__restrict__ c, double *__restrict__ t, double *__restrict__ x,
                                                 double *__restrict__ bsum) {
    pdl_sync();
    double acc = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < mpad; j += (int64_t)gridDim.x * 256) {
        double cs = 1.0, tn = 0.0, lg = 0.0;
        if (j < m) {
            double sn;
            sincos(2.0 * (double)theta[j], &sn, &cs);
            tn = -2.0 * sn / cs;
            // log2 |cos| = log1p(-sin^2) / (2 ln 2), exact to the last bits where the cosine is near 1
            lg = fabs(cs) > 0.5 ? -0.72134752044448170368 * log1p(-sn * sn) : -log2(fabs(cs));
        }
        c[j] = cs;
        t[j] = tn;
        x[j] = copysign(lg, cs);
        acc += lg;  // not finite where the cosine is zero or theta is not finite
    }
    acc = block_sum_f64(acc);
    if (threadIdx.x == 0) bsum[blockIdx.x] = acc;
}

// The grid 2^F of integers whose absolute values sum to less than 2^62, from the
// block sums, for every thread of the block; negative where the sum is not finite,
// past `most`, or 2^62 and more. One warp adds (every thread adding all block sums
// cost 10 us of FP64).
__device__ __forceinline__ int bf_grid(const double *__restrict__ bsum, int nb, double most) {
    __shared__ int F;
    if (threadIdx.x < 32) {
        double s = 0.0;
        for (int b = threadIdx.x; b < nb; b += 32) s += bsum[b];
#pragma unroll
        for (int w = 16; w >= 1; w >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, w);
        if (threadIdx.x == 0) {
            int e = s > 0.0 && s <= most ? ilogb(s) + 1 : 0;  // s < 2^e
            if (e < -960) e = -960;
            F = s <= most ? 62 - e : -1;
        }
    }
    __syncthreads();
    return F;
}

// Integers of the logarithms, sign in bit 63 (q: mpad words); the sums start at zero; *grid = F (or -1).
__global__ void __launch_bounds__(256) k_bf_log_ints(const double *__restrict__ x, int64_t mpad,
                                                     const double *__restrict__ bsum, int nb,
                                                     unsigned long long *__restrict__ q,
                                                     unsigned long long *__restrict__ sums, int64_t l,
                                                     int *__restrict__ grid) {
    pdl_sync();
    const int F = bf_grid(bsum, nb, kBfMaxLog);
    if (blockIdx.x == 0 && threadIdx.x == 0) *grid = F;
    if (F < 0) return;
    const double sc = ldexp(1.0, F);
    for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < mpad; j += (int64_t)gridDim.x * 256) {
        const double v = x[j];
        q[j] = (unsigned long long)llrint(fabs(v) * sc) | (signbit(v) ? 1ull << 63 : 0ull);
    }
    for (int64_t a = blockIdx.x * (int64_t)256 + threadIdx.x; a < l; a += (int64_t)gridDim.x * 256) sums[a] = 0ull;
}

// Integers of v (l values, zero up to lpad); the gates' sums start at zero; *grid = F (negative: a value is not finite, or
// too large); *counter = 0.
__global__ void __launch_bounds__(256) k_bf_value_ints(const double *__restrict__ v, int64_t l, int64_t lpad,
                                                       const double *__restrict__ bsum, int nb,
                                                       unsigned long long *__restrict__ q,
                                                       unsigned long long *__restrict__ sums, int64_t m,
                                                       int *__restrict__ grid, unsigned *__restrict__ counter) {
    pdl_sync();
    const int F = bf_grid(bsum, nb, 1.7e308);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *grid = F;
        *counter = 0u;
    }
    if (F < 0) return;
    for (int64_t a = blockIdx.x * (int64_t)256 + threadIdx.x; a < lpad; a += (int64_t)gridDim.x * 256)
        q[a] = a < l ? (unsigned long long)llrint(ldexp(v[a], F)) : 0ull;
    for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < m; j += (int64_t)gridDim.x * 256) sums[j] = 0ull;
}

// sums[row] += sum (mod 2^64) of q[col] over the set bits of the row's columns [2048 y, + 2048): bits is rows x ld
// words, ld a multiple of 4, q padded with zeros to 64 ld. Block (x, y): rows 512 x.., a row per thread.
__global__ void __launch_bounds__(kBfThreads) k_bf_sums(const uint64_t *__restrict__ bits, int64_t rows, int64_t ld,
                                                        const unsigned long long *__restrict__ q,
                                                        unsigned long long *__restrict__ sums,
                                                        const int *__restrict__ grid) {
    pdl_sync();
    extern __shared__ unsigned long long tab[];
    if (*grid < 0) return;
    const int64_t w0 = blockIdx.y * (int64_t)(kBfCols / 64);
    const int words = (int)(ld - w0 < kBfCols / 64 ? ld - w0 : kBfCols / 64);
    // Table T (columns 4 T..): entry e at 16 T + (e ^ (T & 15)), so that the threads' stores of one entry spread over the banks.
    for (int T = threadIdx.x; T < words * 16; T += kBfThreads) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(q + w0 * 64 + 4 * T);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(q + w0 * 64 + 4 * T + 2);
        const unsigned long long lo[4] = {0ull, a.x, a.y, a.x + a.y}, hi[4] = {0ull, b.x, b.y, b.x + b.y};
#pragma unroll
        for (int e = 0; e < 16; ++e) tab[16 * T + (e ^ (T & 15))] = lo[e & 3] + hi[e >> 2];
    }
    __syncthreads();
    const int64_t row = blockIdx.x * (int64_t)kBfThreads + threadIdx.x;
    if (row >= rows) return;
    const uint64_t *r = bits + row * ld + w0;
    unsigned long long s0 = 0ull, s1 = 0ull;
    for (int w = 0; w < words; w += 2) {  // words is a multiple of 4
        const ulonglong2 v = IQP_IN(row * ld + w0 + w + 1, rows * ld, 92) ? *reinterpret_cast<const ulonglong2 *>(r + w)
                                                                          : make_ulonglong2(0ull, 0ull);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t x = h ? v.y : v.x;
            const unsigned long long *t = tab + 256 * (w + h);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                s0 += t[16 * k + ((int)((x >> (4 * k)) & 15u) ^ k)];
                s1 += t[16 * (k + 1) + ((int)((x >> (4 * k + 4)) & 15u) ^ (k + 1))];
            }
        }
    }
    const unsigned long long s = s0 + s1;
    if (s != 0ull) atomicAdd(sums + row, s);
}

// expval[a] = +-2^-(sum / 2^F) and, with w, v[a] = w[a] expval[a] and the block sums of |v|. Where the integers are not in use
// (grid -1) expval is in place already.
__global__ void __launch_bounds__(256) k_bf_rows_out(const unsigned long long *__restrict__ sums, int64_t l,
                                                     const int *__restrict__ grid, double *__restrict__ expval,
                                                     const double *__restrict__ w, double *__restrict__ v,
                                                     double *__restrict__ bsum) {
    pdl_sync();
    const int F = *grid;
    double acc = 0.0;
    for (int64_t a = blockIdx.x * (int64_t)256 + threadIdx.x; a < l; a += (int64_t)gridDim.x * 256) {
        double e;
        if (F < 0) {
            e = expval[a];
        } else {
            // the sum's whole part and its fraction's top bits, exactly; |sum| < 2^63 of the grid
            const unsigned long long s = sums[a], mag = s & ~(1ull << 63);
            const double whole = F < 63 ? (double)(long long)(mag >> F) : 0.0;
            const unsigned long long fr = F < 63 ? mag & ((1ull << F) - 1ull) : mag;
            e = exp2(-ldexp((double)fr, -F)) * exp2(-whole);
            if (s >> 63) e = -e;
            expval[a] = e;
        }
        if (w != nullptr) {
            const double x = w[a] * e;
            v[a] = x;
            acc += fabs(x);
        }
    }
    if (w != nullptr) {
        acc = block_sum_f64(acc);
        if (threadIdx.x == 0) bsum[blockIdx.x] = acc;
    }
}

// grad[j] = t_j sum / 2^F. The last block to finish compares the grid's error
// with the gradient's norm: each of at most l integers is off by 0.3 2^-F in the
// mean, so the gradient by about 0.3 2^-F sqrt(l sum t_j^2); past 2^-46 of its norm
// (values of very different sizes) *grid = -1 and k_bitflip_grad runs.
__global__ void __launch_bounds__(256) k_bf_grad_out(const unsigned long long *__restrict__ sums, int64_t m, int64_t l,
                                                     int *__restrict__ grid, const double *__restrict__ t,
                                                     double *__restrict__ grad, double *__restrict__ bnorm,
                                                     double *__restrict__ bt, unsigned *__restrict__ counter) {
    pdl_sync();
    __shared__ bool last;
    const int F = *reinterpret_cast<volatile int *>(grid);
    if (F < 0) return;  // k_bitflip_grad runs
    const double sc = ldexp(1.0, -F);
    double n2 = 0.0, t2 = 0.0;
    for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < m; j += (int64_t)gridDim.x * 256) {
        const double g = t[j] * ((double)(long long)sums[j] * sc);
        grad[j] = g;
        n2 = fma(g, g, n2);
        t2 = fma(t[j], t[j], t2);
    }
    n2 = block_sum_f64(n2);
    __syncthreads();
    t2 = block_sum_f64(t2);
    if (threadIdx.x == 0) {
        bnorm[blockIdx.x] = n2;
        bt[blockIdx.x] = t2;
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    double n = 0.0, u = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) {
        n += __ldcg(bnorm + b);
        u += __ldcg(bt + b);
    }
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        n += __shfl_xor_sync(0xFFFFFFFFu, n, w);
        u += __shfl_xor_sync(0xFFFFFFFFu, u, w);
    }
    if (threadIdx.x == 0 && !(0.09 * (double)l * u * sc * sc <= n * 0x1.0p-92)) *grid = -1;
}

// expval[a] = product of c_j over the set bits j of P_A row a. One warp per row.
// grid: null, or run only where it is -1.
__global__ void __launch_bounds__(256) k_bitflip_rows(const uint64_t *__restrict__ PA, int64_t ldp, int64_t l,
                                                       const double *__restrict__ c, double *__restrict__ expval,
                                                       const int *__restrict__ grid) {
    pdl_sync();
    if (grid != nullptr && *grid >= 0) return;
    const int lane = threadIdx.x & 31;
    const int64_t a = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (a >= l) return;
    const uint64_t *row = PA + a * ldp;
    double prod = 1.0;
    for (int64_t w = lane; w < ldp; w += 32) {
        uint64_t bits = row[w];
        while (bits) {
            const int b = __ffsll((long long)bits) - 1;
            bits &= bits - 1ull;
            if (IQP_IN(w * 64 + b, ldp * 64, 90)) prod *= c[w * 64 + b];
        }
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) prod *= __shfl_xor_sync(0xFFFFFFFFu, prod, off);
    if (lane == 0) expval[a] = prod;
}

// v[a] = w[a] * expval[a].
__global__ void k_bitflip_weights(const double *__restrict__ w, const double *__restrict__ ev, int64_t l,
                                  double *__restrict__ v) {
    pdl_sync();
    const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (a < l) v[a] = w[a] * ev[a];
}

// grad[j] = t_j * sum of v[a] over the set bits a of P_A^T row j. One warp per gate.
__global__ void __launch_bounds__(256) k_bitflip_grad(const uint64_t *__restrict__ PAT, int64_t ldlt, int64_t m,
                                                       [[maybe_unused]] int64_t l, const double *__restrict__ v,
                                                       const double *__restrict__ t, double *__restrict__ grad,
                                                       const int *__restrict__ grid) {
    pdl_sync();
    if (grid != nullptr && *grid >= 0) return;
    const int lane = threadIdx.x & 31;
    const int64_t j = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (j >= m) return;
    const uint64_t *row = PAT + j * ldlt;
    double acc = 0.0;
    for (int64_t w = lane; w < ldlt; w += 32) {
        uint64_t bits = row[w];
        while (bits) {
            const int b = __ffsll((long long)bits) - 1;
            bits &= bits - 1ull;
            if (IQP_IN(w * 64 + b, l, 91)) acc += v[w * 64 + b];  // bits past the last observable are zero
        }
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if (lane == 0) grad[j] = t[j] * acc;
}

}  // namespace

cudaError_t launch_bitflip_gates(const float *theta, int64_t m, int64_t mpad, double *c, double *t, cudaStream_t st) {
    int blocks = (int)cdiv(mpad, 256);
    if (blocks > 4096) blocks = 4096;
    LaunchScope ls(IQP_KERNEL_BITFLIP, st);
    launch_pdl(k_bitflip_gates, blocks, 256, 0, st, theta, m, mpad, c, t);
    return cudaGetLastError();
}

cudaError_t launch_bitflip_rows(const uint64_t *PA, int64_t ldp, int64_t l, const double *c, double *expval,
                                cudaStream_t st) {
    LaunchScope ls(IQP_KERNEL_BITFLIP, st);
    launch_pdl(k_bitflip_rows, (unsigned)cdiv(l, 8), 256, 0, st, PA, ldp, l, c, expval, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_bitflip_grad(const uint64_t *PAT, int64_t ldlt, int64_t m, int64_t l, const double *w,
                                const double *ev, double *v, const double *t, double *grad, cudaStream_t st) {
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bitflip_weights, (unsigned)cdiv(l, 256), 256, 0, st, w, ev, l, v);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    LaunchScope ls(IQP_KERNEL_BITFLIP, st);
    launch_pdl(k_bitflip_grad, (unsigned)cdiv(m, 8), 256, 0, st, PAT, ldlt, m, l, v, t, grad, nullptr);
    return cudaGetLastError();
}

namespace {
int bf_blocks(int64_t n) {
    const int64_t b = cdiv(n, 256);
    return (int)(b > kBfBlocks ? kBfBlocks : b);
}
cudaError_t launch_sums(const uint64_t *bits, int64_t rows, int64_t ld, const unsigned long long *q,
                        unsigned long long *sums, const int *grid, cudaStream_t st) {
    static DeviceOnce once;
    const cudaError_t e = allow_smem(once, k_bf_sums, kBfSmem);
    if (e != cudaSuccess) return e;
    const int64_t ny = cdiv(ld, (int64_t)(kBfCols / 64));
    LaunchScope ls(IQP_KERNEL_BITFLIP, st);
    launch_pdl(k_bf_sums, dim3((unsigned)cdiv(rows, (int64_t)kBfThreads), (unsigned)ny), kBfThreads, kBfSmem, st, bits, rows, ld, q,
                                                                                                          sums, grid);
    return cudaGetLastError();
}
}  // namespace

// Whether the integer sums take a problem: enough parity bits that their extra
// launches (about 15 us) are won back (10^9 bits: rows 474 -> 120 us with the
// logarithms, values and gradient 1570 -> 545 us), and column blocks within a grid.
bool bitflip_ints(int64_t m, int64_t l) {
    return (double)m * (double)l >= 33554432.0 && cdiv(m, (int64_t)kBfCols) < 65536 && cdiv(l, (int64_t)kBfCols) < 65536;
}

// Scratch of the integer path in 8-byte words: logarithms or values as numbers
// and integers, the sums, block sums and two grids.
int64_t bitflip_int_words(int64_t m, int64_t l) {
    const int64_t mx = round_up(m, 256) > round_up(l, 256) ? round_up(m, 256) : round_up(l, 256);
    return 3 * mx + 2 * kBfBlocks + 2;
}

// expval (l) and, with w, grad (m). c, t: mpad doubles; v: l doubles; s: the scratch.
cudaError_t launch_bitflip_ints(const uint64_t *PA, int64_t ldp, const uint64_t *PAT, int64_t ldlt, int64_t m, int64_t l,
                                const float *theta, double *c, double *t, int64_t mpad, double *expval, const double *w,
                                double *v, double *grad, double *s, cudaStream_t st) {
    const int64_t mx = mpad > round_up(l, 256) ? mpad : round_up(l, 256);
    double *x = s, *bsum = s + 3 * mx, *bsum2 = bsum + kBfBlocks;
    unsigned long long *q = reinterpret_cast<unsigned long long *>(s + mx), *sums = q + mx;
    int *grid = reinterpret_cast<int *>(bsum2 + kBfBlocks), *grid2 = grid + 2;
    unsigned *counter = reinterpret_cast<unsigned *>(grid + 1);
    const int nb = bf_blocks(mpad), nl = bf_blocks(l);
    cudaError_t e;
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bf_logs, nb, 256, 0, st, theta, m, mpad, c, t, x, bsum);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bf_log_ints, nb > nl ? nb : nl, 256, 0, st, x, mpad, bsum, nb, q, sums, l, grid);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = launch_sums(PA, l, ldp, q, sums, grid, st)) != cudaSuccess) return e;
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bitflip_rows, (unsigned)cdiv(l, 8), 256, 0, st, PA, ldp, l, c, expval, grid);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bf_rows_out, nl, 256, 0, st, sums, l, grid, expval, w, v, bsum2);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (w == nullptr) return cudaSuccess;
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bf_value_ints, nb > nl ? nb : nl, 256, 0, st, v, l, 64 * ldlt, bsum2, nl, q, sums, m, grid2, counter);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = launch_sums(PAT, m, ldlt, q, sums, grid2, st)) != cudaSuccess) return e;
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bf_grad_out, nb, 256, 0, st, sums, m, l, grid2, t, grad, bsum, bsum2, counter);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    LaunchScope ls(IQP_KERNEL_BITFLIP, st);
    launch_pdl(k_bitflip_grad, (unsigned)cdiv(m, 8), 256, 0, st, PAT, ldlt, m, l, v, t, grad, grid2);
    return cudaGetLastError();
}

}  // namespace iqp
