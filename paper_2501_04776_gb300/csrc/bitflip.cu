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
// the product's sign; the value is 2^-(sum). Up to a sum of 512 over all gates the
// grid's error is below the FP64 product's own rounding (2^-53 per factor); past
// it, or where a cosine is zero or not finite, the rows are multiplied instead (a flag
// on the device decides).
// The gradient's w_a <Z_a> are integers on a grid chosen the same way from sum
// |w_a <Z_a>|, and the rest of each a second integer on a grid 2^20 times finer.
// A gate whose sum is too small for the grid's error, at most half a step per
// observable, to stay below 2^-53 of it (less than the FP64 sum's own rounding) is
// summed in FP64: a gate that only meets values 10^-5 of the whole, say (10^4
// observables). Where few values are above that, most gates would be, and all are
// summed in FP64 at once. The integer sums are exact and do not depend on their order.
// Four columns at a time: their 16 partial sums are one table in shared memory
// (128 bytes, each entry in its own pair of banks, so lanes that read different
// entries never collide), a lane takes a row and adds one entry per four bits of
// its words: 5 instructions per four columns whatever bits are set, against about
// 8 and an FP64 operation per set bit. 10^9 bits take 89 us (FP64: 474),
// the gradient's two integers 127 (FP64: 387): bound by the shared-memory reads, 8 bytes
// (12) per four columns and lane.
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
constexpr unsigned kBfMany = 256;              // values (or half of them all) above the bound from which the gradient takes integers
constexpr int kBfLow = 20;                     // bits of the gradient's second integers
// Shared memory of the tables; a second integer is at most 2^19 and a CTA's sum of them below 2^31.
constexpr int bf_smem(bool low) { return kBfCols / 4 * 16 * (low ? 12 : 8); }
static_assert(kBfCols <= 2048 && kBfLow == 20, "sums of the second integers in 32 bits");
constexpr int kBfBlocks = 304, kBfRowBlocks = 2432;  // most blocks of the gates' pass and of the rows', one FP64 sum each
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

// c_j = cos(2 theta_j), t_j = -2 tan(2 theta_j) and sin(2 theta_j). bsum[b] = the block's sum of -log2 |c_j|, from above:
// in FP32, for the grid and the decision alone (10^5 gates' FP64 logarithms took 25 to 45 us, for nothing where the
// products run).
__global__ void __launch_bounds__(256) k_bf_gates(const float *__restrict__ theta, int64_t m, int64_t mpad,
                                                  double *__restrict__ c, double *__restrict__ t, double *__restrict__ sn,
                                                  double *__restrict__ bsum) {
    pdl_sync();
    float sum = 0.f;
    for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < mpad; j += (int64_t)gridDim.x * 256) {
        double cs = 1.0, si = 0.0, tn = 0.0;
        if (j < m) {
            sincos(2.0 * (double)theta[j], &si, &cs);
            tn = -2.0 * si / cs;
            const float fs = (float)si, fc = fabsf((float)cs);
            sum += fc > 0.5f ? -0.72142f * log1pf(-fs * fs) : -1.0001f * log2f(fc);
        }
        c[j] = cs;
        t[j] = tn;
        sn[j] = si;
    }
    const double acc = block_sum_f64((double)sum);  // not finite where a cosine is zero or theta is not finite
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

// Integers of the logarithms, the cosine's sign in bit 63 (q: mpad words); the sums start at zero; *grid = F (or -1),
// *many = 0.
__global__ void __launch_bounds__(256) k_bf_log_ints(const double *__restrict__ c, const double *__restrict__ sn,
                                                     int64_t mpad,
                                                     const double *__restrict__ bsum, int nb,
                                                     unsigned long long *__restrict__ q,
                                                     unsigned long long *__restrict__ sums, int64_t l,
                                                     int *__restrict__ grid, unsigned *__restrict__ many) {
    pdl_sync();
    const int F = bf_grid(bsum, nb, kBfMaxLog);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *grid = F;
        *many = 0u;
    }
    if (F < 0) return;
    const double sc = ldexp(1.0, F);
    for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < mpad; j += (int64_t)gridDim.x * 256) {
        // log2 |cos| = log1p(-sin^2) / (2 ln 2), exact to the last bits where the cosine is near 1
        const double cs = c[j], lg = fabs(cs) > 0.5 ? -0.72134752044448170368 * log1p(-sn[j] * sn[j]) : -log2(fabs(cs));
        q[j] = (unsigned long long)llrint(lg * sc) | (cs < 0.0 ? 1ull << 63 : 0ull);
    }
    for (int64_t a = blockIdx.x * (int64_t)256 + threadIdx.x; a < l; a += (int64_t)gridDim.x * 256) sums[a] = 0ull;
}

// Integers of v (l values, zero up to lpad): q 2^-F + low 2^-(F+20); the gates' sums start at zero; *grid = F (negative:
// a value is not finite, or too large); *many += the values that make the sum of a gate by themselves (twice k_bf_grad_out's
// bound).
__global__ void __launch_bounds__(256) k_bf_value_ints(const double *__restrict__ v, int64_t l, int64_t lpad,
                                                       const double *__restrict__ bsum, int nb,
                                                       unsigned long long *__restrict__ q, int *__restrict__ low,
                                                       unsigned long long *__restrict__ sums,
                                                       unsigned long long *__restrict__ lows, int64_t m,
                                                       int *__restrict__ grid, unsigned *__restrict__ many) {
    pdl_sync();
    const int F = bf_grid(bsum, nb, 1.7e308);
    unsigned above = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) *grid = F;
    if (F < 0) return;
    for (int64_t a = blockIdx.x * (int64_t)256 + threadIdx.x; a < lpad; a += (int64_t)gridDim.x * 256) {
        const double x = a < l ? ldexp(v[a], F) : 0.0;
        const long long h = __double2ll_rn(x);
        q[a] = (unsigned long long)h;
        low[a] = __double2int_rn((x - (double)h) * (double)(1 << kBfLow));  // the difference is exact, at most 1/2
        above += fabs(x) >= (double)l * 0x1.0p33 ? 1u : 0u;
    }
    above = __reduce_add_sync(0xFFFFFFFFu, above);
    if ((threadIdx.x & 31) == 0 && above != 0u) atomicAdd(many, above);
    for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < m; j += (int64_t)gridDim.x * 256) sums[j] = lows[j] = 0ull;
}

// sums[row] += sum (mod 2^64) of q[col] over the set bits of the row's columns [2048 y, + 2048): bits is rows x ld
// words, ld a multiple of 4, q padded with zeros to 64 ld; LOW: likewise lows[row] of low[col]. Block (x, y): rows
// 512 x.., a row per thread.
template <bool LOW>
__global__ void __launch_bounds__(kBfThreads) k_bf_sums(const uint64_t *__restrict__ bits, int64_t rows, int64_t ld,
                                                        const unsigned long long *__restrict__ q,
                                                        unsigned long long *__restrict__ sums,
                                                        const int *__restrict__ low,
                                                        unsigned long long *__restrict__ lows,
                                                        const int *__restrict__ grid, const unsigned *__restrict__ many,
                                                        unsigned least) {
    pdl_sync();
    extern __shared__ unsigned long long tab[];
    [[maybe_unused]] int *ltab = reinterpret_cast<int *>(tab + kBfCols / 4 * 16);
    if (*grid < 0 || (LOW && *many < least)) return;
    const int64_t w0 = blockIdx.y * (int64_t)(kBfCols / 64);
    const int words = (int)(ld - w0 < kBfCols / 64 ? ld - w0 : kBfCols / 64);
    // Table T (columns 4 T..): entry e at 16 T + (e ^ (T & 15)), so that the threads' stores of one entry spread over the banks.
    for (int T = threadIdx.x; T < words * 16; T += kBfThreads) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(q + w0 * 64 + 4 * T);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(q + w0 * 64 + 4 * T + 2);
        const unsigned long long lo[4] = {0ull, a.x, a.y, a.x + a.y}, hi[4] = {0ull, b.x, b.y, b.x + b.y};
#pragma unroll
        for (int e = 0; e < 16; ++e) tab[16 * T + (e ^ (T & 15))] = lo[e & 3] + hi[e >> 2];
        if constexpr (LOW) {
            const int4 v = *reinterpret_cast<const int4 *>(low + w0 * 64 + 4 * T);
            const int l2[4] = {0, v.x, v.y, v.x + v.y}, h2[4] = {0, v.z, v.w, v.z + v.w};
#pragma unroll
            for (int e = 0; e < 16; ++e) ltab[16 * T + (e ^ (T & 15))] = l2[e & 3] + h2[e >> 2];
        }
    }
    __syncthreads();
    const int64_t row = blockIdx.x * (int64_t)kBfThreads + threadIdx.x;
    if (row >= rows) return;
    const uint64_t *r = bits + row * ld + w0;
    unsigned long long s0 = 0ull, s1 = 0ull;
    int t0 = 0;
    for (int w = 0; w < words; w += 2) {  // words is a multiple of 4
        const ulonglong2 v = IQP_IN(row * ld + w0 + w + 1, rows * ld, 92) ? *reinterpret_cast<const ulonglong2 *>(r + w)
                                                                          : make_ulonglong2(0ull, 0ull);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t x = h ? v.y : v.x;
            const unsigned long long *t = tab + 256 * (w + h);
            const int *u = ltab + 256 * (w + h);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const int e0 = 16 * k + ((int)((x >> (4 * k)) & 15u) ^ k);
                const int e1 = 16 * (k + 1) + ((int)((x >> (4 * k + 4)) & 15u) ^ (k + 1));
                s0 += t[e0];
                s1 += t[e1];
                if constexpr (LOW) t0 += u[e0] + u[e1];
            }
        }
    }
    const unsigned long long s = s0 + s1;
    if (s != 0ull) atomicAdd(sums + row, s);
    if (LOW && t0 != 0) atomicAdd(lows + row, (unsigned long long)(long long)t0);
}

// Product of c_j over the set bits j of a row of P_A (word `first` and every `step`-th from there), and sum of v_a over
// those of a row of P_A^T, by one warp (lane-strided, then a shuffle tree); every lane gets it.
__device__ __forceinline__ double row_product(const uint64_t *__restrict__ row, int64_t ldp, const double *__restrict__ c,
                                              int64_t first, int step) {
    double prod = 1.0;
    for (int64_t w = first; w < ldp; w += step) {
        uint64_t bits = row[w];
        while (bits) {
            const int b = __ffsll((long long)bits) - 1;
            bits &= bits - 1ull;
            if (IQP_IN(w * 64 + b, ldp * 64, 90)) prod *= c[w * 64 + b];
        }
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) prod *= __shfl_xor_sync(0xFFFFFFFFu, prod, off);
    return prod;
}
__device__ __forceinline__ double row_sum(const uint64_t *__restrict__ row, int64_t ldlt, [[maybe_unused]] int64_t l,
                                          const double *__restrict__ v, int lane) {
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
    return acc;
}

// expval[a] = +-2^-(sum / 2^F), a row per thread, or, where the integers are not in use (grid -1), the FP64 product: a row
// per warp, or per block where there are no more rows than blocks (500 rows of 10^5 bits and their gradient: 560 -> 380 us,
// 530 by the kernels of the small problems). With w also v[a] = w[a] expval[a] and the block sums of |v|.
__global__ void __launch_bounds__(256) k_bf_rows_out(const unsigned long long *__restrict__ sums, int64_t l,
                                                     const int *__restrict__ grid, const uint64_t *__restrict__ PA,
                                                     int64_t ldp, const double *__restrict__ c,
                                                     double *__restrict__ expval, const double *__restrict__ w,
                                                     double *__restrict__ v, double *__restrict__ bsum) {
    pdl_sync();
    const int F = *grid;
    double acc = 0.0;
    auto put = [&](int64_t a, double e) {
        expval[a] = e;
        if (w != nullptr) {
            const double x = w[a] * e;
            v[a] = x;
            acc += fabs(x);
        }
    };
    if (F < 0) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (l <= gridDim.x) {
            __shared__ double part[8];
            const int64_t a = blockIdx.x;
            const double e = row_product(PA + a * ldp, ldp, c, threadIdx.x, 256);
            if (lane == 0) part[warp] = e;
            __syncthreads();
            if (threadIdx.x == 0)
                put(a, ((part[0] * part[1]) * (part[2] * part[3])) * ((part[4] * part[5]) * (part[6] * part[7])));
        } else {
            for (int64_t a = (int64_t)blockIdx.x * 8 + warp; a < l; a += (int64_t)gridDim.x * 8) {
                const double e = row_product(PA + a * ldp, ldp, c, lane, 32);
                if (lane == 0) put(a, e);
            }
        }
    } else {
        for (int64_t a = blockIdx.x * (int64_t)256 + threadIdx.x; a < l; a += (int64_t)gridDim.x * 256) {
            // the sum's whole part and its fraction's top bits, exactly; |sum| < 2^63 of the grid
            const unsigned long long s = sums[a], mag = s & ~(1ull << 63);
            const double whole = F < 63 ? (double)(long long)(mag >> F) : 0.0;
            const unsigned long long fr = F < 63 ? mag & ((1ull << F) - 1ull) : mag;
            const double e = exp2(-ldexp((double)fr, -F)) * exp2(-whole);
            put(a, s >> 63 ? -e : e);
        }
    }
    if (w != nullptr) {
        acc = block_sum_f64(acc);
        if (threadIdx.x == 0) bsum[blockIdx.x] = acc;
    }
}

// grad[j] = t_j (sums 2^-F + lows 2^-(F+20)), 32 gates per block. The l roundings are half a step at most: a gate for which that
// is more than 2^-53 of its sum, and every gate where the integers are not in use, is summed in FP64, by one of the block's
// warps.
__global__ void __launch_bounds__(256) k_bf_grad_out(const unsigned long long *__restrict__ sums,
                                                     const unsigned long long *__restrict__ lows, int64_t m, int64_t l,
                                                     const int *__restrict__ grid, const unsigned *__restrict__ many,
                                                     unsigned least, const uint64_t *__restrict__ PAT, int64_t ldlt,
                                                     const double *__restrict__ v, const double *__restrict__ t,
                                                     double *__restrict__ grad) {
    pdl_sync();
    __shared__ unsigned marks;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * 32;
    if (warp == 0) {
        const int64_t j = j0 + lane;
        const int F = *many < least ? -1 : *grid;
        bool ok = false;
        if (j < m && F >= 0) {
            const long long h = (long long)sums[j];
            const double d = (double)h, rest = (double)(h - (long long)d);  // |h| < 2^62 + l
            const double sum = fma(d, (double)(1 << kBfLow), fma(rest, (double)(1 << kBfLow), (double)(long long)lows[j]));
            ok = fabs(sum) >= (double)l * 0x1.0p52;
            if (ok) grad[j] = t[j] * (sum * ldexp(1.0, -(F + kBfLow)));
        }
        const unsigned bits = __ballot_sync(0xFFFFFFFFu, j < m && !ok);
        if (lane == 0) marks = bits;
    }
    __syncthreads();
    unsigned todo = marks;
    for (int i = 0; todo; ++i, todo &= todo - 1u) {
        if ((i & 7) != warp) continue;
        const int64_t j = j0 + __ffs(todo) - 1;
        const double x = row_sum(PAT + j * ldlt, ldlt, l, v, lane);
        if (lane == 0) grad[j] = t[j] * x;
    }
}

// expval[a] = product of c_j over the set bits j of P_A row a. One warp per row.
__global__ void __launch_bounds__(256) k_bitflip_rows(const uint64_t *__restrict__ PA, int64_t ldp, int64_t l,
                                                       const double *__restrict__ c, double *__restrict__ expval) {
    pdl_sync();
    const int lane = threadIdx.x & 31;
    const int64_t a = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (a >= l) return;
    const double prod = row_product(PA + a * ldp, ldp, c, lane, 32);
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
__global__ void __launch_bounds__(256) k_bitflip_grad(const uint64_t *__restrict__ PAT, int64_t ldlt, int64_t m, int64_t l,
                                                       const double *__restrict__ v, const double *__restrict__ t,
                                                       double *__restrict__ grad) {
    pdl_sync();
    const int lane = threadIdx.x & 31;
    const int64_t j = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (j >= m) return;
    const double acc = row_sum(PAT + j * ldlt, ldlt, l, v, lane);
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

// The kernels that take a row per warp are not launched as dependents: their few
// blocks would come in while the SMs are full and share the few that free up first, and the FP64
// unit is one per SM (500 rows of 10^5 bits, with their gradient: 594 -> 571 us).
cudaError_t launch_bitflip_rows(const uint64_t *PA, int64_t ldp, int64_t l, const double *c, double *expval,
                                cudaStream_t st) {
    LaunchScope ls(IQP_KERNEL_BITFLIP, st);
    k_bitflip_rows<<<(unsigned)cdiv(l, 8), 256, 0, st>>>(PA, ldp, l, c, expval);
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
    k_bitflip_grad<<<(unsigned)cdiv(m, 8), 256, 0, st>>>(PAT, ldlt, m, l, v, t, grad);
    return cudaGetLastError();
}

namespace {
int bf_blocks(int64_t n) {
    const int64_t b = cdiv(n, 256);
    return (int)(b > kBfBlocks ? kBfBlocks : b);
}
// low, lows, many: null for the rows' logarithms.
template <bool LOW>
cudaError_t launch_sums(const uint64_t *bits, int64_t rows, int64_t ld, const unsigned long long *q,
                        unsigned long long *sums, const int *low, unsigned long long *lows, const int *grid,
                        const unsigned *many, unsigned least, cudaStream_t st) {
    constexpr int smem = bf_smem(LOW);
    static DeviceOnce once;
    const cudaError_t e = allow_smem(once, k_bf_sums<LOW>, smem);
    if (e != cudaSuccess) return e;
    const int64_t ny = cdiv(ld, (int64_t)(kBfCols / 64));
    LaunchScope ls(IQP_KERNEL_BITFLIP, st);
    launch_pdl(k_bf_sums<LOW>, dim3((unsigned)cdiv(rows, (int64_t)kBfThreads), (unsigned)ny), kBfThreads, smem, st, bits, rows,
               ld, q, sums, low, lows, grid, many, least);
    return cudaGetLastError();
}
}  // namespace

// Whether the integer sums take a problem: enough parity bits that their extra
// launches (about 15 us) are won back (10^9 bits: rows 474 -> 120 us with the
// logarithms, values and gradient 1573 -> 570 us, 1498 where the rows are multiplied), and
// column blocks within a grid.
bool bitflip_ints(int64_t m, int64_t l) {
    return (double)m * (double)l >= 33554432.0 && cdiv(m, (int64_t)kBfCols) < 65536 && cdiv(l, (int64_t)kBfCols) < 65536;
}

// Scratch of the integer path in 8-byte words: the sines (later
// the values' second integers), integers, two sums, block sums, two grids and a count.
int64_t bitflip_int_words(int64_t m, int64_t l) {
    const int64_t mx = round_up(m, 256) > round_up(l, 256) ? round_up(m, 256) : round_up(l, 256);
    return 4 * mx + kBfBlocks + kBfRowBlocks + 2;
}

// expval (l) and, with w, grad (m). c, t: mpad doubles; v: l doubles; s: the scratch.
cudaError_t launch_bitflip_ints(const uint64_t *PA, int64_t ldp, const uint64_t *PAT, int64_t ldlt, int64_t m, int64_t l,
                                const float *theta, double *c, double *t, int64_t mpad, double *expval, const double *w,
                                double *v, double *grad, double *s, cudaStream_t st) {
    const int64_t mx = mpad > round_up(l, 256) ? mpad : round_up(l, 256);
    double *sn = s, *bsum = s + 4 * mx, *bsum2 = bsum + kBfBlocks;
    unsigned long long *q = reinterpret_cast<unsigned long long *>(s + mx), *sums = q + mx, *lows = sums + mx;
    int *low = reinterpret_cast<int *>(s);
    int *grid = reinterpret_cast<int *>(bsum2 + kBfRowBlocks), *grid2 = grid + 1;
    unsigned *many = reinterpret_cast<unsigned *>(grid + 2);
    const int nb = bf_blocks(mpad), nl = bf_blocks(l);
    cudaError_t e;
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bf_gates, nb, 256, 0, st, theta, m, mpad, c, t, sn, bsum);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bf_log_ints, nb > nl ? nb : nl, 256, 0, st, c, sn, mpad, bsum, nb, q, sums, l, grid, many);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = launch_sums<false>(PA, l, ldp, q, sums, nullptr, nullptr, grid, nullptr, 0u, st)) != cudaSuccess) return e;
    int64_t nr = l <= kBfRowBlocks ? l : cdiv(l, (int64_t)8);
    if (nr > kBfRowBlocks) nr = kBfRowBlocks;
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        k_bf_rows_out<<<(unsigned)nr, 256, 0, st>>>(sums, l, grid, PA, ldp, c, expval, w, v, bsum2);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (w == nullptr) return cudaSuccess;
    const unsigned least = (unsigned)(l < 2 * kBfMany ? (l + 1) / 2 : kBfMany);
    {
        LaunchScope ls(IQP_KERNEL_BITFLIP, st);
        launch_pdl(k_bf_value_ints, nb > nl ? nb : nl, 256, 0, st, v, l, 64 * ldlt, bsum2, (int)nr, q, low, sums, lows, m, grid2,
                   many);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = launch_sums<true>(PAT, m, ldlt, q, sums, low, lows, grid2, many, least, st)) != cudaSuccess) return e;
    LaunchScope ls(IQP_KERNEL_BITFLIP, st);
    k_bf_grad_out<<<(unsigned)cdiv(m, 32), 256, 0, st>>>(sums, lows, m, l, grid2, many, least, PAT, ldlt, v, t, grad);
    return cudaGetLastError();
}

}  // namespace iqp
