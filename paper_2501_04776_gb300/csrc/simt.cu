// Plain FP32 form on the SIMT cores (small problems, workspaces without the
// tensor form's regions; otherwise tc.cu runs it on the tensor cores), plus the small kernels every form
// shares: theta preparation, the per-observable statistics finalisation, the
// fixed-order gradient reduction and the MMD combine.
//
// Phase contraction (eq. Emat): Phi[a][i] = sum_j c_j P_A[a][j] S_Z[i][j] with
// c_j = 2 theta_j and S_Z = 1 - 2 P_Z, as a 128x128 tile GEMM whose operands
// are expanded from parity bits into shared memory one 32-gate word at a time.
// Gradient (Sec. 2.4): Q[a][j] = sum_i W[a][i] S_Z[i][j], masked by P_A and
// summed over the observables of the tile.
#include "common.cuh"

namespace iqp {

uint32_t check_word_simt() { return take_check_word(); }

namespace {

constexpr int BM = 128, BN = 128, BK = 32, PADF = 4;

// ------------------------------------------------------------ theta split

// c_j, hi_j and lo_j of theta_prep_one for every j < mpad.
__global__ void k_theta_prep(const float *__restrict__ theta, int64_t m, int64_t mpad, float *__restrict__ c32,
                             __nv_bfloat16 *__restrict__ hi, __nv_bfloat16 *__restrict__ lo) {
    pdl_sync();
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < mpad; j += (int64_t)gridDim.x * blockDim.x)
        theta_prep_one(theta, j, m, mpad, c32, hi, lo);
}

// --------------------------------------------------------- FP32 phase GEMM

// MODE 0: per (observable, 128-sample block) partials (S = sum cos, M2 = sum
// (cos - S/n)^2) into part[a * nparts + blockIdx.x].
// MODE 1: W[a][i] = sin Phi (alpha_a + beta_a cos Phi) into W (fp32, ldw).
template <int MODE>
__global__ void __launch_bounds__(256) k_phase_simt(const uint32_t *__restrict__ PA, const uint32_t *__restrict__ PZ,
                                                     int64_t ldp32, const float *__restrict__ c, int64_t l,
                                                     int64_t s, int64_t kwords, double2 *__restrict__ part,
                                                     int64_t nparts, const double *__restrict__ alpha,
                                                     const double *__restrict__ beta, float *__restrict__ W,
                                                     int64_t ldw) {
    pdl_sync();
    __shared__ __align__(16) float As[2][BK][BM + PADF];
    __shared__ __align__(16) float Bs[2][BK][BN + PADF];
    __shared__ float cs[2][BK];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t i0 = (int64_t)blockIdx.x * BN, a0 = (int64_t)blockIdx.y * BM;

    // Row whose bits this thread expands: A rows for tid < 128, B rows above.
    const bool isA = tid < 128;
    const int er = tid & 127;
    const int64_t grow = isA ? a0 + er : i0 + er;
    const bool rvalid = isA ? grow < l : grow < s;
    const uint32_t *src = (isA ? PA : PZ) + (rvalid ? grow : 0) * ldp32;

    float acc[8][8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[r][q] = 0.f;

    const int64_t srows = isA ? l : s;  // rows of the matrix this thread reads
    uint32_t bits = rvalid && IQP_IN((src - (isA ? PA : PZ)) + 0, srows * ldp32, 21) ? src[0] : 0u;
    float cnext = tid < BK ? c[tid] : 0.f;
    for (int64_t kw = 0; kw < kwords; ++kw) {
        const int buf = (int)(kw & 1);
        if (tid < BK) cs[buf][tid] = cnext;
        __syncthreads();
        if (isA) {
#pragma unroll
            for (int k = 0; k < BK; ++k) As[buf][k][er] = ((bits >> k) & 1u) ? cs[buf][k] : 0.f;
        } else {
#pragma unroll
            for (int k = 0; k < BK; ++k) Bs[buf][k][er] = ((bits >> k) & 1u) ? -1.f : 1.f;
        }
        __syncthreads();
        if (kw + 1 < kwords) {
            bits = rvalid && IQP_IN((src - (isA ? PA : PZ)) + kw + 1, srows * ldp32, 22) ? src[kw + 1] : 0u;
            cnext = tid < BK && IQP_IN((kw + 1) * BK + tid, kwords * BK, 23) ? c[(kw + 1) * BK + tid] : 0.f;
        }
#pragma unroll 8
        for (int k = 0; k < BK; ++k) {
            const float4 a_lo = *reinterpret_cast<const float4 *>(&As[buf][k][ty * 4]);
            const float4 a_hi = *reinterpret_cast<const float4 *>(&As[buf][k][64 + ty * 4]);
            const float4 b_lo = *reinterpret_cast<const float4 *>(&Bs[buf][k][tx * 4]);
            const float4 b_hi = *reinterpret_cast<const float4 *>(&Bs[buf][k][64 + tx * 4]);
            const float av[8] = {a_lo.x, a_lo.y, a_lo.z, a_lo.w, a_hi.x, a_hi.y, a_hi.z, a_hi.w};
            const float bv[8] = {b_lo.x, b_lo.y, b_lo.z, b_lo.w, b_hi.x, b_hi.y, b_hi.z, b_hi.w};
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[r][q] = fmaf(av[r], bv[q], acc[r][q]);
        }
    }

#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int64_t a = a0 + (r < 4 ? ty * 4 + r : 64 + ty * 4 + (r - 4));
        if (MODE == 0) {
            float cv[8], sum = 0.f;
            bool ok[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int64_t i = i0 + (q < 4 ? tx * 4 + q : 64 + tx * 4 + (q - 4));
                ok[q] = i < s;
                cv[q] = ok[q] ? cosf(acc[r][q]) : 0.f;
                sum += cv[q];
            }
#pragma unroll
            for (int off = 8; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
            const int64_t ncol = (s - i0) < BN ? (s - i0) : BN;
            const float mean = sum / (float)ncol;
            float m2 = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float d = cv[q] - mean;
                m2 += ok[q] ? d * d : 0.f;
            }
#pragma unroll
            for (int off = 8; off >= 1; off >>= 1) m2 += __shfl_xor_sync(0xFFFFFFFFu, m2, off);
            if (tx == 0 && a < l && IQP_IN(a * nparts + blockIdx.x, l * nparts, 24))
                part[a * nparts + blockIdx.x] = make_double2((double)sum, (double)m2);
        } else {
            if (a < l) {
                const float al = (float)alpha[a];
                const float be = beta ? (float)beta[a] : 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int64_t i = i0 + (q < 4 ? tx * 4 + q : 64 + tx * 4 + (q - 4));
                    if (i < s && IQP_IN(a * ldw + i, l * ldw, 25)) {
                        float sn, cn;
                        sincosf(acc[r][q], &sn, &cn);
                        W[a * ldw + i] = sn * (al + be * cn);
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------- FP32 gradient

// gpart[blockIdx.y * m + j] = sum over the tile's observables a of
//   2 P_A[a][j] * sum_i W[a][i] S_Z[i][j].
__global__ void __launch_bounds__(256) k_grad_simt(const float *__restrict__ W, int64_t ldw,
                                                    const uint32_t *__restrict__ PZ, const uint32_t *__restrict__ PA,
                                                    int64_t ldp32, int64_t l, int64_t s, int64_t m,
                                                    double *__restrict__ gpart) {
    pdl_sync();
    __shared__ __align__(16) float As[BK][BM + PADF];
    __shared__ __align__(16) float Bs[BK][BN + PADF];
    __shared__ float red[16][BN];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t j0 = (int64_t)blockIdx.x * BN, a0 = (int64_t)blockIdx.y * BM;

    float acc[8][8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[r][q] = 0.f;

    // Loader roles: W row (a0 + tid % 128), columns (tid / 128) * 16 .. +16;
    // sign rows: k = tid / 8, 16 gates at (tid % 8) * 16.
    const int wr = tid & 127, wc = (tid >> 7) * 16;
    const int64_t wrow = a0 + wr;
    const int bk = tid >> 3, bg = tid & 7;

    for (int64_t ib = 0; ib < s; ib += BK) {
        // W tile, transposed into k-major.
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = ib + wc + 4 * q;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (wrow < l && IQP_IN(wrow * ldw + (i + 3 < s ? i + 3 : (i < s ? i : 0)), l * ldw, 26)) {
                if (i + 3 < s) {
                    v = *reinterpret_cast<const float4 *>(W + wrow * ldw + i);
                } else {
                    v.x = i < s ? W[wrow * ldw + i] : 0.f;
                    v.y = i + 1 < s ? W[wrow * ldw + i + 1] : 0.f;
                    v.z = i + 2 < s ? W[wrow * ldw + i + 2] : 0.f;
                }
            }
            As[wc + 4 * q + 0][wr] = v.x;
            As[wc + 4 * q + 1][wr] = v.y;
            As[wc + 4 * q + 2][wr] = v.z;
            As[wc + 4 * q + 3][wr] = v.w;
        }
        // Sign tile from P_Z bits.
        {
            const int64_t i = ib + bk;
            uint32_t b = 0u;
            if (i < s && IQP_IN(i * ldp32 + ((j0 + bg * 16) >> 5), s * ldp32, 27))
                b = (PZ[i * ldp32 + ((j0 + bg * 16) >> 5)] >> ((bg & 1) * 16)) & 0xFFFFu;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float4 v;
                v.x = ((b >> (4 * q + 0)) & 1u) ? -1.f : 1.f;
                v.y = ((b >> (4 * q + 1)) & 1u) ? -1.f : 1.f;
                v.z = ((b >> (4 * q + 2)) & 1u) ? -1.f : 1.f;
                v.w = ((b >> (4 * q + 3)) & 1u) ? -1.f : 1.f;
                *reinterpret_cast<float4 *>(&Bs[bk][bg * 16 + 4 * q]) = v;
            }
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < BK; ++k) {
            const float4 a_lo = *reinterpret_cast<const float4 *>(&As[k][ty * 4]);
            const float4 a_hi = *reinterpret_cast<const float4 *>(&As[k][64 + ty * 4]);
            const float4 b_lo = *reinterpret_cast<const float4 *>(&Bs[k][tx * 4]);
            const float4 b_hi = *reinterpret_cast<const float4 *>(&Bs[k][64 + tx * 4]);
            const float av[8] = {a_lo.x, a_lo.y, a_lo.z, a_lo.w, a_hi.x, a_hi.y, a_hi.z, a_hi.w};
            const float bv[8] = {b_lo.x, b_lo.y, b_lo.z, b_lo.w, b_hi.x, b_hi.y, b_hi.z, b_hi.w};
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[r][q] = fmaf(av[r], bv[q], acc[r][q]);
        }
        __syncthreads();
    }

    // Mask by 2 P_A[a][j], sum the thread's 8 rows per column.
    float colsum[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) colsum[q] = 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int64_t a = a0 + (r < 4 ? ty * 4 + r : 64 + ty * 4 + (r - 4));
        if (a < l && IQP_IN(a * ldp32 + ((j0 + 64 + tx * 4) >> 5), l * ldp32, 28)) {
            const uint32_t w_lo = PA[a * ldp32 + ((j0 + tx * 4) >> 5)];
            const uint32_t w_hi = PA[a * ldp32 + ((j0 + 64 + tx * 4) >> 5)];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int64_t j = j0 + (q < 4 ? tx * 4 + q : 64 + tx * 4 + (q - 4));
                const uint32_t wb = q < 4 ? w_lo : w_hi;
                if ((wb >> (j & 31)) & 1u) colsum[q] += 2.f * acc[r][q];
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) red[ty][q < 4 ? tx * 4 + q : 64 + tx * 4 + (q - 4)] = colsum[q];
    __syncthreads();
    if (tid < BN) {
        double t = 0.0;
#pragma unroll
        for (int y = 0; y < 16; ++y) t += (double)red[y][tid];
        const int64_t j = j0 + tid;
        if (j < m && IQP_IN((int64_t)blockIdx.y * m + j, (int64_t)gridDim.y * m, 29)) gpart[(int64_t)blockIdx.y * m + j] = t;
    }
}

// ------------------------------------------------------------ reductions

// Merge the (S, M2) partials of each observable in fixed order (Chan et al.):
// mean = S/s, M2 = sum_k [M2_k + n_k (S_k/n_k - mean)^2].
// Per observable a: the mean of cos Phi over the s samples and its standard
// error from the (sum, M2) partials of pw samples each (Chan's combination),
// plus the sums S1 = sum cos, S2 = sum cos^2 for the MMD loss. One warp per
// observable: lane q takes partials q, q + 32, ... (coalesced 16-byte loads)
// and a fixed xor-shuffle tree combines the lanes, so the result does not
// depend on the launch.
__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, w);
    return v;
}

// Sizes of the partials and the reciprocals the merge needs: an FP64 division or
// square root takes about a microsecond of latency on this GPU, and a warp has
// nothing else to do meanwhile, so the host divides (k_finalize, 777 x 2501: 10.4
// -> 7.2 us).
struct PartSizes {
    int64_t nparts, pw, s;
    double inv_s, inv_pw, inv_last;  // 1 / s, 1 / pw, 1 / (samples of the last partial)
};

// a / b from y = 1 / b: a quotient, and one correction by its exact remainder
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990). Exact where the quotient is a double.
__device__ __forceinline__ double div_by(double a, double b, double y) {
    const double q = a * y;
    return fma(fma(-q, b, a), y, q);
}

// S = sum cos, its mean and M2 = sum (cos - S/s)^2 of one observable's partials, on every lane of the warp.
__device__ __forceinline__ void merge_partials(const double2 *__restrict__ p, const PartSizes &z, int lane, double &S,
                                               double &mean, double &M2) {
    S = 0.0;
    for (int64_t k = lane; k < z.nparts; k += 32) S += p[k].x;
    S = warp_sum_f64(S);
    mean = div_by(S, (double)z.s, z.inv_s);
    M2 = 0.0;
    for (int64_t k = lane; k < z.nparts; k += 32) {
        const bool last = k == z.nparts - 1;
        const double2 v = p[k];
        const double nk = (double)(last ? z.s - k * z.pw : z.pw);
        const double d = div_by(v.x, nk, last ? z.inv_last : z.inv_pw) - mean;
        M2 += v.y + nk * d * d;
    }
    M2 = warp_sum_f64(M2);
}

__global__ void __launch_bounds__(256) k_finalize(const double2 *__restrict__ part, PartSizes z, int64_t l,
                                                  double *__restrict__ expval, double *__restrict__ std_err,
                                                  double *__restrict__ S1, double *__restrict__ S2) {
    pdl_sync();
    const int lane = threadIdx.x & 31;
    const int64_t a = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (a >= l) return;  // whole warps
    if (!IQP_IN(a * z.nparts + z.nparts - 1, l * z.nparts, 30)) return;
    double S, mean, M2;
    merge_partials(part + a * z.nparts, z, lane, S, mean, M2);
    if (lane != 0) return;
    if (expval) expval[a] = mean;
    if (std_err) std_err[a] = sqrt(M2) * z.inv_s;  // sqrt(M2 / s) / sqrt(s)
    if (S1) S1[a] = S;
    if (S2) S2[a] = M2 + S * mean;
}

// grad[j] = sum over observable tiles t of gpart[t * m + j], in order.
__global__ void k_grad_reduce(const double *__restrict__ gpart, int64_t ntiles, int64_t m, double *__restrict__ grad) {
    pdl_sync();
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        double t = 0.0;
        for (int64_t k = 0; k < ntiles; ++k) t += gpart[k * m + j];
        grad[j] = t;
    }
}

// MMD^2 of eq. mmd_estimate and the gradient coefficients alpha, beta.
// sqrt_loss: loss' = sqrt(max(loss, 0)) and alpha, beta scaled by 1/(2 loss')
// (chain rule; zero where loss' = 0).
__global__ void __launch_bounds__(1024) k_mmd_combine(const long long *__restrict__ T, const double *__restrict__ S1,
                                                      const double *__restrict__ S2, int64_t l, int64_t s, int64_t N,
                                                      int unbiased, int sqrt_loss, double *__restrict__ terms,
                                                      double *__restrict__ alpha, double *__restrict__ beta,
                                                      double *__restrict__ loss) {
    pdl_sync();
    __shared__ double red[1024];
    const double ds = (double)s, dN = (double)N, dl = (double)l;
    double acc = 0.0;
    for (int64_t a = threadIdx.x; a < l; a += blockDim.x) {
        const double t = (double)T[a];
        const double p = t / dN, q = S1[a] / ds;
        double term, al, be;
        if (unbiased) {
            const double up = (t * t - dN) / (dN * (dN - 1.0));
            const double uq = (S1[a] * S1[a] - S2[a]) / (ds * (ds - 1.0));
            term = up - 2.0 * p * q + uq;
            al = (2.0 * p / ds - 2.0 * S1[a] / (ds * (ds - 1.0))) / dl;
            be = 2.0 / (ds * (ds - 1.0)) / dl;
        } else {
            term = (p - q) * (p - q);
            al = 2.0 * (p - q) / ds / dl;
            be = 0.0;
        }
        if (terms) terms[a] = term;
        if (alpha) alpha[a] = al;
        if (beta) beta[a] = be;
        acc += term;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w >= 1; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const double L = red[0] / dl;
    if (!sqrt_loss) {
        if (threadIdx.x == 0) *loss = L;
        return;
    }
    const double r = L > 0.0 ? sqrt(L) : 0.0;
    const double f = L > 0.0 ? 0.5 / r : 0.0;
    for (int64_t a = threadIdx.x; a < l; a += blockDim.x) {
        if (alpha) alpha[a] *= f;
        if (beta) beta[a] *= f;
    }
    if (threadIdx.x == 0) *loss = r;
}

// The same from the statistics' partials, one warp per observable over the
// whole grid (the kernel above runs its FP64 divisions, a few hundred thousand
// operations, on one SM: 53 us for 2000 observables; with k_finalize and the
// gradient's scale 71 us, this 19). The last block to finish adds the terms up in a fixed order and,
// with `scale`, sets the fixed-point scale of the gradient's accumulators.
struct MmdConst {
    double inv_s, inv_N, inv_l, inv_ss1, inv_NN1;  // 1 / (s (s - 1)), 1 / (N (N - 1))
};
__global__ void __launch_bounds__(256) k_mmd_terms(const double2 *__restrict__ part, PartSizes z,
                                                   const long long *__restrict__ T, int64_t l, int64_t N,
                                                   int unbiased, int sqrt_loss, MmdConst k, double *__restrict__ terms,
                                                   double *__restrict__ alpha, double *__restrict__ beta,
                                                   double *__restrict__ loss, double *__restrict__ scale,
                                                   uint32_t *__restrict__ counter) {
    pdl_sync();
    const int lane = threadIdx.x & 31;
    const int64_t a = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (a < l && IQP_IN(a * z.nparts + z.nparts - 1, l * z.nparts, 30)) {  // whole warps
        double S, mean, M2;
        merge_partials(part + a * z.nparts, z, lane, S, mean, M2);
        if (lane == 0) {
            const double t = (double)T[a], dN = (double)N;
            const double p = t * k.inv_N, S2 = M2 + S * mean;
            double term, al, be = 0.0;
            if (unbiased) {
                term = (t * t - dN) * k.inv_NN1 - 2.0 * p * mean + (S * S - S2) * k.inv_ss1;
                al = (2.0 * p * k.inv_s - 2.0 * S * k.inv_ss1) * k.inv_l;
                be = 2.0 * k.inv_ss1 * k.inv_l;
            } else {
                term = (p - mean) * (p - mean);
                al = 2.0 * (p - mean) * k.inv_s * k.inv_l;
            }
            terms[a] = term;
            alpha[a] = al;
            beta[a] = be;
        }
    }
    __shared__ bool last;
    __shared__ double red[2][256];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double sum = 0.0, mag = 0.0;
    for (int64_t b = threadIdx.x; b < l; b += 256) {
        sum += __ldcg(terms + b);
        mag += fabs(__ldcg(alpha + b)) + fabs(__ldcg(beta + b));
    }
    red[0][threadIdx.x] = sum;
    red[1][threadIdx.x] = mag;
    __syncthreads();
    for (int w = 128; w >= 1; w >>= 1) {
        if ((int)threadIdx.x < w) {
            red[0][threadIdx.x] += red[0][threadIdx.x + w];
            red[1][threadIdx.x] += red[1][threadIdx.x + w];
        }
        __syncthreads();
    }
    const double L = red[0][0] * k.inv_l;
    double f = 1.0, out = L;
    if (sqrt_loss) {
        out = L > 0.0 ? sqrt(L) : 0.0;
        f = L > 0.0 ? 0.5 / out : 0.0;
        for (int64_t b = threadIdx.x; b < l; b += 256) {
            alpha[b] = __ldcg(alpha + b) * f;
            beta[b] = __ldcg(beta + b) * f;
        }
    }
    if (threadIdx.x == 0) {
        *loss = out;
        if (scale != nullptr) *scale = fixed_scale(2.0 * (double)z.s * red[1][0] * f);
    }
}

}  // namespace

cudaError_t launch_theta_prep(const float *theta, int64_t m, int64_t mpad, float *c32, __nv_bfloat16 *hi,
                              __nv_bfloat16 *lo, cudaStream_t st) {
    int blocks = (int)cdiv(mpad, 256);
    if (blocks > 4096) blocks = 4096;
    LaunchScope ls(IQP_KERNEL_THETA_SPLIT, st);
    launch_pdl(k_theta_prep, blocks, 256, 0, st, theta, m, mpad, c32, hi, lo);
    return cudaGetLastError();
}

cudaError_t launch_phase_simt(int mode, const uint64_t *PA, const uint64_t *PZ, int64_t ldp, const float *c,
                              int64_t l, int64_t s, int64_t m, double2 *part, int64_t nparts, const double *alpha,
                              const double *beta, float *W, int64_t ldw, cudaStream_t st) {
    const int64_t kwords = cdiv(m, 32);
    const int64_t gy_total = cdiv(l, BM);
    for (int64_t y0 = 0; y0 < gy_total; y0 += 65535) {
        const int64_t ny = gy_total - y0 < 65535 ? gy_total - y0 : 65535;
        const int64_t aoff = y0 * BM;
        dim3 grid((unsigned)cdiv(s, BN), (unsigned)ny);
        const uint32_t *pa = reinterpret_cast<const uint32_t *>(PA + aoff * ldp);
        LaunchScope ls(mode == 0 ? IQP_KERNEL_PHASE_FP32 : IQP_KERNEL_RECOMPUTE_FP32, st);
        if (mode == 0)
            launch_pdl(k_phase_simt<0>, grid, 256, 0, st, pa, reinterpret_cast<const uint32_t *>(PZ), 2 * ldp, c, l - aoff,
                                                  s, kwords, part + aoff * nparts, nparts, nullptr, nullptr, nullptr,
                                                  0);
        else
            launch_pdl(k_phase_simt<1>, grid, 256, 0, st, pa, reinterpret_cast<const uint32_t *>(PZ), 2 * ldp, c, l - aoff,
                                                  s, kwords, nullptr, 0, alpha + aoff, beta ? beta + aoff : nullptr,
                                                  W + aoff * ldw, ldw);
    }
    return cudaGetLastError();
}

cudaError_t launch_grad_simt(const float *W, int64_t ldw, const uint64_t *PZ, const uint64_t *PA, int64_t ldp,
                             int64_t l, int64_t s, int64_t m, double *gpart, cudaStream_t st) {
    const int64_t gy_total = cdiv(l, BM);
    for (int64_t y0 = 0; y0 < gy_total; y0 += 65535) {
        const int64_t ny = gy_total - y0 < 65535 ? gy_total - y0 : 65535;
        const int64_t aoff = y0 * BM;
        dim3 grid((unsigned)cdiv(m, BN), (unsigned)ny);
        LaunchScope ls(IQP_KERNEL_GRAD_FP32, st);
        launch_pdl(k_grad_simt, grid, 256, 0, st, W + aoff * ldw, ldw, reinterpret_cast<const uint32_t *>(PZ),
                                          reinterpret_cast<const uint32_t *>(PA + aoff * ldp), 2 * ldp, l - aoff, s,
                                          m, gpart + y0 * m);
    }
    return cudaGetLastError();
}

namespace {
PartSizes part_sizes(int64_t nparts, int64_t pw, int64_t s) {
    return PartSizes{nparts, pw, s, 1.0 / (double)s, 1.0 / (double)pw, 1.0 / (double)(s - (nparts - 1) * pw)};
}
}  // namespace

cudaError_t launch_finalize(const double2 *part, int64_t nparts, int64_t pw, int64_t l, int64_t s, double *expval,
                            double *std_err, double *S1, double *S2, cudaStream_t st) {
    LaunchScope ls(IQP_KERNEL_FINALIZE, st);
    launch_pdl(k_finalize, (unsigned)cdiv(l, 8), 256, 0, st, part, part_sizes(nparts, pw, s), l, expval, std_err, S1, S2);
    return cudaGetLastError();
}

cudaError_t launch_grad_reduce(const double *gpart, int64_t ntiles, int64_t m, double *grad, cudaStream_t st) {
    int blocks = (int)cdiv(m, 256);
    if (blocks > 8192) blocks = 8192;
    LaunchScope ls(IQP_KERNEL_GRAD_REDUCE, st);
    launch_pdl(k_grad_reduce, blocks, 256, 0, st, gpart, ntiles, m, grad);
    return cudaGetLastError();
}

cudaError_t launch_mmd_combine(const int64_t *T, const double *S1, const double *S2, int64_t l, int64_t s, int64_t N,
                               int unbiased, bool sqrt_loss, double *terms, double *alpha, double *beta, double *loss,
                               cudaStream_t st) {
    LaunchScope ls(IQP_KERNEL_MMD_COMBINE, st);
    launch_pdl(k_mmd_combine, 1, 1024, 0, st, reinterpret_cast<const long long *>(T), S1, S2, l, s, N, unbiased,
                                      sqrt_loss ? 1 : 0, terms, alpha, beta, loss);
    return cudaGetLastError();
}

// T, terms, alpha, beta: l each; scale: null or the gradient's fixed-point
// scale; counter: zero (launch_parity_sum_rows leaves it so).
cudaError_t launch_mmd_terms(const double2 *part, int64_t nparts, int64_t pw, const int64_t *T, int64_t l, int64_t s,
                             int64_t N, int unbiased, bool sqrt_loss, double *terms, double *alpha, double *beta,
                             double *loss, double *scale, uint32_t *counter, cudaStream_t st) {
    const double ds = (double)s, dN = (double)N;
    const MmdConst k{1.0 / ds, 1.0 / dN, 1.0 / (double)l, 1.0 / (ds * (ds - 1.0)), 1.0 / (dN * (dN - 1.0))};
    LaunchScope ls(IQP_KERNEL_MMD_COMBINE, st);
    launch_pdl(k_mmd_terms, (unsigned)cdiv(l, 8), 256, 0, st, part, part_sizes(nparts, pw, s),
                                                      reinterpret_cast<const long long *>(T), l, N,
                                                      unbiased, sqrt_loss ? 1 : 0, k, terms, alpha, beta, loss, scale,
                                                      counter);
    return cudaGetLastError();
}

}  // namespace iqp
