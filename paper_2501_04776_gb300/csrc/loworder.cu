// Low-order form: every generator has weight <= 2 (the one- and two-body
// gate sets of Sec. 3.1.1 and Sec. 4). With s_q(i) = (-1)^{z_{i,q}},
// Q_a = supp(a), c_j = 2 theta_j, d_q = sum of c_j over the one-qubit gates
// on q and C_qr = sum of c_j over the gates on {q, r} (symmetric, zero
// diagonal):
//   [g_j.a odd]      = [q in Q_a] for g_j = e_q, [exactly one of q, r in Q_a] for e_q + e_r,
//   1 - 2[g_j.z odd] = s_q(z), or s_q(z) s_r(z),
// so the phase of eq. expvalsample regroups exactly into
//   Phi[a,i] = sum_{q in Q_a} s_q(i) (d_q + M[q,i]) - 2 sum_{q<r in Q_a} C_qr s_q(i) s_r(i),
//   M = C S,  S[r][i] = s_r(i)        (an n x n x s contraction over the pairs with a generator),
// held as X[q,i] = s_q(i) (d_q + M[q,i]), formed in the contraction's epilogue,
// and with W[a,i] = sin Phi (alpha_a + beta_a cos Phi), V[q,i] = sum_{a : q in Q_a} W[a,i]:
//   grad(gate e_q)       = 2 sum_i s_q(i) V[q,i],
//   grad(gate e_q + e_r) = 2 (H[q,r] + H[r,q]) - 4 K[q,r],
//   H[q,r] = sum_i s_q(i) V[q,i] s_r(i)   (needed only for the pairs with a generator),
//   K[q,r] = sum_{a : q, r in Q_a} sum_i W[a,i] s_q(i) s_r(i).
// The work is O(p s + l |Q_a|^2 s), p = number of qubit pairs carrying a
// generator, instead of nnz(P_A) s, and nnz(P_A) is about l |Q_a| n for all
// one- and two-body gates. FP32 arithmetic, FP64
// reductions over samples; C, d and K accumulated in 64-bit fixed point
// (integer atomics, so repeated supports and the gradient are bitwise
// reproducible).
//
// Device-side errors: a generator of weight > 2 records IQP_ERR_ARG, an
// observable of weight > 1024 records IQP_ERR_UNSUPPORTED (in the workspace
// status word); the outputs are then not meaningful.
#include <cstdlib>

#include "common.cuh"

namespace iqp {

namespace {

constexpr int kQMax = 1024;  // observable weight limit (support list in shared memory)
constexpr int kPairMax = 512;  // pairs of Q_a held in shared memory per round
constexpr int kBlk = 256;    // samples per partial, and per block of the heavy observables' kernels
constexpr int kLane = 1024;  // samples per warp in the listed observables' kernels (32 per lane)
constexpr int kQ4 = 256;     // supports up to this size take four sample blocks per pass in k_lo_phase
constexpr unsigned kFull = 0xFFFFFFFFu;

// Optional self-checks (-DIQP_LO_CHECKS, or the library-wide -DIQP_CHECKS):
// an index out of its buffer records status 100 + site in the workspace status
// word and the access is skipped.
#if defined(IQP_CHECKS) && !defined(IQP_LO_CHECKS)
#define IQP_LO_CHECKS
#endif
#ifdef IQP_LO_CHECKS
#define LO_OK(cond, site) ((cond) ? true : (record_status(status_dbg, 100u + (site)), false))
#else
#define LO_OK(cond, site) true
#endif

// d_q, C_qr and E (bits r of row q and q of row r set iff some generator
// acts on {q, r}) from the support list (q0 < q1 < ..., count). Repeated
// supports add their coefficients: each c_j is rounded to a multiple of
// 2^-k, the sums are formed exactly in 64-bit fixed point (integer atomics,
// so their order does not matter) and each is rounded to FP32 once, which
// keeps every result bitwise reproducible.
//
// Scale 2^k of the fixed point, from the largest |c_j| (its float bits, taken
// by an integer atomicMax) and m: m max|c_j| 2^k < 2^62, so no partial sum
// overflows; k is clamped to [-60, 100].
__device__ __forceinline__ int lo_fx_exp(unsigned cmax_bits, int64_t m) {
    const float cm = __uint_as_float(cmax_bits);
    if (!(cm > 0.f) || !(cm < INFINITY)) return 40;
    int e = 0;
    frexp((double)cm * (double)(m > 0 ? m : 1), &e);  // the bound is < 2^e
    const int k = 62 - e;
    return k < -60 ? -60 : (k > 100 ? 100 : k);
}

// Cfx (n x n, upper triangle) and dfx (n): fixed-point sums of c_j = 2 theta_j;
// E bits (upper triangle, both with `full`).
__global__ void k_lo_build(const int4 *__restrict__ sup, const float *__restrict__ theta, int64_t m, int64_t n,
                           unsigned long long *__restrict__ Cfx, unsigned long long *__restrict__ dfx,
                           const unsigned *__restrict__ cmax, unsigned long long *__restrict__ E, int64_t lde, int full,
                           uint32_t *__restrict__ status) {
    pdl_sync();
    [[maybe_unused]] uint32_t *status_dbg = status;
    const float sc = ldexpf(1.0f, lo_fx_exp(*cmax, m));  // |c_j sc| < 2^62
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int4 sp = sup[j];
        if (!LO_OK(sp.w <= 0 || (sp.x >= 0 && sp.x < n && (sp.w < 2 || (sp.y > sp.x && sp.y < n))), 8)) continue;
        if (sp.w == 1 || sp.w == 2) {
            const unsigned long long v = (unsigned long long)to_fixed(2.0f * theta[j], sc);
            if (sp.w == 1) {
                atomicAdd(dfx + sp.x, v);
            } else {
                atomicAdd(Cfx + (int64_t)sp.x * n + sp.y, v);
                atomicOr(E + (int64_t)sp.x * lde + (sp.y >> 6), 1ull << (sp.y & 63));
                if (full) atomicOr(E + (int64_t)sp.y * lde + (sp.x >> 6), 1ull << (sp.x & 63));
            }
        } else if (sp.w > 2) {
            record_status(status, IQP_ERR_ARG);
        }
    }
}

// C from the upper triangle of its fixed-point sums, each rounded to FP32
// once, as the split-BF16 operand (n x kc, zero in columns >= n) and, where the
// contractions run as sums, as FP32 (n x ldc); d (n) likewise. One block per
// pair of 64 x 64 tiles (bi <= bj), which reads the upper tile once and writes
// it and its transpose.
__global__ void __launch_bounds__(256) k_lo_convert(const unsigned long long *__restrict__ Cfx,
                                                    const unsigned long long *__restrict__ dfx,
                                                    const unsigned *__restrict__ cmax, int64_t m, int64_t n, int nb,
                                                    __nv_bfloat16 *__restrict__ hi, __nv_bfloat16 *__restrict__ lo,
                                                    int64_t kc, float *__restrict__ C, int64_t ldc,
                                                    float *__restrict__ d) {
    pdl_sync();
    __shared__ float tile[64][65];
    const float inv = ldexpf(1.0f, -lo_fx_exp(*cmax, m));
    int bi = 0, left = blockIdx.x;  // block number -> (bi, bj), row by row
    while (left >= nb - bi) {
        left -= nb - bi;
        ++bi;
    }
    const int bj = bi + left;
    const int64_t q0 = 64 * (int64_t)bi, r0 = 64 * (int64_t)bj;
    for (int e = threadIdx.x; e < 64 * 64; e += 256) {
        const int64_t q = q0 + (e >> 6), r = r0 + (e & 63);
        tile[e >> 6][e & 63] = q < r && r < n ? __ll2float_rn((long long)Cfx[q * n + r]) * inv : 0.f;
    }
    if (bi == bj && threadIdx.x < 64 && q0 + threadIdx.x < n)
        d[q0 + threadIdx.x] = __ll2float_rn((long long)dfx[q0 + threadIdx.x]) * inv;
    __syncthreads();
    // side 0: rows q0.. (columns r0..); side 1: rows r0.. (columns q0..), the transpose
    for (int side = 0; side < (bi == bj ? 1 : 2); ++side) {
        const int64_t row0 = side ? r0 : q0, col0 = side ? q0 : r0;
        for (int e = threadIdx.x; e < 64 * 8; e += 256) {
            const int a = e >> 3, b = (e & 7) * 8;
            if (row0 + a >= n) continue;
            uint32_t ph[4], pl[4];
            float x[8];
#pragma unroll
            for (int t = 0; t < 8; ++t)
                x[t] = side ? tile[b + t][a] : (bi == bj && b + t < a ? tile[b + t][a] : tile[a][b + t]);
#pragma unroll
            for (int t = 0; t < 8; t += 2) {
                const __nv_bfloat16 h0 = __float2bfloat16_rn(x[t]), h1 = __float2bfloat16_rn(x[t + 1]);
                const __nv_bfloat16 l0 = __float2bfloat16_rn(x[t] - __bfloat162float(h0));
                const __nv_bfloat16 l1 = __float2bfloat16_rn(x[t + 1] - __bfloat162float(h1));
                ph[t / 2] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                pl[t / 2] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
            }
            const int64_t at = (row0 + a) * kc + col0 + b;
            *reinterpret_cast<uint4 *>(hi + at) = make_uint4(ph[0], ph[1], ph[2], ph[3]);
            *reinterpret_cast<uint4 *>(lo + at) = make_uint4(pl[0], pl[1], pl[2], pl[3]);
            if (C != nullptr)
                for (int t = 0; t < 8; ++t)
                    if (col0 + b + t < ldc) C[(row0 + a) * ldc + col0 + b + t] = x[t];
        }
    }
}

// The sample bits in lane order: word (q, 32 b + L) of ZP holds lane L's 32
// samples of the 1024-sample block b, bit 4 k + j being sample
// 1024 b + 128 k + 4 L + j (so that a lane's floats are eight coalesced 16-byte
// words). One warp per (q, b).
__global__ void __launch_bounds__(256) k_lo_zpack(const uint32_t *__restrict__ ZT, int64_t ldzt32, int64_t n, int64_t nb,
                                                  uint32_t *__restrict__ ZP) {
    pdl_sync();
    const int lane = threadIdx.x & 31;
    const int64_t total = n * nb;
    for (int64_t i = (blockIdx.x * (int64_t)256 + threadIdx.x) >> 5; i < total; i += (int64_t)gridDim.x * 8) {
        const int64_t q = i / nb, b = i - q * nb;
        const uint32_t w = 32 * b + lane < ldzt32 ? ZT[q * ldzt32 + 32 * b + lane] : 0u;
        uint32_t o = 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            o |= ((__shfl_sync(kFull, w, 4 * k + (lane >> 3)) >> (4 * (lane & 7))) & 0xFu) << (4 * k);
        ZP[(q * nb + b) * 32 + lane] = o;
    }
}

// Every observable's qubits (in increasing order) and, with C, the pairs among
// them that carry a generator, one warp per observable. One of more than qmax
// (at most kLoQ) qubits or kLoP pairs is left to the heavy observables' kernels: cnt = -1, and
// its number in `heavy` (counted in *nheavy). qmax: the listed kernels take a row of X per
// step and warp, the block kernels several at a time, so where the warps are few (at most four per SM) they take the
// observables from 65 qubits on (30 observables of 120 qubits x
// 100: 158 us before the lists, 188 listed, 129).
constexpr int kListed = 8;  // pairs per lane and round
__global__ void __launch_bounds__(256) k_lo_lists(const uint64_t *__restrict__ A, int64_t lda, int64_t l, int64_t n,
                                                  const unsigned long long *__restrict__ E, int64_t lde,
                                                  const unsigned long long *__restrict__ Cfx,
                                                  const unsigned *__restrict__ cmax, int64_t m, int qmax, int *__restrict__ Lq,
                                                  uint2 *__restrict__ Lp, int *__restrict__ cnt, int *__restrict__ heavy,
                                                  unsigned *__restrict__ nheavy, uint32_t *__restrict__ status) {
    pdl_sync();
    [[maybe_unused]] uint32_t *status_dbg = status;
    __shared__ int sq[8][kLoQ];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t a = (int64_t)blockIdx.x * 8 + warp;
    if (a >= l) return;
    const float inv = ldexpf(1.0f, -lo_fx_exp(*cmax, m));
    const int64_t nw = (n + 63) >> 6;
    int nq = 0;
    for (int64_t wb = 0; wb < nw; wb += 32) {
        uint64_t w = wb + lane < nw ? A[a * lda + wb + lane] : 0ull;
        if (wb + lane == nw - 1 && (n & 63)) w &= (1ull << (n & 63)) - 1ull;  // never a qubit >= n
        const int c = __popcll(w);
        int incl = c;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int u = __shfl_up_sync(kFull, incl, s);
            if (lane >= s) incl += u;
        }
        int p = nq + incl - c;
        while (w) {
            if (p < kLoQ) sq[warp][p] = (int)(64 * (wb + lane)) + __ffsll((long long)w) - 1;
            w &= w - 1ull;
            ++p;
        }
        nq += __shfl_sync(kFull, incl, 31);
    }
    __syncwarp();
    int np = 0;
    if (nq <= qmax) {
        for (int t = lane; t < nq; t += 32) Lq[a * kLoQ + t] = sq[warp][t];
        // the pairs t < u in order, 256 per round: the round's E words are all loaded before the first is used (with all
        // nq^2 candidates, 128 per round, 30 observables of 100 qubits waited 78 rounds, 60 us, on their four SMs)
        const int all = nq * (nq - 1) / 2;
        for (int c0 = 0; c0 < all; c0 += 32 * kListed) {
            int qr[kListed];
            bool ok[kListed];
            unsigned long long ew[kListed];
#pragma unroll
            for (int k = 0; k < kListed; ++k) {
                const int e = c0 + 32 * k + lane;
                ok[k] = e < all;
                // row t holds pairs t (2 nq - t - 1) / 2 ..: the root's rounding is put right by the two steps below
                const float h = (float)(2 * nq - 1);
                int t = ok[k] ? (int)(0.5f * (h - sqrtf(h * h - 8.f * (float)e))) : 0;
                t -= t * (2 * nq - t - 1) / 2 > e ? 1 : 0;
                t += (t + 1) * (2 * nq - t - 2) / 2 <= e ? 1 : 0;
                const int u = ok[k] ? t + 1 + e - t * (2 * nq - t - 1) / 2 : 0;
                const int q = ok[k] ? sq[warp][t] : 0, r = ok[k] ? sq[warp][u] : 0;
                ok[k] = ok[k] && LO_OK(q >= 0 && q < r && r < n, 10);
                qr[k] = q | (r << 16);
                ew[k] = ok[k] ? E[(int64_t)q * lde + (r >> 6)] : 0ull;
            }
#pragma unroll
            for (int k = 0; k < kListed; ++k) {
                const int q = qr[k] & 0xFFFF, r = (int)((unsigned)qr[k] >> 16);
                const bool has = ok[k] && ((ew[k] >> (r & 63)) & 1ull) != 0ull;
                const uint32_t bal = __ballot_sync(kFull, has);
                const int pos = np + __popc(bal & ((1u << lane) - 1u));
                if (has && pos < kLoP) {
                    const float cv = __ll2float_rn((long long)Cfx[(int64_t)q * n + r]) * inv;
                    Lp[a * kLoP + pos] = make_uint2((uint32_t)qr[k], __float_as_uint(-2.0f * cv));
                }
                np += __popc(bal);
            }
        }
    }
    if (lane != 0) return;
    const bool listed = nq <= qmax && np <= kLoP;
    cnt[a] = listed ? nq | (np << 16) : -1;
    if (!listed) {
        const unsigned h = atomicAdd(nheavy, 1u);
        if (h < l) heavy[h] = (int)a;
    }
}

// ------------------------------------------------ pair contractions
// Both n x n x s contractions visit only the pairs that carry a generator
// (the set bits of E): one warp per (qubit q, range of 2048 samples), lane
// l owning the 64 samples of word 32 range + l of every ZT row, each term a
// sign flip and an FP32 add (as in the row-sparse form).

constexpr int kCsBatch = 8;

// fn(r) for every set bit r of E row q, in increasing r, warp-uniformly.
template <class F>
__device__ __forceinline__ void for_each_bit(const unsigned long long *__restrict__ row, int64_t nw, int lane, F &fn) {
    for (int64_t w0 = 0; w0 < nw; w0 += 32) {
        const uint64_t bits = w0 + lane < nw ? row[w0 + lane] : 0ull;
        uint32_t live = __ballot_sync(kFull, bits != 0ull);
        while (live) {
            const int src = __ffs(live) - 1;
            live &= live - 1u;
            uint64_t wb = __shfl_sync(kFull, bits, src);
            const int64_t rb = (w0 + src) * 64;
            while (wb) {
                const int b = __ffsll((long long)wb) - 1;
                wb &= wb - 1ull;
                fn(rb + b);
            }
        }
    }
}

// X[q][i] = s_q(i) (d_q + sum_{r in E_q} C_qr s_r(i)) (C S restricted to the
// pairs with a generator, which is all of C's nonzeros). Grid (n, ranges) x 32 threads.
__global__ void __launch_bounds__(32) k_lo_cs(const unsigned long long *__restrict__ E, int64_t lde,
                                              const float *__restrict__ C, int64_t ldc,
                                              const float *__restrict__ d, const uint64_t *__restrict__ ZT,
                                              int64_t ldzt, int64_t s, float *__restrict__ M, int64_t lds) {
    pdl_sync();
    const int lane = threadIdx.x;
    const int64_t q = blockIdx.x, r0 = blockIdx.y;
    const int64_t vwords = cdiv(s, 64);
    const int64_t wraw = r0 * 32 + lane;
    const int64_t word = wraw < vwords ? wraw : vwords - 1;  // in-bounds load, result unused
    float acc[64];
#pragma unroll
    for (int k = 0; k < 64; ++k) acc[k] = 0.f;
    const float *crow = C + q * ldc;
    auto add = [&](uint64_t z, uint32_t cb) {
        const uint32_t lo = (uint32_t)z, hi = (uint32_t)(z >> 32);
#pragma unroll
        for (int k = 0; k < 32; ++k) acc[k] += __uint_as_float(cb ^ ((lo << (31 - k)) & 0x80000000u));
#pragma unroll
        for (int k = 0; k < 32; ++k) acc[32 + k] += __uint_as_float(cb ^ ((hi << (31 - k)) & 0x80000000u));
    };
    // Pairs are consumed in batches of kCsBatch: the batch's loads are all
    // issued before the first is used (only indices are held while a batch
    // fills), so their latencies overlap.
    int64_t rb[kCsBatch];
    int nb = 0;
#pragma unroll
    for (int t = 0; t < kCsBatch; ++t) rb[t] = 0;
    auto visit = [&](int64_t r) {
#pragma unroll
        for (int t = 0; t + 1 < kCsBatch; ++t) rb[t] = rb[t + 1];
        rb[kCsBatch - 1] = r;
        if (++nb == kCsBatch) {
            uint64_t z[kCsBatch];
            uint32_t cb[kCsBatch];
#pragma unroll
            for (int t = 0; t < kCsBatch; ++t) {
                z[t] = __ldg(ZT + rb[t] * ldzt + word);
                cb[t] = __float_as_uint(__ldg(crow + rb[t]));
            }
#pragma unroll
            for (int t = 0; t < kCsBatch; ++t) add(z[t], cb[t]);
            nb = 0;
        }
    };
    for_each_bit(E + q * lde, lde, lane, visit);
#pragma unroll
    for (int t = 0; t < kCsBatch; ++t)
        if (t >= kCsBatch - nb) add(__ldg(ZT + rb[t] * ldzt + word), __float_as_uint(__ldg(crow + rb[t])));
    if (wraw < vwords) {
        float *mrow = M + q * lds + wraw * 64;  // lds is a multiple of 64
        const uint64_t zq = __ldg(ZT + q * ldzt + word);
        const float dq = d[q];
#pragma unroll
        for (int k = 0; k < 64; ++k) acc[k] = ((zq >> k) & 1ull) ? -(dq + acc[k]) : dq + acc[k];
#pragma unroll
        for (int k = 0; k < 64; k += 4) *reinterpret_cast<float4 *>(mrow + k) = make_float4(acc[k], acc[k + 1], acc[k + 2], acc[k + 3]);
    }
}

// H[q][r] = sum_i s_q(i) V[q][i] s_r(i) for r in E_q. Warp (q, k) takes
// every kHSplit-th set bit of E_q starting at the k-th (listed in shared
// memory, kRMax at a time) and walks the sample ranges in order, so each
// H[q][r] is accumulated by one warp alone (fixed order, FP32 per range, FP64
// across ranges).
constexpr int kHSplit = 8;
constexpr int kRMax = 1024;
constexpr int kHPre = 4;

__global__ void __launch_bounds__(32) k_lo_h(const unsigned long long *__restrict__ E, int64_t lde,
                                             const uint64_t *__restrict__ ZT, int64_t ldzt,
                                             const float *__restrict__ V, int64_t lds, int64_t s,
                                             double *__restrict__ Hd, int64_t ldh) {
    pdl_sync();
    __shared__ int rl[kRMax];
    const int lane = threadIdx.x;
    const int64_t q = blockIdx.x;
    const int split = blockIdx.y;
    const int64_t vwords = cdiv(s, 64);
    const int64_t nranges = cdiv(vwords, 32);
    double *hrow = Hd + q * ldh;
    const unsigned long long *erow = E + q * lde;
    int seen = 0;        // set bits of E_q visited so far
    int64_t w0 = 0;      // next E word to scan
    while (w0 < lde) {
        // list this warp's next pairs
        int nr = 0;
        while (w0 < lde && nr <= kRMax - 64) {
            const uint64_t bits0 = erow[w0];
            uint64_t bits = bits0;
            // bit b of the word is this warp's when (seen + rank of b) % kHSplit == split
            const int rank_start = seen;
            const int cnt = __popcll(bits0);
            if (lane == 0) {
                int rk = rank_start;
                while (bits) {
                    const int b = __ffsll((long long)bits) - 1;
                    bits &= bits - 1ull;
                    if (rk % kHSplit == split) rl[nr++] = (int)(64 * w0 + b);
                    ++rk;
                }
            }
            nr = __shfl_sync(kFull, nr, 0);
            seen += cnt;
            ++w0;
        }
        __syncwarp();
        for (int64_t r0 = 0; r0 < nranges; ++r0) {
            const int64_t wraw = r0 * 32 + lane;
            const bool wvalid = wraw < vwords;
            const int64_t word = wvalid ? wraw : vwords - 1;
            float u[64];
            const uint64_t zq = __ldg(ZT + q * ldzt + word);
            const float *vrow = V + q * lds + word * 64;
#pragma unroll
            for (int k = 0; k < 64; k += 4) {
                const float4 v4 = wvalid ? *reinterpret_cast<const float4 *>(vrow + k) : make_float4(0.f, 0.f, 0.f, 0.f);
                u[k] = v4.x;
                u[k + 1] = v4.y;
                u[k + 2] = v4.z;
                u[k + 3] = v4.w;
            }
#pragma unroll
            for (int k = 0; k < 64; ++k) u[k] = ((zq >> k) & 1ull) ? -u[k] : u[k];
            // loads of the next kHPre pairs are issued ahead of their use
            uint64_t zn[kHPre];
#pragma unroll
            for (int t = 0; t < kHPre; ++t) zn[t] = t < nr ? __ldg(ZT + (int64_t)rl[t] * ldzt + word) : 0ull;
            for (int e0 = 0; e0 < nr; e0 += kHPre) {
                uint64_t zc[kHPre];
#pragma unroll
                for (int t = 0; t < kHPre; ++t) {
                    zc[t] = zn[t];
                    const int en = e0 + kHPre + t;
                    zn[t] = en < nr ? __ldg(ZT + (int64_t)rl[en] * ldzt + word) : 0ull;
                }
#pragma unroll
                for (int t = 0; t < kHPre; ++t) {
                const int e = e0 + t;
                if (e >= nr) break;
                const int64_t r = rl[e];
                const uint64_t z = zc[t];
                const uint32_t lo = (uint32_t)z, hi = (uint32_t)(z >> 32);
                float p[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int k = 0; k < 32; ++k)
                    p[k & 7] += __uint_as_float(__float_as_uint(u[k]) ^ ((lo << (31 - k)) & 0x80000000u));
#pragma unroll
                for (int k = 0; k < 32; ++k)
                    p[k & 7] += __uint_as_float(__float_as_uint(u[32 + k]) ^ ((hi << (31 - k)) & 0x80000000u));
                float dsum = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) dsum += __shfl_xor_sync(kFull, dsum, off);
                if (lane == 0) hrow[r] = r0 == 0 ? (double)dsum : hrow[r] + (double)dsum;
                }
            }
        }
        __syncwarp();
    }
}

// With the tensor cores both contractions are dense GEMMs with one +-1
// operand from bits, M = C S (K = the n qubits r) and H = (s o V) S^T
// (K = the s samples), like the phase contraction; the FP32 operand goes in
// as a hi + lo BF16 split, written by k_lo_convert and k_lo_v.

// Exclusive prefix sum of v over the CTA (every thread calls it); *total
// receives the sum.
__device__ int block_scan(int v, int *scan, int *total) {
    const int tid = threadIdx.x;
    scan[tid] = v;
    __syncthreads();
    for (int off = 1; off < (int)blockDim.x; off <<= 1) {  // inclusive (Hillis-Steele)
        const int u = tid >= off ? scan[tid - off] : 0;
        __syncthreads();
        scan[tid] += u;
        __syncthreads();
    }
    const int incl = scan[tid];
    *total = scan[blockDim.x - 1];
    __syncthreads();
    return incl - v;
}

// The support of observable a in increasing qubit order into Q (shared);
// returns |Q_a| capped at kQMax (recording IQP_ERR_UNSUPPORTED beyond it).
// Every thread of the CTA calls it.
__device__ int support_of_row(const uint64_t *__restrict__ arow, int64_t n, int *Q, int *scan,
                              uint32_t *__restrict__ status) {
    [[maybe_unused]] uint32_t *status_dbg = status;
    const int tid = threadIdx.x;
    const int64_t nw = (n + 63) >> 6;
    int total = 0;
    for (int64_t base = 0; base < nw; base += blockDim.x) {
        uint64_t w = base + tid < nw ? arow[base + tid] : 0ull;
        if (base + tid == nw - 1 && (n & 63)) w &= (1ull << (n & 63)) - 1ull;  // never a qubit >= n
        int sum = 0;
        int pos = total + block_scan(__popcll(w), scan, &sum);
        while (w) {
            const int b = __ffsll((long long)w) - 1;
            w &= w - 1ull;
            if (pos < kQMax && LO_OK(64 * (base + tid) + b < n, 1)) Q[pos] = (int)(64 * (base + tid) + b);
            ++pos;
        }
        total += sum;
    }
    __syncthreads();  // Q is complete before anyone reads it
    if (total > kQMax) {
        if (tid == 0) record_status(status, IQP_ERR_UNSUPPORTED);
        total = kQMax;
    }
    return total;
}

// Shared state of the per-(observable, 256-sample block) kernels.
struct LoShared {
    int Q[kQMax];              // support of the observable
    union alignas(16) {
        uint32_t bits[kQMax][8];    // one 256-sample block: bit (i - i0) of word i/32 for qubit Q[t]
        uint32_t bits4[kQ4][32];    // four blocks at once, for supports of at most kQ4 qubits
    };
    int pr[kPairMax];          // pairs t | u << 16 (t < u) with a generator on {Q[t], Q[u]}
    float pc[kPairMax];        // C restricted to those pairs
    int scan[kBlk];
    int wsum[kBlk / 32];
    float redf[kBlk / 32];
};

// Sample blocks handled by one CTA: the support and, when it fits, the
// pair list are built once and reused for every block.
constexpr int kGroup = 8;    // sample blocks per CTA of k_lo_v (its per-block sums live in registers)
constexpr int kPGroup = 16;  // sample blocks per CTA of k_lo_phase and k_lo_pairs (support and pair list built once)
constexpr int kObsMax = 4096;  // observables of one qubit listed per pass in k_lo_v

// The sample bits of block blk for every support qubit.
__device__ void lo_load_bits(LoShared &sh, int nq, int64_t n, const uint64_t *__restrict__ ZT, int64_t ldzt,
                             int64_t blk, [[maybe_unused]] uint32_t *__restrict__ status_dbg) {
    __syncthreads();  // previous readers of bits are done
    for (int e = threadIdx.x; e < nq * 4; e += kBlk) {
        const int t = e >> 2, k = e & 3;
        const int64_t w = blk * 4 + k;
        const bool okq = LO_OK(t < kQMax && sh.Q[t] >= 0 && sh.Q[t] < n, 2);
        const uint64_t z = (w < ldzt && okq) ? ZT[(int64_t)sh.Q[t] * ldzt + w] : 0ull;
        sh.bits[t][2 * k] = (uint32_t)z;
        sh.bits[t][2 * k + 1] = (uint32_t)(z >> 32);
    }
    __syncthreads();
}

// Appends to the pair list, in (t, u) order, the pairs with a generator
// among the candidates c = t nq + u from *c0 on, 256 per round (compacted
// with warp ballots), until the list holds more than kPairMax - kBlk
// entries or the candidates run out. Returns the list length; every thread
// calls it and gets the same value.
__device__ int lo_fill_pairs(LoShared &sh, int nq, int64_t *c0, const unsigned long long *__restrict__ E,
                             int64_t lde, const unsigned long long *__restrict__ Cfx, float inv, int64_t n,
                             [[maybe_unused]] uint32_t *__restrict__ status_dbg) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t ncand = (int64_t)nq * nq;
    int np = 0;
    while (*c0 < ncand && np <= kPairMax - kBlk) {
        const int64_t c = *c0 + threadIdx.x;
        int t = 0, u = 0;
        bool ok = false;
        if (c < ncand) {
            t = (int)(c / nq);
            u = (int)(c - (int64_t)t * nq);
            if (u > t && LO_OK(t < nq && u < nq, 3)) {
                const int q = sh.Q[t], r = sh.Q[u];
                if (LO_OK(q >= 0 && q < n && r >= 0 && r < n, 4)) ok = (E[(int64_t)q * lde + (r >> 6)] >> (r & 63)) & 1ull;
            }
        }
        const uint32_t bal = __ballot_sync(kFull, ok);
        if (lane == 0) sh.wsum[warp] = __popc(bal);
        __syncthreads();
        int off = np, tot = 0;
#pragma unroll
        for (int w = 0; w < kBlk / 32; ++w) {
            const int v = sh.wsum[w];
            off += w < warp ? v : 0;
            tot += v;
        }
        const int pos = off + __popc(bal & ((1u << lane) - 1u));
        if (ok && LO_OK(pos >= 0 && pos < kPairMax, 5)) {
            sh.pr[pos] = t | (u << 16);
            if (Cfx != nullptr)
                sh.pc[pos] = __ll2float_rn((long long)Cfx[(int64_t)sh.Q[t] * n + sh.Q[u]]) * inv;
        }
        np += tot;
        *c0 += kBlk;
        __syncthreads();
    }
    return np;
}

// v with its sign flipped when bit 31 of y is set.
__device__ __forceinline__ float flip_if(float v, uint32_t y) {
    return __int_as_float(__float_as_int(v) ^ (int)(y & 0x80000000u));
}

// Sum of v over the CTA in FP32 (warp shuffles, then the warps' sums in
// fixed order); every thread gets it. The partial sums of one 256-sample
// block are kept in FP32 and combined across blocks in FP64, as in the
// tensor-core epilogue (FP64 arithmetic runs at 1/64 of the FP32 rate here).
__device__ __forceinline__ float block_sum_f(float v, float *red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kBlk / 32; ++w) t += red[w];
    return t;
}

// The sample bits of blocks blk0 .. blk0 + 3 for every support qubit:
// bits4[t][w] holds samples 32 w .. 32 w + 31 of the 1024. No barriers.
__device__ __forceinline__ void lo_fill_bits4(LoShared &sh, int nq, int64_t n, const uint64_t *__restrict__ ZT,
                                              int64_t ldzt, int64_t blk0,
                                              [[maybe_unused]] uint32_t *__restrict__ status_dbg) {
    for (int e = threadIdx.x; e < nq * 16; e += kBlk) {
        const int t = e >> 4, k = e & 15;
        const int64_t w = blk0 * 4 + k;
        const bool okq = LO_OK(t < kQ4 && sh.Q[t] >= 0 && sh.Q[t] < n, 2);
        const uint64_t z = (w < ldzt && okq) ? ZT[(int64_t)sh.Q[t] * ldzt + w] : 0ull;
        sh.bits4[t][2 * k] = (uint32_t)z;
        sh.bits4[t][2 * k + 1] = (uint32_t)(z >> 32);
    }
}

// lo_fill_bits4 between barriers: previous readers of bits4 are done before
// it, every word is in place after it.
__device__ void lo_load_bits4(LoShared &sh, int nq, int64_t n, const uint64_t *__restrict__ ZT, int64_t ldzt,
                              int64_t blk0, uint32_t *__restrict__ status_dbg) {
    __syncthreads();
    lo_fill_bits4(sh, nq, n, ZT, ldzt, blk0, status_dbg);
    __syncthreads();
}

// The CTA's next work item of the heavy observables' kernels (the first is its block's; the items differ in size, so
// the rest are handed out as CTAs come free). Its barriers also part one item's use of shared memory from the next's.
__device__ __forceinline__ int64_t next_item(unsigned long long *__restrict__ counter) {
    __shared__ unsigned long long item;
    __syncthreads();
    if (threadIdx.x == 0) item = atomicAdd(counter, 1ull);
    __syncthreads();
    return (int64_t)(gridDim.x + item);
}

// The observables too heavy for the lists (or all of them, without lists):
// work item (h, g) is observable heavy[h] (h itself without `heavy`).
// MODE 0: (sum cos, sum (cos - mean)^2) per (observable, 256 samples) into
// part, and Phi itself into phi (row stride ldphi >= lds, columns < lds) when
// phi is not null (a gradient pass follows). MODE 1: W[a][i] = sin Phi
// (alpha_a + beta_a cos Phi), zero for i >= s. MODE 2: the partials and W.
// The pair term visits only the pairs of Q_a that carry a generator (C_qr is
// zero on the others). Item (a, g) takes sample blocks kPGroup g ..
// kPGroup g + kPGroup - 1. For |Q_a| <= kQ4 a thread owns four consecutive
// samples of a 1024-sample pass (four blocks; block b is warps 2b, 2b + 1),
// so every support qubit costs one 16-byte load of M and every pair one
// word pair of sample bits for four samples; larger supports take one block
// per pass, one sample per thread.
constexpr int kPhaseCtas = 5, kPairCtas = 3;  // CTAs per SM of the heavy observables' kernels (45 KB of shared memory each)
template <int MODE>
__global__ void __launch_bounds__(kBlk, kPhaseCtas) k_lo_phase(const uint64_t *__restrict__ A, int64_t lda, int64_t n,
                                                   const uint64_t *__restrict__ ZT, int64_t ldzt,
                                                   const float *__restrict__ X, int64_t lds,
                                                   const unsigned long long *__restrict__ Cfx,
                                                   const unsigned *__restrict__ cmax, int64_t m,
                                                   const unsigned long long *__restrict__ E, int64_t lde, int64_t l,
                                                   const int *__restrict__ heavy, const unsigned *__restrict__ nheavy,
                                                   unsigned long long *__restrict__ counter,
                                                   int64_t s, int64_t nparts, double2 *__restrict__ part,
                                                   const double *__restrict__ alpha, const double *__restrict__ beta,
                                                   float *__restrict__ W, float *__restrict__ phi, int64_t ldphi,
                                                   uint32_t *__restrict__ status) {
    pdl_sync();
    [[maybe_unused]] uint32_t *status_dbg = status;
    __shared__ LoShared sh;
    __shared__ const float *mrow[kQ4];  // X + Q[t] lds (four-block form)
    const int64_t ngroups = cdiv(nparts, (int64_t)kPGroup);
    const int64_t nobs = heavy ? (int64_t)*nheavy : l;
    const float inv = ldexpf(1.0f, -lo_fx_exp(*cmax, m));
    for (int64_t it = blockIdx.x; it < nobs * ngroups; it = next_item(counter)) {
    const int64_t h = it % nobs, a = heavy ? heavy[h] : h;
    const int nq = support_of_row(A + a * lda, n, sh.Q, sh.scan, status);
    const int tid = threadIdx.x, w = tid >> 5, bit = tid & 31;
    const int64_t ncand = (int64_t)nq * nq;
    int64_t c0 = 0;
    int np = lo_fill_pairs(sh, nq, &c0, E, lde, Cfx, inv, n, status);
    const bool complete = c0 >= ncand;  // the whole list fits: reuse it for every block
    const float al = MODE != 0 ? (float)alpha[a] : 0.f;
    const float be = (MODE != 0 && beta) ? (float)beta[a] : 0.f;
    const int64_t bstart = it / nobs * (int64_t)kPGroup;
    const int64_t b1 = bstart + kPGroup < nparts ? bstart + kPGroup : nparts;
    if (nq <= kQ4) {
        for (int t = tid; t < nq; t += kBlk) {
            const int q = sh.Q[t];
            const bool ok = LO_OK(q >= 0 && q < n, 7);
            mrow[t] = X + (ok ? (int64_t)q * lds : 0);
        }
        const int word = tid >> 3;              // bits4 word of this thread's samples
        const int sh4 = 28 - 4 * (tid & 7);     // moves their four bits to bits 28 .. 31
        for (int64_t blk0 = bstart; blk0 < b1; blk0 += 4) {
            lo_load_bits4(sh, nq, n, ZT, ldzt, blk0, status);  // also orders the mrow stores
            const int64_t i0 = blk0 * kBlk + 4 * (int64_t)tid;
            const int64_t blk = blk0 + (tid >> 6);  // this thread's block
            const int64_t i0c = i0 < lds ? i0 : lds - 4;  // lds is a multiple of 64
            float p0 = 0.f, p1 = 0.f, p2 = 0.f, p3 = 0.f;
            for (int t = 0; t < nq; ++t) {
                if (!LO_OK(i0c >= 0 && i0c + 3 < lds, 8)) break;
                const float4 mv = *reinterpret_cast<const float4 *>(mrow[t] + i0c);
                p0 += mv.x;
                p1 += mv.y;
                p2 += mv.z;
                p3 += mv.w;
            }
            float q0 = 0.f, q1 = 0.f, q2 = 0.f, q3 = 0.f;
            if (!complete && blk0 != bstart) {
                c0 = 0;  // the list is rebuilt round by round for every pass
                np = lo_fill_pairs(sh, nq, &c0, E, lde, Cfx, inv, n, status);
            }
            while (true) {
                for (int p = 0; p < np; ++p) {
                    const int pr = sh.pr[p];
                    if (!LO_OK((pr & 0xFFFF) < nq && (pr >> 16) < nq && p < kPairMax, 6)) continue;
                    const uint32_t y = (sh.bits4[pr & 0xFFFF][word] ^ sh.bits4[pr >> 16][word]) << sh4;
                    const float cv = sh.pc[p];
                    q0 = q0 + flip_if(cv, y << 3);
                    q1 = q1 + flip_if(cv, y << 2);
                    q2 = q2 + flip_if(cv, y << 1);
                    q3 = q3 + flip_if(cv, y);
                }
                if (complete || c0 >= ncand) break;
                __syncthreads();
                np = lo_fill_pairs(sh, nq, &c0, E, lde, Cfx, inv, n, status);
            }
            const float ph[4] = {p0 - 2.f * q0, p1 - 2.f * q1, p2 - 2.f * q2, p3 - 2.f * q3};
            bool valid[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) valid[k] = i0 + k < s && blk < b1;
            if (MODE != 1) {
                float cv[4], S1 = 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    cv[k] = valid[k] ? cosf(ph[k]) : 0.f;
                    S1 += cv[k];
                }
                // Block b's sums: its two warps' shuffle sums, in warp order.
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) S1 += __shfl_xor_sync(kFull, S1, off);
                __syncthreads();
                if (bit == 0) sh.redf[w] = S1;
                __syncthreads();
                const float S = sh.redf[w & ~1] + sh.redf[w | 1];
                const int64_t nb = s - blk * kBlk < kBlk ? s - blk * kBlk : kBlk;
                const float mean = nb > 0 ? S / (float)nb : 0.f;
                float M2 = 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float dv = cv[k] - mean;
                    M2 += valid[k] ? dv * dv : 0.f;
                }
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) M2 += __shfl_xor_sync(kFull, M2, off);
                __syncthreads();
                if (bit == 0) sh.redf[w] = M2;
                __syncthreads();
                if ((tid & 63) == 0 && blk < b1)
                    part[a * nparts + blk] = make_double2((double)S, (double)(sh.redf[w] + sh.redf[w + 1]));
                if (MODE == 0 && phi != nullptr && i0 < lds && blk < b1)
                    *reinterpret_cast<float4 *>(phi + a * ldphi + i0) = make_float4(ph[0], ph[1], ph[2], ph[3]);
            }
            if (MODE != 0 && i0 < lds && blk < b1) {
                float o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float sn, cn;
                    sincosf(ph[k], &sn, &cn);
                    o[k] = valid[k] ? sn * (al + be * cn) : 0.f;
                }
                *reinterpret_cast<float4 *>(W + a * lds + i0) = make_float4(o[0], o[1], o[2], o[3]);
            }
        }
        continue;
    }
    for (int64_t blk = bstart; blk < b1; ++blk) {
        lo_load_bits(sh, nq, n, ZT, ldzt, blk, status);
        const int64_t i = blk * kBlk + tid;
        const bool valid = i < s;
        const int64_t ic = valid ? i : s - 1;
        float ph = 0.f;
        for (int t = 0; t < nq; ++t) {
            const int q = sh.Q[t];
            if (!LO_OK(q >= 0 && q < n && ic >= 0 && ic < lds, 7)) continue;
            ph += X[(int64_t)q * lds + ic];
        }
        float pairs = 0.f;
        if (!complete && blk != bstart) {
            c0 = 0;  // the list is rebuilt round by round for every block
            np = lo_fill_pairs(sh, nq, &c0, E, lde, Cfx, inv, n, status);
        }
        while (true) {
            for (int p = 0; p < np; ++p) {
                const int pr = sh.pr[p];
                if (!LO_OK((pr & 0xFFFF) < nq && (pr >> 16) < nq && p < kPairMax, 6)) continue;
                const uint32_t x = sh.bits[pr & 0xFFFF][w] ^ sh.bits[pr >> 16][w];
                const float cv = sh.pc[p];
                pairs += ((x >> bit) & 1u) ? -cv : cv;
            }
            if (complete || c0 >= ncand) break;
            __syncthreads();
            np = lo_fill_pairs(sh, nq, &c0, E, lde, Cfx, inv, n, status);
        }
        ph -= 2.f * pairs;
        if (MODE != 1) {
            const float cv = valid ? cosf(ph) : 0.f;
            const float S = block_sum_f(cv, sh.redf);
            const int64_t nb = s - blk * kBlk < kBlk ? s - blk * kBlk : kBlk;
            const float mean = S / (float)nb;
            const float dv = cv - mean;
            const float M2 = block_sum_f(valid ? dv * dv : 0.f, sh.redf);
            if (tid == 0) part[a * nparts + blk] = make_double2((double)S, (double)M2);
            if (MODE == 0 && phi != nullptr && i < lds) phi[a * ldphi + i] = ph;
        }
        if (MODE != 0) {
            float sn, cn;
            sincosf(ph, &sn, &cn);
            if (i < lds) W[a * lds + i] = valid ? sn * (al + be * cn) : 0.f;
        }
    }
    }  // items
}

// ---------------------------------------------------- the listed observables
// One warp per (observable, 1024 samples), 32 samples per lane, no barriers: the
// observable's qubits and pairs come from its lists (k_lo_lists).
//   Phi: X is added up row by row (eight coalesced 16-byte loads per lane and
// qubit, no sign or addend left to apply); the pair term goes five pairs at a
// time, their 32 sign combinations one per lane, indexed by the lane's transposed
// sample bits (indices5), one shuffle and one add per sample.
//   K (k_lo_k, reading W back; fused with the phase its 16 KB of tables per
// warp left 12 warps per SM to wait for X): W's signed sums over all 16 sign
// patterns of every four samples of a lane are tabulated; a pair then costs
// eight table loads per lane, and the lanes' sums of 32 pairs are combined by
// one reduce-scatter.
// The loads of X from L2 bound the phase where the observables are wide (n =
// 5000, 4096 observables of 50 qubits, 16384 samples): 810 us, against 1868 with
// W in the one-CTA form (18 instructions per qubit and four samples); K 356
// against 1278.
// MODE 0: statistics partials, and Phi into phi when it is not null; 1: W; 2:
// partials and W.
constexpr int kLoWarps = 4;

// The listed observables' phase follows the heavy observables', which waits for all that came before, and shares no output with
// it: where it is launched as its dependent (obs_beside) it runs beside it and waits for it at its end, on every path, so that
// what follows it follows both. A few heavy observables take as long as one of them alone: 2000 observables of about 100 of
// 1000 qubits x 3000, three of more than 128: 412 -> 320 us.
struct AfterHeavy {
    __device__ AfterHeavy() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
    __device__ ~AfterHeavy() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
};
constexpr int kLoTab = 8 * 16 * 32;  // floats of a warp's tables
template <int MODE>
__global__ void __launch_bounds__(32 * kLoWarps) k_lo_obs(
    const int *__restrict__ cnt, const int *__restrict__ Lq, const uint2 *__restrict__ Lp, const uint32_t *__restrict__ ZP,
    int64_t nb, const float *__restrict__ X, int64_t lds, int64_t n, int64_t l, int64_t s, int64_t nparts,
    double2 *__restrict__ part, const double *__restrict__ alpha, const double *__restrict__ beta, float *__restrict__ W,
    float *__restrict__ phi, int64_t ldphi, uint32_t *__restrict__ status) {
    const AfterHeavy after;
    [[maybe_unused]] uint32_t *status_dbg = status;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t a = (int64_t)blockIdx.x * kLoWarps + warp, blk = blockIdx.y;
    if (a >= l) return;
    const int c = cnt[a];
    if (c < 0) return;  // a heavy observable
    const int nq = c & 0xFFFF, np = c >> 16;
    const int64_t i0 = blk * kLane + 4 * lane;  // the lane's samples: i0 + 128 k .. + 3
    const uint32_t *zp = ZP + blk * 32 + lane;
    const uint2 *pairs = Lp + a * kLoP;
    float acc[32];
    {
#pragma unroll
        for (int k = 0; k < 32; ++k) acc[k] = 0.f;
        // The lists are read 32 entries at a time, one per lane, and handed
        // round by shuffles, so that the rows' loads wait for nothing. (Two rows
        // of X at a time in registers, or one: 1100 against 950 us; the warps the
        // extra registers cost matter more.)
        for (int t0 = 0; t0 < nq; t0 += 32) {
            const int mine = t0 + lane < nq ? __ldg(Lq + a * kLoQ + t0 + lane) : 0;
            const int nt = nq - t0 < 32 ? nq - t0 : 32;
#pragma unroll 1
            for (int t = 0; t < nt; ++t) {
                const int q = __shfl_sync(kFull, mine, t);
                if (!LO_OK(q >= 0 && q < n, 11)) continue;
                const float *xr = X + (int64_t)q * lds + i0;
                float4 v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    v[k] = i0 + 128 * k < lds ? __ldg(reinterpret_cast<const float4 *>(xr + 128 * k))
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    acc[4 * k] += v[k].x;
                    acc[4 * k + 1] += v[k].y;
                    acc[4 * k + 2] += v[k].z;
                    acc[4 * k + 3] += v[k].w;
                }
            }
        }
        for (int p0 = 0; p0 < np; p0 += 30) {
            // past the last pair: {0, 0} with C = 0
            const uint2 mine = p0 + lane < np && lane < 30 ? __ldg(pairs + p0 + lane) : make_uint2(0u, 0u);
            const int nt = np - p0 < 30 ? np - p0 : 30;
#pragma unroll 1
            for (int h = 0; h < nt; h += 5) {
                uint32_t z[5], R[8];
                float t = 0.f;
#pragma unroll
                for (int g = 0; g < 5; ++g) {
                    const uint32_t e = __shfl_sync(kFull, mine.x, h + g);
                    const float cv = __uint_as_float(__shfl_sync(kFull, mine.y, h + g));
                    z[g] = __ldg(zp + (int64_t)(e & 0xFFFFu) * nb * 32) ^ __ldg(zp + (int64_t)(e >> 16) * nb * 32);
                    t += ((lane >> g) & 1) ? -cv : cv;
                }
                indices5(z, R);
#pragma unroll
                for (int q = 0; q < 8; ++q)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[8 * k + q] += __shfl_sync(kFull, t, (int)(R[q] >> (8 * k)));
            }
        }
        if (MODE == 0 && phi != nullptr) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (i0 + 128 * k < lds)
                    *reinterpret_cast<float4 *>(phi + a * ldphi + i0 + 128 * k) =
                        make_float4(acc[4 * k], acc[4 * k + 1], acc[4 * k + 2], acc[4 * k + 3]);
        }
    }
    const float al = MODE != 0 ? (float)alpha[a] : 0.f;
    const float be = (MODE != 0 && beta) ? (float)beta[a] : 0.f;
    // The range's four blocks of 256 samples, in a loop that takes the first eight
    // phases and moves the others down: 32 copies of the cosine's code missed the
    // instruction cache for half of the kernel's time (2000 observables x 5000
    // samples: 51 -> 42 us).
    int64_t i = i0;
#pragma unroll 1
    for (int b = 0; b < 4; ++b, i += 256) {
        const int64_t left = s - i;  // phase k of the eight is valid when 128 (k / 4) + k % 4 < left
        float cv[8], S = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const bool valid = 128 * (k / 4) + k % 4 < left;
            if (MODE == 0) {
                cv[k] = valid ? cosf(acc[k]) : 0.f;
            } else {
                float sn, cn;
                sincosf(acc[k], &sn, &cn);
                cv[k] = valid ? cn : 0.f;
                acc[k] = valid ? sn * (al + be * cn) : 0.f;  // W
            }
            S += cv[k];
        }
        if (MODE != 1) {
            const int64_t pb = blk * 4 + b;
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) S += __shfl_xor_sync(kFull, S, off);
            const int64_t nbv = s - pb * kBlk < kBlk ? s - pb * kBlk : kBlk;
            const float mean = nbv > 0 ? S / (float)nbv : 0.f;
            float M2 = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float dv = cv[k] - mean;
                M2 += 128 * (k / 4) + k % 4 < left ? dv * dv : 0.f;
            }
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) M2 += __shfl_xor_sync(kFull, M2, off);
            if (lane == 0 && pb < nparts) part[a * nparts + pb] = make_double2((double)S, (double)M2);
        }
        if (MODE != 0) {
#pragma unroll
            for (int k = 0; k < 8; k += 4)
                if (i + 32 * k < lds)
                    *reinterpret_cast<float4 *>(W + a * lds + i + 32 * k) =
                        make_float4(acc[k], acc[k + 1], acc[k + 2], acc[k + 3]);
        }
#pragma unroll
        for (int k = 0; k < 24; ++k) acc[k] = acc[k + 8];
    }
}

// K[q][r] += sum_i W[a][i] s_q(i) s_r(i) for the listed pairs (see above).
__global__ void __launch_bounds__(32 * kLoWarps) k_lo_k(const int *__restrict__ cnt, const uint2 *__restrict__ Lp,
                                                        const uint32_t *__restrict__ ZP, int64_t nb,
                                                        const float *__restrict__ W, int64_t lds, int64_t n, int64_t l,
                                                        const double *__restrict__ scale,
                                                        unsigned long long *__restrict__ Kfx) {
    pdl_sync();
    extern __shared__ float lo_tab[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t a = (int64_t)blockIdx.x * kLoWarps + warp, blk = blockIdx.y;
    if (a >= l) return;
    const int np = cnt[a] >> 16;
    if (np <= 0) return;  // no pair, or a heavy observable
    const int64_t i0 = blk * kLane + 4 * lane;
    const uint32_t *zp = ZP + blk * 32 + lane;
    const uint2 *pairs = Lp + a * kLoP;
    float *tab = lo_tab + warp * kLoTab + lane;
#pragma unroll
    for (int g = 0; g < 8; ++g) {  // W is zero from s on, up to its row's end
        const float4 w = i0 + 128 * g < lds ? *reinterpret_cast<const float4 *>(W + a * lds + i0 + 128 * g)
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
        const float p01[4] = {w.x + w.y, w.y - w.x, w.x - w.y, -w.x - w.y};
        const float p23[4] = {w.z + w.w, w.w - w.z, w.z - w.w, -w.z - w.w};
#pragma unroll
        for (int e = 0; e < 16; ++e) tab[(g * 16 + e) * 32] = p01[e & 3] + p23[e >> 2];
    }
    const float sc = (float)*scale;
    for (int p0 = 0; p0 < np; p0 += 32) {
        const uint32_t mine = p0 + lane < np ? __ldg(&pairs[p0 + lane].x) : 0u;  // past the last pair: {0, 0}, not used
        float v[32];
#pragma unroll
        for (int h = 0; h < 32; h += 8) {
            if (p0 + h < np) {  // uniform
                uint32_t z[8];
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const uint32_t e = __shfl_sync(kFull, mine, h + g);
                    z[g] = __ldg(zp + (int64_t)(e & 0xFFFFu) * nb * 32) ^ __ldg(zp + (int64_t)(e >> 16) * nb * 32);
                }
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    float u[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        u[k] = tab[(2 * k * 16 + ((z[g] >> (8 * k)) & 15u)) * 32] +
                               tab[((2 * k + 1) * 16 + ((z[g] >> (8 * k + 4)) & 15u)) * 32];
                    v[h + g] = (u[0] + u[1]) + (u[2] + u[3]);
                }
            } else {
#pragma unroll
                for (int g = 0; g < 8; ++g) v[h + g] = 0.f;
            }
        }
        const float d = reduce_scatter(v, lane);
        if (p0 + lane < np) {
            atomicAdd(Kfx + (int64_t)(mine & 0xFFFFu) * n + (mine >> 16), (unsigned long long)to_fixed(d, sc));
        }
    }
}

// V[q][i] = sum over the observables a containing q of W[a][i] (in a order),
// zero for i >= s: s_q V as the hi + lo BF16 operand of H (row stride lds), or V
// itself where H is summed without the tensor cores; gsp[q * nblk + blk] = sum_i s_q(i) V[q][i] over the
// CTA's 256 samples (FP64). A thread owns four consecutive samples of each
// 1024-sample pass (block b of the pass is warps 2b, 2b + 1), so every
// observable costs one 16-byte load of W per thread and pass.
__global__ void __launch_bounds__(kBlk) k_lo_v(const uint64_t *__restrict__ AT, int64_t ldlt,
                                               const uint64_t *__restrict__ ZT, int64_t ldzt,
                                               const float *__restrict__ W, int64_t lds, int64_t s, int64_t nblk,
                                               float *__restrict__ V, __nv_bfloat16 *__restrict__ hi,
                                               __nv_bfloat16 *__restrict__ lo, double *__restrict__ gsp) {
    pdl_sync();
    __shared__ float red[kBlk / 32];
    __shared__ int obs[kObsMax];
    __shared__ int wsum[kBlk / 32];
    constexpr int kPass = kGroup / 4;  // 1024-sample passes per CTA
    const int64_t q = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t *row = AT + q * ldlt;
    const int64_t b0 = blockIdx.y * (int64_t)kGroup;
    const int64_t b1 = b0 + kGroup < nblk ? b0 + kGroup : nblk;
    float4 v[kPass];
#pragma unroll
    for (int g = 0; g < kPass; ++g) v[g] = make_float4(0.f, 0.f, 0.f, 0.f);
    // The observables containing q, kObsMax at a time, in increasing order
    // (each thread compacts one 64-observable word; warps in order).
    for (int64_t w0 = 0; w0 < ldlt; w0 += kObsMax / 64) {
        int no = 0;
        for (int64_t wb = w0; wb < w0 + kObsMax / 64 && wb < ldlt; wb += kBlk) {
            const int64_t wi = wb + threadIdx.x;
            uint64_t bits = (wi < w0 + kObsMax / 64 && wi < ldlt) ? row[wi] : 0ull;
            const int cnt = __popcll(bits);
            int incl = cnt;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int u = __shfl_up_sync(kFull, incl, off);
                if (lane >= off) incl += u;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            int off = no, tot = 0;
#pragma unroll
            for (int k = 0; k < kBlk / 32; ++k) {
                off += k < warp ? wsum[k] : 0;
                tot += wsum[k];
            }
            int pos = off + incl - cnt;
            while (bits) {
                const int b = __ffsll((long long)bits) - 1;
                bits &= bits - 1ull;
                obs[pos++] = (int)(64 * wi + b);
            }
            no += tot;
            __syncthreads();
        }
#pragma unroll
        for (int g = 0; g < kPass; ++g) {
            if (b0 + 4 * g < b1) {  // uniform
                const int64_t i0 = (b0 + 4 * g) * kBlk + 4 * (int64_t)threadIdx.x;
                const int64_t i0c = i0 < lds ? i0 : lds - 4;  // lds is a multiple of 64
                float4 acc = v[g];
                for (int k = 0; k < no; ++k) {
                    const float4 x = *reinterpret_cast<const float4 *>(W + (int64_t)obs[k] * lds + i0c);
                    acc.x += x.x;
                    acc.y += x.y;
                    acc.z += x.z;
                    acc.w += x.w;
                }
                v[g] = acc;
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int g = 0; g < kPass; ++g) {
        if (b0 + 4 * g >= b1) continue;  // uniform
        const int64_t i0 = (b0 + 4 * g) * kBlk + 4 * (int64_t)threadIdx.x;
        const int64_t blk = b0 + 4 * g + (threadIdx.x >> 6);
        const bool in = blk < b1 && i0 < lds;
        const float vv[4] = {in && i0 < s ? v[g].x : 0.f, in && i0 + 1 < s ? v[g].y : 0.f,
                             in && i0 + 2 < s ? v[g].z : 0.f, in && i0 + 3 < s ? v[g].w : 0.f};
        if (in && V != nullptr) *reinterpret_cast<float4 *>(V + q * lds + i0) = make_float4(vv[0], vv[1], vv[2], vv[3]);
        // lds <= 64 ldzt, so the word of i0 is inside row q of ZT when i0 < lds.
        const uint32_t nib = in ? (uint32_t)(ZT[q * ldzt + (i0 >> 6)] >> (i0 & 63)) : 0u;
        float u = 0.f;
        uint32_t ph[4], pl[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float x = ((nib >> k) & 1u) ? -vv[k] : vv[k];
            u += x;
            const __nv_bfloat16 b = __float2bfloat16_rn(x);
            ph[k] = __bfloat16_as_ushort(b);
            pl[k] = __bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(b)));
        }
        if (in && hi != nullptr) {
            *reinterpret_cast<uint2 *>(hi + q * lds + i0) = make_uint2(ph[0] | (ph[1] << 16), ph[2] | (ph[3] << 16));
            *reinterpret_cast<uint2 *>(lo + q * lds + i0) = make_uint2(pl[0] | (pl[1] << 16), pl[2] | (pl[3] << 16));
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) u += __shfl_xor_sync(kFull, u, off);
        __syncthreads();
        if (lane == 0) red[warp] = u;
        __syncthreads();
        if ((threadIdx.x & 63) == 0 && blk < b1) gsp[q * nblk + blk] = (double)(red[warp] + red[warp + 1]);
    }
}

// W[a][i] = sin Phi (alpha_a + beta_a cos Phi) (zero for i >= s) from the
// Phi the statistics pass kept (l x ldphi; phi may be W itself: each
// element is read before it is written, by the same thread), four samples
// per thread: the arithmetic of k_lo_phase<1>, without recomputing Phi.
__global__ void __launch_bounds__(256) k_lo_w(const float *phi, int64_t ldphi, float *W, int64_t lds, int64_t l,
                                             int64_t s, const double *__restrict__ alpha,
                                             const double *__restrict__ beta) {
    pdl_sync();
    const int64_t per_row = lds / 4;
    const int64_t total = l * per_row;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t a = g / per_row, i0 = (g - a * per_row) * 4;
        const float al = (float)alpha[a];
        const float be = beta ? (float)beta[a] : 0.f;
        const float4 f = *reinterpret_cast<const float4 *>(phi + a * ldphi + i0);
        const float v[4] = {f.x, f.y, f.z, f.w};
        float o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float sn, cn;
            sincosf(v[k], &sn, &cn);
            o[k] = i0 + k < s ? sn * (al + be * cn) : 0.f;
        }
        *reinterpret_cast<float4 *>(W + a * lds + i0) = make_float4(o[0], o[1], o[2], o[3]);
    }
}

// K[q][r] += sum over the samples of W[a][i] s_q(i) s_r(i) for the pairs
// q < r of Q_a that carry a generator (the only K entries the gradient
// reads). The pair list is taken kPairPass pairs at a time; warp w owns
// pairs w, w + 8, ... of the pass, each lane eight samples of every block,
// with a running sum per (pair, lane) in registers over the CTA's blocks,
// then one shuffle reduction and one fixed-point atomic per (pair, CTA).
// For supports of at most kQ4 qubits the sample bits and W of four blocks
// are staged per pair of barriers (one block at a time otherwise).
// Work item (a, g) takes blocks kPGroup g ...; heavy observables as in k_lo_phase.
constexpr int kPairPass = 128;
__global__ void __launch_bounds__(kBlk, kPairCtas) k_lo_pairs(const uint64_t *__restrict__ A, int64_t lda, int64_t n,
                                                   const uint64_t *__restrict__ ZT, int64_t ldzt,
                                                   const unsigned long long *__restrict__ E, int64_t lde, int64_t l,
                                                   const int *__restrict__ heavy, const unsigned *__restrict__ nheavy,
                                                   unsigned long long *__restrict__ counter,
                                                   const float *__restrict__ W, int64_t lds, int64_t s,
                                                   int64_t nblk, const double *__restrict__ scale,
                                                   unsigned long long *__restrict__ Kfx,
                                                   uint32_t *__restrict__ status) {
    pdl_sync();
    [[maybe_unused]] uint32_t *status_dbg = status;
    __shared__ LoShared sh;
    __shared__ __align__(16) float wb[4 * kBlk];
    constexpr int kPerWarp = kPairPass / (kBlk / 32);
    const int64_t ngroups = cdiv(nblk, (int64_t)kPGroup);
    const int64_t nobs = heavy ? (int64_t)*nheavy : l;
    for (int64_t it = blockIdx.x; it < nobs * ngroups; it = next_item(counter)) {
    const int64_t h = it % nobs, a = heavy ? heavy[h] : h;
    const int nq = support_of_row(A + a * lda, n, sh.Q, sh.scan, status);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sa = 31 - lane;  // moves this lane's sample bit to bit 31
    const float sc = (float)*scale;
    const int64_t ncand = (int64_t)nq * nq;
    const int64_t b0 = it / nobs * (int64_t)kPGroup;
    const int64_t b1 = b0 + kPGroup < nblk ? b0 + kPGroup : nblk;
    int64_t c0 = 0;
    while (c0 < ncand) {
        const int np = lo_fill_pairs(sh, nq, &c0, E, lde, nullptr, 0.f, n, status);
        for (int p0 = 0; p0 < np; p0 += kPairPass) {
            float acc[kPerWarp];
#pragma unroll
            for (int j = 0; j < kPerWarp; ++j) acc[j] = 0.f;
            // One block's sample-bit rows (8 words per support qubit, at
            // word stride ws of the shared rows) against the lane's 8 W values.
            auto block_pairs = [&](const uint32_t *rows, int ws, const float (&wv)[8]) {
#pragma unroll
                for (int j = 0; j < kPerWarp; ++j) {
                    const int p = p0 + warp + (kBlk / 32) * j;
                    if (p < np) {  // uniform in the warp
                        const int pr = sh.pr[p];
                        const int t = pr & 0xFFFF, u = pr >> 16;
                        if (!LO_OK(t < nq && u < nq && t < kQMax && u < kQMax && p < kPairMax, 9)) continue;
                        const uint4 t0 = *reinterpret_cast<const uint4 *>(rows + t * ws);
                        const uint4 t1 = *reinterpret_cast<const uint4 *>(rows + t * ws + 4);
                        const uint4 u0 = *reinterpret_cast<const uint4 *>(rows + u * ws);
                        const uint4 u1 = *reinterpret_cast<const uint4 *>(rows + u * ws + 4);
                        float v = acc[j];
                        v += flip_if(wv[0], (t0.x ^ u0.x) << sa);
                        v += flip_if(wv[1], (t0.y ^ u0.y) << sa);
                        v += flip_if(wv[2], (t0.z ^ u0.z) << sa);
                        v += flip_if(wv[3], (t0.w ^ u0.w) << sa);
                        v += flip_if(wv[4], (t1.x ^ u1.x) << sa);
                        v += flip_if(wv[5], (t1.y ^ u1.y) << sa);
                        v += flip_if(wv[6], (t1.z ^ u1.z) << sa);
                        v += flip_if(wv[7], (t1.w ^ u1.w) << sa);
                        acc[j] = v;
                    }
                }
            };
            if (nq <= kQ4) {
                for (int64_t blk0 = b0; blk0 < b1; blk0 += 4) {
                    __syncthreads();  // previous readers of bits4 and wb are done
                    lo_fill_bits4(sh, nq, n, ZT, ldzt, blk0, status);
                    {
                        const int64_t i0 = blk0 * kBlk + 4 * (int64_t)threadIdx.x;
                        const bool in = blk0 + (threadIdx.x >> 6) < b1 && i0 < lds;  // lds: a multiple of 64
                        float4 w4 = in ? *reinterpret_cast<const float4 *>(W + a * lds + i0)
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
                        if (i0 >= s) w4.x = 0.f;
                        if (i0 + 1 >= s) w4.y = 0.f;
                        if (i0 + 2 >= s) w4.z = 0.f;
                        if (i0 + 3 >= s) w4.w = 0.f;
                        *reinterpret_cast<float4 *>(&wb[4 * threadIdx.x]) = w4;
                    }
                    __syncthreads();
                    for (int b = 0; b < 4 && blk0 + b < b1; ++b) {  // uniform
                        float wv[8];
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) wv[kk] = wb[kBlk * b + 32 * kk + lane];
                        block_pairs(&sh.bits4[0][8 * b], 32, wv);
                    }
                }
            } else {
                for (int64_t blk = b0; blk < b1; ++blk) {
                    lo_load_bits(sh, nq, n, ZT, ldzt, blk, status);
                    const int64_t i = blk * kBlk + threadIdx.x;
                    wb[threadIdx.x] = i < s ? W[a * lds + i] : 0.f;
                    __syncthreads();
                    float wv[8];
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) wv[kk] = wb[32 * kk + lane];
                    block_pairs(&sh.bits[0][0], 8, wv);
                }
            }
#pragma unroll
            for (int j = 0; j < kPerWarp; ++j) {
                const int p = p0 + warp + (kBlk / 32) * j;
                if (p < np) {  // uniform in the warp
                    float v = acc[j];
#pragma unroll
                    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
                    const int pr = sh.pr[p];
                    if (lane == 0)
                        atomicAdd(Kfx + (int64_t)sh.Q[pr & 0xFFFF] * n + sh.Q[pr >> 16],
                                  (unsigned long long)to_fixed(v, sc));
                }
            }
        }
        __syncthreads();  // the list is read before the next round rebuilds it
    }
    }  // items
}

// Hs[q][r] = sum over the K pieces of H[q][r] + H[r][q], q < r (n x ldh FP64):
// tile by tile, so that the transposed elements are read in rows too (per gate
// they are a cache line each, times the pieces).
__global__ void __launch_bounds__(256) k_lo_hsum(const float *__restrict__ H, int64_t ldh, int64_t n, int hparts, int nb,
                                                 double *__restrict__ Hs) {
    pdl_sync();
    __shared__ float2 tile[32][33];
    int bi = 0, left = blockIdx.x;  // block number -> (bi, bj), bi <= bj
    while (left >= nb - bi) {
        left -= nb - bi;
        ++bi;
    }
    const int64_t q0 = 32 * (int64_t)bi, r0 = 32 * (int64_t)(bi + left);
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    // The pieces in FP32 with their rounding errors added up beside them (the
    // sum to about 2^-46 with one FP64 add per element).
    auto pieces = [&](int64_t row, int64_t col, float &s, float &e) {
        for (int p = 0; p < hparts; ++p) {
            const float v = H[((int64_t)p * n + row) * ldh + col], t = s + v, z = t - s;
            e += (s - (t - z)) + (v - z);
            s = t;
        }
    };
    for (int k = y; k < 32; k += 8) {  // rows r0 + k, columns q0 + x
        float s = 0.f, e = 0.f;
        if (r0 + k < n && q0 + x < n) pieces(r0 + k, q0 + x, s, e);
        tile[k][x] = make_float2(s, e);
    }
    __syncthreads();
    for (int k = y; k < 32; k += 8) {
        const int64_t q = q0 + k, r = r0 + x;
        if (q >= r || r >= n) continue;
        float s = tile[x][k].x, e = tile[x][k].y;
        pieces(q, r, s, e);
        Hs[q * ldh + r] = (double)s + (double)e;
    }
}

// grad_j from the parts above (see the header). H: one piece in FP32 (H), the
// pieces' symmetric sum (Hs), or FP64 sums (Hd).
__global__ void k_lo_grad_out(const int4 *__restrict__ sup, int64_t m, int64_t n, const double *__restrict__ gsp,
                              int64_t nblk, const float *__restrict__ H, int64_t ldh,
                              const double *__restrict__ Hs, const double *__restrict__ Hd,
                              const unsigned long long *__restrict__ Kfx, const double *__restrict__ scale,
                              double *__restrict__ grad) {
    pdl_sync();
    // scale is a power of two; one FP64 division per block, not per thread (500500 gates: 11.8 -> 9.4 us)
    __shared__ double sinv;
    if (threadIdx.x == 0) sinv = -4.0 / *scale;
    __syncthreads();
    const double inv = sinv;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int4 sp = sup[j];
        double g = 0.0;
        if (sp.w == 1) {
            double t = 0.0;
            for (int64_t k = 0; k < nblk; ++k) t += gsp[(int64_t)sp.x * nblk + k];
            g = 2.0 * t;
        } else if (sp.w == 2) {
            const int64_t q = sp.x, r = sp.y;
            const double h = Hs != nullptr   ? Hs[q * ldh + r]
                             : Hd != nullptr ? Hd[q * ldh + r] + Hd[r * ldh + q]
                                             : (double)H[q * ldh + r] + (double)H[r * ldh + q];
            g = fma((double)(long long)Kfx[q * n + r], inv, h + h);  // 2 h - 4 k, rounded once
        }
        grad[j] = g;
    }
}

int grid_1d(int64_t work) {
    int64_t b = cdiv(work, 256);
    if (b < 1) b = 1;
    if (b > 8192) b = 8192;
    return (int)b;
}

}  // namespace

cudaError_t launch_support_list(const uint64_t *G, int64_t m, int64_t ldg, int64_t n, int4 *sup, cudaStream_t st,
                                const float *theta, unsigned *cmax);
cudaError_t launch_bit_transpose_batched(const uint64_t *in, int64_t batch, int64_t in_rows, int64_t in_cols,
                                         int64_t ld_in, uint64_t *out, int64_t ld_out, cudaStream_t st);
cudaError_t launch_fixed_scale(const double *alpha, const double *beta, int64_t l, int64_t s, double *scale,
                               cudaStream_t st);

int64_t lo_part_samples() { return kBlk; }

// The pair contractions on the tensor cores (split BF16) unless IQP_LO_TC=0.
bool lo_tensor() {
    static int v = -1;
    if (v < 0) {
        const char *e = std::getenv("IQP_LO_TC");
        v = (e != nullptr && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

// Elements of the split-BF16 operand buffer (hi and lo) the tensor-core
// contractions need: the larger of C's (n x round_up(n, 64)) and s o V's
// (n x lds), twice.
int64_t lo_split_elems(int64_t n, int64_t lds) {
    const int64_t kc = round_up(n, 64);
    return 2 * n * (kc > lds ? kc : lds);
}

int64_t lo_lde(int64_t n) { return cdiv(n, 64); }

namespace {

unsigned *lo_cmax(const LoArgs &a) { return reinterpret_cast<unsigned *>(a.fx + a.n * a.n + a.n); }
unsigned *lo_nheavy(const LoArgs &a) { return lo_cmax(a) + 1; }
double *lo_scale(const LoArgs &a) { return reinterpret_cast<double *>(a.fx + a.n * a.n); }
unsigned long long *lo_items(const LoArgs &a) { return a.fx + a.n * a.n + a.n + 1; }  // of the phase, of the pairs
const int *lo_heavy(const LoArgs &a) { return a.ZP != nullptr ? a.cnt + a.l : nullptr; }

// Blocks of the heavy observables' kernels: as many as the SMs hold take what
// there is (usually nothing); without lists one per work item. They are not
// launched as dependents: where there are fewer items than the SMs hold, the blocks would come
// in while the contraction before them ends and crowd the SMs that it leaves first (300 observables of
// 300 qubits x 3000: 21 ms, 37 as dependents).
unsigned lo_heavy_blocks(const LoArgs &a, int64_t nblk, int per_sm) {
    int64_t b = a.l * cdiv(nblk, (int64_t)kPGroup);
    if (a.ZP != nullptr && b > per_sm * num_sms()) b = per_sm * num_sms();
    if (b > 0x7FFFFFFF) b = 0x7FFFFFFF;
    return (unsigned)(b < 1 ? 1 : b);
}

// Whether the listed observables' phase runs beside the heavy ones' (AfterHeavy): up to 16384 warps of it (7 per
// scheduler). Past that a few heavy observables' time counts for less than the L1 that their kernel's shared memory
// takes from the first blocks on every SM (4096 x 16384 on 5000 qubits: 4.47 ms in order, 4.56 beside).
bool obs_beside(const LoArgs &a) { return a.l * cdiv(a.s, (int64_t)kLane) <= 16384; }

template <int MODE>
cudaError_t launch_obs(const LoArgs &a, double2 *part, const double *alpha, const double *beta, float *W, float *phi,
                       int64_t ldphi, cudaStream_t st) {
    const int64_t nb = cdiv(a.s, (int64_t)kLane);
    const dim3 grid((unsigned)cdiv(a.l, (int64_t)kLoWarps), (unsigned)nb);
    LaunchScope ls(IQP_KERNEL_LOWORDER, st);
    if (obs_beside(a))
        launch_pdl(k_lo_obs<MODE>, grid, 32 * kLoWarps, 0, st, a.cnt, a.Lq, a.Lp, a.ZP, nb, a.X, a.lds, a.n, a.l, a.s,
                   cdiv(a.s, (int64_t)kBlk), part, alpha, beta, W, phi, ldphi, a.status);
    else
        k_lo_obs<MODE><<<grid, 32 * kLoWarps, 0, st>>>(a.cnt, a.Lq, a.Lp, a.ZP, nb, a.X, a.lds, a.n, a.l, a.s,
                                                       cdiv(a.s, (int64_t)kBlk), part, alpha, beta, W, phi, ldphi, a.status);
    return cudaGetLastError();
}

cudaError_t launch_k(const LoArgs &a, const float *W, cudaStream_t st) {
    constexpr int smem = kLoWarps * kLoTab * 4;
    static DeviceOnce once;
    const cudaError_t e = allow_smem(once, k_lo_k, smem);
    if (e != cudaSuccess) return e;
    const int64_t nb = cdiv(a.s, (int64_t)kLane);
    LaunchScope ls(IQP_KERNEL_LOWORDER, st);
    launch_pdl(k_lo_k, dim3((unsigned)cdiv(a.l, (int64_t)kLoWarps), (unsigned)nb), 32 * kLoWarps, smem, st,
        a.cnt, a.Lp, a.ZP, nb, W, a.lds, a.n, a.l, lo_scale(a), a.fx);
    return cudaGetLastError();
}

template <int MODE>
cudaError_t launch_phase(const LoArgs &a, double2 *part, const double *alpha, const double *beta, float *W, float *phi,
                         int64_t ldphi, cudaStream_t st) {
    const int64_t nblk = cdiv(a.s, (int64_t)kBlk);
    LaunchScope ls(IQP_KERNEL_LOWORDER, st);
    k_lo_phase<MODE><<<lo_heavy_blocks(a, nblk, kPhaseCtas), kBlk, 0, st>>>(
        a.A, a.lda, a.n, a.ZT, a.ldzt, a.X, a.lds, a.fx, lo_cmax(a), a.m, a.E, lo_lde(a.n), a.l, lo_heavy(a), lo_nheavy(a),
        lo_items(a), a.s, nblk, part, alpha, beta, W, phi, ldphi, a.status);
    return cudaGetLastError();
}

}  // namespace

// Supports, C, d, E, the samples transposed, X, and the observables' lists.
cudaError_t launch_lo_prepare(const LoArgs &a, cudaStream_t st) {
    const int64_t n = a.n, m = a.m, lde = lo_lde(n), kc = round_up(n, 64);
    const bool tc = lo_tensor() && a.split != nullptr && a.ldz >= 4 && a.ldz % 2 == 0 &&
                    (reinterpret_cast<uintptr_t>(a.Z) & 15) == 0;
    cudaError_t e;
    // fx: Cfx (n x n), dfx (n), then the largest |c_j| (float bits), the count of heavy observables and the items handed out.
    if ((e = cudaMemsetAsync(a.E, 0, (size_t)n * lde * 8, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(a.fx, 0, (size_t)(n * n + n) * 8 + 24, st)) != cudaSuccess) return e;
    if ((e = launch_support_list(a.G, m, a.ldg, n, a.sup, st, a.theta, lo_cmax(a))) != cudaSuccess) return e;
    if ((e = launch_bit_transpose_batched(a.Z, 1, a.s, n, a.ldz, a.ZT, a.ldzt, st)) != cudaSuccess) return e;
    __nv_bfloat16 *hi = a.split, *lo = a.split + n * kc;
    // dense: the contractions' operand; else C itself and both halves of E, for k_lo_cs and k_lo_h
    auto build = [&](bool dense) {
        LaunchScope ls(IQP_KERNEL_LOWORDER, st);
        launch_pdl(k_lo_build, grid_1d(m), 256, 0, st, a.sup, a.theta, m, n, a.fx, a.fx + n * n, lo_cmax(a), a.E, lde,
                   dense ? 0 : 1, a.status);
        const cudaError_t rc = cudaGetLastError();
        if (rc != cudaSuccess) return rc;
        const int nb = (int)(kc / 64);
        launch_pdl(k_lo_convert, (unsigned)((int64_t)nb * (nb + 1) / 2), 256, 0, st, a.fx, a.fx + n * n, lo_cmax(a), m, n, nb, hi,
                   lo, kc, dense ? nullptr : a.C, a.ldc, a.d);
        return cudaGetLastError();
    };
    if ((e = build(tc)) != cudaSuccess) return e;
    if (a.ZP != nullptr) {
        LaunchScope ls(IQP_KERNEL_LOWORDER, st);
        const int64_t nb = cdiv(a.s, (int64_t)kLane);
        launch_pdl(k_lo_zpack, grid_1d(32 * n * nb), 256, 0, st, reinterpret_cast<const uint32_t *>(a.ZT), 2 * a.ldzt, n, nb, a.ZP);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        launch_pdl(k_lo_lists, (unsigned)cdiv(a.l, (int64_t)8), 256, 0, st, a.A, a.lda, a.l, n, a.E, lde, a.fx, lo_cmax(a), m,
                   a.l * nb <= 4 * (int64_t)num_sms() ? kLoQ / 2 : kLoQ, a.Lq,
                                                                    a.Lp, a.cnt, a.cnt + a.l, lo_nheavy(a), a.status);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // X = s o (d + C S): rows q, columns the samples (Z's rows), K the qubits r.
    if (tc) {
        e = launch_tc_dense(hi, lo, n, kc, n, a.Z, a.s, a.ldz, a.X, a.lds, 1, a.d, a.ZT, a.ldzt, a.status, st);
        if (e != cudaErrorNotSupported) return e;
        // No tensor map for Z (rows 2^40 bytes apart): the sums once more, for the kernel that adds them up.
        if ((e = cudaMemsetAsync(a.fx, 0, (size_t)(n * n + n) * 8, st)) != cudaSuccess) return e;
        if ((e = build(false)) != cudaSuccess) return e;
    }
    LaunchScope ls(IQP_KERNEL_LOWORDER_GEMM, st);
    launch_pdl(k_lo_cs, dim3((unsigned)n, (unsigned)cdiv(a.s, 2048)), 32, 0, st, a.E, lde, a.C, a.ldc, a.d, a.ZT, a.ldzt, a.s, a.X,
                                                                         a.lds);
    return cudaGetLastError();
}

// Statistics partials and, if phi is not null, Phi.
cudaError_t launch_lo_stats(const LoArgs &a, double2 *part, float *phi, int64_t ldphi, cudaStream_t st) {
    const cudaError_t e = launch_phase<0>(a, part, nullptr, nullptr, nullptr, phi, ldphi, st);
    if (e != cudaSuccess || a.ZP == nullptr) return e;
    return launch_obs<0>(a, part, nullptr, nullptr, nullptr, phi, ldphi, st);
}

// The gradient. part: also the statistics partials (one pass over Phi); phi:
// read from there (it may be W) instead of formed; scale_set: the fixed-point
// scale is in place. AT: n x ldlt words (A transposed), W: l x lds, V: n x lds
// (only without the tensor cores), gsp: n x nblk doubles.
cudaError_t launch_lo_grad(const LoArgs &a, double2 *part, const double *alpha, const double *beta, uint64_t *AT,
                           int64_t ldlt, float *W, float *V, double *gsp, double *grad, float *phi, int64_t ldphi,
                           bool scale_set, cudaStream_t st) {
    const int64_t n = a.n, s = a.s, nblk = cdiv(s, (int64_t)kBlk), lde = lo_lde(n);
    const bool listed = a.ZP != nullptr, tc = lo_tensor() && a.split != nullptr;
    cudaError_t e = launch_bit_transpose_batched(a.A, 1, a.l, n, a.lda, AT, ldlt, st);
    if (e != cudaSuccess) return e;
    if (!scale_set && (e = launch_fixed_scale(alpha, beta, a.l, s, lo_scale(a), st)) != cudaSuccess) return e;
    // K's sums take the place of C's, which the heavy observables' phase reads.
    const bool beside = phi == nullptr && obs_beside(a);
    auto clear = [&] { return cudaMemsetAsync(a.fx, 0, (size_t)n * n * sizeof(unsigned long long), st); };
    if (phi == nullptr) {
        e = part != nullptr ? launch_phase<2>(a, part, alpha, beta, W, nullptr, 0, st)
                            : launch_phase<1>(a, nullptr, alpha, beta, W, nullptr, 0, st);
        if (e == cudaSuccess && !beside) e = clear();
        if (e == cudaSuccess && listed)
            e = part != nullptr ? launch_obs<2>(a, part, alpha, beta, W, nullptr, 0, st)
                                : launch_obs<1>(a, nullptr, alpha, beta, W, nullptr, 0, st);
        if (e == cudaSuccess && beside) e = clear();
        if (e != cudaSuccess) return e;
    } else {
        if ((e = clear()) != cudaSuccess) return e;
        LaunchScope ls(IQP_KERNEL_LOWORDER, st);
        launch_pdl(k_lo_w, grid_1d(a.l * (a.lds / 4)), 256, 0, st, phi, ldphi, W, a.lds, a.l, s, alpha, beta);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (listed && (e = launch_k(a, W, st)) != cudaSuccess) return e;
    __nv_bfloat16 *hi = a.split, *lo = a.split + n * a.lds;
    {
        LaunchScope ls(IQP_KERNEL_LOWORDER, st);
        launch_pdl(k_lo_v, dim3((unsigned)n, (unsigned)cdiv(nblk, (int64_t)kGroup)), kBlk, 0, st,
            AT, ldlt, a.ZT, a.ldzt, W, a.lds, s, nblk, tc ? nullptr : V, tc ? hi : nullptr, lo, gsp);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // H = (s o V) S^T: rows q, columns r (ZT's rows), K the samples.
    int hparts = 1;
    if (tc) {
        hparts = a.hparts;
        e = launch_tc_dense(hi, lo, n, a.lds, s, a.ZT, n, a.ldzt, a.H, a.ldc, hparts, nullptr, nullptr, 0, a.status, st);
    } else {
        LaunchScope ls(IQP_KERNEL_LOWORDER_GEMM, st);
        launch_pdl(k_lo_h, dim3((unsigned)n, (unsigned)kHSplit), 32, 0, st, a.E, lde, a.ZT, a.ldzt, V, a.lds, s, a.Hs, a.ldc);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    {
        LaunchScope ls(IQP_KERNEL_LOWORDER, st);
        k_lo_pairs<<<lo_heavy_blocks(a, nblk, kPairCtas), kBlk, 0, st>>>(
            a.A, a.lda, n, a.ZT, a.ldzt, a.E, lde, a.l, lo_heavy(a), lo_nheavy(a), lo_items(a) + 1, W, a.lds, s, nblk,
            lo_scale(a), a.fx, a.status);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (hparts > 1) {
        const int64_t nb = cdiv(n, 32);
        LaunchScope ls(IQP_KERNEL_LOWORDER, st);
        launch_pdl(k_lo_hsum, (unsigned)(nb * (nb + 1) / 2), 256, 0, st, a.H, a.ldc, n, hparts, (int)nb, a.Hs);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    LaunchScope ls(IQP_KERNEL_LOWORDER, st);
    launch_pdl(k_lo_grad_out, grid_1d(a.m), 256, 0, st, a.sup, a.m, n, gsp, nblk, a.H, a.ldc, hparts > 1 ? a.Hs : nullptr,
               tc ? nullptr : a.Hs, a.fx, lo_scale(a), grad);
    return cudaGetLastError();
}

}  // namespace iqp
