// Row-sparse form of the phase contraction and of its gradient, for parity
// matrices P_A of low density (Sec. 2.2 notes that C = 1 - (-1)^{A G^T} is
// sparse when observables and generators have small support).
//
// For one observable a, with J_a = { j : P_A[a][j] = 1 } and c_j = 2 theta_j,
//   Phi[a][i] = sum_{j in J_a} c_j (1 - 2 P_Z[i][j])          (eq. Emat)
// and, for W[a][i] = sin Phi (alpha_a + beta_a cos Phi),
//   grad_j    = sum_{a : j in J_a} 2 sum_i W[a][i] (1 - 2 P_Z[i][j]).
// The work is |J_a| * s per observable instead of m * s: the dense forms
// multiply every zero of P_A too.
//
// Layout: one CTA of 16 warps per (observable, range of 1024 samples). Lane q
// owns the 32 samples of 32-bit word (32 r + q) of every P_Z^T row, so a gate
// costs one coalesced 128-byte load per warp. J_a is listed in shared memory
// (4096 gates at a time) and the warps share it out.
//
// Phase: five gates at a time. Their 32 sign combinations c_1 +- ... are one
// value per lane; each lane transposes the gates' five words into a 5-bit
// index per sample and takes that sample's combination with one shuffle and
// one add, about 30 instructions per gate and word against 160 per gate and
// two words for a sign flip and an add per term. Two batches are added to a pair
// of samples by one packed FP32 add (3.14 -> 2.81 ms of the loss below).
// The warps' partial phases are added in shared memory in a fixed order.
//
// Gradient: W of the range is tabulated, once per CTA, as the signed sums of
// every 8 consecutive samples of a lane over all 256 sign patterns (128 KB,
// each lane's entries in its own bank). A gate's signed dot product is then
// four table loads per lane, indexed by the bytes of its P_Z^T word, and the
// lanes' sums of 32 gates are combined by one reduce-scatter.
//
// Measured, MMD loss and gradient of the n = 1000 one- and two-body circuit
// (500500 gates, 2000 observables, 5000 samples): 18.9 -> 5.6 ms (8.6 with the
// parity words loaded into registers and the list made again for every range);
// independent batches (n = 200, 5000 gates, 256 x 2000 samples), forward and
// backward: 1.43 -> 0.51 ms.
//
// Statistics: (sum cos, sum (cos - mean)^2) partials of 1024 samples (FP32
// within a warp, FP64 across warps), merged by the shared finaliser; where the
// workspace has room for half as many, a CTA takes pairs of ranges and merges their two.
// Gradient sums: the per-range dot products are added into a 64-bit fixed-point
// accumulator per gate with integer atomics. Integer addition is associative,
// so the result does not depend on the order of the atomics: the gradient is
// bitwise reproducible. The fixed-point scale 2^k is chosen per call from the
// bound B = sum_a 2 s (|alpha_a| + |beta_a|) >= |every partial sum| so that
// B 2^k < 2^61: nothing can overflow, and the rounding error per gate is at
// most (number of contributions) * 2^-k / 2.
#include "common.cuh"

namespace iqp {

namespace {

// The lane's P_Z^T word of gate j. Shared batch: a load from P_Z^T.
// Independent batches: the parity is formed here from the observable's own
// transposed samples ZT (n rows of bits over samples) as the XOR of the rows
// of the gate's support (listed for |supp| <= 3, else read from G).
struct ZSource {
    const uint32_t *PZT;  // shared: P_Z^T; independent: this observable's ZT
    int64_t ldzt;         // 32-bit words per row
    int64_t word;
    const int4 *sup;      // independent batches only
    const uint64_t *G;
    int64_t ldg;
    int64_t n;
    int64_t m;            // gates

    template <bool INDEP>
    __device__ __forceinline__ uint32_t get(int64_t j) const {
        if (!IQP_IN(j, m, 70)) return 0u;  // a set parity bit past the last gate
        if (!INDEP) return __ldg(PZT + j * ldzt + word);
        const int4 sp = __ldg(sup + j);
        if (sp.w <= 3) {
            if (!IQP_IN(sp.w > 0 ? sp.x : 0, n, 71) || !IQP_IN(sp.w > 1 ? sp.y : 0, n, 71) ||
                !IQP_IN(sp.w > 2 ? sp.z : 0, n, 71))
                return 0u;
            uint32_t z = 0u;
            if (sp.w > 0) z = __ldg(PZT + (int64_t)sp.x * ldzt + word);
            if (sp.w > 1) z ^= __ldg(PZT + (int64_t)sp.y * ldzt + word);
            if (sp.w > 2) z ^= __ldg(PZT + (int64_t)sp.z * ldzt + word);
            return z;
        }
        uint32_t z = 0u;
        const uint64_t *g = G + j * ldg;
        const int64_t nw = (n + 63) >> 6;
        for (int64_t w = 0; w < nw; ++w) {
            uint64_t gv = __ldg(g + w);
            while (gv) {
                const int b = __ffsll((long long)gv) - 1;
                gv &= gv - 1ull;
                const int64_t q = 64 * w + b;
                if (q >= n) break;
                z ^= __ldg(PZT + q * ldzt + word);
            }
        }
        return z;
    }
};

constexpr int kWarps = 16, kThreads = 32 * kWarps;
constexpr int kRange = 1024;   // samples per CTA: 32 per lane
constexpr int kList = 4096;    // gates of J_a listed at a time
constexpr int kScan = 4;       // P_A words per thread and listing step (ldp is a multiple of 4)
constexpr unsigned kFull = 0xFFFFFFFFu;

// Dynamic shared memory: the list (gate, bits of c), then the partial phases
// (16 x 1024 floats) or the sign tables (4 x 256 x 32 floats) in the same
// place, then W (1024 floats), then the dense words of a listing step, then
// the reductions' words, then (gradient, shared batches) the rings of its
// P_Z^T words. The phase's rings lie in the tables' place.
constexpr int kSmList = 0, kSmTab = kList * 8, kWordBytes = kThreads * kScan * 4;
constexpr int kPartBytes = kWarps * kRange * 4, kTabBytes = 4 * 256 * 32 * 4;
// P_Z^T words in flight: per warp kRing stages of kPhaseStage (kGradStage) gates
// x 128 bytes, brought in by 16-byte asynchronous copies (four gates per warp
// instruction), two stages ahead of their use: 82 KB per SM in the phase. With
// the next five words in registers, 10 to 20 KB per SM, the phase waited on
// them for most of its time.
constexpr int kRing = 3, kPhaseStage = 20, kGradStage = 8;
constexpr int kPhaseRing = kRing * kPhaseStage * 32, kGradRing = kRing * kGradStage * 32;  // words per warp
static_assert(kPhaseStage % 10 == 0 && kWarps * kPhaseRing * 4 <= kTabBytes && kPartBytes <= kTabBytes, "the tables' place");
// bytes of the tables' place, and in all (independent batches stage nothing)
__host__ __device__ constexpr int tab_bytes(bool grad, bool indep) { return grad || !indep ? kTabBytes : kPartBytes; }
constexpr int smem_bytes(bool grad, bool indep) {
    return kSmTab + tab_bytes(grad, indep) + kRange * 4 + kWordBytes + 256 + (grad && !indep ? kWarps * kGradRing * 4 : 0);
}
static_assert(smem_bytes(true, false) <= 232448 && 2 * (smem_bytes(false, true) + 1024) <= 233472, "shared memory");

__device__ __forceinline__ void copy16_async(uint32_t *dst, const uint32_t *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Every group but the newest kRing - 2 of this thread has landed.
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory"); }

// Exclusive prefix sum of v over the CTA; *total receives the sum. Every thread calls it.
__device__ __forceinline__ int block_excl(int v, int *red, int *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += u;
    }
    __syncthreads();  // previous readers of red are done
    if (lane == 31) red[warp] = incl;
    __syncthreads();
    int off = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const int x = red[w];
        off += w < warp ? x : 0;
        tot += x;
    }
    *total = tot;
    return off + incl - v;
}

// Where the listing of a P_A row stands: the step's first word, and how many
// of the step's set bits are listed already.
struct RowCursor {
    int64_t w0;
    int off;
};

// The next gates of the row, at most kList, in increasing order, with c_j;
// returns their number (0 at the row's end). Every thread calls it. A thread
// lists the bits of its own sparse words; a word of more than kFew set bits is
// noted in `dense` and listed by a whole warp (an observable's gates lie in
// runs where the generators are ordered by their qubits).
constexpr int kFew = 3;
__device__ __forceinline__ int list_gates(const uint64_t *__restrict__ row, int64_t ldp, [[maybe_unused]] int64_t m,
                                          const float *__restrict__ c, int2 *list, uint32_t *dense, int *red,
                                          RowCursor &cur) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int *ndense = red + kWarps;
    int n = 0;
    while (cur.w0 < ldp && n < kList) {  // uniform
        const int64_t w = cur.w0 + (int64_t)threadIdx.x * kScan;
        uint64_t bits[kScan];
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < kScan; k += 2) {
            ulonglong2 v = make_ulonglong2(0ull, 0ull);
            if (w + k < ldp) v = *reinterpret_cast<const ulonglong2 *>(row + w + k);  // rows are 32-byte aligned
            bits[k] = v.x;
            bits[k + 1] = v.y;
            cnt += __popcll(v.x) + __popcll(v.y);
        }
        if (threadIdx.x == 0) *ndense = 0;
        int total = 0;
        const int first = block_excl(cnt, red, &total);
        const int take = min(kList - n, total - cur.off);
        if (first + cnt > cur.off && first < cur.off + take) {
            int p = first - cur.off;  // position in this window
#pragma unroll
            for (int k = 0; k < kScan; ++k) {
                uint64_t b = bits[k];
                const int pc = __popcll(b);
                if (pc > kFew) {
                    if (p + pc > 0 && p < take)  // the word's first position in the step, above its number
                        dense[atomicAdd(ndense, 1)] = (uint32_t)((p + cur.off) << 11) | (threadIdx.x * kScan + k);
                    p += pc;
                    continue;
                }
                while (b) {
                    const int64_t j = (w + k) * 64 + __ffsll((long long)b) - 1;
                    b &= b - 1ull;
                    if (p >= 0 && p < take && IQP_IN(j, m, 76))
                        list[n + p] = make_int2((int)j, __float_as_int(__ldg(c + j)));
                    ++p;
                }
            }
        }
        __syncthreads();
        const int nd = *ndense;
        for (int i = warp; i < nd; i += kWarps) {
            const uint32_t e = dense[i];
            const int64_t wi = cur.w0 + (e & 2047u);
            const uint64_t word = __ldg(row + wi);
            const int base = (int)(e >> 11) - cur.off;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int b = lane + 32 * h;
                const int p = base + __popcll(word & ((1ull << b) - 1ull));
                const int64_t j = wi * 64 + b;
                if (((word >> b) & 1ull) && p >= 0 && p < take && IQP_IN(j, m, 77))
                    list[n + p] = make_int2((int)j, __float_as_int(__ldg(c + j)));
            }
        }
        n += take;
        cur.off += take;
        if (cur.off >= total) {
            cur.w0 += (int64_t)kThreads * kScan;
            cur.off = 0;
        }
        __syncthreads();  // the list is in place, `dense` free again
    }
    return n;
}
static_assert(kThreads * kScan <= 2048 && kThreads * kScan * 64 <= (1 << 21), "packing of `dense`");

// acc[k] += sum over this warp's share of the listed gates of +-c_j for
// sample k of the lane (batches of five gates, every 16th batch; the next
// batch's words are loaded before the current one is used). A short last
// batch takes gates of c = 0.
template <bool INDEP>
__device__ __forceinline__ void phase_list(float (&acc)[32], const int2 *list, int n, const ZSource &zs, int warp,
                                           int lane) {
    uint32_t z[5];
    float t = 0.f;
    auto load = [&](int b, uint32_t (&zz)[5], float &tt) {
        tt = 0.f;
#pragma unroll
        for (int g = 0; g < 5; ++g) {
            const int e = 5 * b + g;
            zz[g] = 0u;
            if (e < n) {  // uniform in the warp
                const int2 jc = list[e];
                zz[g] = zs.get<INDEP>((int64_t)(uint32_t)jc.x);
                const float cv = __int_as_float(jc.y);
                tt += ((lane >> g) & 1) ? -cv : cv;
            }
        }
    };
    if (5 * warp < n) load(warp, z, t);
    for (int b = warp; 5 * b < n; b += kWarps) {
        uint32_t zn[5], R[8];
        float tn = 0.f;
#pragma unroll
        for (int g = 0; g < 5; ++g) zn[g] = 0u;
        if (5 * (b + kWarps) < n) load(b + kWarps, zn, tn);
        indices5(z, R);
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[8 * k + q] += __shfl_sync(kFull, t, (int)(R[q] >> (8 * k)));
#pragma unroll
        for (int g = 0; g < 5; ++g) z[g] = zn[g];
        t = tn;
    }
}

// Adds 2 scale sum_i W_i s_ij of this warp's share of the listed gates into
// their accumulators: batches of 32 gates, every 16th batch. sc = 2 scale, a
// power of two in [2^-119, 2^119].
template <bool INDEP>
__device__ __forceinline__ void grad_list(const int2 *list, int n, const ZSource &zs, const float *tab,
                                          unsigned long long *__restrict__ gfx, float sc, int warp, int lane) {
    const float *tl = tab + lane;
    for (int b = warp; 32 * b < n; b += kWarps) {
        const int e0 = 32 * b;
        float v[32];
#pragma unroll
        for (int h = 0; h < 32; h += 8) {
            uint32_t z[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) z[g] = e0 + h + g < n ? zs.get<INDEP>((int64_t)(uint32_t)list[e0 + h + g].x) : 0u;
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const float a0 = tl[(z[g] & 0xFFu) * 32], a1 = tl[8192 + ((z[g] >> 8) & 0xFFu) * 32];
                const float a2 = tl[16384 + ((z[g] >> 16) & 0xFFu) * 32], a3 = tl[24576 + (z[g] >> 24) * 32];
                v[h + g] = (a0 + a1) + (a2 + a3);
            }
        }
        const float d = reduce_scatter(v, lane);
        if (e0 + lane < n) {
            const int64_t j = (int64_t)(uint32_t)list[e0 + lane].x;
            const long long q = to_fixed(d, sc);
            if (IQP_IN(j, zs.m, 72)) atomicAdd(gfx + j, (unsigned long long)q);
        }
    }
}

// The words of gates e0 .. e0 + STAGE - 1 (below `end`) of the list into `dst`
// (STAGE x 32 words): 16-byte piece c of a gate's 128 bytes where c < nch.
template <int STAGE>
__device__ __forceinline__ void fetch_stage(uint32_t *dst, const int2 *list, int e0, int end, const uint32_t *pzt,
                                            int64_t ldzt, int nch, [[maybe_unused]] int64_t m, int lane) {
#pragma unroll
    for (int i = 0; i < STAGE / 4; ++i) {
        const int g = 4 * i + (lane >> 3), c = lane & 7;
        if (e0 + g < end && c < nch) {
            const int64_t j = (int64_t)(uint32_t)list[e0 + g].x;
            if (IQP_IN(j, m, 70)) copy16_async(dst + g * 32 + 4 * c, pzt + j * ldzt + 4 * c);
        }
    }
    copy_commit();
}

// Two FP32 adds in one instruction, each rounded to nearest like a scalar add.
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, float lo, float hi) {
    uint64_t b, d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(b) : "f"(lo), "f"(hi));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// phase_list for shared batches: this warp's share of the list is a run of
// gates, its words staged in `ring`. pzt: P_Z^T at this range's words. acc: pair
// t holds samples 2 t and 2 t + 1 of the lane. Two batches of five at a time, so
// that one's index and shuffle latencies lie behind the other's.
__device__ __forceinline__ void phase_list_staged(uint64_t (&acc)[16], const int2 *list, int n, const uint32_t *pzt,
                                                  int64_t ldzt, int nch, int64_t m, uint32_t *ring, int warp, int lane) {
    const int per = 5 * ((n + 5 * kWarps - 1) / (5 * kWarps));
    const int b0 = warp * per, end = b0 + per < n ? b0 + per : n;
    uint32_t sign[5];
#pragma unroll
    for (int g = 0; g < 5; ++g) sign[g] = (uint32_t)((lane >> g) & 1) << 31;
#pragma unroll
    for (int k = 0; k < kRing - 1; ++k)
        fetch_stage<kPhaseStage>(ring + k * kPhaseStage * 32, list, b0 + k * kPhaseStage, end, pzt, ldzt, nch, m, lane);
    // a batch's five words and this lane's sign combination of its c_j; gates past the end count as c = 0
    auto load = [&](const uint32_t *zw, const int2 *lp, int left, uint32_t (&z)[5]) {
        float t = 0.f;
#pragma unroll
        for (int g = 0; g < 5; ++g) {
            z[g] = zw[g * 32];
            const uint32_t cb = g < left ? (uint32_t)lp[g].y : 0u;
            t += __uint_as_float(cb ^ sign[g]);
        }
        return t;
    };
    int st = 0;
    for (int e0 = b0; e0 < end; e0 += kPhaseStage) {
        copy_wait();
        __syncwarp();
        const uint32_t *zw = ring + st * kPhaseStage * 32 + lane;
#pragma unroll 1
        for (int h = 0; h < kPhaseStage && e0 + h < end; h += 10) {
            uint32_t z0[5], z1[5], R0[8], R1[8];
            const float t0 = load(zw + h * 32, list + e0 + h, end - e0 - h, z0);
            const float t1 = load(zw + (h + 5) * 32, list + e0 + h + 5, end - e0 - h - 5, z1);
            indices5(z0, R0);
            indices5(z1, R1);
#pragma unroll
            for (int q = 0; q < 8; q += 2)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float a0 = __shfl_sync(kFull, t0, (int)(R0[q] >> (8 * k)));
                    const float a1 = __shfl_sync(kFull, t0, (int)(R0[q + 1] >> (8 * k)));
                    const float c0 = __shfl_sync(kFull, t1, (int)(R1[q] >> (8 * k)));
                    const float c1 = __shfl_sync(kFull, t1, (int)(R1[q + 1] >> (8 * k)));
                    acc[4 * k + q / 2] = add_f32x2(add_f32x2(acc[4 * k + q / 2], a0, a1), c0, c1);
                }
        }
        __syncwarp();  // every lane has read the stage that comes free
        const int nx = st == 0 ? kRing - 1 : st - 1;
        fetch_stage<kPhaseStage>(ring + nx * kPhaseStage * 32, list, e0 + (kRing - 1) * kPhaseStage, end, pzt, ldzt, nch, m,
                                 lane);
        st = st + 1 == kRing ? 0 : st + 1;
    }
}

// grad_list for shared batches, staged likewise.
__device__ __forceinline__ void grad_list_staged(const int2 *list, int n, const uint32_t *pzt, int64_t ldzt, int nch,
                                                 int64_t m, uint32_t *ring, const float *tab,
                                                 unsigned long long *__restrict__ gfx, float sc, int warp, int lane) {
    const float *tl = tab + lane;
    const int per = 8 * ((n + 8 * kWarps - 1) / (8 * kWarps));
    const int b0 = warp * per, end = b0 + per < n ? b0 + per : n;
#pragma unroll
    for (int k = 0; k < kRing - 1; ++k)
        fetch_stage<kGradStage>(ring + k * kGradStage * 32, list, b0 + k * kGradStage, end, pzt, ldzt, nch, m, lane);
    int st = 0;
    for (int e0 = b0; e0 < end; e0 += 32) {
        float v[32];
#pragma unroll
        for (int h = 0; h < 32; h += kGradStage) {
            copy_wait();
            __syncwarp();
            const uint32_t *zw = ring + st * kGradStage * 32 + lane;
#pragma unroll
            for (int g = 0; g < kGradStage; ++g) {
                const uint32_t z = e0 + h + g < end ? zw[g * 32] : 0u;
                const float a0 = tl[(z & 0xFFu) * 32], a1 = tl[8192 + ((z >> 8) & 0xFFu) * 32];
                const float a2 = tl[16384 + ((z >> 16) & 0xFFu) * 32], a3 = tl[24576 + (z >> 24) * 32];
                v[h + g] = (a0 + a1) + (a2 + a3);
            }
            __syncwarp();
            const int nx = st == 0 ? kRing - 1 : st - 1;
            fetch_stage<kGradStage>(ring + nx * kGradStage * 32, list, e0 + h + (kRing - 1) * kGradStage, end, pzt, ldzt, nch,
                                    m, lane);
            st = st + 1 == kRing ? 0 : st + 1;
        }
        const float d = reduce_scatter(v, lane);
        if (e0 + lane < end) {
            const int64_t j = (int64_t)(uint32_t)list[e0 + lane].x;
            if (IQP_IN(j, m, 72)) atomicAdd(gfx + j, (unsigned long long)to_fixed(d, sc));
        }
    }
}

// Sum of v over the CTA: shuffles in FP32 within a warp, the warps' sums in
// FP64 in a fixed order, by warp 0 alone (16 FP64 adds by every warp took a
// tenth of the statistics pass). Every thread calls it; warp 0 gets the sum.
__device__ __forceinline__ double block_sum(float v, float *red) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
#pragma unroll
        for (int w = 0; w < kWarps; ++w) t += (double)red[w];
    }
    return t;
}

// MODE 0: statistics partials, and Phi itself into phi (l x ldphi FP32) when
// phi is not null (a gradient pass follows). MODE 1: W from Phi (read from
// phi when not null, else recomputed), then the gradient contributions of
// every gate of J_a. MODE 2: both from one Phi (gradient coefficients known
// in advance). Independent batches always recompute.
// INDEP: PZT holds every observable's transposed samples (n x ldzt words
// each, observable a at PZT + a n ldzt) and the parities are formed on the fly.
// phi: element e = 32-sample position k, lane q of a range's nl valid lanes at
// range start + k nl + q.
// nparts: ranges of 1024 samples; pair: partials of 2048 (rpc and r0 are even).
template <int MODE, bool INDEP>
__global__ void __launch_bounds__(kThreads, MODE == 0 && INDEP ? 2 : 1)
    k_sparse(const uint64_t *__restrict__ PA, int64_t ldp, const uint64_t *__restrict__ PZT, int64_t ldzt,
             int64_t m, const float *__restrict__ c, int64_t s, int64_t nparts, double2 *__restrict__ part,
             const double *__restrict__ alpha, const double *__restrict__ beta, const double *__restrict__ scale,
             unsigned long long *__restrict__ gfx, const int4 *__restrict__ sup, const uint64_t *__restrict__ G,
             int64_t ldg, int64_t n, float *__restrict__ phi, int64_t ldphi, int64_t r0,
             int64_t rpc, int pair) {
    pdl_sync();
    extern __shared__ __align__(16) uint8_t sm[];
    int2 *list = reinterpret_cast<int2 *>(sm + kSmList);
    float *tab = reinterpret_cast<float *>(sm + kSmTab);
    float *wsm = reinterpret_cast<float *>(sm + kSmTab + tab_bytes(MODE != 0, INDEP));
    uint32_t *dense = reinterpret_cast<uint32_t *>(wsm + kRange);
    int *red = reinterpret_cast<int *>(dense + kThreads * kScan);
    [[maybe_unused]] uint32_t *ring = reinterpret_cast<uint32_t *>(red + 64);  // the gradient's
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t a = blockIdx.x;
    const int64_t vwords = cdiv(s, 32);
    const uint64_t *parow = PA + a * ldp;
    [[maybe_unused]] const int64_t l = gridDim.x;
    int held = -1;  // gates in the list when it holds all of J_a: listed once for all of the CTA's ranges
    const int64_t rbeg = r0 + blockIdx.y * rpc, rend = rbeg + rpc < nparts ? rbeg + rpc : nparts;
    for (int64_t r = rbeg; r < rend; ++r) {
    if (r > rbeg) __syncthreads();  // the previous range is done with shared memory
    const int nl = (int)(vwords - r * 32 < 32 ? vwords - r * 32 : 32);  // lanes with samples
    const int64_t word = r * 32 + (lane < nl ? lane : nl - 1);          // in-bounds load, result masked
    const ZSource zs{reinterpret_cast<const uint32_t *>(INDEP ? PZT + a * n * ldzt : PZT), 2 * ldzt, word, sup, G, ldg, n, m};
    // shared batches: this range's words of P_Z^T row 0, and its 16-byte pieces inside a row (2 ldzt is a multiple of 8)
    const uint32_t *pzt = reinterpret_cast<const uint32_t *>(PZT) + r * 32;
    const int nch = (int)(2 * ldzt - r * 32 < 32 ? (2 * ldzt - r * 32) / 4 : 8);

    // Phi of elements tid and tid + 512 (element e: sample 32 (e % 32) + e / 32 of the range)
    float ph[2];
    const bool kept = MODE == 1 && !INDEP && phi != nullptr;
    float *prow = phi == nullptr ? nullptr : phi + a * ldphi + r * kRange;
    if (kept) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = tid + kThreads * h;
            const bool in = lane < nl && IQP_IN(a * ldphi + r * kRange + (e >> 5) * nl + lane, l * ldphi, 73);
            ph[h] = in ? prow[(e >> 5) * nl + lane] : 0.f;
        }
    } else {
        float acc[32];
        uint64_t acc2[16];
#pragma unroll
        for (int k = 0; k < 32; ++k) acc[k] = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) acc2[k] = 0ull;
        auto phase = [&](int cnt) {
            if constexpr (INDEP)
                phase_list<true>(acc, list, cnt, zs, warp, lane);
            else
                phase_list_staged(acc2, list, cnt, pzt, 2 * ldzt, nch, m, reinterpret_cast<uint32_t *>(tab) + warp * kPhaseRing,
                                  warp, lane);
        };
        if (held >= 0) {
            phase(held);
        } else {
            RowCursor cur{0, 0};
            for (bool first = true;; first = false) {
                const int cnt = list_gates(parow, ldp, m, c, list, dense, red, cur);
                phase(cnt);
                if (cur.w0 >= ldp) {
                    if (first) held = cnt;
                    break;
                }
                __syncthreads();  // the list is read before it is filled again
            }
        }
        __syncthreads();  // the partial phases lie where other warps' rings were
        if constexpr (!INDEP) {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                acc[2 * k] = __uint_as_float((uint32_t)acc2[k]);
                acc[2 * k + 1] = __uint_as_float((uint32_t)(acc2[k] >> 32));
            }
        }
#pragma unroll
        for (int k = 0; k < 32; ++k) tab[warp * kRange + k * 32 + lane] = acc[k];
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = tid + kThreads * h;
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) v += tab[w * kRange + e];
            ph[h] = v;
            if (MODE == 0 && !INDEP && phi != nullptr && lane < nl &&
                IQP_IN(a * ldphi + r * kRange + (e >> 5) * nl + lane, l * ldphi, 74))
                prow[(e >> 5) * nl + lane] = v;
        }
    }
    const int64_t left = s - r * kRange;  // samples of this range, from here on
    bool valid[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) valid[h] = lane * 32 + (tid >> 5) + kWarps * h < left;

    if (MODE == 0 || MODE == 2) {
        float cv[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) cv[h] = valid[h] ? cosf(ph[h]) : 0.f;
        float *redf = reinterpret_cast<float *>(red);
        const double S = block_sum(cv[0] + cv[1], redf);
        if (tid == 0) redf[kWarps] = (float)(S / (double)(left < kRange ? left : kRange));
        __syncthreads();
        const float mean = redf[kWarps];
        float m2 = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float d = cv[h] - mean;
            m2 += valid[h] ? d * d : 0.f;
        }
        const double M2 = block_sum(m2, redf);
        if (tid == 0 && !pair) {
            if (IQP_IN(a * nparts + r, l * nparts, 75)) part[a * nparts + r] = make_double2(S, M2);
        } else if (tid == 0) {
            double *held = reinterpret_cast<double *>(red + 32);  // the even range's
            if ((r & 1) != 0) {  // Chan et al.: the even range has all its samples
                const double nk = (double)(left < kRange ? left : kRange), d = S / nk - held[0] / kRange;
                held[1] += M2 + d * d * (kRange * nk / (kRange + nk));
                held[0] += S;
            } else {
                held[0] = S;
                held[1] = M2;
            }
            const int64_t np = (nparts + 1) / 2;
            if (((r & 1) != 0 || r + 1 == nparts) && IQP_IN(a * np + r / 2, l * np, 75))
                part[a * np + r / 2] = make_double2(held[0], held[1]);
        }
    }
    if (MODE != 0) {
        const float al = (float)alpha[a];
        const float be = beta ? (float)beta[a] : 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float sn, cn;
            sincosf(ph[h], &sn, &cn);
            wsm[tid + kThreads * h] = valid[h] ? sn * (al + be * cn) : 0.f;
        }
        __syncthreads();  // W is in place, the partial phases are read
        // Table of byte b: thread (warp, lane) fills the 16 entries whose high
        // four bits are `warp`, each the sum of its two halves' signed sums.
#pragma unroll 1
        for (int b = 0; b < 4; ++b) {
            float w[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) w[k] = wsm[(8 * b + k) * 32 + lane];
            float hi = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) hi += ((warp >> k) & 1) ? -w[4 + k] : w[4 + k];
            float *t = tab + (b * 256 + warp * 16) * 32 + lane;
            const float p01[4] = {w[0] + w[1], w[1] - w[0], w[0] - w[1], -w[0] - w[1]};
            const float p23[4] = {w[2] + w[3], w[3] - w[2], w[2] - w[3], -w[2] - w[3]};
#pragma unroll
            for (int e = 0; e < 16; ++e) t[e * 32] = hi + (p01[e & 3] + p23[e >> 2]);
        }
        const float sc = (float)(2.0 * *scale);
        auto grad = [&](int cnt) {
            if constexpr (INDEP)
                grad_list<true>(list, cnt, zs, tab, gfx, sc, warp, lane);
            else
                grad_list_staged(list, cnt, pzt, 2 * ldzt, nch, m, ring + warp * kGradRing, tab, gfx, sc, warp, lane);
        };
        if (held >= 0) {
            __syncthreads();
            grad(held);
        } else {
            RowCursor cur{0, 0};
            for (bool first = true;; first = false) {
                const int cnt = list_gates(parow, ldp, m, c, list, dense, red, cur);  // its barriers also publish the tables
                grad(cnt);
                if (cur.w0 >= ldp) {
                    if (first) held = cnt;
                    break;
                }
                __syncthreads();
            }
        }
    }
    }  // ranges
}

// scale = 2^k with B 2^k < 2^61, B = sum_a 2 s (|alpha_a| + |beta_a|)
// (fixed-order FP64 sum).
__global__ void __launch_bounds__(256) k_sparse_scale(const double *__restrict__ alpha,
                                                      const double *__restrict__ beta, int64_t l, int64_t s,
                                                      double *__restrict__ scale) {
    pdl_sync();
    __shared__ double red[256];
    double acc = 0.0;
    for (int64_t a = threadIdx.x; a < l; a += 256) acc += fabs(alpha[a]) + (beta ? fabs(beta[a]) : 0.0);
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w >= 1; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *scale = fixed_scale(2.0 * (double)s * red[0]);
    }
}

// grad[j] = fixed-point accumulator / scale.
__global__ void k_sparse_grad_out(const unsigned long long *__restrict__ gfx, int64_t m,
                                  const double *__restrict__ scale, double *__restrict__ grad) {
    pdl_sync();
    const double inv = 1.0 / *scale;  // a power of two: exact
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x)
        grad[j] = (double)(long long)gfx[j] * inv;
}

// npart: partials per observable, one per range or per two.
template <int MODE, bool INDEP>
cudaError_t launch_k(int64_t l, int64_t npart, int kernel, const uint64_t *PA, int64_t ldp, const uint64_t *PZT,
                     int64_t ldzt, int64_t m, const float *c, int64_t s, double2 *part, const double *alpha,
                     const double *beta, const double *scale, unsigned long long *gfx, const SparseIndep *ind, float *phi,
                     int64_t ldphi, cudaStream_t st) {
    constexpr int smem = smem_bytes(MODE != 0, INDEP);
    static DeviceOnce once;
    cudaError_t e = allow_smem(once, k_sparse<MODE, INDEP>, smem);
    if (e != cudaSuccess) return e;
    // Observables on grid x (the CTAs running at once share a range's P_Z^T
    // segments in L2), ranges on y: a CTA takes as many of them as leave four
    // CTAs per SM, so that J_a is listed once for them all (5% of the time where
    // P_A's density is 0.008), at most 65535 blocks per launch.
    const int64_t nparts = cdiv(s, (int64_t)kRange);
    const bool pair = part != nullptr && npart < nparts;
    int64_t rpc = l * nparts / (4 * (int64_t)num_sms() + 1);
    rpc = rpc < 1 ? 1 : (rpc > nparts ? nparts : rpc);
    rpc = cdiv(nparts, cdiv(nparts, rpc));  // equal shares
    if (pair) rpc = round_up(rpc, 2);
    for (int64_t r0 = 0; r0 < nparts; r0 += 65535 * rpc) {
        const int64_t nr = cdiv(nparts - r0, rpc) < 65535 ? cdiv(nparts - r0, rpc) : 65535;
        LaunchScope ls(kernel, st);
        launch_pdl(k_sparse<MODE, INDEP>, dim3((unsigned)l, (unsigned)nr), kThreads, smem, st,
            PA, ldp, PZT, ldzt, m, c, s, nparts, part, alpha, beta, scale, gfx, ind ? ind->sup : nullptr,
            ind ? ind->G : nullptr, ind ? ind->ldg : 0, ind ? ind->n : 0, phi, ldphi, r0, rpc, pair ? 1 : 0);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

int64_t sparse_part_samples() { return kRange; }
uint32_t check_word_sparse() { return take_check_word(); }

// Statistics partials and the gradient from one pass over Phi (shared
// batches; alpha, beta known before the estimates): k_sparse<2>.
cudaError_t launch_sparse_value_grad(const uint64_t *PA, int64_t ldp, const uint64_t *PZT, int64_t ldzt,
                                     const float *c, int64_t l, int64_t s, int64_t m, int64_t nparts, double2 *part,
                                     const double *alpha, const double *beta, double *scale, unsigned long long *gfx,
                                     double *grad, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(gfx, 0, (size_t)m * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    {
        LaunchScope ls(IQP_KERNEL_GRAD_SPARSE, st);
        launch_pdl(k_sparse_scale, 1, 256, 0, st, alpha, beta, l, s, scale);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    e = launch_k<2, false>(l, nparts, IQP_KERNEL_PHASE_SPARSE, PA, ldp, PZT, ldzt, m, c, s, part, alpha, beta, scale, gfx,
                           nullptr, nullptr, 0, st);
    if (e != cudaSuccess) return e;
    int blocks = (int)cdiv(m, 256);
    if (blocks > 8192) blocks = 8192;
    LaunchScope ls(IQP_KERNEL_GRAD_SPARSE, st);
    launch_pdl(k_sparse_grad_out, blocks, 256, 0, st, gfx, m, scale, grad);
    return cudaGetLastError();
}

// scale (one double) = 2^k with sum_a 2 s (|alpha_a| + |beta_a|) 2^k < 2^61;
// used by every fixed-point gradient accumulation.
cudaError_t launch_fixed_scale(const double *alpha, const double *beta, int64_t l, int64_t s, double *scale,
                               cudaStream_t st) {
    LaunchScope ls(IQP_KERNEL_GRAD_SPARSE, st);
    launch_pdl(k_sparse_scale, 1, 256, 0, st, alpha, beta, l, s, scale);
    return cudaGetLastError();
}

// indep != nullptr: independent batches (PZT = every observable's ZT).
// phi != nullptr: Phi is kept there (l x ldphi FP32, ldphi a multiple of 64).
cudaError_t launch_sparse_stats(const uint64_t *PA, int64_t ldp, const uint64_t *PZT, int64_t ldzt, const float *c,
                                int64_t l, int64_t s, int64_t m, double2 *part, int64_t nparts,
                                const SparseIndep *indep, float *phi, int64_t ldphi, cudaStream_t st) {
    if (indep)
        return launch_k<0, true>(l, nparts, IQP_KERNEL_PHASE_SPARSE, PA, ldp, PZT, ldzt, m, c, s, part, nullptr, nullptr,
                                 nullptr, nullptr, indep, nullptr, 0, st);
    return launch_k<0, false>(l, nparts, IQP_KERNEL_PHASE_SPARSE, PA, ldp, PZT, ldzt, m, c, s, part, nullptr, nullptr,
                              nullptr, nullptr, nullptr, phi, ldphi, st);
}

cudaError_t launch_sparse_grad(const uint64_t *PA, int64_t ldp, const uint64_t *PZT, int64_t ldzt, const float *c,
                               int64_t l, int64_t s, int64_t m, int64_t nparts, const double *alpha,
                               const double *beta, double *scale, unsigned long long *gfx, double *grad,
                               const SparseIndep *indep, const float *phi, int64_t ldphi, bool scale_set, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(gfx, 0, (size_t)m * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    if (!scale_set) {
        LaunchScope ls(IQP_KERNEL_GRAD_SPARSE, st);
        launch_pdl(k_sparse_scale, 1, 256, 0, st, alpha, beta, l, s, scale);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (indep)
        e = launch_k<1, true>(l, nparts, IQP_KERNEL_GRAD_SPARSE, PA, ldp, PZT, ldzt, m, c, s, nullptr, alpha, beta, scale,
                              gfx, indep, nullptr, 0, st);
    else
        e = launch_k<1, false>(l, nparts, IQP_KERNEL_GRAD_SPARSE, PA, ldp, PZT, ldzt, m, c, s, nullptr, alpha, beta, scale,
                               gfx, nullptr, const_cast<float *>(phi), ldphi, st);
    if (e != cudaSuccess) return e;
    int blocks = (int)cdiv(m, 256);
    if (blocks > 8192) blocks = 8192;
    LaunchScope ls(IQP_KERNEL_GRAD_SPARSE, st);
    launch_pdl(k_sparse_grad_out, blocks, 256, 0, st, gfx, m, scale, grad);
    return cudaGetLastError();
}

}  // namespace iqp
