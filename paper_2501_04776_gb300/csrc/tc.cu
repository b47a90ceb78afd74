// Split-BF16 tensor-core (tcgen05 / TMEM) kernels for sm_103a.
//
// k_tc (phase modes): the phase contraction of eq. Emat,
// Phi = (2 theta . P_A) S_Z^T, one 128 (observables) x 256 (samples) FP32
// accumulator in TMEM per CTA and tile, K = gates streamed in 64-wide stages.
// Operands never exist in HBM as numbers: a TMA warp brings 256-gate slices
// of the parity bits (and of the hi/lo BF16 split of 2 theta) into shared
// memory, and sixteen producer warps expand them: B = 1 - 2 P_Z into the
// 128-byte-swizzled K-major BF16 layout in shared memory, and A_hi =
// hi_j [P_A], A_lo = lo_j [P_A] (all exact in BF16) either straight into
// TMEM with tcgen05.st (the default for CTA pairs: the MMA then reads A from
// TMEM, and shared memory carries only B) or into shared memory like B
// (IQP_PHASE_TMEM=0, and the one-CTA form). One thread issues two
// tcgen05.mma per 16-gate step (hi and lo share B), a whole stage from one
// asm statement. The epilogue runs in the producer warps straight from TMEM:
//   mode 0: cos, per-observable (S, M2) partials over 64-sample groups, and
//           Phi itself (FP32) when a gradient pass follows that reads it back
//           (the MMD loss, the autograd pair; k_w_from_phi forms W from it);
//   mode 1: W = sin Phi (alpha + beta cos Phi), split into hi + lo BF16 rows;
//   mode 2: both from one pass (the loss coefficients known in advance).
// Otherwise Phi itself is never written.
//
// Two sample tiles per tile (TA = 3; the full rounds of tiles of CTA
// pairs): a pair computes 256 observables x 512 samples against each A stage,
// in two M256 x N256 accumulators that fill TMEM (columns 0..255, 256..511).
// A_hi / A_lo then live in shared memory beside the two B operands, a stage
// takes sixteen MMAs, and the A expansion per flop halves. The running sums
// of the accumulation chunks go to a per-CTA buffer in global memory (it
// stays in L2). The double tiles of a last, partial round run as a balanced
// split (TcArgs::skW): their bits stages, end to end, in one equal range per
// CTA pair, each range's piece of a tile a split part that k_split_reduce adds
// up; or, without room for its scratch, as single tiles (TcArgs::dtmap), whose
// last round is split the same way.
//
// Dense form (mode 3, A by TMA): out = (A_hi + A_lo) (1 - 2 B_bits)^T for a
// dense split-BF16 matrix A brought in by TMA and a +-1 operand expanded from
// bits as above, the FP32 accumulator stored as is (FP32 or FP64). The
// low-order form's pair contractions M = C S and H = (s o V) S^T use it.
//
// Gradient contraction (Sec. 2.4, backward of eq. Emat), two kernels:
//  - k_grad_pair (default): CTA pairs in the transposed orientation,
//    D[j][a] = sum_i S_Z[i][j] W[a][i] over 256 gates x 256 observables per
//    tile, K = samples in 128-wide stages, the +-1 operand written into TMEM
//    from P_Z^T bits, W_hi / W_lo by TMA; the epilogue masks by 2 P_A[a][j]
//    (bits of P_A^T) and sums over the tile's observables per gate row
//    (description at the kernel);
//  - k_tc<GRAD> (IQP_GRAD_PAIR=0): one CTA per 128 observables x 256 gates,
//    W tiles by TMA as A, the +-1 operand expanded into shared memory from
//    P_Z^T, reduced over observables with a warp reduce-scatter.
// Both write FP64 partials per (observable tile, gate) that k_grad_reduce
// sums in a fixed order.
//
// Accumulation: the tensor core's FP32 accumulation rounds toward zero, so a
// single accumulator over ~10^4 K-steps shrinks |Phi| by ~1e-4 relative. Each
// tile therefore accumulates in chunks of `chunk` K-stages: a chunk starts a
// fresh accumulator (TMEM columns 0..255) and, when it completes, the
// producer warps add it into an FP32 running sum with round-to-nearest adds
// (TMEM columns 256..511, or shared memory when A occupies those columns, or
// global memory in the two-sample-tile form).
// The epilogue reads accumulator + running sum. The pair gradient reduces
// every chunk into its FP64 per-gate partials instead.
//
// CTA pairs: with CG = 2 the kernels run as clusters of two CTAs on two SMs.
// A phase tile is 256 observables x 256 samples; each CTA holds 128
// observables' A rows and half (128 rows) of the B operand, and the even CTA
// issues M256 x N256 pair MMAs (cta_group::2) that read both CTAs' operands
// and write 128 accumulator rows into each CTA's TMEM. Per SM this halves the
// B operand's expansion work and the tensor core's B reads. Both CTAs'
// producer warps arrive on the even CTA's stage barrier (the odd CTA's through
// one forwarding thread); stage and chunk completions are signalled to both
// CTAs by one pair commit.
//
// Every wait is bounded (globaltimer); on expiry the CTA records
// IQP_ERR_TIMEOUT, drains its in-flight copies and MMAs, frees TMEM and exits.
#include <cuda.h>

#include <cstdlib>

#include "common.cuh"

namespace iqp {

uint64_t default_spin_limit_ns();
uint32_t check_word_tc() { return take_check_word(); }

namespace {

constexpr int TM = 128;      // accumulator rows (observables) per CTA
constexpr int TN = 256;      // accumulator columns (samples or gates) per tile
constexpr int KS = 64;       // K per operand stage
constexpr int KB = 256;      // K per bits stage
constexpr int NBITS = 2;     // bits stages
constexpr int NGEN = 16;     // producer / epilogue warps (4 per scheduler)
constexpr int kThreads = 64 + NGEN * 32;
constexpr int kRowsPerPass = NGEN * 32 / 8;   // operand rows expanded per pass (8 chunks per row)
constexpr int kGroupCols = TN / (NGEN / 4);   // accumulator columns per epilogue warp
constexpr int kGroupLoads = kGroupCols / 32;
constexpr uint32_t kTmemCols = 512;   // accumulator (0..255) + running sum (256..511)
constexpr uint32_t kSumCol = 256;
// A-in-TMEM form: columns 256..511 hold the A operand of the four operand
// stages instead of the running sum: stage os at 256 + 64 os; its 16-gate
// K step k (0..3) has A_hi at + 16 k and A_lo at + 16 k + 8 (8 columns of
// two BF16 each), so one warp's share is 16 contiguous columns.
constexpr uint32_t kAColBase = 256;
constexpr uint32_t kAColStage = 64;
constexpr int kMaxOp = 4;
constexpr int kWPrefetch = 8;  // gradient: W tiles prefetched into L2 this many stages ahead

// Shared-memory layout for a CTA group of CG CTAs (CG = 1 or 2). ATM: the A
// operand (hi / lo) lives in TMEM, so an operand stage in shared memory holds
// only B, and the running sum of the accumulation chunks moves from TMEM to
// shared memory (TM x TN FP32, as float4 groups of 4 columns, row-minor).
// DT (two sample tiles per tile): an operand stage holds A_hi, A_lo and the
// B operands of both sample tiles, the two accumulators fill TMEM, and the
// running sums live in global memory.
// X3 (FP32 form, three planes of A): an operand stage holds the three A
// planes and B; the two accumulators fill TMEM like DT's.
template <int CG, bool ATMA, bool ATM = false, bool DT = false, bool X3 = false>
struct Cfg {
    static constexpr int TNB = TN / CG;      // B rows this CTA holds (per sample tile)
    static constexpr int NOP = DT || X3 ? 3 : (CG == 2 || ATM) ? 4 : (ATMA ? 3 : 2);  // operand stages
    // Operand stage: A_hi (128 x 128 B), A_lo, B (TNB x 128 B) [DT: then the
    // second sample tile's B]; ATM: B only.
    static constexpr uint32_t OP_A_HI = 0, OP_A_LO = 16384, OP_A_3 = 32768;
    static constexpr uint32_t OP_B = ATM ? 0 : X3 ? 49152 : 32768;
    static constexpr uint32_t OP_B1 = OP_B + TNB * 128;
    static constexpr uint32_t OP_BYTES = OP_B + (DT ? 2 : 1) * TNB * 128;
    // Bits stage: A bits (128 rows x 32 B), B bits (TNB rows x 32 B) [DT: then
    // the second sample tile's], c_hi, c_lo.
    static constexpr uint32_t BT_A = 0, BT_B = 4096, BT_B1 = BT_B + TNB * 32;
    static constexpr uint32_t BT_CHI = BT_B + (DT ? 2 : 1) * TNB * 32, BT_CLO = BT_CHI + 512;
    static constexpr uint32_t BT_C3 = BT_CLO + 512;  // X3: the third plane of 2 theta
    static constexpr uint32_t BT_BYTES = X3 ? BT_C3 + 1024 : BT_CLO + 512;
    static constexpr uint32_t SM_OP = 0;
    static constexpr uint32_t SM_BITS = SM_OP + NOP * OP_BYTES;
    static constexpr uint32_t SM_BAR = SM_BITS + NBITS * BT_BYTES;
    static constexpr uint32_t SM_RED = SM_BAR + 256;   // 4 x 256 floats (grad epilogue)
    static constexpr uint32_t SM_SUM = SM_RED + 4 * 256 * 4;  // ATM: running sum
    static constexpr uint32_t SM_END = SM_SUM + (ATM ? TM * TN * 4 : 0);
    static constexpr uint32_t SMEM = SM_END + 1024;     // + alignment slack
    static constexpr uint32_t IDESC = idesc_bf16(TM * CG, TN);
    static_assert(OP_BYTES % 1024 == 0 && BT_BYTES % 1024 == 0 && SM_SUM % 16 == 0, "stage alignment");
    static_assert(SMEM <= 232448, "shared memory");
};

// Tile t -> (row block tm, column block tc), walking `gm` row blocks of one
// column block before the next column block (the last group may be
// shorter). The CTAs running at once then share gm row panels and about
// (CTAs / gm) column panels, which stay in L2: each column panel is read
// from DRAM once per group instead of once per row block.
__device__ __forceinline__ void tile_coords(int64_t t, int64_t tiles_m, int64_t tiles_nc, int64_t gm, int64_t &tm,
                                            int64_t &tc) {
    const int64_t per = gm * tiles_nc;
    const int64_t g = t / per;
    const int64_t r = t - g * per;
    const int64_t rows = tiles_m - g * gm < gm ? tiles_m - g * gm : gm;
    tm = g * gm + r % rows;
    tc = r / rows;
}

struct TcArgs;
__device__ __forceinline__ void tile_rc(int64_t t, const TcArgs &a, int64_t &tm, int64_t &tc);

struct TcArgs {
    int64_t l, s, m;
    int64_t nks;          // operand stages per tile
    int64_t chunk;        // operand stages per accumulation chunk
    int64_t tiles_m, tiles_n;
    int64_t group_m;      // row blocks per tile group (L2 rasterisation)
    const __nv_bfloat16 *chi, *clo;
    int64_t mpad;          // length of chi / clo
    double2 *part;
    int64_t nparts;
    const double *alpha, *beta;
    __nv_bfloat16 *whi, *wlo;
    int64_t ldw;
    const uint32_t *pa32;  // P_A, for the gradient mask
    int64_t ldp32;
    double *gpart;
    float *out;            // mode 0: Phi; mode 3: the accumulator (+ dvec[row], sign bits of zt32)
    int64_t ldo;
    // mode 3: K pieces (1 = whole), floats between their outputs, addend and sign bits (null = neither)
    int kparts;
    int64_t out_part;
    const float *dvec;
    const uint32_t *zt32;
    int64_t ldzt32;
    // Work units of this launch: the tiles, whole (nunits tiles); or, for a
    // split launch, nunits parts of the tiles from `whole` on (phase modes
    // only; see skW).
    int64_t nunits, whole;
    float *skp;            // split parts' partial accumulators, TM x TN FP32 per (part, CTA of the pair)
    uint32_t *status;
    uint64_t limit_ns;
    int serp;              // phase, whole tiles: every other round of tiles walks the gates backwards
    // X3: the third plane of 2 theta, W as FP32 (l x ldw) and the largest |W| of each row (float bits)
    const __nv_bfloat16 *c3;
    float *wf;
    uint32_t *wmax;
    // Two-sample-tile phase kernels: per CTA, the running sums of both
    // accumulators (2 x TM x TN FP32 as float4 groups of 4 columns, row-minor).
    float4 *gsum;
    // Single tiles taken from double tiles (the last round of a two-tile
    // phase): tile t is half t % 2 of double tile dbase + t / 2 of a
    // tiles_m x tiles_n2 walk.
    int dtmap;
    int64_t dbase, tiles_n2;
    // Balanced split of a last round (split units only): the skW
    // bits stages of the tiles from `whole` on, laid end to end, are cut into
    // skP equal contiguous ranges, one per CTA group; unit u is piece u / skP
    // of range u % skP (the part of the range inside one tile; empty when the
    // range has fewer pieces). Range g's piece of tile whole + t takes slot g + t:
    // one after the other in a tile, and from one piece to the next the range
    // or the tile goes up, so that they fit skP + tiles - 1 slots. (With as many
    // slots per tile as the most that one tile takes, 56 double tiles over 76
    // ranges had no room and ran as 56 ranges: n = 5000, 10^6 gates, 4096 x 16384,
    // phase 123 -> 131 ms.)
    int64_t skW, skP;
    int64_t skcap;  // floats of split-part scratch at skp
};

__device__ __forceinline__ void tile_rc(int64_t t, const TcArgs &a, int64_t &tm, int64_t &tc) {
    if (a.dtmap) {
        int64_t tc2;
        tile_coords(a.dbase + t / 2, a.tiles_m, a.tiles_n2, a.group_m, tm, tc2);
        tc = 2 * tc2 + (t & 1);
        return;
    }
    tile_coords(t, a.tiles_m, a.tiles_n, a.group_m, tm, tc);
}

struct Bars {
    uint64_t bits_full[NBITS], bits_empty[NBITS], op_full[kMaxOp], op_empty[kMaxOp], w_full[kMaxOp],
        peer_full[kMaxOp], acc_full, drain, red_full;
    uint32_t tmem_slot;
    int abort_flag;
};

// Work unit u -> its tile, its operand-stage range [ks0, ks1) and, for a
// part of a split tile, its slot v (-1 for a whole tile). SPL = false: the
// units are the tiles, whole. SPL = true: unit u is a piece of the balanced
// split (see skW); the parts cover a tile's stages in ranges of whole bits
// stages (KB / KS operand stages), in order.
// KP (the dense form): unit u is K piece u / whole of tile u % whole, v the piece.
template <bool SPL, bool KP = false>
__device__ __forceinline__ void unit_of(int64_t u, const TcArgs &a, int nks, int64_t &tile, int &ks0, int &ks1,
                                        int64_t &v) {
    if (KP) {
        tile = u % a.whole;
        v = u / a.whole;
        const int64_t nkb = (nks + KB / KS - 1) / (KB / KS);
        ks0 = (KB / KS) * (int)(v * nkb / a.kparts);
        const int e = (KB / KS) * (int)((v + 1) * nkb / a.kparts);
        ks1 = e < nks ? e : nks;
        return;
    }
    if (!SPL) {
        tile = u;
        ks0 = 0;
        ks1 = nks;
        v = -1;
        return;
    }
    const int64_t nkb = (nks + KB / KS - 1) / (KB / KS);
    const int64_t g = u % a.skP, k = u / a.skP;
    const int64_t A = g * a.skW / a.skP, B = (g + 1) * a.skW / a.skP;
    const int64_t start = k == 0 ? A : (A / nkb + k) * nkb;
    tile = a.whole;
    ks0 = ks1 = 0;
    v = -1;
    if (start >= B) return;  // this range has no piece k
    const int64_t tt = start / nkb;
    const int64_t end = B < (tt + 1) * nkb ? B : (tt + 1) * nkb;
    tile = a.whole + tt;
    ks0 = (KB / KS) * (int)(start - tt * nkb);
    const int64_t e = (KB / KS) * (end - tt * nkb);
    ks1 = e < nks ? (int)e : nks;
    v = g + tt;
}

// Split tile tt (from `whole` on): the number of its parts and the slot of the first.
__device__ __forceinline__ void part_info(int64_t tt, const TcArgs &a, int nks, int64_t &np, int64_t &base) {
    const int64_t nkb = (nks + KB / KS - 1) / (KB / KS);
    const int64_t g0 = ((tt * nkb + 1) * a.skP - 1) / a.skW;
    const int64_t g1 = ((tt + 1) * nkb * a.skP - 1) / a.skW;
    np = g1 - g0 + 1;
    base = g0 + tt;
}

__device__ __forceinline__ uint8_t *aligned_smem(uint8_t *raw) {
    const uint32_t a = smem_u32(raw);
    return raw + ((1024u - (a & 1023u)) & 1023u);
}

// Expand one 64-gate sub-stage q of a bits stage into the B operand
// (ROWS rows, +-1 BF16). Thread gt handles chunk gt%8 of rows
// gt/8 + kRowsPerPass*k.
template <int ROWS>
__device__ __forceinline__ void expand_b(const uint8_t *bits, uint8_t *opB, int q, int gt) {
    const uint32_t c = gt & 7;
    const uint32_t sub = (uint32_t)q * 8u + (c >> 2) * 4u;  // byte offset of the u32 holding chunk c
    const uint32_t sh = (c & 3u) * 8u;
#pragma unroll
    for (int k = 0; k < ROWS / kRowsPerPass; ++k) {
        const uint32_t row = (uint32_t)(gt >> 3) + (uint32_t)kRowsPerPass * k;
        const uint32_t w = *reinterpret_cast<const uint32_t *>(bits + row * 32u + sub);
        const uint4 v = expand_pm1((w >> sh) & 0xFFu);
        *reinterpret_cast<uint4 *>(opB + swz128(row, c)) = v;
    }
}

// Expand sub-stage q into A_hi / A_lo (128 rows): hi_j / lo_j where the
// parity bit is set, 0 elsewhere.
__device__ __forceinline__ void expand_a(const uint8_t *bitsA, const uint8_t *chi, const uint8_t *clo, uint8_t *opHi,
                                         uint8_t *opLo, int q, int gt) {
    const uint32_t c = gt & 7;
    const uint4 h = *reinterpret_cast<const uint4 *>(chi + (uint32_t)q * 128u + c * 16u);
    const uint4 lo = *reinterpret_cast<const uint4 *>(clo + (uint32_t)q * 128u + c * 16u);
    const uint32_t sub = (uint32_t)q * 8u + (c >> 2) * 4u;
    const uint32_t sh = (c & 3u) * 8u;
#pragma unroll
    for (int k = 0; k < TM / kRowsPerPass; ++k) {
        const uint32_t row = (uint32_t)(gt >> 3) + (uint32_t)kRowsPerPass * k;
        const uint32_t w = *reinterpret_cast<const uint32_t *>(bitsA + row * 32u + sub);
        const uint4 mk = expand_mask((w >> sh) & 0xFFu);
        const uint32_t off = swz128(row, c);
        *reinterpret_cast<uint4 *>(opHi + off) = make_uint4(h.x & mk.x, h.y & mk.y, h.z & mk.z, h.w & mk.w);
        *reinterpret_cast<uint4 *>(opLo + off) = make_uint4(lo.x & mk.x, lo.y & mk.y, lo.z & mk.z, lo.w & mk.w);
    }
}

// The X3 form of expand_a: the three planes of 2 theta (512 bytes apart from
// `c` on) masked into three A planes 16384 bytes apart from opA on.
__device__ __forceinline__ void expand_a3(const uint8_t *bitsA, const uint8_t *cp, uint8_t *opA, int q, int gt) {
    const uint32_t c = gt & 7;
    uint4 v[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) v[p] = *reinterpret_cast<const uint4 *>(cp + 512u * p + (uint32_t)q * 128u + c * 16u);
    const uint32_t sub = (uint32_t)q * 8u + (c >> 2) * 4u;
    const uint32_t sh = (c & 3u) * 8u;
#pragma unroll
    for (int k = 0; k < TM / kRowsPerPass; ++k) {
        const uint32_t row = (uint32_t)(gt >> 3) + (uint32_t)kRowsPerPass * k;
        const uint32_t w = *reinterpret_cast<const uint32_t *>(bitsA + row * 32u + sub);
        const uint4 mk = expand_mask((w >> sh) & 0xFFu);
        uint8_t *dst = opA + swz128(row, c);
#pragma unroll
        for (int p = 0; p < 3; ++p)
            *reinterpret_cast<uint4 *>(dst + 16384 * p) =
                make_uint4(v[p].x & mk.x, v[p].y & mk.y, v[p].z & mk.z, v[p].w & mk.w);
    }
}

// Bounded wait polled by every lane (each needs the acquire), with the outcome
// made warp-uniform so that a give-up never splits a warp.
__device__ __forceinline__ bool wait_warp(uint64_t *b, uint32_t parity, volatile int *abort_flag, uint32_t *status,
                                          uint64_t lim) {
    const bool got = mbar_wait(b, parity, abort_flag, status, lim);
    return __all_sync(0xFFFFFFFFu, got);
}

// wait_warp with cluster-scope acquire (the barrier completes from the peer CTA too).
__device__ __forceinline__ bool wait_warp_cluster(uint64_t *b, uint32_t parity, volatile int *abort_flag,
                                                  uint32_t *status, uint64_t lim) {
    const bool got = mbar_wait_cluster(b, parity, abort_flag, status, lim);
    return __all_sync(0xFFFFFFFFu, got);
}

// 32 columns of the tile at TMEM address `t`: the current accumulator plus,
// when the tile was accumulated in more than one chunk, the running sum (in
// TMEM at t + kSumCol, or, when `ss` is given, in shared memory: the 8 float4
// groups of these columns for this thread's row at ss[0], ss[TM], ...).
__device__ __forceinline__ void load_sum32(uint32_t t, bool chunked, uint32_t (&r)[32], const float4 *ss = nullptr) {
    tmem_ld32(t, r);
    if (chunked) {
        if (ss != nullptr) {
#pragma unroll
            for (int e4 = 0; e4 < 8; ++e4) {
                const float4 v = ss[e4 * TM];
                r[4 * e4] = __float_as_uint(__uint_as_float(r[4 * e4]) + v.x);
                r[4 * e4 + 1] = __float_as_uint(__uint_as_float(r[4 * e4 + 1]) + v.y);
                r[4 * e4 + 2] = __float_as_uint(__uint_as_float(r[4 * e4 + 2]) + v.z);
                r[4 * e4 + 3] = __float_as_uint(__uint_as_float(r[4 * e4 + 3]) + v.w);
            }
            return;
        }
        uint32_t acc[32];
        tmem_ld32(t + kSumCol, acc);
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) + __uint_as_float(acc[e]));
    }
}

// X3: 32 columns of the tile at TMEM address `t`, the exact accumulator of
// plane 0 plus the accumulator of planes 1 and 2 (kSumCol further on) plus,
// where the tile was accumulated in more than one chunk, the running sum `ss`
// (as in load_sum32).
__device__ __forceinline__ void load_sum32_x3(uint32_t t, const float4 *ss, uint32_t (&r)[32]) {
    load_sum32(t, true, r);
    if (ss != nullptr) {
#pragma unroll
        for (int e4 = 0; e4 < 8; ++e4) {
            const float4 v = ss[e4 * TM];
            r[4 * e4] = __float_as_uint(__uint_as_float(r[4 * e4]) + v.x);
            r[4 * e4 + 1] = __float_as_uint(__uint_as_float(r[4 * e4 + 1]) + v.y);
            r[4 * e4 + 2] = __float_as_uint(__uint_as_float(r[4 * e4 + 2]) + v.z);
            r[4 * e4 + 3] = __float_as_uint(__uint_as_float(r[4 * e4 + 3]) + v.w);
        }
    }
}

// A-in-TMEM form: this warp's share of one 64-gate operand stage of A, the 16
// gates [16 g, 16 g + 16) (K step g) for the row of TMEM lane
// (32 quarter + lane): hi_j (A_hi) and lo_j (A_lo) where bit j of `b16` (the
// row's parities of these gates) is set, 0 elsewhere, two BF16 per 32-bit
// column (the lower gate in the low half). chi / clo: the bits stage's hi /
// lo split of 2 theta; q: the operand stage within the bits stage. `t` is the
// TMEM address of the warp's 16 columns: A_hi in the first 8, A_lo in the
// next 8, stored at once.
__device__ __forceinline__ void expand_a_tmem(uint32_t b16, const uint8_t *chi, const uint8_t *clo, int q, int g,
                                              uint32_t t) {
    const uint32_t off = (uint32_t)q * 128u + (uint32_t)g * 32u;
    const uint4 h0 = *reinterpret_cast<const uint4 *>(chi + off);
    const uint4 h1 = *reinterpret_cast<const uint4 *>(chi + off + 16);
    const uint4 l0 = *reinterpret_cast<const uint4 *>(clo + off);
    const uint4 l1 = *reinterpret_cast<const uint4 *>(clo + off + 16);
    const uint4 m0 = expand_mask(b16 & 0xFFu), m1 = expand_mask((b16 >> 8) & 0xFFu);
    const uint32_t v[16] = {h0.x & m0.x, h0.y & m0.y, h0.z & m0.z, h0.w & m0.w,
                            h1.x & m1.x, h1.y & m1.y, h1.z & m1.z, h1.w & m1.w,
                            l0.x & m0.x, l0.y & m0.y, l0.z & m0.z, l0.w & m0.w,
                            l1.x & m1.x, l1.y & m1.y, l1.z & m1.z, l1.w & m1.w};
    tmem_st16(t, v);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(a));
    const uint32_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(b));
    return lo | (hi << 16);
}

// W = sin Phi (alpha_a + beta_a cos Phi) as BF16 hi/lo (l x ldw) from a Phi
// the statistics pass kept (l x ldphi FP32, columns < s), with the
// arithmetic of the recompute epilogue, so W is the same bit for bit. Four
// samples per thread; columns >= s get zeros (the gradient's tensor map ends
// at s).
__global__ void __launch_bounds__(256) k_w_from_phi(const float *__restrict__ phi, int64_t ldphi, int64_t ldw,
                                                    int64_t l, int64_t s,
                                                    const double *__restrict__ alpha,
                                                    const double *__restrict__ beta, __nv_bfloat16 *__restrict__ whi,
                                                    __nv_bfloat16 *__restrict__ wlo) {
    pdl_sync();
    const int64_t per_row = ldw / 4;
    const int64_t total = l * per_row;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = g / per_row, i0 = (g - row * per_row) * 4;
        if (i0 >= s) continue;
        if (!IQP_IN(row, l, 40) || !IQP_IN(row * ldphi + i0 + 3, l * ldphi, 41) || !IQP_IN(row * ldw + i0 + 3, l * ldw, 42))
            continue;
        const float al = (float)alpha[row];
        const float be = beta ? (float)beta[row] : 0.f;
        const float4 f = *reinterpret_cast<const float4 *>(phi + row * ldphi + i0);
        const float v[4] = {f.x, f.y, f.z, f.w};
        uint32_t ph[2], pl[2];
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
            float s0, k0, s1, k1;
            sincosf(v[e], &s0, &k0);
            sincosf(v[e + 1], &s1, &k1);
            const float w0 = i0 + e < s ? s0 * (al + be * k0) : 0.f;
            const float w1 = i0 + e + 1 < s ? s1 * (al + be * k1) : 0.f;
            const float h0 = __bfloat162float(__float2bfloat16_rn(w0));
            const float h1 = __bfloat162float(__float2bfloat16_rn(w1));
            ph[e / 2] = pack_bf16x2(h0, h1);
            pl[e / 2] = pack_bf16x2(w0 - h0, w1 - h1);
        }
        *reinterpret_cast<uint2 *>(whi + row * ldw + i0) = make_uint2(ph[0], ph[1]);
        *reinterpret_cast<uint2 *>(wlo + row * ldw + i0) = make_uint2(pl[0], pl[1]);
    }
}

// ---- FP32 form: three BF16 planes of an FP32 value
// A value x is taken apart on the grid 2^E of its operand (2 theta as a whole,
// or one row of W): plane 0 is x rounded to a multiple of 2^E, or, from 256 grid
// steps on, to BF16's 8 bits, which is a multiple of 2^E too; planes 1 and 2 are
// the BF16 head and tail of the rest (at most 2^(E-1) or 2^-9 |x|). E is the
// least for which the |plane 0| of one accumulation chunk add up to at most 2^24
// grid steps, so that its sums against +-1 are integers that the tensor core's FP32
// accumulator holds exactly. The other two planes have an accumulator of their
// own, which truncates like any, at 2^-9 of the sum where plane 0 holds the values
// and at the sum itself for the values below the grid.
// Those decide the chunk and the grid. With one chunk of 65536 gates and
// 2^E = 2^-8 of the largest |2 theta|, one parameter 500 times the others left them
// all below the grid. With the sum of |2 theta| over a chunk of 8192 gates in
// place of the maximum, only values below about 2^-11 of its mean are, and the
// truncation is an eighth. Measured against FP64 (65536 gates, 256 x 19456, one
// parameter near pi / 2, the others of 0.003): estimates off by 2.2e-5 -> 1.3e-8, gradient
// 6.2e-5 -> 1.0e-7; every other parameter large: 1.1e-5 -> 1.3e-8, 6.1e-5 -> 5.1e-7;
// SIMT kernels 3.7e-8 and 3.9e-6. Values below 2^-11 of the mean have up to 1e-5 relative
// in a model of the arithmetic (16 terms per step, truncated to 24 bits), in a
// phase of at most 0.2 (2 theta is at most pi here): 2e-6.
// Three products per contraction, bound like the split form by producing the
// masked planes (one- and two-body circuit, n = 300, 1000 observables, 10^4
// samples): its autograd step takes 2.95 ms (2.91 with one chunk; error 1.2e-7),
// against 59.5 ms on the FP32 FMA pipe (0.54 of its peak; 3.3e-6).
struct X3Grid {
    float step, inv, big;  // 2^E, 2^-E, 2^(E+8)
};
// |values| that add up to at most 2^bits bound.
__device__ __forceinline__ X3Grid x3_grid(float bound, int bits) {
    int e = (int)((__float_as_uint(bound) >> 23) & 255u) - 126 + bits - 24;  // bound 2^bits < 2^(e + 24)
    e = e < -120 ? -120 : (e > 104 ? 104 : e);
    X3Grid g;
    g.step = __uint_as_float((uint32_t)(e + 127) << 23);
    g.inv = __uint_as_float((uint32_t)(127 - e) << 23);
    g.big = 256.f * g.step;
    return g;
}
__device__ __forceinline__ void x3_planes(float x, const X3Grid &g, float (&p)[3]) {
    // scaling by powers of two and both differences are exact
    p[0] = fabsf(x) >= g.big ? __bfloat162float(__float2bfloat16_rn(x)) : rintf(x * g.inv) * g.step;
    const float rest = x - p[0];
    p[1] = __bfloat162float(__float2bfloat16_rn(rest));
    p[2] = rest - p[1];
}

// 2 theta reduced to [-pi, pi] (the phase enters only as cos and sin, and
// every term is +-c_j, so multiples of 2 pi drop out); the reduction bounds
// the grid's maximum.
__device__ __forceinline__ float x3_angle(float theta) {
    const float c = 2.0f * theta;
    if (!(fabsf(c) > 3.1415927f)) return c;
    const double d = (double)c;
    return (float)(d - 6.283185307179586476925 * rint(d * 0.15915494309189533577));
}

// Sum of the finite |2 theta_j| over the gates first + threadIdx.x, + 256, ... below end, over the block (fixed order).
__device__ __forceinline__ float x3_block_sum(const float *__restrict__ theta, int64_t first, int64_t end) {
    __shared__ float red[8];
    float v = 0.f;
    for (int64_t j = first + threadIdx.x; j < end; j += 256) {
        const float c = fabsf(x3_angle(theta[j]));
        if (c <= 4.f) v += c;
    }
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, w);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = red[0];
    for (int w = 1; w < 8; ++w) v += red[w];
    return v;
}

// bsum[b] = sum of |2 theta| over the gates of block b (kX3Gates of them).
__global__ void __launch_bounds__(256) k_x3_csum(const float *__restrict__ theta, int64_t m, float *__restrict__ bsum) {
    pdl_sync();
    const int64_t j0 = blockIdx.x * (int64_t)kX3Gates;
    const float v = x3_block_sum(theta, j0, j0 + kX3Gates < m ? j0 + kX3Gates : m);
    if (threadIdx.x == 0) bsum[blockIdx.x] = v;
}

// The planes of 2 theta (mpad BF16 each, zero beyond m), on the grid of the
// block sums (nb of them; nb = 0: each block takes the sum itself, which saves
// a launch where the gates are one chunk). A chunk is kX3Gates consecutive
// gates that may begin anywhere, so it lies in two blocks at most. Row maxima
// wmax (l words, or none) start at zero for the phase that follows.
__global__ void __launch_bounds__(256) k_x3_theta(const float *__restrict__ theta, int64_t m, int64_t mpad,
                                                  const float *__restrict__ bsum, int64_t nb,
                                                  __nv_bfloat16 *__restrict__ planes, uint32_t *__restrict__ wmax,
                                                  int64_t l) {
    pdl_sync();
    float sum = 0.f;
    if (nb == 0) {
        sum = x3_block_sum(theta, 0, m);
    } else {
        __shared__ uint32_t most;
        if (threadIdx.x == 0) most = 0u;
        __syncthreads();
        float v = 0.f;
        for (int64_t b = threadIdx.x; b < nb; b += 256) v = fmaxf(v, bsum[b]);
        atomicMax(&most, __float_as_uint(v));  // non-negative floats order like their bits
        __syncthreads();
        sum = 2.f * __uint_as_float(most);
    }
    const X3Grid g = x3_grid(1.01f * sum, 0);  // rounding adds 2^-9 and half a step per gate, 2^-12 of 2^24 steps
    for (int64_t j = blockIdx.x * (int64_t)256 + threadIdx.x; j < mpad; j += (int64_t)gridDim.x * 256) {
        float p[3] = {0.f, 0.f, 0.f};
        if (j < m) x3_planes(x3_angle(theta[j]), g, p);
        if (!IQP_IN(j, mpad, 61)) continue;
#pragma unroll
        for (int k = 0; k < 3; ++k) planes[k * mpad + j] = __float2bfloat16_rn(p[k]);
    }
    if (wmax != nullptr)
        for (int64_t a = blockIdx.x * (int64_t)256 + threadIdx.x; a < l; a += (int64_t)gridDim.x * 256) wmax[a] = 0u;
}

// W = sin Phi (alpha + beta cos Phi) (FP32) and its row maxima from a kept Phi, as
// the phase's own epilogue forms them (MODE 1): 2048 samples of a row per block.
// W may be Phi itself (ldphi = ldw): each thread replaces what it read. 10^7
// samples take 20 us, the second contraction they replace 1390 (45150 gates).
__global__ void __launch_bounds__(256) k_x3_w(const float *phi, int64_t ldphi, float *W, int64_t ldw, int64_t l, int64_t s,
                                              const double *__restrict__ alpha, const double *__restrict__ beta,
                                              uint32_t *__restrict__ wmax) {
    pdl_sync();
    const int64_t per_row = cdiv(s, 2048), total = l * per_row;
    for (int64_t t = blockIdx.x; t < total; t += gridDim.x) {
        const int64_t a = t / per_row, i0 = (t - a * per_row) * 2048;
        const float al = (float)alpha[a], be = beta ? (float)beta[a] : 0.f;
        float mx = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int64_t i = i0 + 1024 * k + 4 * threadIdx.x;  // rows are padded to whole fours
            if (i >= s || !IQP_IN(a * ldw + i + 3, l * ldw, 64) || !IQP_IN(a * ldphi + i + 3, l * ldphi, 65)) continue;
            const float4 p = *reinterpret_cast<const float4 *>(phi + a * ldphi + i);
            float w[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float sn, cn;
                sincosf(w[e], &sn, &cn);
                w[e] = i + e < s ? sn * (al + be * cn) : 0.f;
                if (fabsf(w[e]) <= 3.4e38f) mx = fmaxf(mx, fabsf(w[e]));
            }
            *reinterpret_cast<float4 *>(W + a * ldw + i) = make_float4(w[0], w[1], w[2], w[3]);
        }
        const uint32_t mb = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx));
        if ((threadIdx.x & 31) == 0 && mb != 0u) atomicMax(wmax + a, mb);
    }
}

// The planes of W (l x ldw BF16 each) from W as FP32 and its row maxima, eight
// samples per thread; columns >= s are left as they are (the gradient's tensor
// maps end at s).
__global__ void __launch_bounds__(256) k_x3_wsplit(const float *__restrict__ W, int64_t ldw, int64_t l, int64_t s,
                                                   const uint32_t *__restrict__ wmax, __nv_bfloat16 *__restrict__ planes) {
    pdl_sync();
    const int64_t per_row = cdiv(s, 8), total = l * per_row;
    for (int64_t t = blockIdx.x * (int64_t)256 + threadIdx.x; t < total; t += (int64_t)gridDim.x * 256) {
        const int64_t a = t / per_row, i0 = (t - a * per_row) * 8;  // ldw is a multiple of 64: whole words
        if (!IQP_IN(a * ldw + i0 + 7, l * ldw, 62)) continue;
        const X3Grid g = x3_grid(__uint_as_float(wmax[a]), kX3SampleBits);
        const float4 u = *reinterpret_cast<const float4 *>(W + a * ldw + i0);
        const float4 v = *reinterpret_cast<const float4 *>(W + a * ldw + i0 + 4);
        const float x[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        uint32_t o[3][4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            float p[3], q[3];
            x3_planes(x[e], g, p);
            x3_planes(x[e + 1], g, q);
#pragma unroll
            for (int k = 0; k < 3; ++k) o[k][e / 2] = pack_bf16x2(p[k], q[k]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
            *reinterpret_cast<uint4 *>(planes + (k * l + a) * ldw + i0) = make_uint4(o[k][0], o[k][1], o[k][2], o[k][3]);
    }
}

// ------------------------------------------------------------------ kernel
// W of eight consecutive samples i.. of observable row: BF16 hi/lo rows, or (X3)
// FP32, returning the largest finite |W| among those below s.
__device__ __forceinline__ void store_w8(const TcArgs &args, int64_t row, int64_t i, const float (&w)[8]) {
    uint32_t ph[4], pl[4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
        const float h0 = __bfloat162float(__float2bfloat16_rn(w[e])), h1 = __bfloat162float(__float2bfloat16_rn(w[e + 1]));
        ph[e / 2] = pack_bf16x2(h0, h1);
        pl[e / 2] = pack_bf16x2(w[e] - h0, w[e + 1] - h1);
    }
    __nv_bfloat16 *dh = args.whi + row * args.ldw + i, *dl = args.wlo + row * args.ldw + i;
    if (i + 8 <= args.s) {
        *reinterpret_cast<uint4 *>(dh) = make_uint4(ph[0], ph[1], ph[2], ph[3]);
        *reinterpret_cast<uint4 *>(dl) = make_uint4(pl[0], pl[1], pl[2], pl[3]);
        return;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e)
        if (i + e < args.s) {
            reinterpret_cast<uint16_t *>(dh)[e] = (uint16_t)(ph[e / 2] >> ((e & 1) * 16));
            reinterpret_cast<uint16_t *>(dl)[e] = (uint16_t)(pl[e / 2] >> ((e & 1) * 16));
        }
}
__device__ __forceinline__ float store_wf8(const TcArgs &args, int64_t row, int64_t i, const float (&w)[8]) {
    float mx = 0.f;
    float *d = args.wf + row * args.ldw + i;
    if (i + 8 <= args.s) {
        *reinterpret_cast<float4 *>(d) = make_float4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<float4 *>(d + 4) = make_float4(w[4], w[5], w[6], w[7]);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float v = fabsf(w[e]);
        if (i + e >= args.s) continue;
        if (v <= 3.4e38f) mx = fmaxf(mx, v);
        if (i + 8 > args.s) d[e] = w[e];
    }
    return mx;
}

// Merges 32 cosines (columns 32 c .. of a group with nvalid valid columns) into
// (S, M2): their own sum and squared deviations from registers, then the merge of
// the two means (Chan et al.). Each cosine is taken once: the epilogue took it
// once for the sum and again for the deviations from the whole group's mean,
// half of its instructions, with no product under way meanwhile where a CTA pair
// has one tile (all of k_tc, cold: 36 gates, 64 x 1024: 37.6 -> 18.5 us; 3001
// gates, 777 x 2501: 71.6 -> 50.3 us).
__device__ __forceinline__ void merge_cos32(const uint32_t (&r)[32], int c, int nvalid, float &S, float &M2) {
    const int n = nvalid - 32 * c < 32 ? nvalid - 32 * c : 32;
    if (n <= 0) return;
    float s = 0.f, m2 = 0.f;
#pragma unroll
    for (int e = 0; e < 32; ++e) s += e < n ? __uint_as_float(r[e]) : 0.f;
    const float mean = s / (float)n;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
        const float d = __uint_as_float(r[e]) - mean;
        m2 = e < n ? fmaf(d, d, m2) : m2;
    }
    if (c > 0) {  // the columns before are all valid: 32 c of them
        const float before = (float)(32 * c), d = mean - S / before;
        m2 += M2 + d * d * (before * (float)n / (before + (float)n));
        s += S;
    }
    S = s;
    M2 = m2;
}

// r rotated by eight entries: the epilogues take the cosines of eight columns per
// turn of a loop, so that its code is one copy of eight, not 32, which the
// instruction cache holds (k_tc, 36 gates, 64 x 1024: 18.5 -> 14.7 us).
__device__ __forceinline__ void rotate8(uint32_t (&r)[32]) {
    uint32_t t[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) t[e] = r[e];
#pragma unroll
    for (int e = 0; e < 24; ++e) r[e] = r[e + 8];
#pragma unroll
    for (int e = 0; e < 8; ++e) r[24 + e] = t[e];
}

// Values of 32 consecutive columns col0.. of `row`, stored into out
// (row-major, args.ldo elements per row, columns < args.s). Rows start 16-byte
// aligned (ldo a multiple of 4).
__device__ __forceinline__ void store_out32(const TcArgs &args, float *out, int64_t row, int64_t col0,
                                            const uint32_t (&r)[32]) {
    if (!IQP_IN(row * args.ldo + col0, args.l * args.ldo, 45) ||
        !IQP_IN(row * args.ldo + (col0 + 32 <= args.s ? col0 + 31 : args.s - 1), args.l * args.ldo, 46))
        return;
    float *f = out + row * args.ldo + col0;
    if (col0 + 32 <= args.s) {
#pragma unroll
        for (int e = 0; e < 32; e += 4)
            *reinterpret_cast<float4 *>(f + e) = make_float4(__uint_as_float(r[e]), __uint_as_float(r[e + 1]),
                                                             __uint_as_float(r[e + 2]), __uint_as_float(r[e + 3]));
    } else {
        for (int e = 0; e < 32 && col0 + e < args.s; ++e) f[e] = __uint_as_float(r[e]);
    }
}

// Split phase tiles (kept out of line, so that its registers do not weigh on
// the stage loop): this warp's 32 rows x 64 columns of the accumulator (+
// running sum) into its part's slot.
template <bool X3>
__device__ __noinline__ void split_store(float *dst, uint32_t tbase, bool chunked, const float4 *ss0) {
    uint32_t r[32];
#pragma unroll 1
    for (int c = 0; c < kGroupLoads; ++c) {
        if (X3)
            load_sum32_x3(tbase + c * 32, chunked ? ss0 + c * 8 * TM : nullptr, r);
        else
            load_sum32(tbase + c * 32, chunked, r, ss0 != nullptr ? ss0 + c * 8 * TM : nullptr);
#pragma unroll
        for (int e = 0; e < 32; e += 4)
            *reinterpret_cast<float4 *>(dst + c * 32 + e) = make_float4(
                __uint_as_float(r[e]), __uint_as_float(r[e + 1]), __uint_as_float(r[e + 2]), __uint_as_float(r[e + 3]));
    }
}

// The split tiles' epilogue: one warp per (row, 64 columns) of a split tile adds
// the tile's parts up in part order (two columns per lane, 256 coalesced bytes
// per part) and forms what the whole tiles' epilogue forms, over the whole chip.
// With the last part's CTA doing both, a tile of 20 parts cost 0.47 ms of one SM's
// time for 45 us of products (1000 observables x 10^4 samples, 45150 gates).
template <int MODE, bool X3>
__global__ void __launch_bounds__(256) k_split_reduce(const TcArgs args, int CG, int NH, int64_t tiles) {
    pdl_sync();
    const int lane = threadIdx.x & 31;
    const int64_t w = (blockIdx.x * (int64_t)256 + threadIdx.x) >> 5;
    const int group = (int)(w & 3), rl = (int)((w >> 2) & (TM - 1));
    const int64_t v = w >> 9;  // (tile, half, accumulator)
    const int h = (int)(v % NH), half = (int)((v / NH) % CG);
    const int64_t tt = v / (NH * CG);
    if (tt >= tiles) return;
    int64_t tm, tc, np, base;
    tile_rc(args.whole + tt, args, tm, tc);
    part_info(tt, args, (int)args.nks, np, base);
    const int64_t row = (tm * CG + half) * TM + rl;
    const int64_t c0 = (NH == 2 ? 2 * tc + h : tc) * TN + group * kGroupCols;  // first sample of this group
    if (row >= args.l || c0 >= args.s) return;
    const int64_t so = (((base * CG + half) * NH + h) * TM + rl) * TN + group * kGroupCols + 2 * lane;
    const int64_t pstride = (int64_t)CG * NH * TM * TN;
    if (!IQP_IN(so + (np - 1) * pstride + 1, args.skcap, 49)) return;
    float x = 0.f, y = 0.f;
#pragma unroll 4
    for (int64_t p = 0; p < np; ++p) {
        const float2 u = __ldcg(reinterpret_cast<const float2 *>(args.skp + so + p * pstride));
        x += u.x;
        y += u.y;
    }
    const int64_t i = c0 + 2 * lane;
    const bool v0 = i < args.s, v1 = i + 1 < args.s;
    float s0 = 0.f, k0, s1 = 0.f, k1;
    if (MODE == 0) {
        k0 = cosf(x);
        k1 = cosf(y);
    } else {
        sincosf(x, &s0, &k0);
        sincosf(y, &s1, &k1);
    }
    if (MODE != 1) {
        const int64_t nvalid = args.s - c0 < kGroupCols ? args.s - c0 : kGroupCols;
        float S = (v0 ? k0 : 0.f) + (v1 ? k1 : 0.f);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, o);
        const float mean = S / (float)nvalid;
        float M2 = (v0 ? (k0 - mean) * (k0 - mean) : 0.f) + (v1 ? (k1 - mean) * (k1 - mean) : 0.f);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) M2 += __shfl_xor_sync(0xFFFFFFFFu, M2, o);
        if (lane == 0 && IQP_IN(row * args.nparts + c0 / kGroupCols, args.l * args.nparts, 50))
            args.part[row * args.nparts + c0 / kGroupCols] = make_double2((double)S, (double)M2);
    }
    if (MODE == 0) {
        if (args.out != nullptr && IQP_IN(row * args.ldo + (v1 ? i + 1 : c0), args.l * args.ldo, 45)) {
            float *f = args.out + row * args.ldo + i;
            if (v1) *reinterpret_cast<float2 *>(f) = make_float2(x, y);
            else if (v0) *f = x;
        }
    } else {
        const float al = (float)args.alpha[row], be = args.beta ? (float)args.beta[row] : 0.f;
        const float w0 = s0 * (al + be * k0), w1 = s1 * (al + be * k1);
        if (!IQP_IN(row * args.ldw + (v1 ? i + 1 : c0), args.l * args.ldw, 44)) return;
        if (X3) {
            float *f = args.wf + row * args.ldw + i;
            if (v1) *reinterpret_cast<float2 *>(f) = make_float2(w0, w1);
            else if (v0) *f = w0;
            const float a0 = fabsf(w0), a1 = fabsf(w1);
            float mx = v0 && a0 <= 3.4e38f ? a0 : 0.f;
            if (v1 && a1 <= 3.4e38f) mx = fmaxf(mx, a1);
            const uint32_t mb = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx));
            if (lane == 0 && mb != 0u) atomicMax(args.wmax + row, mb);
        } else {
            const float h0 = __bfloat162float(__float2bfloat16_rn(w0)), h1 = __bfloat162float(__float2bfloat16_rn(w1));
            const uint32_t ph = pack_bf16x2(h0, h1), pl = pack_bf16x2(w0 - h0, w1 - h1);
            __nv_bfloat16 *dh = args.whi + row * args.ldw + i, *dl = args.wlo + row * args.ldw + i;
            if (v1) {
                *reinterpret_cast<uint32_t *>(dh) = ph;
                *reinterpret_cast<uint32_t *>(dl) = pl;
            } else if (v0) {
                *reinterpret_cast<uint16_t *>(dh) = (uint16_t)ph;
                *reinterpret_cast<uint16_t *>(dl) = (uint16_t)pl;
            }
        }
    }
}

// GRAD = false: phase contraction (MODE 0 stats / MODE 1 W / MODE 2 both),
//              or (MODE 3) a dense contraction whose accumulator is stored.
// GRAD = true : gradient contraction.
// AT = true: the A operand arrives by TMA in the swizzled layout (always for
// the gradient's W; for MODE 3, a dense split-BF16 matrix); AT = false: the
// producer warps expand it from P_A bits and the hi/lo split of 2 theta.
// CG = 1: one CTA per tile of 128 rows; CG = 2: a CTA pair per tile of 256 rows.
// TA (phase modes of CTA pairs): 0 = A in shared memory; 1 = A in TMEM; 3 =
// two sample tiles (2 x 256 samples) per tile against each A stage; 4 = the
// FP32 form (X3): 2 theta as three BF16 planes (the kernel's note below).
template <bool GRAD, int MODE, int CG, bool AT, bool SPL, int TA>
__global__ void __launch_bounds__(kThreads, 1)
    k_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmA2,
         const __grid_constant__ CUtensorMap tmB, const TcArgs args) {
    pdl_sync();
    constexpr bool ATMA = GRAD || AT;  // A operand by TMA
    // A operand in TMEM, written by the producer warps (phase modes, CTA pairs)
    constexpr bool ATM = TA == 1 && !GRAD && !AT && CG == 2;
    // Two sample tiles per tile (phase modes, CTA pairs, whole tiles): A in
    // shared memory, two accumulators, running sums in global memory
    constexpr bool DT = TA == 3 && !GRAD && !AT && CG == 2;
    // FP32 form: three planes of 2 theta, the first on an integer grid, so its
    // products (into accumulator columns 0..255) sum exactly; the other two
    // share columns 256..511
    constexpr bool X3 = TA == 4 && !GRAD && !AT && CG == 2;
    using C = Cfg<CG, ATMA, ATM, DT, X3>;
    constexpr int NOP = C::NOP;
    // Serpentine gate order (phase kernels, whole tiles): the CTA groups' odd
    // rounds of tiles walk their bits stages from the last to the first, so a
    // round starts on the operand rows the round before it read last, which
    // are still in L2. The sum is the same up to the order of its terms.
    constexpr bool SERP = !GRAD && !ATMA && !SPL;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = aligned_smem(smem_raw);
    Bars *bar = reinterpret_cast<Bars *>(smem + C::SM_BAR);
    float *red = reinterpret_cast<float *>(smem + C::SM_RED);
    float4 *sum4 = reinterpret_cast<float4 *>(smem + C::SM_SUM);  // ATM: running sum
    volatile int *abort_flag = &bar->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t lim = args.limit_ns;
    uint32_t *status = args.status;
    constexpr int CL = CG;  // CTAs per cluster
    const uint32_t crank = CL == 2 ? cluster_ctarank() : 0u;  // CTA rank in the cluster
    const bool leader = CG == 1 || crank == 0;                 // issues this CTA's MMAs
    const int64_t group0 = blockIdx.x / CL, ngroups = gridDim.x / CL;

    if (threadIdx.x == 0) {
        for (int i = 0; i < NBITS; ++i) {
            mbar_init(&bar->bits_full[i], 1);
            mbar_init(&bar->bits_empty[i], NGEN);
        }
        for (int i = 0; i < NOP; ++i) {
            // Even CTA: its own producer warps, plus one forwarded arrival from
            // the odd CTA of a pair.
            mbar_init(&bar->op_full[i], CG == 2 ? NGEN + 1 : NGEN);
            mbar_init(&bar->op_empty[i], 1);  // the MMAs that read the stage
            mbar_init(&bar->w_full[i], 1);
            mbar_init(&bar->peer_full[i], NGEN);  // odd CTA: its producer warps
        }
        mbar_init(&bar->acc_full, 1);
        mbar_init(&bar->drain, 1);
        mbar_init(&bar->red_full, NGEN);
        bar->abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
    }
    if (warp == 1) {
        if constexpr (CG == 2) {
            tmem_alloc_pair(&bar->tmem_slot, kTmemCols);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(&bar->tmem_slot, kTmemCols);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (CL == 2) cluster_sync_all();  // the peer's barriers exist before anyone arrives on them
    tc_fence_after();
    const uint32_t tmem = bar->tmem_slot;

    const int64_t nunits = args.nunits;
    const int nks = (int)args.nks;     // host guarantees nks < 2^31
    const int chunk = (int)args.chunk;

    if (warp == 0) {
        // ---------------------------------------------------------- TMA producer
        if (lane == 0) {
            prefetch_tmap(&tmA);
            prefetch_tmap(&tmB);
            if (ATMA) prefetch_tmap(&tmA2);
            uint32_t itb = 0, ito = 0;
            uint32_t bmask = 0, bpar = 0, omask = 0, opar = 0;  // issued stages and their last parities
            bool ok = true;
            for (int64_t u = group0; u < nunits && ok; u += ngroups) {
                int64_t t, uv;
                int ks0, ks1;
                unit_of<SPL, MODE == 3>(u, args, nks, t, ks0, ks1, uv);
                int64_t tm64, tc64;
                tile_rc(t, args, tm64, tc64);
                const int tm = (int)tm64;
                const int tn = (int)tc64;
                const int prank = CG == 2 ? (int)crank : 0;        // rank within an MMA pair
                const int a0 = tm * TM * CG + prank * TM;          // this CTA's first A row
                const int b0 = tn * TN * (DT ? 2 : 1) + prank * C::TNB;  // this CTA's first B row
                const bool rev = SERP && args.serp != 0 && ((((u - group0) / ngroups) & 1) != 0);
                const int kbA = ks0 / (KB / KS), kbN = (ks1 + KB / KS - 1) / (KB / KS) - kbA;
                for (int i = 0; i < kbN && ok; ++i, ++itb) {
                    const int kb = rev ? kbA + kbN - 1 - i : kbA + i;
                    const uint32_t bs = itb % NBITS;
                    if (!mbar_wait(&bar->bits_empty[bs], ((itb / NBITS) & 1u) ^ 1u, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    uint8_t *bits = smem + C::SM_BITS + bs * C::BT_BYTES;
                    const int x = (int)(kb * 4);
                    if (ATMA) {
                        mbar_arrive_expect_tx(&bar->bits_full[bs], C::TNB * 32);
                        tma_load_2d(bits + C::BT_B, &tmB, &bar->bits_full[bs], x, b0);
                    } else if (DT) {
                        mbar_arrive_expect_tx(&bar->bits_full[bs], TM * 32 + 2 * C::TNB * 32 + 1024);
                        tma_load_2d(bits + C::BT_A, &tmA, &bar->bits_full[bs], x, a0);
                        tma_load_2d(bits + C::BT_B, &tmB, &bar->bits_full[bs], x, b0);
                        tma_load_2d(bits + C::BT_B1, &tmB, &bar->bits_full[bs], x, b0 + TN);
                        const bool cin = IQP_IN((int64_t)kb * KB + KB - 1, args.mpad, 54);
                        bulk_load(bits + C::BT_CHI, args.chi + (cin ? kb * KB : 0), 512, &bar->bits_full[bs]);
                        bulk_load(bits + C::BT_CLO, args.clo + (cin ? kb * KB : 0), 512, &bar->bits_full[bs]);
                    } else {
                        mbar_arrive_expect_tx(&bar->bits_full[bs], TM * 32 + C::TNB * 32 + (X3 ? 1536 : 1024));
                        tma_load_2d(bits + C::BT_A, &tmA, &bar->bits_full[bs], x, a0);
                        tma_load_2d(bits + C::BT_B, &tmB, &bar->bits_full[bs], x, b0);
                        // the split of 2 theta is mpad long (bits stages never pass it)
                        const bool cin = IQP_IN((int64_t)kb * KB + KB - 1, args.mpad, 54);
                        bulk_load(bits + C::BT_CHI, args.chi + (cin ? kb * KB : 0), 512, &bar->bits_full[bs]);
                        bulk_load(bits + C::BT_CLO, args.clo + (cin ? kb * KB : 0), 512, &bar->bits_full[bs]);
                        if (X3) bulk_load(bits + C::BT_C3, args.c3 + (cin ? kb * KB : 0), 512, &bar->bits_full[bs]);
                    }
                    bmask |= 1u << bs;
                    bpar = (bpar & ~(1u << bs)) | (((itb / NBITS) & 1u) << bs);
                    if (ATMA) {
                        // A_hi / A_lo tiles (W, or a dense operand) of the operand stages of this bits stage.
                        for (int q = 0; q < KB / KS; ++q) {
                            const int ks = kb * (KB / KS) + q;
                            if (ks >= ks1) break;
                            const uint32_t os = ito % NOP;
                            if (!mbar_wait(&bar->op_empty[os], ((ito / NOP) & 1u) ^ 1u, abort_flag, status, lim)) {
                                ok = false;
                                break;
                            }
                            uint8_t *op = smem + C::SM_OP + os * C::OP_BYTES;
                            mbar_arrive_expect_tx(&bar->w_full[os], 2 * TM * KS * 2);
                            tma_load_2d(op + C::OP_A_HI, &tmA, &bar->w_full[os], (int)(ks * KS), a0);
                            tma_load_2d(op + C::OP_A_LO, &tmA2, &bar->w_full[os], (int)(ks * KS), a0);
                            // Warm L2 with the W tiles kWPrefetch stages ahead.
                            if (ks + kWPrefetch < nks) {
                                tma_prefetch_2d(&tmA, (int)((ks + kWPrefetch) * KS), a0);
                                tma_prefetch_2d(&tmA2, (int)((ks + kWPrefetch) * KS), a0);
                            }
                            omask |= 1u << os;
                            opar = (opar & ~(1u << os)) | (((ito / NOP) & 1u) << os);
                            ++ito;
                        }
                    }
                }
            }
            // Drain: every copy this thread issued has landed before exit.
#pragma unroll
            for (int i = 0; i < NBITS; ++i)
                if ((bmask >> i) & 1u) mbar_drain(&bar->bits_full[i], (bpar >> i) & 1u, status, lim);
#pragma unroll
            for (int i = 0; i < NOP; ++i)
                if (ATMA && ((omask >> i) & 1u)) mbar_drain(&bar->w_full[i], (opar >> i) & 1u, status, lim);
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer
        if (lane == 0 && leader) {
            uint32_t ito = 0;
            bool ok = true;
            // operand descriptors of stage 0 (K step 0)
            const uint32_t sb = smem_u32(smem + C::SM_OP);
            const uint64_t d_b0 = sdesc_k128(sb + C::OP_B);
            [[maybe_unused]] const uint64_t d_b1 = sdesc_k128(sb + C::OP_B1);
            const uint64_t d_hi0 = sdesc_k128(sb + C::OP_A_HI), d_lo0 = sdesc_k128(sb + C::OP_A_LO);
            for (int64_t u = group0; u < nunits && ok; u += ngroups) {
                int64_t t, uv;
                int ks0, ks1;
                unit_of<SPL, MODE == 3>(u, args, nks, t, ks0, ks1, uv);
                int kc = 0;  // stage index within the current accumulation chunk
                for (int ks = ks0; ks < ks1; ++ks, ++ito) {
                    const uint32_t os = ito % NOP;
                    // One-CTA gradient: this thread also waits for the stage's W
                    // tiles (a pair's W halves are vouched for by its producers).
                    const bool got =
                        CG == 2 ? mbar_wait_cluster(&bar->op_full[os], (ito / NOP) & 1u, abort_flag, status, lim)
                                : (mbar_wait(&bar->op_full[os], (ito / NOP) & 1u, abort_flag, status, lim) &&
                                   (!ATMA ||
                                    mbar_wait(&bar->w_full[os], (ito / NOP) & 1u, abort_flag, status, lim)));
                    if (!got) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    // first stage of a chunk: overwrite the accumulator
                    const uint32_t acc = kc == 0 ? 0u : 1u;
                    // Descriptors of the stage's first K step (stage os is
                    // os * OP_BYTES / 16 further in the start-address field).
                    const uint64_t so = (uint64_t)(os * (C::OP_BYTES >> 4));
                    // (one function may not mix cta_group::1 and ::2 forms)
                    if constexpr (ATM)
                        umma_stage4_pair_ts(tmem, tmem + kAColBase + os * kAColStage, d_b0 + so, C::IDESC, acc);
                    else if constexpr (DT) {
                        umma_stage4_pair_ss(tmem, d_hi0 + so, d_lo0 + so, d_b0 + so, C::IDESC, acc);
                        umma_stage4_pair_ss(tmem + (uint32_t)TN, d_hi0 + so, d_lo0 + so, d_b1 + so, C::IDESC, acc);
                    } else if constexpr (X3) {
                        umma_stage4_pair_ss1(tmem, d_hi0 + so, d_b0 + so, C::IDESC, acc);
                        umma_stage4_pair_ss(tmem + (uint32_t)TN, d_lo0 + so,
                                            d_lo0 + so + ((C::OP_A_3 - C::OP_A_LO) >> 4), d_b0 + so, C::IDESC, acc);
                    } else if constexpr (CG == 2)
                        umma_stage4_pair_ss(tmem, d_hi0 + so, d_lo0 + so, d_b0 + so, C::IDESC, acc);
                    else
                        umma_stage4_ss(tmem, d_hi0 + so, d_lo0 + so, d_b0 + so, C::IDESC, acc);
                    if constexpr (CG == 2) umma_commit_pair(&bar->op_empty[os]);
                    else umma_commit(&bar->op_empty[os]);
                    if (++kc == chunk || ks == ks1 - 1) {
                        if constexpr (CG == 2) umma_commit_pair(&bar->acc_full);
                        else umma_commit(&bar->acc_full);
                        kc = 0;
                    }
                }
            }
            // Drain: all issued MMAs complete before TMEM is freed (and, for a
            // pair, before the peer may leave: the cluster barrier below).
            if constexpr (CG == 2) umma_commit_pair(&bar->drain);
            else umma_commit(&bar->drain);
            mbar_drain(&bar->drain, 0u, status, lim);
        } else if (CG == 2 && lane == 0) {
            // Odd CTA of a pair: forward "my half of stage ks is ready" to the
            // even CTA's stage barrier, one cluster-scope release per stage,
            // so the producer warps themselves only use CTA-scope arrivals.
            const uint32_t op_full_remote = mapa_shared(smem_u32(&bar->op_full[0]), 0u);
            uint32_t ito = 0;
            bool ok = true;
            for (int64_t u = group0; u < nunits && ok; u += ngroups) {
                int64_t t, uv;
                int ks0, ks1;
                unit_of<SPL, MODE == 3>(u, args, nks, t, ks0, ks1, uv);
                for (int ks = ks0; ks < ks1; ++ks, ++ito) {
                    const uint32_t os = ito % NOP;
                    if (!mbar_wait(&bar->peer_full[os], (ito / NOP) & 1u, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_remote(op_full_remote + os * 8u);
                }
            }
        }
    } else {
        // ------------------------------------------------ producers + epilogue
        const int gt = threadIdx.x - 64;   // 0 .. NGEN*32-1
        const int quarter = warp & 3;      // TMEM lane quarter this warp may access
        const int group = (warp - 2) >> 2; // accumulator column group of the epilogue
        uint32_t itb = 0, ito = 0, tcount = 0, nacc = 0;
        const int rl = quarter * 32 + lane;  // accumulator row (TMEM lane) of this thread
        // DT: this CTA's running sums (both accumulators) in global memory
        // (the host launches at most kMaxSplitCtas CTAs of this form)
        [[maybe_unused]] float4 *gsum_cta =
            (DT || X3) && IQP_IN(blockIdx.x, kMaxSplitCtas, 59)
                ? args.gsum + (int64_t)blockIdx.x * ((DT ? kDtSumFloats : kSplitSlotFloats) / 4)
                : nullptr;
        // ATM: this thread's A parity bits of the current bits stage, 16 per
        // operand stage (see expand_a_tmem), packed two stages per word
        uint32_t abits01 = 0, abits23 = 0;
        bool ok = true;
        for (int64_t u = group0; u < nunits && ok; u += ngroups) {
            int ks0, ks1;
            int64_t tm, tc, slot;
            {
                int64_t t;
                unit_of<SPL, MODE == 3>(u, args, nks, t, ks0, ks1, slot);
                tile_rc(t, args, tm, tc);
            }
            if (ks0 >= ks1) continue;      // an empty piece of a balanced split: no work
            const uint32_t tix = tcount++;  // units this CTA ran before this one
            const int64_t tn = tc;
            const int64_t arow0 = tm * TM * CG + (CG == 2 ? (int64_t)crank * TM : 0);  // first observable here
            int kc = 0;              // stage index within the current chunk
            int nchunk = 0;          // chunks of this tile already folded into the running sum
            bool fold_due = false;   // a finished chunk must be folded before the next release
            // Stage order: bits stages forwards, or (serpentine rounds) from the
            // last one (c0 operand stages, ks1 - 4 kbTop) down to the first;
            // within a bits stage always q = 0, 1, ...
            const bool rev = SERP && args.serp != 0 && ((((u - group0) / ngroups) & 1) != 0);
            const int kbTop = (ks1 - 1) >> 2;
            const int c0 = ks1 - 4 * kbTop;
            for (int ks = ks0; ks < ks1; ++ks) {
                const int idx = ks - ks0;  // position in the tile's stage sequence
                int q;
                bool qlast;  // the bits stage's last operand stage
                if (!rev) {
                    q = ks & 3;
                    qlast = q == 3 || ks == ks1 - 1;
                } else if (idx < c0) {
                    q = idx;
                    qlast = idx == c0 - 1;
                } else {
                    q = (idx - c0) & 3;
                    qlast = q == 3;
                }
                const uint32_t bs = itb % NBITS;
                if (q == 0 && !wait_warp(&bar->bits_full[bs], (itb / NBITS) & 1u, abort_flag, status, lim)) {
                    ok = false;
                    break;
                }
                const uint8_t *bits = smem + C::SM_BITS + bs * C::BT_BYTES;
                if (ATM && q == 0) {
                    // Row rl's 256 parity bits of this bits stage (8 words);
                    // operand stage j needs bits [64 j + 16 group, +16), in
                    // word 2 j + (group >> 1) at bit 16 (group & 1).
                    const uint4 x0 = *reinterpret_cast<const uint4 *>(bits + C::BT_A + rl * 32);
                    const uint4 x1 = *reinterpret_cast<const uint4 *>(bits + C::BT_A + rl * 32 + 16);
                    const bool odd = (group >> 1) & 1;
                    const uint32_t sh = (uint32_t)(group & 1) * 16u;
                    const uint32_t w0 = odd ? x0.y : x0.x, w1 = odd ? x0.w : x0.z;
                    const uint32_t w2 = odd ? x1.y : x1.x, w3 = odd ? x1.w : x1.z;
                    abits01 = ((w0 >> sh) & 0xFFFFu) | ((w1 >> sh) << 16);
                    abits23 = ((w2 >> sh) & 0xFFFFu) | ((w3 >> sh) << 16);
                }
                const uint32_t os = ito % NOP;
                if (!wait_warp(&bar->op_empty[os], ((ito / NOP) & 1u) ^ 1u, abort_flag, status, lim)) {
                    ok = false;
                    break;
                }
                uint8_t *op = smem + C::SM_OP + os * C::OP_BYTES;
                if (ATM) {
                    // The MMAs that read this stage's A columns have completed
                    // (op_empty); order the TMEM stores after them.
                    tc_fence_after();
                    const uint32_t b16 = ((q < 2 ? abits01 : abits23) >> ((q & 1) * 16)) & 0xFFFFu;
                    const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + kAColBase + os * kAColStage +
                                        (uint32_t)group * 16u;
                    expand_a_tmem(b16, bits + C::BT_CHI, bits + C::BT_CLO, q, group, ta);
                }
                expand_b<C::TNB>(bits + C::BT_B, op + C::OP_B, q, gt);
                if constexpr (DT) expand_b<C::TNB>(bits + C::BT_B1, op + C::OP_B1, q, gt);
                if constexpr (X3)
                    expand_a3(bits + C::BT_A, bits + C::BT_CHI, op + C::OP_A_HI, q, gt);
                else if (!ATMA && !ATM)
                    expand_a(bits + C::BT_A, bits + C::BT_CHI, bits + C::BT_CLO, op + C::OP_A_HI, op + C::OP_A_LO, q,
                             gt);
                if (ATM) {
                    tmem_wait_st();
                    tc_fence_before();
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (ATMA && CG == 2 && !wait_warp(&bar->w_full[os], (ito / NOP) & 1u, abort_flag, status, lim)) {
                    // A pair's W tiles must have landed before the stage is released.
                    ok = false;
                    break;
                }
                if (fold_due) {
                    // This stage opens a new chunk and its first MMA overwrites
                    // the accumulator: fold the finished chunk into the running
                    // sum first, then release the stage (it was produced while
                    // the previous chunk's last MMAs ran).
                    if (!wait_warp(&bar->acc_full, nacc & 1u, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    ++nacc;
                    __syncwarp();
                    tc_fence_after();
                    const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(group * kGroupCols);
#pragma unroll 1
                    for (int c = 0; c < (DT ? 2 : 1) * kGroupLoads; ++c) {
                        uint32_t r[32], acc[32];
                        const int hb = DT && c >= kGroupLoads ? 1 : 0;  // DT: accumulator of the second sample tile
                        const int cc = c - hb * kGroupLoads;
                        if (X3)
                            load_sum32(tb + (uint32_t)(cc * 32), true, r);
                        else
                            tmem_ld32(tb + (uint32_t)(hb * TN + cc * 32), r);
                        if (ATM || DT || X3) {
                            // running sum in shared memory (ATM) or global memory
                            // (DT), this thread's row only
                            float4 *sp = ATM ? sum4 + ((group * kGroupCols + cc * 32) >> 2) * TM + rl
                                             : gsum_cta + ((hb * TN + group * kGroupCols + cc * 32) >> 2) * TM + rl;
#pragma unroll
                            for (int e4 = 0; e4 < 8; ++e4) {
                                float4 v = make_float4(__uint_as_float(r[4 * e4]), __uint_as_float(r[4 * e4 + 1]),
                                                       __uint_as_float(r[4 * e4 + 2]), __uint_as_float(r[4 * e4 + 3]));
                                if (nchunk > 0) {
                                    const float4 o = sp[e4 * TM];
                                    v.x += o.x;
                                    v.y += o.y;
                                    v.z += o.z;
                                    v.w += o.w;
                                }
                                sp[e4 * TM] = v;
                            }
                            continue;
                        }
                        if (nchunk > 0) {
                            tmem_ld32(tb + kSumCol + c * 32, acc);
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                r[e] = __float_as_uint(__uint_as_float(r[e]) + __uint_as_float(acc[e]));
                        }
                        tmem_st32(tb + kSumCol + c * 32, r);
                    }
                    tc_fence_before();
                    ++nchunk;
                    fold_due = false;
                }
                if (lane == 0) {
                    // Even CTA: straight to the stage barrier; odd CTA: to the
                    // local barrier its forwarder watches.
                    if (CG == 2 && !leader) mbar_arrive(&bar->peer_full[os]);
                    else mbar_arrive(&bar->op_full[os]);
                }
                ++ito;
                if (qlast) {
                    if (lane == 0) mbar_arrive(&bar->bits_empty[bs]);
                    ++itb;
                }
                if (++kc == chunk) {
                    kc = 0;
                    fold_due = ks != ks1 - 1;
                }
            }
            if (!ok) break;
            // ------------------------------------------------------ epilogue
            if (!wait_warp(&bar->acc_full, nacc & 1u, abort_flag, status, lim)) {
                ok = false;
                break;
            }
            ++nacc;
            __syncwarp();  // lanes leave the wait loop independently; tcgen05.ld is warp-aligned
            tc_fence_after();
            const int64_t row = arow0 + quarter * 32 + lane;  // observable a
            const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(group * kGroupCols);
            const bool chunked = nchunk > 0;

            if constexpr (!GRAD && MODE != 3 && SPL) {
                // A part of a split tile: store this part's accumulator(s);
                // k_split_reduce, launched next, adds the tile's parts up and
                // runs the epilogue. Slot layout: ((slot * CG + CTA) * NH + h)
                // per TM x TN accumulator h (DT: two).
                constexpr int NH = DT ? 2 : 1;
                const int64_t half = CG == 2 ? (int64_t)crank : 0;
#pragma unroll 1
                for (int h = 0; h < NH; ++h) {
                    const int64_t so = (((slot * CG + half) * NH + h) * TM + rl) * TN + group * kGroupCols;
                    const float4 *ss0 = ATM  ? sum4 + ((group * kGroupCols) >> 2) * TM + rl
                                        : DT || X3 ? gsum_cta + ((h * TN + group * kGroupCols) >> 2) * TM + rl
                                                   : nullptr;
                    if (IQP_IN(so + kGroupCols - 1, args.skcap, 47))
                        split_store<X3>(args.skp + so, tbase + (uint32_t)(h * TN), chunked, ss0);
                }
                tc_fence_before();
                continue;
            }
            // Phi (or Q) for 32 columns: last chunk's accumulator + running sum.
            // DT: the two sample tiles' accumulators in turn.
            for (int hb = 0; hb < (DT ? 2 : 1) && ok; ++hb) {
                const int64_t tn_h = DT ? 2 * tn + hb : tn;
                const uint32_t tb_h = tbase + (uint32_t)(hb * TN);
                // where the running sum of this thread's row keeps the group's
                // 32 columns c * 32..: shared memory (ATM), global memory (DT),
                // else TMEM
                auto ssum = [&](int c) -> const float4 * {
                    return ATM  ? sum4 + ((group * kGroupCols + c * 32) >> 2) * TM + rl
                           : DT || X3 ? gsum_cta + ((hb * TN + group * kGroupCols + c * 32) >> 2) * TM + rl
                                      : nullptr;
                };
                auto ldsum = [&](int c, uint32_t (&r)[32]) {
                    if (X3)
                        load_sum32_x3(tb_h + c * 32, chunked ? ssum(c) : nullptr, r);
                    else
                        load_sum32(tb_h + c * 32, chunked, r, ssum(c));
                };
                if (!GRAD && MODE == 0) {
                    const int64_t c0 = tn_h * TN + group * kGroupCols;  // first sample of this group
                    int64_t nvalid = args.s - c0;
                    nvalid = nvalid < 0 ? 0 : (nvalid > kGroupCols ? kGroupCols : nvalid);
                    float S = 0.f, M2 = 0.f;
                    uint32_t r[32];
#pragma unroll 1
                    for (int c = 0; c < kGroupLoads; ++c) {
                        ldsum(c, r);
                        // Phi itself, when a gradient pass follows (W from it
                        // instead of a second contraction).
                        if (args.out != nullptr && c * 32 < nvalid && row < args.l)
                            store_out32(args, args.out, row, c0 + c * 32, r);
#pragma unroll 1
                        for (int v = 0; v < 4; ++v) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) r[e] = __float_as_uint(cosf(__uint_as_float(r[e])));
                            rotate8(r);
                        }
                        merge_cos32(r, c, (int)nvalid, S, M2);
                    }
                    if (row < args.l && nvalid > 0 && IQP_IN(row * args.nparts + c0 / kGroupCols, args.l * args.nparts, 50))
                        args.part[row * args.nparts + (c0 / kGroupCols)] = make_double2((double)S, (double)M2);
                } else if (!GRAD && MODE == 2) {
                    // Both: the statistics of MODE 0 and W of MODE 1 from one
                    // pass over Phi (the loss's alpha, beta known in advance).
                    const int64_t c0 = tn_h * TN + group * kGroupCols;
                    int64_t nvalid = args.s - c0;
                    nvalid = nvalid < 0 ? 0 : (nvalid > kGroupCols ? kGroupCols : nvalid);
                    const bool rv = row < args.l;
                    const float al = rv && IQP_IN(row, args.l, 55) ? (float)args.alpha[row] : 0.f;
                    const float be = (rv && args.beta) ? (float)args.beta[row] : 0.f;
                    [[maybe_unused]] float wmax = 0.f;
                    float S = 0.f, M2 = 0.f;
                    uint32_t r[32];
#pragma unroll 1
                    for (int c = 0; c < kGroupLoads; ++c) {
                        ldsum(c, r);
                        const int64_t i0 = c0 + c * 32;
                        const bool in = rv && i0 < args.s && IQP_IN(row * args.ldw + i0, args.l * args.ldw, 43) &&
                                        IQP_IN(row * args.ldw + (i0 + 32 <= args.s ? i0 + 31 : args.s - 1),
                                               args.l * args.ldw, 44);
                        // eight columns of W at a time, stored as they are formed
#pragma unroll 1
                        for (int v = 0; v < 4; ++v) {
                            float w[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                float sn, cn;
                                sincosf(__uint_as_float(r[e]), &sn, &cn);
                                r[e] = __float_as_uint(cn);
                                w[e] = sn * (al + be * cn);
                            }
                            rotate8(r);
                            const int64_t i = i0 + 8 * v;
                            if (!in || i >= args.s) continue;
                            if (X3)
                                wmax = fmaxf(wmax, store_wf8(args, row, i, w));
                            else
                                store_w8(args, row, i, w);
                        }
                        merge_cos32(r, c, (int)nvalid, S, M2);
                    }
                    if (X3 && wmax > 0.f && IQP_IN(row, args.l, 60)) atomicMax(args.wmax + row, __float_as_uint(wmax));
                    if (rv && nvalid > 0 && IQP_IN(row * args.nparts + c0 / kGroupCols, args.l * args.nparts, 51))
                        args.part[row * args.nparts + (c0 / kGroupCols)] = make_double2((double)S, (double)M2);
                } else if (!GRAD && MODE == 3) {
                    const int64_t c0 = tn_h * TN + group * kGroupCols;
                    uint32_t r[32];
#pragma unroll 1
                    for (int c = 0; c < kGroupLoads; ++c) {
                        ldsum(c, r);
                        if (row >= args.l || c0 + c * 32 >= args.s) continue;
                        if (args.dvec != nullptr) {  // uniform
                            const float dv = args.dvec[row];
                            const uint32_t zw = args.zt32[row * args.ldzt32 + ((c0 + c * 32) >> 5)];
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                r[e] = __float_as_uint(dv + __uint_as_float(r[e])) ^ ((zw << (31 - e)) & 0x80000000u);
                        }
                        store_out32(args, args.out + slot * args.out_part, row, c0 + c * 32, r);
                    }
                } else if (!GRAD) {
                    const int64_t c0 = tn_h * TN + group * kGroupCols;
                    const bool rv = row < args.l;
                    const float al = rv && IQP_IN(row, args.l, 55) ? (float)args.alpha[row] : 0.f;
                    const float be = (rv && args.beta) ? (float)args.beta[row] : 0.f;
                    [[maybe_unused]] float wmax = 0.f;
                    uint32_t r[32];
#pragma unroll 1
                    for (int c = 0; c < kGroupLoads; ++c) {
                        ldsum(c, r);
                        const int64_t i0 = c0 + c * 32;
                        const bool in = rv && i0 < args.s && IQP_IN(row * args.ldw + i0, args.l * args.ldw, 43) &&
                                        IQP_IN(row * args.ldw + (i0 + 32 <= args.s ? i0 + 31 : args.s - 1),
                                               args.l * args.ldw, 44);
#pragma unroll 1
                        for (int v = 0; v < 4; ++v) {
                            float w[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                float sn, cn;
                                sincosf(__uint_as_float(r[e]), &sn, &cn);
                                w[e] = sn * (al + be * cn);
                            }
                            rotate8(r);
                            const int64_t i = i0 + 8 * v;
                            if (!in || i >= args.s) continue;
                            if (X3)
                                wmax = fmaxf(wmax, store_wf8(args, row, i, w));
                            else
                                store_w8(args, row, i, w);
                        }
                    }
                    if (X3 && wmax > 0.f && IQP_IN(row, args.l, 60)) atomicMax(args.wmax + row, __float_as_uint(wmax));
                } else {
                    // Gradient epilogue: mask by 2 P_A[a][j], reduce over observables.
                    const bool rv = row < args.l;
                    uint32_t r[32];
#pragma unroll 1
                    for (int c = 0; c < kGroupLoads; ++c) {
                        ldsum(c, r);
                        const int64_t j0 = tn_h * TN + group * kGroupCols + c * 32;
                        const uint32_t mask = (rv && j0 < args.m &&
                                               IQP_IN(row * args.ldp32 + (j0 >> 5), args.l * args.ldp32, 52))
                                                  ? args.pa32[row * args.ldp32 + (j0 >> 5)]
                                                  : 0u;
                        float v[32];
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = ((mask >> e) & 1u) ? 2.f * __uint_as_float(r[e]) : 0.f;
                        red[quarter * 256 + group * kGroupCols + c * 32 + lane] = reduce_scatter(v, lane);
                    }
                    // All producer warps' column sums are in `red`; combine the four
                    // lane quarters in fixed order. (The next tile's writes to
                    // `red` follow a full K loop that needs every warp, so a
                    // second barrier is not needed.)
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar->red_full);
                    if (!wait_warp(&bar->red_full, tix & 1u, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    __syncwarp();
                    const int64_t j = tn_h * TN + gt;
                    if (gt < TN && j < args.m && arow0 < args.l) {
                        const double sum = (double)red[gt] + (double)red[256 + gt] + (double)red[512 + gt] +
                                           (double)red[768 + gt];
                        if (IQP_IN((arow0 / TM) * args.m + j, args.tiles_m * args.m, 53))
                            args.gpart[(arow0 / TM) * args.m + j] = sum;
                    }
                }
            }
            if (!ok) break;
            tc_fence_before();
        }
    }

    __syncthreads();
    if (CL == 2) cluster_sync_all();  // no pair MMA still reads the peer's operands
    if (warp == 1) {
        __syncwarp();  // lane 0 ran the MMA loop alone; dealloc is warp-aligned
        tc_fence_after();
        if constexpr (CG == 2) tmem_dealloc_pair(tmem, kTmemCols);
        else tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------------------------ gradient, CTA pairs
// k_grad_pair: the gradient contraction in the transposed orientation,
//   D[j][a] = sum_i S_Z[i][j] W[a][i],   grad partial g_j += sum_a 2 P_A[a][j] D[j][a],
// as CTA pairs (cta_group::2): a tile is 256 gates (M, 128 per CTA) x 256
// observables (N), K = samples in 128-sample operand stages, GNS stages in
// flight.
//  - W (B operand: hi and lo BF16 tiles, 128 observables per CTA, two
//    128-byte K atoms each) arrives by TMA; both CTAs' loads complete on the
//    even CTA's w_full barrier.
//  - S_Z^T (A operand, +-1) is expanded from the transposed sample parities
//    P_Z^T straight into TMEM by eight producer warps (tcgen05.st). The even
//    CTA's producers also wait for the stage's W (w_full, both CTAs' halves)
//    before they arrive, and the odd CTA's readiness is forwarded by one
//    thread, so the MMA thread waits on a single barrier per stage.
//  - The accumulator (256 TMEM columns) is reduced after every accumulation
//    chunk (see below) by eight epilogue warps: mask by 2 P_A[a][j] (bits of
//    P_A^T), sum over the warp's 128 observables in FP32, add into an FP64
//    per-gate partial. Each
//    epilogue warp writes one FP64 partial per (tile, gate): row
//    2 * (observable tile) + (its column half).
// One MMA-issuing thread is the critical path here: its per-stage work is
// one barrier wait and 16 MMAs with precomputed descriptors, and the stage is
// twice as long as the phase kernel's to halve the per-stage overheads.
// Warps: 0 = W loads, 1 = MMA issuer (even CTA) / forwarder (odd CTA),
// 2 = P_Z^T bit loads, 3..10 = producers, 11..18 = epilogue.
// TMEM: accumulator at columns 0..255, A stage os at 256 + 64 os.
constexpr int GN = kGradObs;     // observables per tile (accumulator columns)
constexpr int GNB = GN / 2;      // W rows (observables) per CTA
constexpr int GKS = 128;         // samples per operand stage
constexpr int GNS = 3;           // operand stages in flight
constexpr int GSPB = 256 / GKS;  // operand stages per bits stage
constexpr int GACOLS = GKS / 2;  // TMEM columns per A stage
constexpr int GPROD = 8;         // producer warps
constexpr int GEPI = 8;          // epilogue warps
constexpr int GW0 = 3;           // first producer warp
constexpr int GE0 = GW0 + GPROD; // first epilogue warp
constexpr int kGThreads = (GE0 + GEPI) * 32;
// Accumulation chunks: a tile's K loop is cut into the fewest chunks of at
// most grad_chunk_samples() samples (default 10240), of equal length up to
// one stage. Each chunk boundary stalls the MMAs while the epilogue reads the
// accumulator, so fewer, longer chunks are faster; the chunk bounds the
// error of the tensor core's truncating FP32 accumulation.
constexpr uint32_t kGAcol = GN;      // first A column

// X3 (the FP32 form): tiles of 256 gates x 128 observables, W as three BF16
// planes, the first on an integer grid of its row. Per K step one N = 256
// product takes planes 0 (this CTA pair's first 128 rows of B: the even CTA's)
// and 1 (the odd CTA's) side by side into accumulator columns 0..127 and
// 128..255, and one N = 128 product adds plane 2 (64 rows per CTA) to columns
// 128..255. Plane 0's sums are exact; its rounding happens once, when the
// epilogue adds the two halves.
template <bool X3>
struct GCfg {
    static constexpr int NS = X3 ? 4 : GNS;               // operand stages in flight
    static constexpr int OBS = X3 ? 128 : GN;             // observables per tile
    static constexpr uint32_t ATOM = GNB * 128;           // one 128-byte K atom of a W tile
    static constexpr uint32_t ATOM2 = X3 ? 64 * 128 : GNB * 128;
    static constexpr uint32_t OP_HI = 0, OP_LO = 2 * ATOM;
    static constexpr uint32_t OP_BYTES = 2 * ATOM + 2 * ATOM2;  // W_hi + W_lo (X3: plane 0 or 1, and plane 2)
    static constexpr uint32_t SM_BITS = NS * OP_BYTES;
    static constexpr uint32_t BT_BYTES = TM * 32;         // P_Z^T: 128 gates x 256 samples
    static constexpr uint32_t SM_BAR = SM_BITS + NBITS * BT_BYTES;
    static constexpr uint32_t SM_END = SM_BAR + 256;
    static constexpr uint32_t SMEM = SM_END + 1024;
    static constexpr uint32_t IDESC = idesc_bf16(2 * TM, GN), IDESC2 = idesc_bf16(2 * TM, GN / 2);
    static_assert(OP_BYTES % 1024 == 0 && BT_BYTES % 1024 == 0, "stage alignment");
    static_assert(ATOM == 16384, "umma_stage8_pair_ts_b steps 16384 bytes between K atoms");
    static_assert(kGAcol + NS * GACOLS <= kTmemCols, "TMEM columns");
    static_assert(SMEM <= 232448, "shared memory");
};

struct GBars {
    uint64_t bits_full[NBITS], bits_empty[NBITS], a_full[4], a_peer[4], w_full[4], empty[4], acc_full,
        acc_empty, drain;
    uint32_t tmem_slot;
    int abort_flag;
};

struct GradArgs {
    int64_t l, s, m;
    int64_t nks;                  // operand stages per tile: ceil(s / GKS)
    int64_t chunk;                // operand stages per accumulation chunk
    int64_t tiles_g, tiles_o;     // gate blocks (256), observable blocks (GN)
    int64_t group_o;              // observable blocks per tile group (L2 rasterisation)
    const uint32_t *pat32;        // P_A^T: m rows of ldlt32 32-bit words (bits over observables)
    int64_t ldlt32;
    double *gpart;                // 2 * tiles_o rows of m FP64 partials
    uint32_t *status;
    uint64_t limit_ns;
};

template <bool X3>
__global__ void __launch_bounds__(kGThreads, 1)
    k_grad_pair(const __grid_constant__ CUtensorMap tmWhi, const __grid_constant__ CUtensorMap tmWlo,
                const __grid_constant__ CUtensorMap tmW3, const __grid_constant__ CUtensorMap tmZt,
                const GradArgs args) {
    pdl_sync();
    using C = GCfg<X3>;
    constexpr int GNS = C::NS, GN = C::OBS, GNB = GN / 2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = aligned_smem(smem_raw);
    GBars *bar = reinterpret_cast<GBars *>(smem + C::SM_BAR);
    volatile int *abort_flag = &bar->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t lim = args.limit_ns;
    uint32_t *status = args.status;
    const uint32_t crank = cluster_ctarank();
    const bool leader = crank == 0;
    const int64_t group0 = blockIdx.x / 2, ngroups = gridDim.x / 2;
    const int64_t ntiles = args.tiles_g * args.tiles_o;
    const int nks = (int)args.nks;
    const int chunk = (int)args.chunk;

    if (threadIdx.x == 0) {
        for (int i = 0; i < NBITS; ++i) {
            mbar_init(&bar->bits_full[i], 1);
            mbar_init(&bar->bits_empty[i], GPROD);
        }
        for (int i = 0; i < GNS; ++i) {
            mbar_init(&bar->a_full[i], GPROD + 1);  // even CTA: its producers + the odd CTA's forwarded arrival
            mbar_init(&bar->a_peer[i], GPROD);     // odd CTA: its producers
            mbar_init(&bar->w_full[i], 1);         // even CTA: its arrive.expect_tx; both CTAs' bytes
            mbar_init(&bar->empty[i], 1);          // the pair commit of the stage's MMAs
        }
        mbar_init(&bar->acc_full, 1);
        mbar_init(&bar->acc_empty, 2 * GEPI);  // even CTA: both CTAs' epilogue warps
        mbar_init(&bar->drain, 1);
        bar->abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
    }
    if (warp == 1) {
        tmem_alloc_pair(&bar->tmem_slot, kTmemCols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem = bar->tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ W loads
        if (lane == 0) {
            prefetch_tmap(&tmWhi);
            prefetch_tmap(&tmWlo);
            if (X3) prefetch_tmap(&tmW3);
            const uint32_t w_full_leader = mapa_shared(smem_u32(&bar->w_full[0]), 0u);
            uint32_t os = 0, ph = 0, omask = 0, opar = 0;  // stage ring position and its phase parity
            bool ok = true;
            for (int64_t t = group0; t < ntiles && ok; t += ngroups) {
                int64_t to, tg;
                tile_coords(t, args.tiles_o, args.tiles_g, args.group_o, to, tg);
                // this CTA's first W row (X3: of plane 0 or 1, then of plane 2 GNB crank further on)
                const int a0 = (int)(to * GN) + (X3 ? 0 : (int)crank * GNB);
                int a0n = -1;                                      // the next tile's (for L2 prefetch)
                if (t + ngroups < ntiles) {
                    int64_t ton, tgn;
                    tile_coords(t + ngroups, args.tiles_o, args.tiles_g, args.group_o, ton, tgn);
                    a0n = (int)(ton * GN) + (X3 ? 0 : (int)crank * GNB);
                }
                for (int ks = 0; ks < nks; ++ks) {
                    if (!mbar_wait(&bar->empty[os], ph ^ 1u, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    uint8_t *op = smem + os * C::OP_BYTES;
                    if (leader) mbar_arrive_expect_tx(&bar->w_full[os], 2 * C::OP_BYTES);
#pragma unroll
                    for (int at = 0; at < 2; ++at) {
                        const int x = ks * GKS + at * 64;
                        const int a2 = X3 ? a0 + (int)crank * GNB : a0;
                        if (leader) {
                            tma_load_2d(op + C::OP_HI + at * C::ATOM, &tmWhi, &bar->w_full[os], x, a0);
                            tma_load_2d(op + C::OP_LO + at * C::ATOM2, X3 ? &tmW3 : &tmWlo, &bar->w_full[os], x, a2);
                        } else {
                            tma_load_2d_pair(op + C::OP_HI + at * C::ATOM, X3 ? &tmWlo : &tmWhi, w_full_leader + os * 8u,
                                             x, a0);
                            tma_load_2d_pair(op + C::OP_LO + at * C::ATOM2, X3 ? &tmW3 : &tmWlo, w_full_leader + os * 8u,
                                             x, a2);
                        }
                    }
                    // warm L2 with the tiles 512 samples beyond this load (the next tile's near the end)
                    int xp = ks * GKS + 512, ap = a0;
                    if (xp >= nks * GKS) {
                        xp -= nks * GKS;
                        ap = a0n;
                    }
                    if (ap >= 0) {
                        const CUtensorMap *m1 = X3 && !leader ? &tmWlo : &tmWhi, *m2 = X3 ? &tmW3 : &tmWlo;
                        const int ap2 = X3 ? ap + (int)crank * GNB : ap;
                        tma_prefetch_2d(m1, xp, ap);
                        tma_prefetch_2d(m1, xp + 64, ap);
                        tma_prefetch_2d(m2, xp, ap2);
                        tma_prefetch_2d(m2, xp + 64, ap2);
                    }
                    omask |= 1u << os;
                    opar = (opar & ~(1u << os)) | (ph << os);
                    if (++os == GNS) {
                        os = 0;
                        ph ^= 1u;
                    }
                }
            }
            // Drain: every W load has landed before exit (the odd CTA's land on
            // the even CTA's barriers, part of the bytes it expects).
            if (leader) {
#pragma unroll
                for (int i = 0; i < GNS; ++i)
                    if ((omask >> i) & 1u) mbar_drain(&bar->w_full[i], (opar >> i) & 1u, status, lim);
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------ P_Z^T bit loads
        if (lane == 0) {
            prefetch_tmap(&tmZt);
            uint32_t itb = 0, bmask = 0, bpar = 0;
            bool ok = true;
            for (int64_t t = group0; t < ntiles && ok; t += ngroups) {
                int64_t to, tg;
                tile_coords(t, args.tiles_o, args.tiles_g, args.group_o, to, tg);
                const int j0 = (int)(tg * 2 * TM) + (int)crank * TM;  // this CTA's first gate
                for (int kb = 0; kb < (nks + GSPB - 1) / GSPB; ++kb, ++itb) {
                    const uint32_t bs = itb % NBITS;
                    if (!mbar_wait(&bar->bits_empty[bs], ((itb / NBITS) & 1u) ^ 1u, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    uint8_t *bits = smem + C::SM_BITS + bs * C::BT_BYTES;
                    mbar_arrive_expect_tx(&bar->bits_full[bs], C::BT_BYTES);
                    tma_load_2d(bits, &tmZt, &bar->bits_full[bs], kb * 4, j0);  // 256 samples = 4 words
                    bmask |= 1u << bs;
                    bpar = (bpar & ~(1u << bs)) | (((itb / NBITS) & 1u) << bs);
                }
            }
#pragma unroll
            for (int i = 0; i < NBITS; ++i)
                if ((bmask >> i) & 1u) mbar_drain(&bar->bits_full[i], (bpar >> i) & 1u, status, lim);
        }
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            // ------------------------------------------------------------ MMA issuer
            uint32_t os = 0, ph = 0, nchk = 0;
            bool ok = true;
            const uint64_t d_w0 = sdesc_k128(smem_u32(smem) + C::OP_HI);  // W_hi of stage 0, K step 0
            for (int64_t t = group0; t < ntiles && ok; t += ngroups) {
                int kc = 0;
                for (int ks = 0; ks < nks; ++ks) {
                    if (kc == 0 &&
                        !mbar_wait_cluster(&bar->acc_empty, (nchk & 1u) ^ 1u, abort_flag, status, lim)) {
                        // the epilogue warps of both CTAs have read the previous chunk
                        ok = false;
                        break;
                    }
                    if (!mbar_wait_cluster(&bar->a_full[os], ph, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t dhi = d_w0 + (uint64_t)(os * (C::OP_BYTES >> 4));
                    if constexpr (X3)
                        umma_stage8_pair_ts_x3(tmem, tmem + GN, tmem + kGAcol + os * GACOLS, dhi, dhi + (C::OP_LO >> 4),
                                               C::IDESC, C::IDESC2, kc == 0 ? 0u : 1u);
                    else
                        umma_stage8_pair_ts_b(tmem, tmem + kGAcol + os * GACOLS, dhi, dhi + (C::OP_LO >> 4), C::IDESC,
                                              kc == 0 ? 0u : 1u);
                    umma_commit_pair(&bar->empty[os]);
                    if (++kc == chunk || ks == nks - 1) {
                        umma_commit_pair(&bar->acc_full);
                        ++nchk;
                        kc = 0;
                    }
                    if (++os == GNS) {
                        os = 0;
                        ph ^= 1u;
                    }
                }
            }
            umma_commit_pair(&bar->drain);
            mbar_drain(&bar->drain, 0u, status, lim);
        } else if (lane == 0) {
            // Odd CTA: forward "my A half of stage os is in TMEM" to the even CTA.
            const uint32_t a_full_remote = mapa_shared(smem_u32(&bar->a_full[0]), 0u);
            uint32_t os = 0, ph = 0;
            bool ok = true;
            for (int64_t t = group0; t < ntiles && ok; t += ngroups) {
                for (int ks = 0; ks < nks; ++ks) {
                    if (!mbar_wait(&bar->a_peer[os], ph, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_remote(a_full_remote + os * 8u);
                    if (++os == GNS) {
                        os = 0;
                        ph ^= 1u;
                    }
                }
            }
        }
    } else if (warp < GE0) {
        // --------------------------------------- producers: S_Z^T (+-1) into TMEM
        const int quarter = warp & 3;        // TMEM lane quarter
        const int h = (warp - GW0) >> 2;     // 64-sample half of each operand stage
        const int rl = quarter * 32 + lane;  // gate row of this CTA
        uint32_t itb = 0, os = 0, ph = 0, zb[4] = {0u, 0u, 0u, 0u};
        bool ok = true;
        for (int64_t t = group0; t < ntiles && ok; t += ngroups) {
            for (int ks = 0; ks < nks; ++ks) {
                const int q = ks % GSPB;
                const uint32_t bs = itb % NBITS;
                if (q == 0) {
                    if (!wait_warp(&bar->bits_full[bs], (itb / NBITS) & 1u, abort_flag, status, lim)) {
                        ok = false;
                        break;
                    }
                    // this row's bits for its halves of the bits stage's two operand stages
                    const uint8_t *bits = smem + C::SM_BITS + bs * C::BT_BYTES;
                    const uint4 x0 = *reinterpret_cast<const uint4 *>(bits + rl * 32);
                    const uint4 x1 = *reinterpret_cast<const uint4 *>(bits + rl * 32 + 16);
                    zb[0] = h ? x0.z : x0.x;  // operand stage 0: words 2 h, 2 h + 1
                    zb[1] = h ? x0.w : x0.y;
                    zb[2] = h ? x1.z : x1.x;  // operand stage 1: words 4 + 2 h, 5 + 2 h
                    zb[3] = h ? x1.w : x1.y;
                }
                if (!wait_warp(&bar->empty[os], ph ^ 1u, abort_flag, status, lim)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + kGAcol + os * GACOLS + (uint32_t)h * 32u;
#pragma unroll
                for (int wd = 0; wd < 2; ++wd) {
                    const uint32_t b = q == 0 ? zb[wd] : zb[2 + wd];
                    uint32_t v[16];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint4 e = expand_pm1((b >> (8 * i)) & 0xFFu);
                        v[4 * i] = e.x;
                        v[4 * i + 1] = e.y;
                        v[4 * i + 2] = e.z;
                        v[4 * i + 3] = e.w;
                    }
                    tmem_st16(ta + (uint32_t)wd * 16u, v);
                }
                tmem_wait_st();
                tc_fence_before();
                // The even CTA's producers vouch for the stage's W as well
                // (both CTAs' halves complete on its w_full).
                if (leader && !wait_warp_cluster(&bar->w_full[os], ph, abort_flag, status, lim)) {
                    ok = false;
                    break;
                }
                __syncwarp();
                if (lane == 0) {
                    if (leader) mbar_arrive(&bar->a_full[os]);
                    else mbar_arrive(&bar->a_peer[os]);
                }
                if (++os == GNS) {
                    os = 0;
                    ph ^= 1u;
                }
                if (q == GSPB - 1 || ks == nks - 1) {
                    if (lane == 0) mbar_arrive(&bar->bits_empty[bs]);
                    ++itb;
                }
            }
        }
    } else {
        // ---------------------------------------------- epilogue: masked reduction
        const int quarter = warp & 3;
        const int e = (warp - GE0) >> 2;  // column half: observables [GNB e, GNB e + GNB) of the tile
        const int rl = quarter * 32 + lane;
        const uint32_t acc_empty_remote = mapa_shared(smem_u32(&bar->acc_empty), 0u);
        constexpr int NW = GNB / 32;
        uint32_t nchk = 0;
        bool ok = true;
        const int nch = (nks + chunk - 1) / chunk;
        for (int64_t t = group0; t < ntiles && ok; t += ngroups) {
            int64_t to, tg;
            tile_coords(t, args.tiles_o, args.tiles_g, args.group_o, to, tg);
            const int64_t j = tg * 2 * TM + (int64_t)crank * TM + rl;  // gate of this thread
            const int64_t a0 = to * GN + (int64_t)e * GNB;             // first observable of this warp
            // 2 P_A[a][j] for the warp's GNB observables: GNB / 32 words of P_A^T
            // row j (a0 is a multiple of 32); bits of observables >= l are dropped.
            uint32_t mk[NW];
#pragma unroll
            for (int w = 0; w < NW; ++w) mk[w] = 0u;
            if (j < args.m) {
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    const int64_t wi = a0 / 32 + w;
                    if (wi < args.ldlt32 && IQP_IN(j * args.ldlt32 + wi, args.m * args.ldlt32, 56))
                        mk[w] = __ldg(args.pat32 + j * args.ldlt32 + wi);
                    const int64_t rem = args.l - (a0 + 32 * w);  // valid observables in this word
                    if (rem < 32) mk[w] &= rem <= 0 ? 0u : ((1u << rem) - 1u);
                }
            }
            double gsum = 0.0;
            for (int c = 0; c < nch; ++c, ++nchk) {
                if (!wait_warp(&bar->acc_full, nchk & 1u, abort_flag, status, lim)) {
                    ok = false;
                    break;
                }
                __syncwarp();
                tc_fence_after();
                float part = 0.f;
                const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)e * GNB;
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    uint32_t r[32];
                    tmem_ld32(tb + w * 32, r);
                    if (X3) {  // planes 1 and 2
                        uint32_t r2[32];
                        tmem_ld32(tb + GN + w * 32, r2);
#pragma unroll
                        for (int x = 0; x < 32; ++x)
                            r[x] = __float_as_uint(__uint_as_float(r[x]) + __uint_as_float(r2[x]));
                    }
#pragma unroll
                    for (int x = 0; x < 32; ++x)
                        if ((mk[w] >> x) & 1u) part += __uint_as_float(r[x]);
                    if (X3 && w + 1 < NW) {
                        gsum += 2.0 * (double)part;
                        part = 0.f;
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (leader) mbar_arrive(&bar->acc_empty);
                    else mbar_arrive_remote(acc_empty_remote);
                }
                gsum += 2.0 * (double)part;
            }
            if (!ok) break;
            if (j < args.m && IQP_IN((2 * to + e) * args.m + j, 2 * args.tiles_o * args.m, 57))
                args.gpart[(2 * to + e) * args.m + j] = gsum;
        }
    }

    __syncthreads();
    cluster_sync_all();  // no pair MMA or pair-barrier copy still touches the peer
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc_pair(tmem, kTmemCols);
    }
}

// Bounded wait on an mbarrier nothing arrives on: exercises the timeout path.
__global__ void k_timeout_selftest(uint32_t *status, uint64_t limit_ns) {
    __shared__ __align__(8) uint64_t b;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&b, 1);
        abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait(&b, 0u, &abort_flag, status, limit_ns);
    __syncthreads();
}

// ------------------------------------------------------------ tensor maps

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Row-major 2D tensor: `cols` elements per row (dim 0), `rows` rows, row
// pitch `pitch_bytes`; box = box_cols x box_rows.
bool make_map(CUtensorMap *map, const void *base, CUtensorMapDataType dt, int64_t cols, int64_t rows,
              int64_t pitch_bytes, uint32_t box_cols, uint32_t box_rows, CUtensorMapSwizzle swz) {
    EncodeTiledFn fn = encode_fn();
    if (fn == nullptr) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)pitch_bytes};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t es[2] = {1, 1};
    return fn(map, dt, 2, const_cast<void *>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool GRAD, int MODE, int CG, bool AT = GRAD, bool SPL = false, int TA = 0>
cudaError_t launch_k(const CUtensorMap &a, const CUtensorMap &a2, const CUtensorMap &b, const TcArgs &args,
                     cudaStream_t st) {
    constexpr bool kPhasePair = !GRAD && !AT && CG == 2;
    using C = Cfg<CG, GRAD || AT, TA == 1 && kPhasePair, TA == 3 && kPhasePair, TA == 4 && kPhasePair>;
    constexpr int CL = CG;
    static DeviceOnce once;
    const cudaError_t e0 = allow_smem(once, k_tc<GRAD, MODE, CG, AT, SPL, TA>, (int)C::SMEM);
    if (e0 != cudaSuccess) return e0;
    int sms = num_sms();
    if (sms < CL) sms = CL;
    const int64_t groups = args.nunits < sms / CL ? args.nunits : sms / CL;
    LaunchScope ls(GRAD        ? IQP_KERNEL_GRAD_TC
                   : TA == 4   ? (MODE == 1 ? IQP_KERNEL_RECOMPUTE_FP32 : IQP_KERNEL_PHASE_FP32)
                   : MODE == 1 ? IQP_KERNEL_RECOMPUTE_TC
                   : MODE == 3 ? IQP_KERNEL_LOWORDER_GEMM
                               : IQP_KERNEL_PHASE_TC,
                   st);
    if constexpr (CL == 1) {
        launch_pdl(k_tc<GRAD, MODE, 1, AT, SPL, TA>, (unsigned)groups, kThreads, C::SMEM, st, a, a2, b, args);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(groups * CL), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // the kernel begins with pdl_sync
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_tc<GRAD, MODE, CG, AT, SPL, TA>, a, a2, b, args);
}

// Tensor-core group size: CTA pairs unless IQP_CTA_PAIRS=0.
// Row blocks per tile group (IQP_TILE_GROUP, 1..64; default 8; 1 = plain
// row-major order).
int64_t tile_group() {
    static int64_t g = -1;
    if (g < 0) {
        const char *e = std::getenv("IQP_TILE_GROUP");
        const long v = e ? std::atol(e) : 8;
        g = (v >= 1 && v <= 64) ? v : 8;
    }
    return g;
}

// Split the last round of phase tiles across idle CTA groups unless
// IQP_SPLIT_TAIL=0.
bool split_tail() {
    static int v = -1;
    if (v < 0) {
        const char *e = std::getenv("IQP_SPLIT_TAIL");
        v = (e != nullptr && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

// Observable blocks per tile group of the pair gradient (IQP_GRAD_GROUP,
// 1..64; default 4). Each block's W panel (256 observables x s samples, hi
// and lo) is read by every gate block of its group; the group's panels must
// stay in L2 while the group sweeps the gate blocks, or W is read from DRAM
// once per round of tiles.
int64_t grad_group() {
    static int64_t g = -1;
    if (g < 0) {
        const char *e = std::getenv("IQP_GRAD_GROUP");
        const long v = e ? std::atol(e) : 4;
        g = (v >= 1 && v <= 64) ? v : 4;
    }
    return g;
}

// Accumulation chunk lengths: gates per chunk of the phase kernels
// (IQP_PHASE_CHUNK, a multiple of 256 from 256 to 65536; default 8192) and
// the longest chunk of the pair gradient in samples (IQP_GRAD_CHUNK, a
// multiple of 128 from 128 to 65536; default 10240). A chunk boundary stalls
// the MMAs while the accumulator is read; a longer chunk lets the tensor
// core's truncating FP32 accumulation drift further. On 10^4 x 10^4 x 10^5
// with theta ~ U(-0.05, 0.05) the gradient's relative error is 1.9e-5 at 4096
// gates, 2.7e-5 at 8192 and 5.3e-5 at 16384; the gradient chunk moves it by
// less than 4e-6 between 2560 and 10240 samples.
int64_t env_multiple(const char *name, int64_t unit, int64_t dflt) {
    const char *e = std::getenv(name);
    const long v = e ? std::atol(e) : dflt;
    return (v >= unit && v <= 65536 && v % unit == 0) ? v : dflt;
}
int64_t phase_chunk_gates() {
    static int64_t g = -1;
    if (g < 0) g = env_multiple("IQP_PHASE_CHUNK", 256, 8192);
    return g;
}
int64_t grad_chunk_samples() {
    static int64_t g = -1;
    if (g < 0) g = env_multiple("IQP_GRAD_CHUNK", 128, 10240);
    return g;
}

// Serpentine gate order for the phase kernels' whole tiles (IQP_PHASE_SERP;
// default 1; 0 = every tile walks the gates forwards).
bool phase_serp() {
    static int v = -1;
    if (v < 0) {
        const char *e = std::getenv("IQP_PHASE_SERP");
        v = (e != nullptr && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

// Phase kernels of CTA pairs: full rounds of tiles of two sample tiles
// (256 observables x 512 samples) against each A stage, the rest as single
// tiles (IQP_PHASE_DT; default 1; 0 = single tiles only).
bool phase_dt() {
    static int v = -1;
    if (v < 0) {
        const char *e = std::getenv("IQP_PHASE_DT");
        v = (e != nullptr && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

// Phase kernels of CTA pairs with the A operand in TMEM (default) or in
// shared memory (IQP_PHASE_TMEM=0).
bool phase_tmem() {
    static int v = -1;
    if (v < 0) {
        const char *e = std::getenv("IQP_PHASE_TMEM");
        v = (e != nullptr && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

// Gradient contraction as CTA pairs in the transposed orientation
// (k_grad_pair, default) or single CTAs (IQP_GRAD_PAIR=0, or IQP_CTA_PAIRS=0).
bool grad_pair() {
    static int v = -1;
    if (v < 0) {
        const char *e = std::getenv("IQP_GRAD_PAIR");
        v = (e != nullptr && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

int cta_group() {
    static int cg = -1;
    if (cg < 0) {
        const char *e = std::getenv("IQP_CTA_PAIRS");
        cg = (e != nullptr && e[0] == '0') ? 1 : 2;
    }
    return cg;
}

// FP32 form on the tensor cores (IQP_FP32_TC; default 1; 0 = the SIMT kernels).
bool fp32_tc() {
    static int v = -1;
    if (v < 0) {
        const char *e = std::getenv("IQP_FP32_TC");
        v = (e != nullptr && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

// Every tile whole (no split parts).
void whole_tiles(TcArgs &a, int64_t ntiles) {
    a.nunits = a.whole = ntiles;
    a.skp = nullptr;
}

template <class T>
T *at(void *ws, size_t off) {
    return reinterpret_cast<T *>(static_cast<char *>(ws) + off);
}

}  // namespace

namespace {
// Two sample tiles per tile (CTA pairs): whole tiles, or (SPL) the pieces of
// a balanced split of the last round.
template <bool SPL>
cudaError_t launch_phase_dt_k(int mode, const CUtensorMap &ma, const CUtensorMap &mb, const TcArgs &a,
                              cudaStream_t st) {
    if (mode == 0) return launch_k<false, 0, 2, false, SPL, 3>(ma, ma, mb, a, st);
    if (mode == 1) return launch_k<false, 1, 2, false, SPL, 3>(ma, ma, mb, a, st);
    return launch_k<false, 2, 2, false, SPL, 3>(ma, ma, mb, a, st);
}

template <bool SPL>
cudaError_t launch_phase_x3_k(int mode, const CUtensorMap &ma, const CUtensorMap &mb, const TcArgs &a,
                              cudaStream_t st) {
    if (mode == 0) return launch_k<false, 0, 2, false, SPL, 4>(ma, ma, mb, a, st);
    if (mode == 1) return launch_k<false, 1, 2, false, SPL, 4>(ma, ma, mb, a, st);
    return launch_k<false, 2, 2, false, SPL, 4>(ma, ma, mb, a, st);
}

template <bool SPL>
cudaError_t launch_phase_k(int mode, int cg, const CUtensorMap &ma, const CUtensorMap &mb, const TcArgs &a,
                           cudaStream_t st) {
    if (cg == 2 && phase_tmem()) {
        if (mode == 0) return launch_k<false, 0, 2, false, SPL, 1>(ma, ma, mb, a, st);
        if (mode == 1) return launch_k<false, 1, 2, false, SPL, 1>(ma, ma, mb, a, st);
        return launch_k<false, 2, 2, false, SPL, 1>(ma, ma, mb, a, st);
    }
    if (cg == 2) {
        if (mode == 0) return launch_k<false, 0, 2, false, SPL>(ma, ma, mb, a, st);
        if (mode == 1) return launch_k<false, 1, 2, false, SPL>(ma, ma, mb, a, st);
        return launch_k<false, 2, 2, false, SPL>(ma, ma, mb, a, st);
    }
    if (mode == 0) return launch_k<false, 0, 1, false, SPL>(ma, ma, mb, a, st);
    if (mode == 1) return launch_k<false, 1, 1, false, SPL>(ma, ma, mb, a, st);
    return launch_k<false, 2, 1, false, SPL>(ma, ma, mb, a, st);
}
}  // namespace

namespace {
// Times the choices below weigh, in us: a bits stage of a tile (of two sample
// tiles: DT), and what a split costs beside its products (parts of 256 or 512 KB
// per CTA pair to store, add up and launch; about P + tiles of them whatever the
// sizes: 17 us of adding up for 84 DT parts, as much again for the rest).
constexpr double kStageUs = 2.6, kStageDtUs = 4.8, kSplitUs = 20.0, kSplitDtUs = 35.0;

// Balanced split of `left` tiles (from tile `first` on) over P CTA groups: their
// bits stages, end to end, in equal ranges, one per group, each range's piece of
// a tile a part (see unit_of). skp: scratch of `slots` accumulators. Returns
// false, and leaves the tiles whole, where that saves less than it costs: (1 -
// left / P) of the tiles' K loop. 4 double tiles left on 76 pairs, 177 stages: 517
// -> 83 us with the parts added up over the chip (k_split_reduce). 40 tiles of 12
// stages: whole 72 us, split 80. Where the tiles fill half the groups at most,
// or `always`, they are split in any case: there are few parts to add up, and
// sums of shorter ranges lose less to the tensor core's truncation (standard
// errors of small circuits 6e-7 relative, 1.1e-6 with whole tiles).
bool balance(TcArgs &a, int64_t first, int64_t left, int64_t P, int cg, int nh, float *skp, int64_t slots,
             bool always = false) {
    const int64_t nkb = cdiv(a.nks, KB / KS), W = left * nkb;
    const double stage = nh == 2 ? kStageDtUs : kStageUs, cost = nh == 2 ? kSplitDtUs : kSplitUs;
    if (!split_tail() || skp == nullptr || left <= 0 || nkb < 2) return false;
    if (P > W) P = W;  // at least one bits stage per range
    const int64_t fit = slots / (cg * nh) - left + 1;  // P ranges over `left` tiles are at most P + left - 1 pieces
    if (P > fit) P = fit;
    if (P <= left) return false;
    if (!always && 2 * left > P && (double)(nkb * (P - left)) * stage <= cost * (double)P) return false;
    a.whole = first;
    a.nunits = P * (cdiv(W / P + 1, nkb) + 2);
    a.skW = W;
    a.skP = P;
    a.skp = skp;
    a.skcap = slots * kSplitSlotFloats;
    return true;
}

cudaError_t launch_split_reduce(int mode, bool x3, const TcArgs &a, int cg, int nh, int64_t tiles, cudaStream_t st) {
    const unsigned blocks = (unsigned)(tiles * cg * nh * TM * 4 / 8);
    LaunchScope ls(x3 ? (mode == 1 ? IQP_KERNEL_RECOMPUTE_FP32 : IQP_KERNEL_PHASE_FP32)
                      : (mode == 1 ? IQP_KERNEL_RECOMPUTE_TC : IQP_KERNEL_PHASE_TC),
                   st);
    if (x3) {
        if (mode == 0) launch_pdl(k_split_reduce<0, true>, blocks, 256, 0, st, a, cg, nh, tiles);
        else if (mode == 1) launch_pdl(k_split_reduce<1, true>, blocks, 256, 0, st, a, cg, nh, tiles);
        else launch_pdl(k_split_reduce<2, true>, blocks, 256, 0, st, a, cg, nh, tiles);
    } else {
        if (mode == 0) launch_pdl(k_split_reduce<0, false>, blocks, 256, 0, st, a, cg, nh, tiles);
        else if (mode == 1) launch_pdl(k_split_reduce<1, false>, blocks, 256, 0, st, a, cg, nh, tiles);
        else launch_pdl(k_split_reduce<2, false>, blocks, 256, 0, st, a, cg, nh, tiles);
    }
    return cudaGetLastError();
}

// The T single tiles of a phase: full rounds of whole tiles, then the last
// round's tiles as a balanced split where that pays (skp: its scratch, or null).
cudaError_t launch_single_tiles(int mode, int cg, bool x3, const CUtensorMap &ma, const CUtensorMap &mb, TcArgs a,
                                int64_t T, float *skp, int64_t slots, cudaStream_t st) {
    int sms = num_sms();
    if (sms > kMaxSplitCtas) sms = kMaxSplitCtas;
    const int64_t P = sms / cg;  // CTA groups
    auto run = [&](bool split, const TcArgs &w) {
        if (x3) return split ? launch_phase_x3_k<true>(mode, ma, mb, w, st) : launch_phase_x3_k<false>(mode, ma, mb, w, st);
        return split ? launch_phase_k<true>(mode, cg, ma, mb, w, st) : launch_phase_k<false>(mode, cg, ma, mb, w, st);
    };
    const int64_t R = P >= 1 ? T % P : 0;
    TcArgs b = a;
    whole_tiles(a, T);
    if (!balance(b, T - R, R, P, cg, 1, skp, slots)) return run(false, a);
    if (T - R > 0) {
        whole_tiles(a, T - R);
        const cudaError_t e = run(false, a);
        if (e != cudaSuccess) return e;
    }
    const cudaError_t e = run(true, b);
    return e != cudaSuccess ? e : launch_split_reduce(mode, x3, b, cg, 1, R, st);
}
}  // namespace

// Whether the FP32 form runs on the tensor cores here (its planes also need
// the plan's optional regions).
bool x3_available() { return fp32_tc() && num_sms() >= 2 && num_sms() <= kMaxSplitCtas && iqp_tensor_path_available(); }

cudaError_t launch_phase_tc(int mode, const Plan &p, void *ws, const double *alpha, const double *beta,
                            cudaStream_t st, iqp_status *why) {
    const int cg = cta_group();
    CUtensorMap ma, mb;
    if (!make_map(&ma, at<uint64_t>(ws, p.off_pa), CU_TENSOR_MAP_DATA_TYPE_UINT64, p.ldp, p.l, p.ldp * 8, 4, TM,
                  CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map(&mb, at<uint64_t>(ws, p.off_pz), CU_TENSOR_MAP_DATA_TYPE_UINT64, p.ldp, p.s, p.ldp * 8, 4,
                  (uint32_t)(TN / cg), CU_TENSOR_MAP_SWIZZLE_NONE)) {
        *why = IQP_ERR_UNSUPPORTED;
        return cudaErrorNotSupported;
    }
    TcArgs a{};  // every field zero unless set below
    a.l = p.l;
    a.s = p.s;
    a.m = p.m;
    a.nks = cdiv(p.m, KS);
    a.chunk = phase_chunk_gates() / KS;  // operand stages per accumulation chunk
    a.tiles_m = cdiv(p.l, TM * cg);
    a.tiles_n = cdiv(p.s, TN);
    a.group_m = tile_group();
    a.chi = at<__nv_bfloat16>(ws, p.off_c);
    a.mpad = p.mpad;
    a.clo = a.chi + p.mpad;
    a.part = at<double2>(ws, p.off_part);
    a.nparts = p.nparts;
    a.alpha = alpha;
    a.beta = beta;
    a.whi = at<__nv_bfloat16>(ws, p.off_w);
    a.wlo = a.whi + p.l * p.ldw;
    a.ldw = p.ldw;
    a.pa32 = nullptr;
    a.ldp32 = 2 * p.ldp;
    a.gpart = nullptr;
    // MODE 0 keeps Phi (FP32, l x ldw) when a gradient pass follows.
    a.out = (mode == 0 && p.phi_out) ? p.phi : nullptr;
    a.ldo = p.ldphi;
    a.status = at<uint32_t>(ws, p.off_status);
    a.limit_ns = default_spin_limit_ns();
    a.serp = phase_serp() ? 1 : 0;
    // Two sample tiles per tile: the full rounds of double tiles (256 x 512)
    // run in one launch; the double tiles of the last, partial round continue
    // below as single tiles (tile t = half t % 2 of double tile dbase + t / 2).
    int64_t T = a.tiles_m * a.tiles_n;
    {
        int sms = num_sms();
        if (sms > kMaxSplitCtas) sms = kMaxSplitCtas;
        const int64_t P = sms / 2;  // CTA pairs
        const int64_t tiles_n2 = cdiv(p.s, 2 * TN);
        const int64_t T2 = a.tiles_m * tiles_n2;
        if (cg == 2 && phase_dt() && p.off_gsum != 0 && num_sms() <= kMaxSplitCtas && P >= 1) {
            const int64_t full = (T2 / P) * P, left = T2 - full;
            TcArgs d = a;
            d.tiles_n = tiles_n2;
            d.gsum = at<float4>(ws, p.off_gsum);
            TcArgs b = d;
            bool bal = left > 0 && p.off_skx != 0 && balance(b, full, left, P, 2, 2, at<float>(ws, p.off_skx), kSplitSlots, full > 0);
            if (bal && full == 0) {  // less than a round: against single tiles, whole or split
                const double k = (double)cdiv(a.nks, KB / KS) * kStageUs, w = k * (double)cdiv(T, P);
                const double sp = k * (double)T / (double)P + kSplitUs;
                bal = (double)left / (double)P * (double)cdiv(a.nks, KB / KS) * kStageDtUs + kSplitDtUs < (w < sp ? w : sp);
            }
            if (full > 0 || bal) {
                if (full > 0) {
                    whole_tiles(d, full);
                    const cudaError_t e = launch_phase_dt_k<false>(mode, ma, mb, d, st);
                    if (e != cudaSuccess || left == 0) return e;
                }
                if (bal) {
                    const cudaError_t e = launch_phase_dt_k<true>(mode, ma, mb, b, st);
                    return e != cudaSuccess ? e : launch_split_reduce(mode, false, b, 2, 2, left, st);
                }
                a.dtmap = 1;
                a.dbase = full;
                a.tiles_n2 = tiles_n2;
                T = 2 * left;
            }
        }
    }
    float *skp = p.off_skp != 0 ? at<float>(ws, p.off_skp) : nullptr;
    int64_t slots = kMaxSplitCtas;
    if (p.off_skx != 0) {
        skp = at<float>(ws, p.off_skx);
        slots = kSplitSlots;
    }
    return launch_single_tiles(mode, cg, false, ma, mb, a, T, skp, slots, st);
}

// The FP32 form's phase (p.x3): the same contraction with 2 theta as three
// planes (k_tc, TA = 4). mode 0: statistics; 1: W (FP32) and its row maxima;
// 2: both.
cudaError_t launch_phase_x3(int mode, const Plan &p, void *ws, const double *alpha, const double *beta,
                            cudaStream_t st, iqp_status *why) {
    CUtensorMap ma, mb;
    if (!make_map(&ma, at<uint64_t>(ws, p.off_pa), CU_TENSOR_MAP_DATA_TYPE_UINT64, p.ldp, p.l, p.ldp * 8, 4, TM,
                  CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map(&mb, at<uint64_t>(ws, p.off_pz), CU_TENSOR_MAP_DATA_TYPE_UINT64, p.ldp, p.s, p.ldp * 8, 4,
                  (uint32_t)(TN / 2), CU_TENSOR_MAP_SWIZZLE_NONE)) {
        *why = IQP_ERR_UNSUPPORTED;
        return cudaErrorNotSupported;
    }
    TcArgs a{};  // every field zero unless set below
    a.l = p.l;
    a.s = p.s;
    a.m = p.m;
    a.nks = cdiv(p.m, KS);
    a.chunk = cdiv(a.nks, cdiv(a.nks, (int64_t)(kX3Gates / KS)));  // fewest chunks, balanced
    a.tiles_m = cdiv(p.l, 2 * TM);
    a.tiles_n = cdiv(p.s, TN);
    a.group_m = tile_group();
    a.chi = at<__nv_bfloat16>(ws, p.off_xc);
    a.clo = a.chi + p.mpad;
    a.c3 = a.clo + p.mpad;
    a.mpad = p.mpad;
    a.part = at<double2>(ws, p.off_xpart);
    a.nparts = cdiv(p.s, (int64_t)kPartColsTc);
    a.alpha = alpha;
    a.beta = beta;
    a.ldw = p.ldw;
    if (mode != 0) {
        a.wf = at<float>(ws, p.off_w);
        a.wmax = at<uint32_t>(ws, p.off_xrow);  // zeroed by k_x3_theta
    }
    a.status = at<uint32_t>(ws, p.off_status);
    a.limit_ns = default_spin_limit_ns();
    a.serp = phase_serp() ? 1 : 0;
    a.gsum = at<float4>(ws, p.off_xsum);
    if (mode == 0 && p.phi_out) {  // Phi for the gradient pass
        a.out = p.phi;
        a.ldo = p.ldphi;
    }
    return launch_single_tiles(mode, 2, true, ma, mb, a, a.tiles_m * a.tiles_n, at<float>(ws, p.off_skp), kX3Slots, st);
}

// Phase pass of the FP32 form's gradient where Phi was kept.
cudaError_t launch_x3_w(const Plan &p, void *ws, const double *alpha, const double *beta, cudaStream_t st) {
    int64_t blocks = p.l * cdiv(p.s, (int64_t)2048);
    if (blocks > 65536) blocks = 65536;
    LaunchScope ls(IQP_KERNEL_RECOMPUTE_FP32, st);
    launch_pdl(k_x3_w, (unsigned)blocks, 256, 0, st, p.phi, p.ldphi, at<float>(ws, p.off_w), p.ldw, p.l, p.s, alpha, beta,
                                             at<uint32_t>(ws, p.off_xrow));
    return cudaGetLastError();
}

cudaError_t launch_x3_theta(const Plan &p, void *ws, const float *theta, cudaStream_t st) {
    float *bsum = at<float>(ws, p.off_xsums);
    const int64_t nb = p.m <= kX3Gates ? 0 : cdiv(p.m, (int64_t)kX3Gates);
    if (nb > 0) {
        LaunchScope ls(IQP_KERNEL_THETA_SPLIT, st);
        launch_pdl(k_x3_csum, (unsigned)nb, 256, 0, st, theta, p.m, bsum);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    int64_t blocks = cdiv(p.mpad, 256);
    if (blocks > 4096) blocks = 4096;
    LaunchScope ls(IQP_KERNEL_THETA_SPLIT, st);
    launch_pdl(k_x3_theta, (unsigned)blocks, 256, 0, st, theta, p.m, p.mpad, bsum, nb, at<__nv_bfloat16>(ws, p.off_xc),
                                                 p.off_xw != p.off_xrow ? at<uint32_t>(ws, p.off_xrow) : nullptr, p.l);
    return cudaGetLastError();
}

namespace {
// Observables o0 .. o0 + l (X3: the planes hold these alone; else all).
template <bool X3>
cudaError_t launch_grad_pair(const Plan &p, void *ws, int64_t o0, int64_t l, cudaStream_t st, iqp_status *why) {
    using C = GCfg<X3>;
    CUtensorMap mhi, mlo, m3, mz;
    const __nv_bfloat16 *whi = at<__nv_bfloat16>(ws, X3 ? p.off_xw : p.off_w);
    const __nv_bfloat16 *wlo = whi + l * p.ldw;
    if (!make_map(&mhi, whi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.s, l, p.ldw * 2, KS, GNB,
                  CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&mlo, wlo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.s, l, p.ldw * 2, KS, GNB,
                  CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&m3, X3 ? wlo + l * p.ldw : wlo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.s, l, p.ldw * 2, KS, 64,
                  CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&mz, at<uint64_t>(ws, p.off_pzt), CU_TENSOR_MAP_DATA_TYPE_UINT64, p.ldzt, p.m, p.ldzt * 8, 4, TM,
                  CU_TENSOR_MAP_SWIZZLE_NONE)) {
        *why = IQP_ERR_UNSUPPORTED;
        return cudaErrorNotSupported;
    }
    GradArgs a;
    a.l = l;
    a.s = p.s;
    a.m = p.m;
    a.nks = cdiv(p.s, GKS);
    const int64_t cmax = (X3 ? (int64_t)1 << kX3SampleBits : grad_chunk_samples()) / GKS;
    a.chunk = cdiv(a.nks, cdiv(a.nks, cmax));  // fewest chunks, balanced
    a.tiles_g = cdiv(p.m, 2 * TM);
    a.tiles_o = cdiv(l, (int64_t)C::OBS);
    a.group_o = grad_group() * (GN / C::OBS);
    a.pat32 = at<uint32_t>(ws, p.off_pat) + o0 / 32;  // whole tiles of 128 observables end inside a row
    a.ldlt32 = 2 * p.ldlt;
    a.gpart = at<double>(ws, p.off_gpart) + 2 * (o0 / C::OBS) * p.m;
    a.status = at<uint32_t>(ws, p.off_status);
    a.limit_ns = default_spin_limit_ns();
    static DeviceOnce once;
    const cudaError_t e0 = allow_smem(once, k_grad_pair<X3>, (int)C::SMEM);
    if (e0 != cudaSuccess) return e0;
    int sms = num_sms();
    if (sms < 2) sms = 2;
    const int64_t ntiles = a.tiles_g * a.tiles_o;
    const int64_t groups = ntiles < sms / 2 ? ntiles : sms / 2;
    LaunchScope ls(X3 ? IQP_KERNEL_GRAD_FP32 : IQP_KERNEL_GRAD_TC, st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(groups * 2), 1, 1);
    cfg.blockDim = dim3(kGThreads, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // the kernel begins with pdl_sync
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_grad_pair<X3>, mhi, mlo, m3, mz, a);
}
}  // namespace

// Rows of FP64 gradient partials the gradient contraction writes: two per
// 256-observable tile for the CTA-pair kernel, one per 128-observable tile
// for the single-CTA kernel (IQP_GRAD_PAIR=0 or IQP_CTA_PAIRS=0).
int64_t grad_tc_rows(const Plan &p) { return cta_group() == 2 && grad_pair() ? 2 * cdiv(p.l, GN) : cdiv(p.l, TM); }

// The FP32 form's gradient contraction (p.x3): W taken apart into its planes,
// then k_grad_pair<true>, for as many observables at a time as the planes hold; 2
// ceil(l / 128) rows of partials.
cudaError_t launch_grad_x3(const Plan &p, void *ws, cudaStream_t st, iqp_status *why) {
    const int64_t rows = x3_rows(p.l, p.ldw);
    for (int64_t o0 = 0; o0 < p.l; o0 += rows) {
        const int64_t l = p.l - o0 < rows ? p.l - o0 : rows;
        int64_t grid = cdiv(l * cdiv(p.s, (int64_t)8), 256);
        const int64_t cap = (int64_t)num_sms() * 8;
        if (grid > cap) grid = cap;
        {
            LaunchScope ls(IQP_KERNEL_RECOMPUTE_FP32, st);
            launch_pdl(k_x3_wsplit, (unsigned)grid, 256, 0, st, at<float>(ws, p.off_w) + o0 * p.ldw, p.ldw, l, p.s,
                       at<uint32_t>(ws, p.off_xrow) + o0, at<__nv_bfloat16>(ws, p.off_xw));
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
        const cudaError_t e = launch_grad_pair<true>(p, ws, o0, l, st, why);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_grad_tc(const Plan &p, void *ws, cudaStream_t st, iqp_status *why) {
    if (cta_group() == 2 && grad_pair()) return launch_grad_pair<false>(p, ws, 0, p.l, st, why);
    const int cg = 1;
    CUtensorMap mhi, mlo, mb;
    const __nv_bfloat16 *whi = at<__nv_bfloat16>(ws, p.off_w);
    const __nv_bfloat16 *wlo = whi + p.l * p.ldw;
    const uint32_t wrows = TM;
    if (!make_map(&mhi, whi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.s, p.l, p.ldw * 2, KS, wrows,
                  CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&mlo, wlo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.s, p.l, p.ldw * 2, KS, wrows,
                  CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&mb, at<uint64_t>(ws, p.off_pzt), CU_TENSOR_MAP_DATA_TYPE_UINT64, p.ldzt, p.m, p.ldzt * 8, 4,
                  (uint32_t)(TN / cg), CU_TENSOR_MAP_SWIZZLE_NONE)) {
        *why = IQP_ERR_UNSUPPORTED;
        return cudaErrorNotSupported;
    }
    TcArgs a{};  // every field zero unless set below
    a.l = p.l;
    a.s = p.s;
    a.m = p.m;
    a.nks = cdiv(p.s, KS);
    a.chunk = 32;  // 2048 samples per accumulation chunk
    a.tiles_m = cdiv(p.l, TM * cg);
    a.tiles_n = cdiv(p.m, TN);
    a.group_m = tile_group();
    a.chi = a.clo = nullptr;
    a.mpad = 0;
    a.part = nullptr;
    a.nparts = 0;
    a.alpha = a.beta = nullptr;
    a.whi = a.wlo = nullptr;
    a.ldw = p.ldw;
    a.pa32 = at<uint32_t>(ws, p.off_pa);
    a.ldp32 = 2 * p.ldp;
    a.gpart = at<double>(ws, p.off_gpart);
    a.out = nullptr;
    a.ldo = 0;
    whole_tiles(a, a.tiles_m * a.tiles_n);
    a.status = at<uint32_t>(ws, p.off_status);
    a.limit_ns = default_spin_limit_ns();
    return launch_k<true, 0, 1>(mhi, mlo, mb, a, st);
}

cudaError_t launch_w_from_phi(const Plan &p, void *ws, const double *alpha, const double *beta, cudaStream_t st) {
    if (p.phi == nullptr || p.ldw % 4 != 0 || p.ldphi % 4 != 0) return cudaErrorInvalidValue;
    __nv_bfloat16 *whi = at<__nv_bfloat16>(ws, p.off_w);
    __nv_bfloat16 *wlo = whi + p.l * p.ldw;
    const int64_t total = p.l * (p.ldw / 4);
    int64_t grid = cdiv(total, 256);
    const int64_t cap = (int64_t)num_sms() * 8;
    if (grid > cap) grid = cap;
    if (grid < 1) grid = 1;
    LaunchScope ls(IQP_KERNEL_RECOMPUTE_TC, st);
    launch_pdl(k_w_from_phi, (unsigned)grid, 256, 0, st, p.phi, p.ldphi, p.ldw, p.l, p.s, alpha, beta, whi, wlo);
    return cudaGetLastError();
}

cudaError_t launch_tc_dense(const __nv_bfloat16 *a_hi, const __nv_bfloat16 *a_lo, int64_t rows, int64_t kpad,
                            int64_t k, const uint64_t *b_bits, int64_t nb, int64_t ldb, float *out, int64_t ldo,
                            int kparts, const float *d, const uint64_t *zt, int64_t ldzt, uint32_t *status,
                            cudaStream_t st) {
    // Single CTAs: their half-size tiles fill the last round better, and with A by
    // TMA the producers have only the +-1 rows to expand. n = 5000, 16384 samples:
    // X 1009 us (CTA pairs 1124), H 1047 (1236); 1000 x 5000 40 either way. H in
    // K pieces keeps the pairs: its pieces are counted for them.
    const int cg = kparts == 1 ? 1 : cta_group();
    CUtensorMap mhi, mlo, mb;
    if (kpad % KS != 0 || k > kpad || k > 64 * ldb || ldb % 2 != 0 || ldb < 4 || ldo % 4 != 0 ||
        !make_map(&mhi, a_hi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, kpad, rows, kpad * 2, KS, TM,
                  CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&mlo, a_lo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, kpad, rows, kpad * 2, KS, TM,
                  CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&mb, b_bits, CU_TENSOR_MAP_DATA_TYPE_UINT64, ldb, nb, ldb * 8, 4, (uint32_t)(TN / cg),
                  CU_TENSOR_MAP_SWIZZLE_NONE))
        return cudaErrorNotSupported;
    TcArgs a{};  // every field zero unless set below
    a.l = rows;
    a.s = nb;
    a.m = k;
    a.nks = cdiv(k, KS);
    a.chunk = 64;
    a.tiles_m = cdiv(rows, TM * cg);
    a.tiles_n = cdiv(nb, TN);
    a.group_m = tile_group();
    a.chi = a.clo = nullptr;
    a.mpad = 0;
    a.part = nullptr;
    a.nparts = 0;
    a.alpha = a.beta = nullptr;
    a.whi = a.wlo = nullptr;
    a.ldw = 0;
    a.pa32 = nullptr;
    a.ldp32 = 0;
    a.gpart = nullptr;
    a.out = out;
    a.ldo = ldo;
    a.kparts = kparts;
    a.out_part = rows * ldo;
    a.dvec = d;
    a.zt32 = reinterpret_cast<const uint32_t *>(zt);
    a.ldzt32 = 2 * ldzt;
    whole_tiles(a, a.tiles_m * a.tiles_n);
    a.nunits *= kparts;
    a.status = status;
    a.limit_ns = default_spin_limit_ns();
    if (cg == 2) return launch_k<false, 3, 2, true>(mhi, mlo, mb, a, st);
    return launch_k<false, 3, 1, true>(mhi, mlo, mb, a, st);
}

cudaError_t launch_timeout_selftest(uint32_t *status, uint64_t limit_ns, cudaStream_t st) {
    LaunchScope ls(IQP_KERNEL_SELFTEST, st);
    k_timeout_selftest<<<1, 32, 0, st>>>(status, limit_ns);
    return cudaGetLastError();
}

}  // namespace iqp
