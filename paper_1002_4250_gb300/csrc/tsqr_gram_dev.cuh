// Device code of the exact-Gram reduction (tsqr_gram.cuh has the method): digits of a slab of
// rows into tensor-core operands, their exact sums, the tree over the slabs, and the
// fixed-point Cholesky factor of the whole.
#pragma once

#include <type_traits>

#include "tsqr_fold.cuh"
#include "tsqr_gram.cuh"
#include "tsqr_tc.cuh"

namespace tsqr {
namespace gram {

typedef unsigned long long u64;
typedef __int128 i128;
typedef unsigned __int128 u128;

constexpr int kDigits = 8;       // of a column
constexpr int kBlock = 32;       // columns of a block
// The least pivot a column may keep, relative to its square (2^-kPivotBits).
constexpr int kPivotBits = 64;
// Biased exponents a column's largest entry may have: outside, squares leave FP64's range (or
// come near it) and the Householder reduction decides what R is.  A slab's exponent word goes no
// lower than kLeastD, whatever its entries; a column that is there in every slab has lost digits
// (2^-430: half of them), or is zero, and is not served.
constexpr int kExpLo = 1023 - 400, kExpHi = 1023 + 400;
constexpr int kLeastD = kExpLo + 4;
constexpr int kUnit = -1086;     // |x| = Q 2^(D + kUnit) for a column's exponent word D

constexpr int cmin(int a, int b) { return a < b ? a : b; }
constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Shape of a column set: NI columns against themselves (NJ = 0), or against NJ others.
// Operand rows: digit s of column i at s NI + i, then digit t of column j at S NI + t NJ + j.
template <int NI, int NJ>
struct Shape {
    static constexpr int S = kDigits;
    static constexpr bool kCross = NJ > 0;
    static constexpr int MN = S * (NI + NJ);
    // Row tiles of 128 accumulator lanes: TS digits of the NI columns each.  A block against
    // itself needs a second tile only for its low digits against each other, (s, t) and (t, s)
    // being mirrors: tile 1 takes digits TS .. S-1 against TS .. TE-1 (FP64: digits 4 to 7 against
    // 4 and 5; what is left out, both digits 6 or 7, is below 2^-96 of the product).
    static constexpr int TS = NI > 16 ? 4 : S;
    static constexpr int kTiles = TS < S ? 2 : 1;
    static constexpr int TE = kCross || kTiles == 1 ? S : 6;
    static constexpr int NR = kCross ? NJ : NI;            // columns of a right-hand digit
    static constexpr int N0 = S * NR;
    static constexpr int N1 = kTiles == 1 ? 0 : kCross ? N0 : (TE - TS) * NI;
    // Narrow sets put two 64-row blocks into one product: block k+1's operand rows follow block
    // k's, so a 128-row tile against twice the columns holds both blocks' sums on its diagonal
    // (a product takes some 95 cycles however few its columns).
    static constexpr int kPair = !kCross && MN <= 64 ? 2 : 1;
    static constexpr int kCols = kPair * N0 + N1;          // tensor-memory columns
    static constexpr int kSets = cmin(8, 512 / kCols);     // accumulator sets, 1,024 rows each
    static_assert((kSets & (kSets - 1)) == 0, "a power of two");
    static_assert(kCols <= 512 && (kTiles == 1 || 2 * TS >= S), "accumulators fit");
    // Slicing: a task is four columns of a 64-row block, each warp has one a round.
    static constexpr int kGroups = (NI + NJ) / 4;
    static constexpr int kRoundKb = kGramSlicers / kGroups;
    static_assert(kRoundKb >= 1, "a block a round");
    static constexpr int kKbBytes = MN * 128;              // 64 FP16 per operand row
    static constexpr int kStage = kRoundKb * kKbBytes;
    static constexpr int kRaw = kGramSlicers * 2048;         // a round of A: 64 bytes a lane
    static constexpr int kRaws = 2;                        // rounds on their way
    // Flush: partial sums (64-bit) of JP columns at a time over the stages, [half][row digit]
    // [j][i]; halves: digits 0-3 and 4-7 of the right-hand columns.
    static constexpr bool kMirror = !kCross && kTiles == 2;
    static constexpr int kRowDigits = kCross ? S : TS;
    static constexpr int kLd = NI + 1;
    static constexpr int per_j() {
        return (kPair * kRowDigits * 2 + (kMirror ? S - TS : 0)) * kLd * 8;
    }
    static constexpr int kStages = 2 * kStage;
    static constexpr int jp() {
        int j = NR;
        while (j * per_j() > kStages) j = (j / 2 + 7) / 8 * 8;
        return j;
    }
    static constexpr int JP = jp();
    static_assert(JP % 8 == 0 && NR % JP == 0 && JP * per_j() <= kStages, "flush buffers");
    static constexpr int kU = NI * NR * 16;                // the 128-bit sums
};

struct alignas(16) Smem {   // beside the stages
    uint64_t full[2];       // a stage is sliced: one arrival a warp
    uint64_t free[2];       // a stage is multiplied: the tensor cores' commit
    uint64_t drain;         // all tensor-core work so far is done
    uint32_t tmem;
    int flag, bad, item;
    int above[2];           // a stage's round has an entry above its column's range
    int stop;               // the round that was not multiplied for it; -1: none
    int D[128], E[128], Dnew[128];
};

// Shared memory: Smem, stages, raw rounds, U.  (Tile reads past the last operand row fall into
// the raw rounds: rows and columns that no one reads back.)
constexpr int kHead = 2048;
static_assert(sizeof(Smem) <= kHead, "the stages start at a multiple of 1,024 bytes");
template <typename Sh>
constexpr size_t smem_bytes() {
    return kHead + Sh::kStages + Sh::kRaws * Sh::kRaw + Sh::kU;
}

// ------------------------------------------------------------------------------------------
// Digits.  One entry in fixed point: |x| = Q units, d = D - exponent >= 2 (so Q fills at most
// 62 of 64 bits), plus 128 in every byte: byte k minus 128 is then the balanced digit
// of weight 256^k.  (A shift by the word's size or more gives 0: zero and subnormal entries.)
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ u64 fix64(const double x, const int D, int &dmin) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int d = D - ((hi >> 20) & 0x7ff);
    dmin = min(dmin, d);
    const u64 mant = ((u64)(unsigned)((hi & 0xfffff) | 0x100000) << 43) | ((u64)(unsigned)lo << 11);
    u64 q;
    asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(mant), "r"((unsigned)d));
    return q + 0x8080808080808080ull;
}
__device__ __forceinline__ uint32_t hfma2_u(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// The four digits (FP16 pairs of two rows) of a 32-bit word of each row, most significant
// first: a byte b under 0x64 is the FP16 1024 + b; sgn (1024 + b) - sgn 1152 is the signed digit.
__device__ __forceinline__ void digits4(const uint32_t w0, const uint32_t w1, const uint32_t sgn,
                                        const uint32_t off, uint32_t &s0, uint32_t &s1,
                                        uint32_t &s2, uint32_t &s3) {
    const uint32_t t = __byte_perm(w0, w1, 0x6273), b = __byte_perm(w0, w1, 0x4051);
    s0 = hfma2_u(__byte_perm(t, 0x64646464u, 0x4140), sgn, off);
    s1 = hfma2_u(__byte_perm(t, 0x64646464u, 0x4342), sgn, off);
    s2 = hfma2_u(__byte_perm(b, 0x64646464u, 0x4140), sgn, off);
    s3 = hfma2_u(__byte_perm(b, 0x64646464u, 0x4342), sgn, off);
}

// ------------------------------------------------------------------------------------------
// Rows of a lane in a 64-row block: 16 q + 2 c8 + {0, 1}, q = 0..3 (eight lanes read 128
// consecutive bytes), the same for every column: the operand's rows are the block's in another
// order, which the sums do not see.  Piece q of the lane goes to raw + 512 q (the warp's q-th
// pieces side by side) and only the lane itself reads it, so no barrier stands between; 8-byte
// copies where A is not 16-byte aligned.  Rows past the end read as zeros (any: an address to name
// where there is nothing to copy).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ void copy16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(tc::smem_u32(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_rows(unsigned char *raw, const double *p, const int64_t left,
                                          const int c8, const bool vec, const double *any) {
    if (left >= 64 && vec) {
#pragma unroll
        for (int q = 0; q < 4; ++q) copy16(raw + 512 * q, p + 16 * q + 2 * c8);
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int r = 16 * (e >> 1) + 2 * c8 + (e & 1);
            cp_async8(raw + 512 * (e >> 1) + 8 * (e & 1), r < left ? p + r : any, r < left ? 8 : 0);
        }
    }
}
// Largest biased exponent of the lane's eight entries.
__device__ __forceinline__ int max_exponent(const unsigned char *raw) {
    int e = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const double2 v = *reinterpret_cast<const double2 *>(raw + 512 * p);
        e = max(e, max((__double2hiint(v.x) >> 20) & 0x7ff, (__double2hiint(v.y) >> 20) & 0x7ff));
    }
    return e;
}
// The lane's eight entries as digits: digit s to dst + s step.
__device__ __forceinline__ void slice8(const unsigned char *raw, const int D, int &dmin,
                                       unsigned char *dst, const int step) {
    uint32_t o[kDigits][4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const double2 v = *reinterpret_cast<const double2 *>(raw + 512 * p);
        const u64 q0 = fix64(v.x, D, dmin), q1 = fix64(v.y, D, dmin);
        const uint32_t sg =
            __byte_perm(__double2hiint(v.x), __double2hiint(v.y), 0x7632) & 0x80008000u;
        const uint32_t sgn = sg | 0x3c003c00u, off = sg ^ 0xe480e480u;
        digits4((uint32_t)(q0 >> 32), (uint32_t)(q1 >> 32), sgn, off, o[0][p], o[1][p], o[2][p],
                o[3][p]);
        digits4((uint32_t)q0, (uint32_t)q1, sgn, off, o[4][p], o[5][p], o[6][p], o[7][p]);
    }
#pragma unroll
    for (int s = 0; s < kDigits; ++s)
        *reinterpret_cast<uint4 *>(dst + s * step) = make_uint4(o[s][0], o[s][1], o[s][2], o[s][3]);
}

// ------------------------------------------------------------------------------------------
// 128-bit integers
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ i128 shr128(const i128 x, const int s) {
    return s == 0 ? x : s >= 127 ? (x < 0 ? (i128)-1 : (i128)0) : x >> s;
}
__device__ __forceinline__ i128 shift128(const i128 x, const int s) {  // left for s > 0
    return s >= 0 ? (i128)((u128)x << (s > 127 ? 127 : s)) : shr128(x, -s);
}
struct alignas(16) Q128 {
    u64 lo, hi;
};
__device__ __forceinline__ i128 unpack(const Q128 q) { return (i128)(((u128)q.hi << 64) | q.lo); }
__device__ __forceinline__ Q128 pack(const i128 x) {
    Q128 q;
    q.lo = (u64)x;
    q.hi = (u64)((u128)x >> 64);
    return q;
}
__device__ __forceinline__ i128 ldcg128(const void *p) {
    const ulonglong2 t = __ldcg(reinterpret_cast<const ulonglong2 *>(p));
    return (i128)(((u128)t.y << 64) | t.x);
}
// (i, j), i <= j, of packed index o = j (j + 1) / 2 + i.
__device__ __forceinline__ void unpack_index(const int o, int &i, int &j) {
    j = (int)((sqrtf(8.0f * (float)o + 1.0f) - 1.0f) * 0.5f);
    while ((j + 1) * (j + 2) / 2 <= o) ++j;
    while (j * (j + 1) / 2 > o) --j;
    i = o - j * (j + 1) / 2;
}

// ------------------------------------------------------------------------------------------
// One work item's view of the CTA: shared memory, tensor memory and the barriers' state.
// ------------------------------------------------------------------------------------------
struct Cta {
    Smem *sm;
    Q128 *U;           // the current item's sums
    unsigned char *stages;
    uint32_t tmem;
    bool ok;           // no wait has given up
};
template <typename Sh>
__device__ __forceinline__ Q128 *sums_of(const Cta &c) {
    return reinterpret_cast<Q128 *>(c.stages + Sh::kStages + Sh::kRaws * Sh::kRaw);
}

// Columns of an item: local column l < NI is column i0 + l of the matrix (l < ni), NI + l is j0 + l.
struct Cols {
    int i0, ni, j0, nj;
};

// The sums of one set over the 64-row blocks [kb0, kb1): in c.U (the lower half of a block
// against itself holds what its mirror adds), exponents in sm.D, sm.bad where the rows cannot be
// served.  Every thread of the CTA; all copies and tensor-core work have ended on return.
template <int NI, int NJ>
__device__ __noinline__ void sum_rows(const GramProblem &p, const Cols cols, const int64_t kb0,
                                         const int64_t kb1, Cta &c) {
    using Sh = Shape<NI, NJ>;
    constexpr int S = Sh::S;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Smem &sm = *c.sm;
    c.U = sums_of<Sh>(c);
    if (tid == 0) sm.bad = 0;
    if (tid < 128) sm.D[tid] = sm.E[tid] = 0;
    for (int o = tid; o < NI * Sh::NR; o += kGramThreads) c.U[o] = Q128{0, 0};

    const int rounds = (int)((kb1 - kb0 + Sh::kRoundKb - 1) / Sh::kRoundKb);
    const double *A = p.A, *B = p.B;
    const int c8 = lane & 7;

    // The lane's column, block and operand address.  A warp takes four columns, with an odd leading
    // dimension of one parity: every other column is 16-byte aligned then, and the warps that have
    // those copy them in half as many pieces (1,000,000 x 50: 661 us without, 626 so).
    const int kbo = warp / Sh::kGroups, group = warp % Sh::kGroups;
    const int lc = (p.lda | (B ? p.ldb : 0)) & 1
                       ? 8 * (group >> 1) + 2 * (lane >> 3) + (group & 1)
                       : 4 * group + (lane >> 3);
    const bool right = NJ > 0 && lc >= NI;
    const bool mine = warp < Sh::kRoundKb * Sh::kGroups &&
                      (right ? lc - NI < cols.nj : lc < cols.ni);
    const int gcol = right ? cols.j0 + lc - NI : cols.i0 + lc;
    const double *const src = (gcol < p.na ? A + (int64_t)gcol * p.lda
                                           : B + (int64_t)(gcol - p.na) * p.ldb) + (kb0 + kbo) * 64;
    const bool vec = __all_sync(0xffffffffu, ((uintptr_t)src & 15) == 0) != 0;
    const int row0 = right ? S * NI + lc - NI : lc;  // operand row of digit 0
    unsigned char *const dst = c.stages + kbo * Sh::kKbBytes + (row0 >> 3) * 1024 +
                               (row0 & 7) * 128 + ((c8 ^ (row0 & 7)) << 4);
    const int step = (right ? NJ : NI) * 128;        // from digit to digit
    unsigned char *const raw0 = c.stages + Sh::kStages + warp * 2048 + lane * 16;
    auto raw_of = [&](const int r) { return raw0 + (r % Sh::kRaws) * Sh::kRaw; };
    // Round r of A on its way to shared memory (one cp.async group a round, empty at the end).
    auto load_round = [&](const int r) {
        if (mine && r < rounds) {
            const int64_t kb = kb0 + kbo + (int64_t)r * Sh::kRoundKb;
            copy_rows(raw_of(r), src + (int64_t)r * (64 * Sh::kRoundKb),
                      kb < kb1 ? p.m - kb * 64 : 0, c8, vec, A);
        }
        cp_async_commit();
    };
    // The column exponents block kb of round r (64 rows) needs, to sm.Dnew: a column whose largest
    // entry there is out of its range gets that entry's exponent and two bits to spare, the others
    // keep theirs.  A column's exponents so follow from its slab alone, whatever set it is in: the
    // sets of a matrix sum the digits of one and the same matrix.  True if any column changes.
    auto scan_block = [&](const int r, const int kb) {
        const bool here = mine && kbo == kb;
        int top = here ? max_exponent(raw_of(r)) : 0;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        if (c8 == 0 && here) atomicMax(&sm.E[lc], top);
        __syncthreads();
        bool up = false;
        if (tid < NI + NJ) {
            const int e = sm.E[tid];
            if (e > kExpHi) sm.bad = 1;
            up = e + 2 > sm.D[tid];
            sm.Dnew[tid] = up ? max(e + 4, kLeastD) : sm.D[tid];
            sm.E[tid] = 0;
        }
        return __syncthreads_or(up) != 0;
    };
    auto zero_stages = [&]() {  // columns past the matrix's read as zeros
        for (int i = tid; i < Sh::kStages / 16; i += kGramThreads)
            reinterpret_cast<uint4 *>(c.stages)[i] = make_uint4(0, 0, 0, 0);
        tc::fence_proxy_async();
        __syncthreads();
    };
    const bool padded = cols.ni < NI || cols.nj < NJ;

    constexpr uint32_t idesc0 = tc::instr_desc(0, 128, Sh::kPair * Sh::N0, false, false);
    constexpr uint32_t idesc1 = Sh::kTiles == 2 ? tc::instr_desc(0, 128, Sh::N1, false, false) : 0;
    const uint64_t desc0 = tc::smem_desc(tc::smem_u32(c.stages), 16, 1024, tc::kSw128);
    const bool issuer = tid == kGramThreads - 32;  // the thread that issues the tensor-core work
    constexpr long long kPolls = 1LL << 22;
    volatile int *const above = sm.above, *const stop = &sm.stop;
    int blocks = 0;                 // 64-row blocks in the accumulators
    int used[2] = {0, 0};           // rounds given to each stage since the barriers' last start
    uint32_t drained = 0;           // completions of sm.drain since then
    auto restart_barriers = [&]() {  // between two CTA barriers; nothing is in flight
        if (tid == 0) {
            for (int b = 0; b < 2; ++b) {
                tc::mbar_inval(&sm.full[b]);
                tc::mbar_init(&sm.full[b], kGramSlicers);
                tc::mbar_inval(&sm.free[b]);
                tc::mbar_init(&sm.free[b], 1);
            }
            tc::mbar_inval(&sm.drain);
            tc::mbar_init(&sm.drain, 1);
            tc::fence_mbar_init();
            above[0] = above[1] = 0;
            *stop = -1;
        }
        used[0] = used[1] = 0;
        drained = 0;
    };
    // Waits for a barrier's phase, or for the stop: true where the phase is complete (the same for
    // the warp's lanes).
    auto wait_or_stop = [&](uint64_t *bar, const uint32_t parity) {
        bool done = !c.ok;  // a wait that gave up: no further one holds the CTA up
        for (long long it = 0; !done; ++it) {
            done = tc::mbar_test(bar, parity);
            if (!done && *stop >= 0) break;
            if (it >= kPolls) {
                c.ok = false;
                done = true;
            }
        }
        return __any_sync(0xffffffffu, done) != 0;
    };
    // The last commits to the stages' barriers (the multiplying warp, which has counted the rounds it
    // issued): a commit that arrives after its barrier is gone would write to memory that is another's.
    auto settle = [&]() {
        if (warp == kGramSlicers)
            for (int b = 0; b < 2; ++b)
                if (used[b] > 0 && c.ok) c.ok = tc::mbar_wait(&sm.free[b], (used[b] - 1) & 1, kPolls);
    };
    auto drain = [&]() {  // every thread; the issuer's work so far
        if (issuer) tc::mma_commit(&sm.drain);
        if (c.ok) c.ok = tc::mbar_wait(&sm.drain, drained & 1, kPolls);
        ++drained;
    };

    // Accumulators into U: every digit product's sum, weighted.  The tensor cores are drained
    // before, and the stages are free on return.
    auto flush = [&]() {
        tc::fence_after_sync();
        __syncthreads();
        const int part = warp >> 2, lrow = (32 * (warp & 3) + lane) % (128 / Sh::kPair);
        const int s = lrow / NI, i = lrow - s * NI;
        // (a pair's second block: the second half of the lanes and of the columns)
        const int second = Sh::kPair == 2 ? (warp & 3) >> 1 : 0;
        const uint32_t lanes = c.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + second * Sh::N0;
        long long *buf = reinterpret_cast<long long *>(c.stages);
        constexpr int kHalf = Sh::kRowDigits * Sh::JP * Sh::kLd;     // words of a half
        constexpr int kL1 = 2 * kHalf;                               // then tile 1's, [s - TS][j][i]
        constexpr int kSecond = 2 * kHalf;                           // (or a pair's second block)
        // sum over the sets of K <= 4 digits of columns at .. at + 7, weighted 256^(3 - t)
        auto digits = [&](auto K, long long (&x)[8], const uint32_t at) {
            int v[K][8];
#pragma unroll
            for (int t = 0; t < K; ++t)
#pragma unroll
                for (int e = 0; e < 8; ++e) v[t][e] = 0;
#pragma unroll 1
            for (int set = 0; set < cmin(Sh::kSets, 4 * blocks / Sh::kPair); ++set) {
                float f[K][8];
#pragma unroll
                for (int t = 0; t < K; ++t) tc::tmem_ld8(at + set * Sh::kCols + t * Sh::NR, f[t]);
                tc::tmem_ld_wait();
#pragma unroll
                for (int t = 0; t < K; ++t)
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[t][e] += __float2int_rn(f[t][e]);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                long long y = 0;
#pragma unroll
                for (int t = 0; t < K; ++t) y = y * 256 + v[t][e];
                x[e] = y << (8 * (4 - K));
            }
        };
        auto put = [&](const int at, const long long (&x)[8]) {
#pragma unroll
            for (int e = 0; e < 8; ++e) buf[at + e * Sh::kLd + i] = x[e];
        };
        for (int jb = 0; jb < Sh::NR; jb += Sh::JP) {
            constexpr int kJ = Sh::JP / 8;
            // a task: four right-hand digits of eight columns; tile 0's halves, then tile 1's
            constexpr int kTasks = Sh::kMirror ? 3 * kJ : 2 * Sh::kTiles * kJ;
            for (int task = part; task < kTasks && part < 4; task += 4) {
                const int which = task / kJ, jl = 8 * (task - which * kJ);
                const int tile = which >> 1, half = which & 1;
                const uint32_t at = lanes + (tile ? Sh::N0 : 0) + jb + jl + half * (4 * Sh::NR);
                long long x[8];
                if (Sh::kMirror && tile == 1) {
                    digits(std::integral_constant<int, Sh::kMirror ? Sh::TE - Sh::TS : 4>(), x, at);
                    if (s < S - Sh::TS) put(kL1 + (s * Sh::JP + jl) * Sh::kLd, x);
                } else {
                    const int sr = s + tile * Sh::TS;  // the row's digit
                    digits(std::integral_constant<int, 4>(), x, at);
                    if (s < Sh::TS && sr < Sh::kRowDigits)
                        put(second * kSecond + half * kHalf + (sr * Sh::JP + jl) * Sh::kLd, x);
                }
            }
            tc::fence_before_sync();
            __syncthreads();
            // weights: row digit s, word ending in digit e: 256^(7 - s) 256^(7 - e), in units of 2^24
            auto add = [&](i128 &g, const long long x, const int sh) {
                g += sh >= 0 ? (i128)x << (sh >= 0 ? sh : 0) : (i128)(x >> (sh < 0 ? -sh : 0));
            };
            for (int o = tid; o < NI * Sh::JP; o += kGramThreads) {
                const int ii = o % NI, jl = o / NI, j = jb + jl;
                i128 g = 0, mir = 0;
#pragma unroll
                for (int sr = 0; sr < Sh::kRowDigits; ++sr) {
                    const int at = (sr * Sh::JP + jl) * Sh::kLd + ii;
                    add(g, buf[at] + (Sh::kPair == 2 ? buf[kSecond + at] : 0), 64 - 8 * sr);
                    add(mir, buf[kHalf + at] + (Sh::kPair == 2 ? buf[kSecond + kHalf + at] : 0),
                        32 - 8 * sr);
                }
                if (Sh::kMirror) {
#pragma unroll
                    for (int sr = Sh::TS; sr < S; ++sr) {
                        const long long x = buf[kL1 + ((sr - Sh::TS) * Sh::JP + jl) * Sh::kLd + ii];
                        const int sh = 32 - 8 * sr;
                        if (sr < Sh::TE)
                            add(g, x, sh);
                        else
                            add(mir, x, sh);
                    }
                    g = (ii <= j ? g : 0) + (ii == j ? 2 * mir : mir);
                } else {
                    g = NJ > 0 || ii <= j ? g + mir : 0;
                }
                Q128 *u = c.U + ii * Sh::NR + j;
                *u = pack(unpack(*u) + g);
            }
            __syncthreads();
        }
        blocks = 0;
    };

    // Tensor-core work of blocks [k0, k1) of the round in stage b (the issuer).  The 16-row steps go
    // round the accumulator sets.  (Descriptors by addition: their low bits hold the address over
    // 16; built from addresses they cost more than the products.)
    auto multiply = [&](const int b, const int k0, const int k1) {
        tc::fence_after_sync();
        uint64_t ad = desc0 + (uint32_t)((b * Sh::kStage + k0 * Sh::kKbBytes) >> 4);
#pragma unroll 1
        for (int kb = k0; kb < k1; kb += Sh::kPair, ad += Sh::kPair * Sh::kKbBytes >> 4) {
            const int step0 = 4 * (blocks + kb - k0) / Sh::kPair;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                const uint32_t d0 = c.tmem + (uint32_t)((step0 + ks) % Sh::kSets) * Sh::kCols;
                const bool add = step0 + ks >= Sh::kSets;
                const uint64_t bd = ad + 2 * ks + (NJ > 0 ? S * NI * 8 : 0);
                tc::mma_f16(d0, ad + 2 * ks, bd, idesc0, add);
                if (Sh::kTiles == 2)
                    tc::mma_f16(d0 + Sh::N0, ad + 2 * ks + Sh::TS * NI * 8,
                                NJ > 0 ? bd : ad + 2 * ks + Sh::TS * NI * 8, idesc1, add);
            }
        }
    };

    // Rounds run without a CTA barrier: a warp slices its task of a round into the round's stage as
    // soon as the tensor cores are done with the round before the last (free), and the last warp,
    // which slices nothing, issues a round's products once all have arrived (full).  A warp that meets an entry
    // above its column's range says so of the round's stage before it arrives; the last warp then
    // issues nothing for that round and sets the stop, which every wait watches, and the whole CTA
    // takes that round block by block.
    restart_barriers();
#pragma unroll 1
    for (int r = 0; r < Sh::kRaws; ++r) load_round(r);
    cp_async_wait<Sh::kRaws - 1>();
    __syncthreads();
    scan_block(0, 0);
    if (tid < NI + NJ) sm.D[tid] = sm.Dnew[tid];
    if (padded)
        zero_stages();
    else
        __syncthreads();
    int r = 0;
    int r_at = 0, blocks_at = 0;  // blocks in the accumulators before round r_at
    while (r < rounds && !sm.bad) {
        const int b = r & 1;
        bool go;
        if (warp < kGramSlicers) {
            cp_async_wait<Sh::kRaws - 1>();
            go = used[b] == 0 || wait_or_stop(&sm.free[b], (used[b] - 1) & 1);
            if (go) {
                int dmin = 2;
                if (mine) slice8(raw_of(r), sm.D[lc], dmin, dst + b * Sh::kStage, step);
                if (__any_sync(0xffffffffu, dmin < 2) && lane == 0) above[b] = 1;
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.full[b]);
            }
        } else {
            if (c.ok) c.ok = tc::mbar_wait(&sm.full[b], used[b] & 1, kPolls);
            __syncwarp();
            // (round r's word alone: another warp may be saying so of the next round, in the other
            // stage, and where the rounds break off decides where the sums are cut, which has to
            // follow from the data; no warp is in round r + 2 before round r is multiplied.  One
            // word with the least round number, by shared-memory atomics: 7,203 us at 4,194,304 x
            // 128, 7,115 so)
            go = above[b] == 0;
            if (issuer) {
                if (go) {
                    multiply(b, 0, Sh::kRoundKb);
                    tc::mma_commit(&sm.free[b]);
                } else {
                    *stop = r;
                }
            }
            __syncwarp();
        }
        if (go) {
            ++used[b];
            blocks += Sh::kRoundKb;
            load_round(r + Sh::kRaws);
            if (r + 1 == rounds || blocks + Sh::kRoundKb > 16 * Sh::kSets * Sh::kPair) {
                if (issuer) tc::mma_commit(&sm.drain);
                __syncwarp();
                go = wait_or_stop(&sm.drain, drained & 1);
                if (go) {
                    ++drained;
                    flush();
                    if (r + 1 < rounds && padded) zero_stages();
                    r_at = r + 1;
                    blocks_at = 0;
                }
            }
        }
        if (go) {
            ++r;
            continue;
        }
        // ---- round *stop block by block: where an entry is above its column's range, what is
        //      accumulated goes to U, then the exponents rise and U's entries follow
        __syncthreads();
        r = *stop;
        blocks = blocks_at + (r - r_at) * Sh::kRoundKb;
        settle();
        drain();
        cp_async_wait_all();
        __syncthreads();
        restart_barriers();
#pragma unroll 1
        for (int q = 0; q < Sh::kRaws; ++q) load_round(r + q);
        cp_async_wait<Sh::kRaws - 1>();
        if (Sh::kPair == 2) zero_stages();
        __syncthreads();
#pragma unroll 1
        for (int kb = 0; kb < Sh::kRoundKb; ++kb) {
            const bool up = scan_block(r, kb);
            if (sm.bad) break;
            if (up) {
                if (blocks > 0) flush();
                for (int o = tid; o < NI * Sh::NR; o += kGramThreads) {
                    const int i = o / Sh::NR, j = (NJ > 0 ? NI : 0) + o % Sh::NR;
                    c.U[o] =
                        pack(shr128(unpack(c.U[o]), sm.Dnew[i] - sm.D[i] + sm.Dnew[j] - sm.D[j]));
                }
                __syncthreads();
                if (tid < NI + NJ) sm.D[tid] = sm.Dnew[tid];
                if (padded || Sh::kPair == 2)
                    zero_stages();
                else
                    __syncthreads();
            }
            int dmin = 2;
            // (in block 0 of stage 0; a pair's second block reads as zeros)
            if (mine && kbo == kb)
                slice8(raw_of(r), sm.D[lc], dmin, dst - kbo * Sh::kKbBytes, step);
            tc::fence_proxy_async();
            __syncthreads();
            if (issuer) multiply(0, 0, 1);
            blocks += Sh::kPair;
            drain();
            if (blocks + Sh::kRoundKb > 16 * Sh::kSets * Sh::kPair) {
                flush();
                if (padded || Sh::kPair == 2) zero_stages();
            }
        }
        if (sm.bad) break;
        load_round(r + Sh::kRaws);
        ++r;
        if (r == rounds) flush();
        r_at = r;
        blocks_at = blocks;
        __syncthreads();
    }
    cp_async_wait_all();
    settle();
    if (__syncthreads_or(!c.ok) && tid == 0) sm.bad = 1;
    __syncthreads();
}

// ------------------------------------------------------------------------------------------
// The tree over a set's slabs.  Publishes the leaf (exponents, sums); the last child of a node to
// arrive adds its siblings, aligned to the largest exponents, and climbs on.  Returns true in the
// CTA that has written the set's sum (the last slot of the set's tree).
// ------------------------------------------------------------------------------------------
template <int NI, int NJ, int NR>
__device__ __noinline__ bool climb(const GramProblem &p, const Cols cols, const int set, const int slab,
                      const size_t slot_bytes, Cta &c) {
    const int tid = threadIdx.x, lane = tid & 31;
    Smem &sm = *c.sm;
    const int inner = gram_inner_nodes(p.nslab, p.n);
    unsigned int *counters = p.counters + (size_t)set * inner;
    unsigned char *slots = p.slots + (size_t)set * (p.nslab + inner) * slot_bytes;
    const int nout = NJ > 0 ? cols.ni * cols.nj : cols.ni * (cols.ni + 1) / 2;
    auto decode = [&](const int o, int &i, int &j) {  // local columns of output o
        if (NJ > 0) {
            i = o / cols.nj;
            j = o - i * cols.nj;
        } else {
            unpack_index(o, i, j);
        }
    };
    {
        unsigned char *mine = slots + (size_t)slab * slot_bytes;
        int *head = reinterpret_cast<int *>(mine);
        if (tid < 128) {
            const int l = tid < 64 ? tid : NI + tid - 64;
            head[tid] = (tid < 64 ? tid < cols.ni : tid - 64 < cols.nj) ? sm.D[l] : 0;
        }
        if (tid == 0) head[kGramSlotHead / 4 - 1] = sm.bad;
        for (int o = tid; o < nout; o += kGramThreads) {
            int i, j;
            decode(o, i, j);
            i128 g = unpack(c.U[i * NR + j]);
            if (NJ == 0 && i < j) g += unpack(c.U[j * NR + i]);
            reinterpret_cast<Q128 *>(mine + kGramSlotHead)[o] = pack(g >> p.guard);
        }
    }
    int cnt = p.nslab, off = 0, t = slab, cidx = 0;
    constexpr int kHeads = NJ > 0 ? 64 : 32;  // exponents of a child: block I's, then block J's
    const int arity = gram_arity(p.n);
    int *kd = reinterpret_cast<int *>(c.stages);  // the node's exponents, then its children's
    while (cnt > 1) {
        const int next_cnt = (cnt + arity - 1) / arity;
        const int parent = t / arity, first = parent * arity;
        const int nchild = min(arity, cnt - first);
        __threadfence();
        __syncthreads();
        if (tid == 0) sm.flag = atomicAdd(&counters[cidx + parent], 1u) + 1 == (unsigned)nchild;
        __syncthreads();
        if (!sm.flag) return false;
        __threadfence();
        const unsigned char *kids = slots + (size_t)(off + first) * slot_bytes;
        unsigned char *node = slots + (size_t)(off + cnt + parent) * slot_bytes;
        if (tid == 0) sm.bad = 0;
        for (int e = tid; e < kHeads * nchild; e += kGramThreads) {
            const int l = e % kHeads;
            kd[kHeads + e] = __ldcg(reinterpret_cast<const int *>(kids + e / kHeads * slot_bytes) +
                                    (l < 32 ? l : 32 + l));
        }
        int bad = 0;
        if (tid < nchild)
            bad = __ldcg(reinterpret_cast<const int *>(kids + tid * slot_bytes) + kGramSlotHead / 4 - 1);
        __syncthreads();
        if (bad) sm.bad = 1;
        if (tid < kHeads) {
            int d = 0;
            for (int ch = 1; ch <= nchild; ++ch) d = max(d, kd[kHeads * ch + tid]);
            kd[tid] = d;
            reinterpret_cast<int *>(node)[tid < 32 ? tid : 32 + tid] = d;
        }
        __syncthreads();
        if (tid == 0) reinterpret_cast<int *>(node)[kGramSlotHead / 4 - 1] = sm.bad;
        // an output's children go to as many threads as there are for it
        const int parts = max(1, min(nchild, kGramThreads / nout));
        Q128 *part = reinterpret_cast<Q128 *>(c.stages + (((arity + 1) * kHeads * 4 + 15) & ~15));
        for (int u = tid; u < nout * parts; u += kGramThreads) {
            const int o = u % nout;
            int i, j;
            decode(o, i, j);
            const int jj = NJ > 0 ? 32 + j : j;
            const int dij = kd[i] + kd[jj];
            const unsigned char *e = kids + kGramSlotHead + (size_t)o * 16;
            i128 g = 0;
#pragma unroll 8
            for (int ch = u / nout; ch < nchild; ch += parts)
                g += shr128(ldcg128(e + ch * slot_bytes),
                            dij - kd[kHeads * (ch + 1) + i] - kd[kHeads * (ch + 1) + jj]);
            (parts > 1 ? part[u] : reinterpret_cast<Q128 *>(node + kGramSlotHead)[o]) = pack(g);
        }
        if (parts > 1) {
            __syncthreads();
            for (int o = tid; o < nout; o += kGramThreads) {
                i128 g = 0;
                for (int q = 0; q < parts; ++q) g += unpack(part[q * nout + o]);
                reinterpret_cast<Q128 *>(node + kGramSlotHead)[o] = pack(g);
            }
        }
        off += cnt;
        cidx += next_cnt;
        cnt = next_cnt;
        t = parent;
    }
    __threadfence();
    __syncthreads();
    return true;
}

// ------------------------------------------------------------------------------------------
// Root: the Cholesky factor of the summed Gram in fixed point.  Columns are scaled by powers of
// two so that every diagonal lies in [1/4, 1); values are integers over 2^122.  Step k works on
// row k scaled by 2^z (pivot in [1/4, 1) again): l = C(k, j) / pivot in [-2, 2], to about 2^-90
// from a 46-bit reciprocal and one residual, then C(i, j) -= l_i C(k, j).  R(k, j) = l_j sqrt(pivot).
// ------------------------------------------------------------------------------------------
// (a b) >> 122 to 2^8 (2^-114: far below the columns' own rounding), a, b < 2^124: one full product
// of words and the high halves of two.
__device__ __forceinline__ u128 mul122(const u128 a, const u128 b) {
    const u64 ah = (u64)(a >> 64), al = (u64)a, bh = (u64)(b >> 64), bl = (u64)b;
    return ((u128)ah * bh + __umul64hi(ah, bl) + __umul64hi(al, bh)) << 6;
}
// 2^60 (2^122 / d) to about 46 bits, d in [2^120, 2^122): the hardware's FP32 reciprocal and one
// Newton step.
__device__ __forceinline__ u64 recip60(const u128 d) {
    const u64 x = (u64)(d >> 58);  // d / 2^122 = x / 2^64
    const float f = __uint2float_rz((uint32_t)(x >> 32)) * 2.3283064365386963e-10f;
    float y;
    asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(f));
    const uint32_t yb = __float_as_uint(y);  // y in (1, 4]
    const u64 r = (u64)((yb & 0x7fffff) | 0x800000) << (37 + (int)(yb >> 23) - 127);
    const long long e = (1ll << 60) - (long long)__umul64hi(x, r);
    return r + (u64)(__mul64hi((long long)r, e) << 4);
}
// 2^122 c / d to about 2^-90 from r = recip60(d): 46 bits, then the residual's quotient; c <= 2 d.
__device__ __forceinline__ u128 quotient(const u128 c, const u128 d, const u64 r) {
    const u64 q = __umul64hi((u64)(c >> 60), r);  // of weight 2^64
    const u128 qd = (((u128)q * (u64)(d >> 64)) << 6) + (((u128)q * (u64)d) >> 58);
    const long long res = (long long)((i128)(c - qd) >> 16);  // below 2^62
    return ((u128)q << 64) + (u128)((i128)__mul64hi(res, (long long)r) << 20);
}
// x / 2^122 as a sum of two doubles (the second below the first's last place).
struct D2 {
    double hi, lo;
};
__device__ __forceinline__ D2 to_double(const i128 x) {
    const long long top = (long long)(x >> 64);
    const double h = (double)top;
    const double r = (double)(top - (long long)h);
    return D2{h * 0x1p-58, r * 0x1p-58 + (double)(u64)x * 0x1p-122};
}
__device__ __forceinline__ D2 sqrt2(const D2 x) {
    const double s = sqrt(x.hi + x.lo);
    return D2{s, (fma(-s, s, x.hi) + x.lo) / (2.0 * s)};
}

__device__ __forceinline__ int bits128(const u128 x) {
    const u64 h = (u64)(x >> 64);
    return h ? 128 - __clzll((long long)h) : 64 - __clzll((long long)(u64)x);
}
// 2^64 sqrt(d / 2^122) to about 2^-62 of it, d in [2^120, 2^122): the hardware's FP32 reciprocal
// square root, two Newton steps, and the residual's share.
__device__ __forceinline__ u64 sqrt64(const u128 d) {
    const u64 x = (u64)(d >> 58);
    const float f = __uint2float_rz((uint32_t)(x >> 32)) * 2.3283064365386963e-10f;
    float yf;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(yf) : "f"(f));
    const uint32_t yb = __float_as_uint(yf);  // in [1, 2]
    u64 y = (u64)((yb & 0x7fffff) | 0x800000) << (39 + (int)(yb >> 23) - 127);
#pragma unroll
    for (int it = 0; it < 2; ++it) {
        const long long e = (1ll << 62) - (long long)__umul64hi(x, __umul64hi(y, y) << 2);
        y += (u64)(__mul64hi((long long)y, e) << 1);
    }
    const u64 q = __umul64hi(x, y);  // of 2^62
    const long long res = (long long)((i128)((d << 2) - (u128)q * q) >> 8);
    const u64 v = (q << 2) + (u64)(__mul64hi(res, (long long)y) >> 51);
    return v >> 62 ? v : ~0ull;
}
// p 2^e, p in [2^62, 2^64), rounded to FP64 (in range).
__device__ __forceinline__ double round64(u64 p, int e, const bool neg) {
    if (!(p >> 63)) {
        p <<= 1;
        --e;
    }
    const u64 m = (p >> 11) + ((p >> 10) & 1);
    return __longlong_as_double((long long)((((u64)(1023 + 52 + 11 - 1 + e) << 52) + m) |
                                            ((u64)neg << 63)));
}

// l sqrt(d) 2^g from s = sqrt64(d).
__device__ __forceinline__ double r_entry(const i128 l, const u64 s, const int g) {
    const u128 a = (u128)(l < 0 ? -l : l);
    const int b = bits128(a);
    const u64 top = b > 64 ? (u64)(a >> (b - 64)) : (u64)a << ((64 - b) & 63);
    return b ? round64(__umul64hi(top, s), b - 186 + g, l < 0) : 0.0;
}

// C: packed upper rows (row k at rowoff(n, k) - k + j); row k's l replaces it, k < np (the rows
// below are not done: a right-hand side in the matrix's range has no pivot).  rowv: 3 n
// entries of scratch (the scaled pivots stay in the last n).  Thread k < np returns pivot k, scaled,
// and its shift.  Returns false if a pivot is too small (*low: zero on entry, then non-zero).
//
// A chain of np steps, each a reciprocal, a quotient and a multiplication deep.  The first n threads
// hold column j = tid: row k's l are theirs, and while the others take row k off the rows below they
// find the next pivot (from the diagonal as it was and l's own share) and its reciprocal.  Up to 32
// columns the trailing matrix stays in registers.  (1,000 x 32, with what follows here: 53 us a call,
// 72 with full products, the reciprocal in the chain and R in double-double.)
static __device__ __noinline__ bool factor_chain(Q128 *C, Q128 *rowv, const int n, const int np,
                                                 int *low, u128 &mine, int &myz) {
    const int tid = threadIdx.x, nt = kGramThreads, warp = tid >> 5, lane = tid & 31;
    constexpr i128 kLeast = (i128)1 << (122 - kPivotBits);
    Q128 *Lq = rowv, *Cp = rowv + n, *dv = rowv + 2 * n;
    // Up to 32 columns a thread keeps its entry (ti, tj) of C in registers until its row's turn.
    const bool owns = n <= kGramMaxN;
    int ti = -1, tj = 0;
    i128 own = 0;
    if (owns && tid < n * (n + 1) / 2) {
        int a, b;
        unpack_index(n * (n + 1) / 2 - 1 - tid, a, b);
        ti = n - 1 - b;
        tj = n - 1 - a;
        own = unpack(C[tid]);
    }
    i128 diag = tid < n ? unpack(C[rowoff(n, tid)]) : (i128)0;
    u128 d = 0;  // the pivot scaled to [1/4, 1)
    u64 r = 0;
    int z = 0;
    mine = 0;
    myz = 0;
    auto pivot = [&](const i128 d0) {
        z = (122 - bits128((u128)d0)) >> 1;
        d = (u128)d0 << (2 * z);
        r = recip60(d);
    };
    {
        const i128 d0 = unpack(C[0]);
        if (d0 < kLeast) return false;  // the same for every thread
        if (tid < n) pivot(d0);
    }
    for (int k = 0; k < np; ++k) {
        Q128 *Ck = C + rowoff(n, k) - k;
        u128 lm = 0, cm = 0;  // |l| and |c| of the thread's column
        if (tid < n) {
            if (tid == k) {
                dv[k] = pack((i128)d);
                mine = d;
                myz = z;
            } else if (tid > k) {
                const i128 c0 = unpack(Ck[tid]);
                const bool neg = c0 < 0;
                cm = (u128)(neg ? -c0 : c0) << z;
                lm = quotient(cm, d, r);
                const Q128 l = pack(neg ? -(i128)lm : (i128)lm);
                Lq[tid] = l;
                Ck[tid] = l;
                Cp[tid] = pack(neg ? -(i128)cm : (i128)cm);
                if (tid == k + 1) Lq[k] = pack(diag);
            }
        }
        if (k + 1 == np) break;
        __syncthreads();
        if (tid < n) {
            const i128 a = unpack(Lq[k + 1]), b = unpack(Cp[k + 1]);
            const i128 d0 = unpack(Lq[k]) -
                            (i128)mul122((u128)(a < 0 ? -a : a), (u128)(b < 0 ? -b : b));
            if (d0 < kLeast) *low = 1;
            diag -= (i128)mul122(lm, cm);
            pivot(d0 < kLeast ? kLeast : d0);
        }
        // trailing update, (i, j) with k < i <= j: a thread an entry, or a warp a row
        if (ti > k) {
            const i128 a = unpack(Lq[ti]), b = unpack(Cp[tj]);
            const u128 q = mul122((u128)(a < 0 ? -a : a), (u128)(b < 0 ? -b : b));
            own = (a < 0) != (b < 0) ? own + (i128)q : own - (i128)q;
            if (ti == k + 1) C[tid] = pack(own);
        }
        for (int i = k + 1 + (nt >> 5) - 1 - warp; i < n && !owns; i += nt >> 5) {
            const i128 a = unpack(Lq[i]);
            const u128 am = (u128)(a < 0 ? -a : a);
            Q128 *Ci = C + rowoff(n, i) - i;
            for (int jj = i + lane; jj < n; jj += 32) {
                const i128 b = unpack(Cp[jj]);
                const u128 q = mul122(am, (u128)(b < 0 ? -b : b));
                const i128 x = unpack(Ci[jj]);
                Ci[jj] = pack((a < 0) != (b < 0) ? x + (i128)q : x - (i128)q);
            }
        }
        __syncthreads();
        if (*low) return false;
    }
    return true;
}

// R from the chain's l and pivots: R(k, k) = sqrt(d_k) 2^-z_k, R(k, j) = l sqrt(d_k), g[j] the power
// of two of column j; in integers to the last (the chip has two FP64 lanes an SM).
static __device__ __noinline__ bool factor_root(Q128 *C, Q128 *rowv, const int n, const int np,
                                                const int *g, double *R, const int64_t ldr, int *low) {
    const int tid = threadIdx.x, nt = kGramThreads;
    Q128 *Lq = rowv;
    u128 mine;
    int myz;
    if (!factor_chain(C, rowv, n, np, low, mine, myz)) return false;
    __syncthreads();
    if (tid < np) Lq[tid] = Q128{sqrt64(mine), (u64)myz};
    __syncthreads();
    for (int o = tid; o < n * n; o += nt) {
        const int col = o / n, row = o - col * n;
        double v = 0.0;
        if (row >= np) {
            // (not done, not wanted)
        } else if (row < col) {
            v = r_entry(unpack(C[rowoff(n, row) - row + col]), Lq[row].lo, g[col]);
        } else if (row == col) {
            v = round64(Lq[row].lo, g[col] - 64 - (int)Lq[row].hi, false);
        }
        R[row + (int64_t)col * ldr] = v;
    }
    return true;
}

// The inverse of the factor just formed, for Q = A R^-1 (p.Q): R = diag(rho) M 2^g by columns, with
// M(k, k) = 2^-z_k and M(k, j) = l, so column j of the inverse is M^-1 e_j / rho_j: a warp a
// column, its entries one a lane, 110 bits after the point through the substitution (which a
// growth past 2^11 ends), then 62 bits against the column's largest entry.  Q's columns come
// out with an error of about sqrt(m n) 2^(F - 73): sm.bad where that is above 2^-47 (a
// bound; what Q^T Q - I shows is 2^-50, as with reflectors), an A whose Q the reflectors give.
static __device__ __noinline__ void invert_root(const GramProblem &p, const Q128 *C, const Q128 *dv,
                                                Smem &sm) {
    const int n = p.n, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned all = 0xffffffffu;
    const int limit = 52 - (64 - __clzll((long long)(p.m * n - 1)));  // of 2 F
    for (int j = warp; j < kGramMaxN; j += kGramThreads >> 5) {
        if (j >= n) {  // a column of zeros
            p.Q->w[kGramMaxN * j + lane] = 0;
            if (lane == 0) {
                p.Q->D[j] = 2047 + 64;
                p.Q->F[j] = 0;
            }
            continue;
        }
        const int z = lane < n ? (bits128((u128)unpack(dv[lane])) -
                                  bits128((u128)unpack(C[rowoff(n, lane)]))) >> 1 : 0;
        i128 x = lane == j ? (i128)1 << 110 : (i128)0;
        bool bad = false;
        for (int k = j; k >= 0; --k) {
            if (lane == k) {
                if (bits128((u128)(x < 0 ? -x : x)) + z > 121) {
                    bad = true;
                    x = 0;
                }
                x = (i128)((u128)x << z);
            }
            const u64 hi = __shfl_sync(all, (u64)((u128)x >> 64), k), lo = __shfl_sync(all, (u64)x, k);
            if (lane < k) {
                const i128 xk = (i128)(((u128)hi << 64) | lo);
                const i128 l = unpack(C[rowoff(n, lane) - lane + k]);
                const u128 q = mul122((u128)(l < 0 ? -l : l), (u128)(xk < 0 ? -xk : xk));
                x = (l < 0) != (xk < 0) ? (i128)((u128)x + q) : (i128)((u128)x - q);
            }
        }
        // 1 / rho, in (1, 2], times 2^62
        const D2 rho = sqrt2(to_double(unpack(dv[j])));
        const double y = 1.0 / rho.hi, dy = y * (fma(-y, rho.hi, 1.0) - y * rho.lo);
        const u64 inv = __double2ull_rn(y * 0x1p62) + (u64)__double2ll_rn(dy * 0x1p62);
        const u128 ax = (u128)(x < 0 ? -x : x);
        const u128 v = (((u128)(u64)(ax >> 64) * inv) << 2) + (((u128)(u64)ax * inv) >> 62);
        const int e = lane <= j ? sm.E[lane] - p.guard / 2 : 0;
        int F = v ? bits128(v) - 110 + e : -1000;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) F = max(F, __shfl_xor_sync(all, F, o));
        const int s = e - 48 - F;  // v 2^(e - 110) in units of 2^(F - 62)
        long long w;
        if (s >= 0)
            w = (long long)(v << min(s, 64));
        else
            w = s < -126 ? 0 : (long long)((v + ((u128)1 << (-s - 1))) >> -s);
        p.Q->w[kGramMaxN * j + lane] = x < 0 ? -w : w;
        if (lane == 0) {
            p.Q->D[j] = sm.D[j];
            p.Q->F[j] = F;
        }
        if (__any_sync(all, bad || 2 * F > limit) && lane == 0) sm.bad = 1;
    }
}

// Every set's sum (all written): gathered, scaled and factored; R written.  False: not served.
static __device__ __noinline__ bool finish(const GramProblem &p, const size_t slot_bytes, Smem *smp,
                                    unsigned char *base) {
    constexpr int NB = kBlock;
    const int tid = threadIdx.x, n = p.n;
    Smem &sm = *smp;
    Q128 *C = reinterpret_cast<Q128 *>(base);
    Q128 *rowv = C + n * (n + 1) / 2;
    const int per_set = p.nslab + gram_inner_nodes(p.nslab, p.n), nset = gram_sets(p.nb);
    auto top = [&](const int set) {
        return p.slots + ((size_t)(set + 1) * per_set - 1) * slot_bytes;
    };
    auto set_of = [&](const int I, const int J) {
        return I == J ? I : p.nb + J * (J - 1) / 2 + I;
    };
    __syncthreads();
    if (tid == 0) sm.bad = 0;
    __syncthreads();
    for (int s = tid; s < nset; s += kGramThreads)
        if (__ldcg(reinterpret_cast<const int *>(top(s)) + kGramSlotHead / 4 - 1)) sm.bad = 1;
    if (tid < n) {  // column exponents: the largest of the column's sets
        const int b = tid / NB, l = tid - b * NB;
        int d = 0;
        for (int o = 0; o < p.nb; ++o) {
            const int s = set_of(min(o, b), max(o, b));
            d = max(d, __ldcg(reinterpret_cast<const int *>(top(s)) + (o < b ? 64 : 0) + l));
        }
        sm.D[tid] = d;
        if (d <= kLeastD) sm.bad = 1;
    }
    __syncthreads();
    if (sm.bad) return false;
    auto entry = [&](const int i, const int j) {  // the sum (i, j), i <= j, aligned to sm.D
        const int I = i / NB, J = j / NB, li = i - I * NB, lj = j - J * NB;
        const unsigned char *t = top(set_of(I, J));
        const int *h = reinterpret_cast<const int *>(t);
        const int nj = min(NB, n - J * NB);
        const size_t o = I == J ? (size_t)(lj * (lj + 1) / 2 + li) : (size_t)(li * nj + lj);
        const i128 x = ldcg128(t + kGramSlotHead + o * 16);
        return shr128(x, sm.D[i] + sm.D[j] - __ldcg(h + li) - __ldcg(h + (I == J ? lj : 64 + lj)));
    };
    if (tid < n) {
        const i128 d = entry(tid, tid);
        const u64 dh = (u64)((u128)d >> 64);
        const int len = dh ? 128 - __clzll((long long)dh) : 64 - __clzll((long long)(u64)d);
        sm.E[tid] = d > 0 ? (122 - len) >> 1 : 0;  // shift of the column
        if (!(d > 0) && tid < p.np) sm.bad = 1;
        sm.Dnew[tid] = 73 - sm.E[tid] + sm.D[tid] + kUnit + p.guard / 2;
    }
    __syncthreads();
    if (sm.bad) return false;
    for (int o = tid; o < n * (n + 1) / 2; o += kGramThreads) {
        int i, j;
        unpack_index(o, i, j);
        C[rowoff(n, i) - i + j] = pack(shift128(entry(i, j), sm.E[i] + sm.E[j]));
    }
    __syncthreads();
    if (!factor_root(C, rowv, n, p.np, sm.Dnew, p.R, p.ldr, &sm.bad)) return false;
    if (p.Q) {
        invert_root(p, C, rowv + 2 * n, sm);
        __syncthreads();
    }
    return !sm.bad;
}

// One work item: its rows' sums and the climb.  True in the CTA that has written the set's sum.
template <int NI, int NJ>
__device__ __forceinline__ bool item_of(const GramProblem &p, const Cols cols, const int set,
                                        const int slab, const size_t slot_bytes, Cta &c) {
    const int64_t kb0 = (int64_t)slab * p.nkb / p.nslab, kb1 = (int64_t)(slab + 1) * p.nkb / p.nslab;
    sum_rows<NI, NJ>(p, cols, kb0, kb1, c);
    return climb<NI, NJ, Shape<NI, NJ>::NR>(p, cols, set, slab, slot_bytes, c);
}

// Tensor memory and barriers of the CTA; smem: its dynamic shared memory.
__device__ __forceinline__ void cta_begin(Cta &c, unsigned char *smem) {
    c.sm = reinterpret_cast<Smem *>(smem);
    c.stages = smem + kHead;
    if (threadIdx.x >> 5 == kGramSlicers) tc::tmem_alloc(&c.sm->tmem, 512);
    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&c.sm->full[b], kGramSlicers);
            tc::mbar_init(&c.sm->free[b], 1);
        }
        tc::mbar_init(&c.sm->drain, 1);
        tc::fence_mbar_init();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    c.tmem = c.sm->tmem;
    c.ok = true;
}
// (The barriers' lives end too: what follows in the same launch, the Householder reduction, takes the
// memory they stand in.  A CTA barrier stands between this and that.)
__device__ __forceinline__ void cta_end(const Cta &c) {
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            tc::mbar_inval(&c.sm->full[b]);
            tc::mbar_inval(&c.sm->free[b]);
        }
        tc::mbar_inval(&c.sm->drain);
    }
    if (threadIdx.x >> 5 == kGramSlicers) {
        tc::tmem_relinquish();
        tc::tmem_dealloc(c.tmem, 512);
    }
}

}  // namespace gram
}  // namespace tsqr
