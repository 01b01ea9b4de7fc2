// Q = A R^-1 on the tensor cores, for matrices the exact-Gram reduction served (tsqr_qr): A and
// the inverse as whole numbers (GramQForm), their digit products summed exactly, one rounding.
//
// A tile of A (128 lanes of 32 columns) is cut into 8 digits, which lie along the reduction (K = 256,
// digit s of column k at 32 s + k); the inverse is the other operand, digit w - s of its entry
// (k, j) at column 32 w + j, so that accumulator column 32 w + j collects all products of weight
// w = 0 .. 7 (at most 256 products of two digits: below 2^22).  What is left out, weights 8 to
// 14, is below 2^-62 of the largest product.
//
// A tile is 32 KB in and 32 KB out (320 us of copy rate at 4,194,304 x 32) against some 25
// instructions an entry to cut it and 40 to put its eight sums together and round them to FP64,
// in integers: the chip's FP64 units would take longer than the tile's memory traffic.  The shift
// and logic unit bounds it (63% busy when the pass took 630 us), so sums and shifts that a
// multiply-add can do go there, and whole tiles go without bounds checks: 530 us (840 with the
// sums in 64-bit multiply-adds and a 64-bit leading-zero count).  The reflectors' passes, bound by
// FP64, took 14 ms.  One 128-row tile whatever the width took 2.4 ms at 16,777,216 x 8, four side
// by side take 0.5 ms.
#pragma once

#include "tsqr_gram_dev.cuh"

namespace tsqr {

namespace gram {

constexpr int kQStage = 128 * 512;            // a tile's digits: four 128-byte lines a row
constexpr int kQInverse = 640 * 128;          // the inverse: lines of digits 2a, 2a + 1 for w >= 2a
constexpr int kQHead = 1024;
constexpr size_t kQSmem = kQHead + kQInverse + 2 * kQStage;

struct alignas(16) QSmem {
    uint64_t full[2], done[2];
    uint32_t tmem, p8;
    int D[kGramMaxN], F[kGramMaxN];
};
static_assert(sizeof(QSmem) <= kQHead, "the operands start at a multiple of 1,024 bytes");

// Multipliers the compiler must not see as shifts: the unit that shifts and adds is the busy one
// (63% against the multiplier's 20), and a multiply-add does both.
struct Powers {
    uint32_t p8, p16, m20;  // 2^8, 2^16, -2^20
};
__device__ __forceinline__ uint32_t mad_u32(const uint32_t a, const uint32_t b, const uint32_t c) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// Four accumulators of weights 256^3 .. 1 as a 64-bit number times 2^16.  (f + 1.5 2^23: f, a
// whole number below 2^22, in the low bits; two of them fit 32, with their offsets 32 unsigned.)
__device__ __forceinline__ long long word4(const float f0, const float f1, const float f2,
                                           const float f3, const Powers &c) {
    constexpr float kMagic = 12582912.0f;
    constexpr u64 kBits = 0x4B400000u, kBias = (kBits * 256 + kBits) & 0xffffffffu;
    constexpr u64 kOff = 0 - (kBias << 32) - (kBias << 16);
    const uint32_t a = mad_u32(__float_as_uint(f0 + kMagic), c.p8, __float_as_uint(f1 + kMagic));
    const uint32_t b = mad_u32(__float_as_uint(f2 + kMagic), c.p8, __float_as_uint(f3 + kMagic));
    const u64 hi = ((u64)(a + (uint32_t)(kOff >> 32)) << 32) | (uint32_t)kOff;
    u64 r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(b), "r"(c.p16), "l"(hi));
    return (long long)r;
}
// (H 2^32 + L) 2^(e - 16), rounded to FP64 (H, L: word4's; e20: e's place in the exponent field).  Integers throughout: the 96-bit sum
// is shifted until its sign bit is the top one, cut to 64 bits and rounded to 53.  small: a sum
// below 2^48, whose leading bits need another word.
__device__ __forceinline__ double round_sum(const long long H, const long long L,
                                            const uint32_t e20, const Powers &c, bool &small) {
    const long long hi = H + (L >> 32);  // 2^32 of it
    const uint32_t w2 = (uint32_t)((u64)hi >> 32), w1 = (uint32_t)hi, w0 = (uint32_t)L;
    const uint32_t s = (uint32_t)((int)w2 >> 31), x = w2 ^ s;
    small = x == 0;
    const int sh = __clz((int)x) - 1;
    const uint32_t t1 = __funnelshift_l(w1, w2, sh) ^ s, t0 = __funnelshift_l(w0, w1, sh) ^ s;
    const u64 m = ((((u64)t1 << 32) | t0) + 512) >> 10;  // 2^52 .. 2^53
    const uint32_t top = mad_u32((uint32_t)sh, c.m20, (uint32_t)(m >> 32) + e20);
    return __hiloint2double((int)(top | (s & 0x80000000u)), (int)(uint32_t)m);
}
__device__ __noinline__ double round_small(const long long H, const long long L,
                                            const uint32_t e20) {
    const int e = (int)(e20 >> 20);
    // 64 bits and the sign hold the sum (in units of 2^-16)
    const u64 v = ((u64)H << 32) + (u64)L;
    const bool neg = H + (L >> 32) < 0;
    if (v == 0 && !neg) return 0.0;
    const u64 a = !neg ? v : v ? 0 - v : ~0ull;
    const int sh = __clzll((long long)a);
    u64 m = a << sh;
    m = (m >> 11) + ((m >> 10) & 1);
    const u64 bits = m + ((u64)(e - sh - 31) << 52);
    return __longlong_as_double((long long)(bits | ((u64)neg << 63)));
}

__device__ __forceinline__ void q_rows(const GramQArgs &a, unsigned char *smem) {
    QSmem &sm = *reinterpret_cast<QSmem *>(smem);
    unsigned char *const inv = smem + kQHead, *const stages = inv + kQInverse;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr long long kPolls = 1LL << 22;
    // groups of eight columns of A in a tile; up to 16 columns, as many copies of the inverse as there
    // are blocks stand on the other operand's diagonal
    const int rows = gram_q_rows(a.n), groups = 512 / rows;
    if (blockIdx.x >= a.ntiles) return;
    if (warp == kGramSlicers) tc::tmem_alloc(&sm.tmem, 512);
    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&sm.full[b], kGramSlicers);
            tc::mbar_init(&sm.done[b], 1);
        }
        tc::fence_mbar_init();
        *(volatile uint32_t *)&sm.p8 = 256;
    }
    if (tid < kGramMaxN) {
        sm.D[tid] = a.form->D[tid];
        sm.F[tid] = a.form->F[tid];
    }
    long long *const w = reinterpret_cast<long long *>(stages);
    for (int i = tid; i < kGramMaxN * kGramMaxN; i += kGramThreads) w[i] = a.form->w[i];
    __syncthreads();
    // 16-byte chunks (eight rows k of one digit of a column j) of the inverse's lines
    for (int o = tid; o < 640 * 8; o += kGramThreads) {
        const int line = o >> 3, chunk = o & 7;
        const int t = line < 256 ? 0 : line < 448 ? 1 : line < 576 ? 2 : 3;  // digits 2t, 2t + 1
        const int l = line - (t == 0 ? 0 : t == 1 ? 256 : t == 2 ? 448 : 576);
        const int d = (l >> 5) - (chunk >> 2), j = l & 31;                   // digit w - s
        uint32_t v[4] = {0, 0, 0, 0};
        if (d >= 0 && (j >> 3) / groups == (chunk & 3) / groups) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const u64 q = (u64)w[kGramMaxN * (j % (8 * groups)) + 8 * ((chunk & 3) % groups) + e] +
                              0x8080808080808080ull;
                const int digit = (int)((q >> (56 - 8 * d)) & 255) - 128;
                const uint32_t hf = __half_as_ushort(__int2half_rn(digit));
                v[e >> 1] |= hf << (16 * (e & 1));
            }
        }
        *reinterpret_cast<uint4 *>(inv + line * 128 + ((chunk ^ (line & 7)) << 4)) =
            make_uint4(v[0], v[1], v[2], v[3]);
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = sm.tmem;
    bool ok = true;

    if (warp == kGramSlicers) {  // the products
        const uint64_t bd0 = tc::smem_desc(tc::smem_u32(inv), 16, 1024, tc::kSw128);
        const uint64_t ad0 = tc::smem_desc(tc::smem_u32(stages), 16, 1024, tc::kSw128);
        int k = 0;
        for (int64_t t = blockIdx.x; t < a.ntiles; t += gridDim.x, ++k) {
            const int b = k & 1;
            if (ok) ok = tc::mbar_wait(&sm.full[b], (k >> 1) & 1, kPolls);
            __syncwarp();
            tc::fence_after_sync();
            if (lane == 0 && ok) {
                constexpr int kLine[4] = {0, 256, 448, 576};
#pragma unroll
                for (int s = 0; s < kDigits; ++s) {
                    const uint32_t idesc = tc::instr_desc(0, 128, 32 * (kDigits - s), false, false);
                    const uint64_t ad = ad0 + ((b * kQStage + (s >> 1) * 16384 + (s & 1) * 64) >> 4);
                    const uint64_t bd = bd0 + (((kLine[s >> 1] + 32 * (s & 1)) * 128 + (s & 1) * 64) >> 4);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        tc::mma_f16(tmem + b * 256 + 32 * s, ad + 2 * h, bd + 2 * h, idesc, s + h > 0);
                }
                tc::mma_commit(&sm.done[b]);
            }
            __syncwarp();
        }
    } else {
        // the thread's row of 8 columns; lane of the operand and place of the columns in it
        const int lr = 32 * (warp & 3) + lane, place = warp >> 2;
        const int r = 128 * (place / groups) + lr, c0 = 8 * (place % groups);
        Powers pw;
        pw.p8 = *(volatile uint32_t *)&sm.p8;
        pw.p16 = pw.p8 * pw.p8;
        pw.m20 = 0u - pw.p16 * 16;
        int D[8];
        uint32_t F[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            D[e] = sm.D[c0 + e];
            F[e] = (uint32_t)(1023 + 52 - 1 + 42 - 16 - 79 + sm.F[c0 + e]) << 20;
        }
        const bool whole = c0 + 8 <= a.n;  // no column of the thread is missing
        double v[8];
        auto load = [&](const int64_t t) {
            const int64_t row = t * rows + r;
            const bool in = t < a.ntiles && row < a.m;
            const double *p = a.A + row + c0 * a.lda;
            if (whole && (t + 1) * rows <= a.m) {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = p[e * a.lda];
                return;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = in && c0 + e < a.n ? p[e * a.lda] : 0.0;
        };
        unsigned char *const dst = stages + lr * 128;
        // the rows of tile t (the k-th here) from its sums
        auto store = [&](const int64_t t, const int k) {
            const int b = k & 1;
            if (ok) ok = tc::mbar_wait(&sm.done[b], (k >> 1) & 1, kPolls);
            __syncwarp();
            tc::fence_after_sync();
            if (c0 < a.n) {
                const uint32_t at = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + b * 256 + 8 * place;
                long long half[2][8];
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    float f[4][8];
#pragma unroll
                    for (int d = 0; d < 4; ++d) tc::tmem_ld8(at + 32 * (4 * g + d), f[d]);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 8; ++e) half[g][e] = word4(f[0][e], f[1][e], f[2][e], f[3][e], pw);
                }
                const int64_t row = t * rows + r;
                double *q = a.Q + row + c0 * a.ldq;
                double x[8];
                bool any = false;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    bool small;
                    x[e] = round_sum(half[0][e], half[1][e], F[e], pw, small);
                    any |= small;
                }
                if (any) {  // (seldom; which of them, again)
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        bool small;
                        round_sum(half[0][e], half[1][e], F[e], pw, small);
                        if (small) x[e] = round_small(half[0][e], half[1][e], F[e]);
                    }
                }
                if (whole && (t + 1) * rows <= a.m) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) q[e * a.ldq] = x[e];
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (row < a.m && c0 + e < a.n) q[e * a.ldq] = x[e];
                }
            }
            tc::fence_before_sync();
        };
        load(blockIdx.x);
        int k = 0;
        int64_t t = blockIdx.x;
        // Stage and accumulators b = k % 2 were last read for tile k - 2, whose rows every warp has
        // written before it arrives here.
        for (; t < a.ntiles; t += gridDim.x, ++k) {
            const int b = k & 1;
            uint32_t o[kDigits][4];
            int unused = 0;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const double x = v[2 * p], y = v[2 * p + 1];
                const u64 q0 = fix64(x, D[2 * p], unused), q1 = fix64(y, D[2 * p + 1], unused);
                const uint32_t sg = __byte_perm(__double2hiint(x), __double2hiint(y), 0x7632) & 0x80008000u;
                const uint32_t sgn = sg | 0x3c003c00u, off = sg ^ 0xe480e480u;
                digits4((uint32_t)(q0 >> 32), (uint32_t)(q1 >> 32), sgn, off, o[0][p], o[1][p],
                        o[2][p], o[3][p]);
                digits4((uint32_t)q0, (uint32_t)q1, sgn, off, o[4][p], o[5][p], o[6][p], o[7][p]);
            }
#pragma unroll
            for (int s = 0; s < kDigits; ++s)
                *reinterpret_cast<uint4 *>(dst + b * kQStage + (s >> 1) * 16384 +
                                           (((4 * (s & 1) + place) ^ (lr & 7)) << 4)) =
                    make_uint4(o[s][0], o[s][1], o[s][2], o[s][3]);
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sm.full[b]);
            load(t + gridDim.x);
            if (k > 0) store(t - gridDim.x, k - 1);
        }
        store(t - gridDim.x, k - 1);
    }
    if (__syncthreads_or(!ok) && tid == 0) atomicOr(a.status, kStatusTimeoutBit);
    if (warp == kGramSlicers) {
        tc::tmem_relinquish();
        tc::tmem_dealloc(tmem, 512);
    }
}

}  // namespace gram
}  // namespace tsqr
