// Exact-Gram reduction on the tensor cores (tsqr_gram.cuh has the method).
#include <cstring>

#include "tsqr_gram.cuh"
#define TSQR_FOLD_THREADS (32 * (kGramFoldWarps + 1))
#include "tsqr_fold.cuh"
#include "tsqr_tc.cuh"

namespace tsqr {

namespace {

typedef unsigned long long u64;
typedef __int128 i128;
typedef unsigned __int128 u128;

constexpr int kGramPivotBits = 64;
// Biased FP64 exponents a column's largest entry may have: outside, squares leave FP64's range
// (or come near it) and the Householder reduction decides what R is.
constexpr int kExpLo = 1023 - 400, kExpHi = 1023 + 400;
constexpr long long kVerdictPolls = 1LL << 27;  // of at least 0.2 us each

// Shape of one width class: NB columns, S digits a column.
template <int NB, int S>
struct Shape {
    static constexpr int MN = NB * S;                    // operand rows (digit s of column j at s NB + j)
    static constexpr bool kTwoTiles = MN > 128;          // digits 0-3 in tile 0, the rest in tile 1
    static constexpr int N0 = MN;                        // tile 0: against every digit
    static constexpr int N1 = kTwoTiles ? 2 * NB : 0;    // tile 1: against digits 4 and 5
    static constexpr int kCols = N0 + N1;                // tensor-memory columns of one accumulator set
    static constexpr int kSets = 512 / kCols < 8 ? 512 / kCols : 8;  // sets, 1,024 rows each
    static constexpr int kGroups = NB / 4;               // column groups of a slicing task
    static constexpr int kRoundKb = NB == 24 ? 2 : kGramWarps / kGroups;  // 64-row blocks a round
    static constexpr int kSlicers = kRoundKb * kGroups;  // warps with a task (all but 4 at 24)
    static constexpr int kSetRounds = 16 / kRoundKb;     // rounds of at most 1,024 rows
    static constexpr int kKbBytes = MN * 128;            // 64 FP16 per operand row
    static constexpr int kStage = kRoundKb * kKbBytes;
    static constexpr int kPad = 8192;                    // rows tile 0 or 1 reads past the last block
    static constexpr int kStages = 2 * kStage + kPad;
    static constexpr int kRaw = kSlicers * 2048;         // a round of A: 64 bytes a lane
    static constexpr int kRaws = 2;                      // rounds on their way
    static_assert(kSlicers <= kGramWarps, "one task a warp");
    // flush buffers (over the stages): 64-bit partial sums [row digit][column j][column i], one
    // word of padding a row (the transposed reads of the mirrored digits would share a bank)
    static constexpr int kLd = NB + 1;
    static constexpr int kRowDigits0 = kTwoTiles ? 4 : S;
    static constexpr int kHi = 0;
    static constexpr int kLo = kRowDigits0 * NB * kLd * 8;
    static constexpr int kL1 = 2 * kLo;
    static constexpr int kFlush = kL1 + (kTwoTiles ? (S - 4) * NB * kLd * 8 : 0);
    static_assert(S == 8 && kFlush <= kStages, "flush buffers fit the stages");
};

struct alignas(16) GramSmem {  // after the stages
    uint64_t bar[2];
    uint32_t tmem;
    int flag;
    int bad;
    int D[32];
    int E[32];
    int Dnew[32];
};

// ------------------------------------------------------------------------------------------
// One entry in fixed point: |x| = Q 2^(D - 1086), Q < 2^62, d = D - exponent >= 2.  Returns Q
// plus 128 in every byte: byte k minus 128 is then the balanced digit of weight 256^k.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ u64 fix64(const double x, const int D, int &dmin) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int d = D - ((hi >> 20) & 0x7ff);
    dmin = min(dmin, d);
    const u64 mant = ((u64)(unsigned)((hi & 0xfffff) | 0x100000) << 43) | ((u64)(unsigned)lo << 11);
    u64 q;
    // (a shift of 64 or more gives 0: zero and subnormal entries, whose D - 0 is above 64)
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

// Rows of a lane in a 64-row block: 16 q + 2 c8 + {0, 1}, q = 0..3 (eight lanes read 128
// consecutive bytes); the same order for every column, so the operand's rows are the block's in
// another order, which the sums do not see.  The lane's 16-byte pieces go to dst + 512 q (the
// warp's q-th pieces side by side) and only the lane itself reads them; rows past the end are
// zeros.
__device__ __forceinline__ void copy16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(tc::smem_u32(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_rows(unsigned char *dst, const double *p, const int64_t left,
                                          const int c8, const bool vec) {
    if (left >= 64 && vec) {
#pragma unroll
        for (int q = 0; q < 4; ++q) copy16(dst + 512 * q, p + 16 * q + 2 * c8);
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int r = 16 * (e >> 1) + 2 * c8 + (e & 1);
            cp_async8(dst + 512 * (e >> 1) + 8 * (e & 1), r < left ? p + r : p, r < left ? 8 : 0);
        }
    }
}

// The lane's eight rows of one column as digits in the operand: digit s in row s NB + column,
// 16-byte unit c8 (128-byte rows, swizzled).
template <int NB, int S>
__device__ __forceinline__ void slice8(const unsigned char *raw, const int D, int &dmin,
                                       unsigned char *dst) {
    uint32_t o[8][4];
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
    for (int s = 0; s < S; ++s)
        *reinterpret_cast<uint4 *>(dst + s * NB * 128) = make_uint4(o[s][0], o[s][1], o[s][2], o[s][3]);
}

__device__ __forceinline__ i128 shr128(const i128 x, const int s) {
    return s >= 127 ? (x < 0 ? (i128)-1 : (i128)0) : x >> s;
}
__device__ __forceinline__ i128 shift128(const i128 x, const int s) {  // left for s > 0
    return s >= 0 ? (i128)((u128)x << (s > 127 ? 127 : s)) : shr128(x, -s);
}

struct alignas(16) Q128 {
    u64 lo, hi;
};
__device__ __forceinline__ i128 unpack(const Q128 q) {
    return (i128)(((u128)q.hi << 64) | q.lo);
}
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
// Root: the Cholesky factor of the summed Gram in fixed point.  Columns are scaled by powers of
// two so that every diagonal lies in [1/4, 1); values are integers over 2^122.  Step k works on
// row k scaled by 2^z (pivot in [1/4, 1) again): l = C(k, j) / pivot in [-2, 2], to about 2^-112
// from a 64-bit reciprocal and one residual, then C(i, j) -= l_i C(k, j).  R(k, j) = l_j sqrt(pivot).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ u128 mul122(const u128 a, const u128 b) {  // (a b) >> 122; a, b < 2^124
    const u64 ah = (u64)(a >> 64), al = (u64)a, bh = (u64)(b >> 64), bl = (u64)b;
    const u128 mid = (u128)ah * bl + (u128)al * bh + __umul64hi(al, bl);
    return (((u128)ah * bh) << 6) + (mid >> 58);
}
__device__ __forceinline__ u128 mul60(const u128 a, const u64 r) {  // (a r) >> 60
    return (((u128)(u64)(a >> 64) * r) << 4) + (((u128)(u64)a * r) >> 60);
}
__device__ __forceinline__ u64 recip60(const u128 d) {  // 2^60 (2^122 / d), d in [2^120, 2^122)
    const u64 x = (u64)(d >> 58);                       // d / 2^122 = x / 2^64
    const float f = __uint2float_rz((uint32_t)(x >> 32)) * 2.3283064365386963e-10f;
    float y;
    asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(f));
    u64 r = (u64)(y * 1152921504606846976.0f);
#pragma unroll
    for (int it = 0; it < 2; ++it) {
        const long long e = (1ll << 60) - (long long)__umul64hi(x, r);
        r += (u64)(__mul64hi((long long)r, e) << 4);
    }
    return r;
}
__device__ __forceinline__ double to_double(const i128 x) {  // x / 2^122, correctly rounded enough
    return (double)(long long)(x >> 64) * 0x1p-58 + (double)(u64)x * 0x1p-122;
}

// C: n x n (row k at C + k n), upper part used; row k's l replaces it.  rowv: 3 n entries of
// scratch.  Returns false if a pivot is too small.
__device__ __noinline__ bool factor_root(Q128 *C, Q128 *rowv, const int n, const int *g, double *R,
                                         const int64_t ldr) {
    const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31;
    Q128 *Lq = rowv, *Cp = rowv + n, *dv = rowv + 2 * n;
    for (int k = 0; k < n; ++k) {
        const i128 d0 = unpack(C[k * n + k]);
        if (d0 < ((i128)1 << (122 - kGramPivotBits))) return false;  // the same for every thread
        const u64 dh = (u64)((u128)d0 >> 64);
        const int len = dh ? 128 - __clzll((long long)dh) : 64 - __clzll((long long)(u64)d0);
        const int z = (122 - len) >> 1;
        const int j = k + 1 + tid;
        if (j < n || tid == 0) {
            const u128 d = (u128)d0 << (2 * z);
            if (tid == 0) dv[k] = pack((i128)d);
            if (j < n) {
                const i128 c0 = unpack(C[k * n + j]);
                const bool neg = c0 < 0;
                const u128 c = (u128)(neg ? -c0 : c0) << z;
                const u64 r = recip60(d);
                u128 q = mul60(c, r);
                const i128 res = (i128)(c - mul122(q, d));
                const u128 dq = mul60((u128)(res < 0 ? -res : res), r);
                q = res < 0 ? q - dq : q + dq;
                const Q128 l = pack(neg ? -(i128)q : (i128)q);
                Lq[j] = l;
                C[k * n + j] = l;
                Cp[j] = pack(neg ? -(i128)c : (i128)c);
            }
        }
        __syncthreads();
        // trailing update, (i, j) with k < i <= j: a warp a row
        for (int i = k + 1 + warp; i < n; i += nt >> 5) {
            const i128 a = unpack(Lq[i]);
            const u128 am = (u128)(a < 0 ? -a : a);
            for (int jj = i + lane; jj < n; jj += 32) {
                const i128 b = unpack(Cp[jj]);
                const u128 p = mul122(am, (u128)(b < 0 ? -b : b));
                const i128 c = unpack(C[i * n + jj]);
                C[i * n + jj] = pack((a < 0) != (b < 0) ? c + (i128)p : c - (i128)p);
            }
        }
        __syncthreads();
    }
    // R(k, k) = 2^-z sqrt(d), with d0 = C(k, k) = 2^-2z d still in place; R(k, j) = l sqrt(d)
    double *sd = reinterpret_cast<double *>(Lq);
    for (int k = tid; k < n; k += nt) sd[k] = sqrt(to_double(unpack(dv[k])));
    __syncthreads();
    for (int o = tid; o < n * n; o += nt) {
        const int col = o / n, row = o - col * n;
        double v = 0.0;
        if (row == col)
            v = sqrt(to_double(unpack(C[row * n + row])));
        else if (row < col)
            v = to_double(unpack(C[row * n + col])) * sd[row];
        R[row + (int64_t)col * ldr] = row <= col ? scalbn(v, g[col]) : 0.0;
    }
    return true;
}

// The Householder reduction of the same CTA (12 bulk warps and the reducer; the other warps have
// left), kept out of line: it runs only where the Gram sum cannot serve.
__device__ __noinline__ void fold_job(const F64Args &f, const int leaf) {
    leaf_tree_job<double, double, 2, 1, false>(f, f.A, f.ldS, f.ldS * f.n, leaf);
}

// ------------------------------------------------------------------------------------------
// The kernel.  One CTA per SM, at most one leaf each; launched cooperatively (every CTA waits
// for the root's verdict).
// ------------------------------------------------------------------------------------------
template <int NB, int S>
__global__ void __launch_bounds__(kGramThreads, 1) tsqr_gram_f64_kernel(const __grid_constant__ GramArgs a) {
    using Sh = Shape<NB, S>;
    extern __shared__ __align__(1024) double smem_d[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(smem_d);
    GramSmem &sm = *reinterpret_cast<GramSmem *>(smem + Sh::kStages + Sh::kRaws * Sh::kRaw);
    Q128 *acc = reinterpret_cast<Q128 *>(smem + Sh::kStages + Sh::kRaws * Sh::kRaw + sizeof(GramSmem));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n = a.n, npair = n * (n + 1) / 2;
    const int c = blockIdx.x;

    if (c < a.ctas) {
        // ---- set-up
        if (warp == kGramWarps - 1) tc::tmem_alloc(&sm.tmem, 512);
        if (tid == 0) {
            tc::mbar_init(&sm.bar[0], 1);
            tc::mbar_init(&sm.bar[1], 1);
            tc::fence_mbar_init();
            sm.bad = 0;
        }
        if (tid < 32) sm.D[tid] = sm.E[tid] = 0;
        for (int i = tid; i < Sh::kStages / 16; i += kGramThreads)
            reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0, 0, 0, 0);
        for (int o = tid; o < npair; o += kGramThreads) acc[o] = Q128{0, 0};
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        const uint32_t tmem = sm.tmem;

        const int64_t kb0 = (int64_t)c * a.nkb / a.ctas, kb1 = (int64_t)(c + 1) * a.nkb / a.ctas;
        const int rounds = (int)((kb1 - kb0 + Sh::kRoundKb - 1) / Sh::kRoundKb);
        const double *A = (const double *)a.A, *B = (const double *)a.B;
        const bool vec = ((a.lda | (B ? a.ldb : 0)) & 1) == 0 &&
                         (((uintptr_t)A | (uintptr_t)B) & 15) == 0;
        const int c8 = lane & 7;

        // the lane's column, block and operand address
        const bool slicer = warp < Sh::kSlicers;
        const int kbo = warp / Sh::kGroups;
        const int col = 4 * (warp % Sh::kGroups) + (lane >> 3);
        const double *src = (col < a.na ? A + (int64_t)col * a.lda
                                        : B + (int64_t)(col - a.na) * a.ldb) + (kb0 + kbo) * 64;
        const bool mine = slicer && col < n;
        unsigned char *const dst = smem + kbo * Sh::kKbBytes + (col >> 3) * 1024 +
                                   (col & 7) * 128 + ((c8 ^ (col & 7)) << 4);
        const int my_rounds = mine ? (int)((kb1 - kb0 - kbo + Sh::kRoundKb - 1) / Sh::kRoundKb) : 0;
        const int64_t left0 = a.m - (kb0 + kbo) * 64;
        unsigned char *const raw = smem + Sh::kStages + warp * 2048 + lane * 16;
        // Round r of A on its way to shared memory (one cp.async group a round, empty at the end).
        auto load_round = [&](const int r) {
            if (mine && r < rounds) {
                const int64_t row = (int64_t)r * (64 * Sh::kRoundKb);
                copy_rows(raw + (r % Sh::kRaws) * Sh::kRaw, src + row,
                          r < my_rounds ? left0 - row : 0, c8, vec);
            }
            cp_async_commit();
        };
        // Column exponents raised to what round r needs (one bit to spare); old ones stay
        // in sm.D until the caller has flushed.
        auto scan_round = [&](const int r) {
            int e = 0;
            if (mine) {
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const double2 v = *reinterpret_cast<const double2 *>(
                        raw + (r % Sh::kRaws) * Sh::kRaw + 512 * p);
                    e = max(e, max((__double2hiint(v.x) >> 20) & 0x7ff,
                                   (__double2hiint(v.y) >> 20) & 0x7ff));
                }
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
            if (c8 == 0 && mine) atomicMax(&sm.E[col], e);
            __syncthreads();
            if (tid < NB) {
                e = sm.E[tid];
                if (e > kExpHi) sm.bad = 1;
                sm.Dnew[tid] = max(sm.D[tid], max(e, kExpLo) + 3);
                sm.E[tid] = 0;
            }
            __syncthreads();
        };
        constexpr uint32_t idesc0 = tc::instr_desc(0, 128, Sh::N0, false, false);
        constexpr uint32_t idesc1 = Sh::kTwoTiles ? tc::instr_desc(0, 128, Sh::N1, false, false) : 0;
        const uint32_t sbase = tc::smem_u32(smem);
        uint32_t par[2] = {0, 0};   // parity of the next completion of each stage's barrier
        bool pend[2] = {false, false};
        int sets = 0, in_set = 0;   // accumulator sets begun, rounds in the current one
        bool ok = true;
        auto wait_stage = [&](const int b) {
            if (pend[b]) {
                ok &= tc::mbar_wait(&sm.bar[b], par[b], 1LL << 24);
                par[b] ^= 1;
                pend[b] = false;
            }
        };
        // Accumulators into acc: every digit product's sum, weighted.  All tensor-core work is
        // waited for; the stages are free on return.
        auto flush = [&]() {
            wait_stage(0);
            wait_stage(1);
            tc::fence_after_sync();
            __syncthreads();
            {
                const int q = warp & 3, part = warp >> 2;
                const int p = 32 * q + lane, s = p / NB, i = p - s * NB;
                const uint32_t lanes = tmem + ((uint32_t)(32 * q) << 16);
                long long *hib = reinterpret_cast<long long *>(smem + Sh::kHi);
                long long *lob = reinterpret_cast<long long *>(smem + Sh::kLo);
                long long *l1b = reinterpret_cast<long long *>(smem + Sh::kL1);
                // sum over the sets of digits t .. t + 3 of columns j0 .. j0 + 7, weighted 256^(3 - t)
                auto four = [&](long long (&x)[8], const uint32_t at) {
                    int v[4][8];
#pragma unroll
                    for (int t = 0; t < 4; ++t)
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[t][e] = 0;
                    for (int set = 0; set < sets; ++set) {
                        float f[4][8];
#pragma unroll
                        for (int t = 0; t < 4; ++t)
                            tc::tmem_ld8(at + set * Sh::kCols + t * NB, f[t]);
                        tc::tmem_ld_wait();
#pragma unroll
                        for (int t = 0; t < 4; ++t)
#pragma unroll
                            for (int e = 0; e < 8; ++e) v[t][e] += __float2int_rn(f[t][e]);
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        x[e] = ((long long)v[0][e] * 256 + v[1][e]) * 65536 +
                               ((long long)v[2][e] * 256 + v[3][e]);
                };
                auto pair = [&](long long (&x)[8], const uint32_t at) {
                    float f[2][8];
                    tc::tmem_ld8(at, f[0]);
                    tc::tmem_ld8(at + NB, f[1]);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        x[e] = ((long long)__float2int_rn(f[0][e]) * 256 + __float2int_rn(f[1][e])) *
                               65536;
                };
                auto put = [&](long long *buf, const long long (&x)[8], const int j0) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) buf[(s * NB + j0 + e) * Sh::kLd + i] = x[e];
                };
                constexpr int kJ = NB / 8;
                for (int task = part; task < (Sh::kTwoTiles ? 2 : 1) * kJ; task += 4) {
                    const bool t1 = task >= kJ;
                    const int j0 = 8 * (t1 ? task - kJ : task);
                    const uint32_t at = lanes + j0;
                    long long x[8];
                    if (!t1) {
                        four(x, at);
                        if (s < Sh::kRowDigits0) put(hib, x, j0);
                        four(x, at + 4 * NB);
                        if (s < Sh::kRowDigits0) put(lob, x, j0);
                    } else if (sets == 1) {
                        pair(x, at + Sh::N0);
                        if (s < S - 4) put(l1b, x, j0);
                    } else {
                        long long y[8];
                        pair(x, at + Sh::N0);
                        for (int set = 1; set < sets; ++set) {
                            pair(y, at + Sh::N0 + set * Sh::kCols);
#pragma unroll
                            for (int e = 0; e < 8; ++e) x[e] += y[e];
                        }
                        if (s < S - 4) put(l1b, x, j0);
                    }
                }
                tc::fence_before_sync();
            }
            __syncthreads();
            const long long *hib = reinterpret_cast<const long long *>(smem + Sh::kHi);
            const long long *lob = reinterpret_cast<const long long *>(smem + Sh::kLo);
            const long long *l1b = reinterpret_cast<const long long *>(smem + Sh::kL1);
            for (int o = tid; o < npair; o += kGramThreads) {
                int i, j;
                unpack_index(o, i, j);
                i128 g = 0;
#pragma unroll
                for (int s = 0; s < Sh::kRowDigits0; ++s) {
                    const int ij = (s * NB + j) * Sh::kLd + i, ji = (s * NB + i) * Sh::kLd + j;
                    long long l = lob[ij];
                    if (Sh::kTwoTiles) l += lob[ji];
                    g += (i128)hib[ij] << (64 - 8 * s);
                    g += s <= 4 ? (i128)l << (s <= 4 ? 32 - 8 * s : 0)
                                : (i128)(l >> (s > 4 ? 8 * s - 32 : 0));
                }
                if (Sh::kTwoTiles) {
#pragma unroll
                    for (int s = 4; s < S; ++s) {
                        const int ij = ((s - 4) * NB + j) * Sh::kLd + i;
                        const int ji = ((s - 4) * NB + i) * Sh::kLd + j;
                        long long l = l1b[ij];
                        if (s >= 6) l += l1b[ji];
                        g += (i128)(l >> (8 * s - 32));
                    }
                }
                acc[o] = pack(unpack(acc[o]) + g);
            }
            sets = 0;
            in_set = 0;
            __syncthreads();
        };

        auto zero_stages = [&]() {  // columns past n read as zeros
            for (int i = tid; i < Sh::kStages / 16; i += kGramThreads)
                reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0, 0, 0, 0);
            tc::fence_proxy_async();
            __syncthreads();
        };
#pragma unroll
        for (int r = 0; r < Sh::kRaws; ++r) load_round(r);
        cp_async_wait<Sh::kRaws - 1>();
        scan_round(0);
        if (tid < NB) sm.D[tid] = sm.Dnew[tid];
        zero_stages();
        for (int r = 0; r < rounds && !sm.bad; ++r) {
            const int b = r & 1;
            cp_async_wait<Sh::kRaws - 1>();
            wait_stage(b);
            for (;;) {
                int dmin = 2;
                if (mine) {
                    slice8<NB, S>(raw + (r % Sh::kRaws) * Sh::kRaw, sm.D[col], dmin,
                                  dst + b * Sh::kStage);
                    tc::fence_proxy_async();
                }
                if (!__syncthreads_or(dmin < 2)) break;
                // an entry above its column's range: what is accumulated goes to acc, then the
                // exponents rise and acc's entries follow
                scan_round(r);
                if (sm.bad) break;
                if (sets > 0) flush();
                for (int o = tid; o < npair; o += kGramThreads) {
                    int i, j;
                    unpack_index(o, i, j);
                    acc[o] = pack(shr128(unpack(acc[o]), sm.Dnew[i] - sm.D[i] + sm.Dnew[j] - sm.D[j]));
                }
                __syncthreads();
                if (tid < NB) sm.D[tid] = sm.Dnew[tid];
                zero_stages();
            }
            if (sm.bad) break;
            if (in_set == 0) ++sets;
            if (tid == kGramThreads - 32) {
                tc::fence_after_sync();
                const uint32_t d0 = tmem + (uint32_t)(sets - 1) * Sh::kCols;
                for (int kb = 0; kb < Sh::kRoundKb; ++kb) {
                    const uint32_t base = sbase + b * Sh::kStage + kb * Sh::kKbBytes;
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        const bool add = in_set > 0 || kb > 0 || ks > 0;
                        const uint64_t bd = tc::smem_desc(base + 32 * ks, 16, 1024, tc::kSw128);
                        tc::mma_f16(d0, bd, bd, idesc0, add);
                        if (Sh::kTwoTiles) {
                            const uint64_t b1 = tc::smem_desc(base + 4 * NB * 128 + 32 * ks, 16, 1024,
                                                              tc::kSw128);
                            tc::mma_f16(d0 + Sh::N0, b1, b1, idesc1, add);
                        }
                    }
                }
                tc::mma_commit(&sm.bar[b]);
            }
            pend[b] = true;
            if (++in_set == Sh::kSetRounds) in_set = 0;
            load_round(r + Sh::kRaws);
            if (r + 1 == rounds || (in_set == 0 && sets == Sh::kSets)) {
                flush();
                if (r + 1 < rounds && n < NB) zero_stages();
            }
        }
        cp_async_wait_all();
        wait_stage(0);
        wait_stage(1);
        __syncthreads();
        if (warp == kGramWarps - 1) {
            tc::tmem_relinquish();
            tc::tmem_dealloc(tmem, 512);
        }
        if (__syncthreads_or(!ok)) {  // a wait gave up: reported, the Householder reduction runs
            if (tid == 0) {
                sm.bad = 1;
                atomicOr(a.status, kStatusTimeoutBit);
            }
            __syncthreads();
        }

        // ---- the tree: publish (exponents, sums), the last child to arrive adds its siblings
        int cnt = a.ctas, off = 0, t = c, cidx = 0;
        bool root = false;
        for (;;) {
            if (cnt == 1) {
                root = true;
                break;
            }
            const int next_cnt = (cnt + kGramArity - 1) / kGramArity;
            const int parent = t / kGramArity, first = parent * kGramArity;
            const int nchild = min(kGramArity, cnt - first);
            unsigned char *mine = a.slots + (size_t)(off + t) * a.slot_bytes;
            if (tid < 32) reinterpret_cast<int *>(mine)[tid] = tid < n ? sm.D[tid] : 0;
            if (tid == 0) reinterpret_cast<int *>(mine)[kGramSlotHead / 4 - 1] = sm.bad;
            for (int o = tid; o < npair; o += kGramThreads)
                reinterpret_cast<Q128 *>(mine + kGramSlotHead)[o] = acc[o];
            __threadfence();
            __syncthreads();
            if (tid == 0) sm.flag = atomicAdd(&a.counters[cidx + parent], 1u) + 1 == (unsigned)nchild;
            __syncthreads();
            if (!sm.flag) break;
            __threadfence();
            const unsigned char *kids = a.slots + (size_t)(off + first) * a.slot_bytes;
            // the children's exponents (and whether one cannot be served), then the sums
            int *kd = reinterpret_cast<int *>(smem);
            if (tid < 32 * kGramArity) {
                const int ch = tid >> 5;
                kd[tid] = ch < nchild ? __ldcg(reinterpret_cast<const int *>(kids + ch * a.slot_bytes) + lane)
                                      : 0;
            }
            if (tid == 0) sm.bad = 0;
            __syncthreads();
            if (tid < 32) {
                int d = 0;
                for (int ch = 0; ch < kGramArity; ++ch) d = max(d, kd[32 * ch + tid]);
                sm.D[tid] = d;
            } else if (tid < 32 + nchild) {
                if (__ldcg(reinterpret_cast<const int *>(kids + (tid - 32) * a.slot_bytes) +
                           kGramSlotHead / 4 - 1))
                    sm.bad = 1;
            }
            __syncthreads();
            for (int o = tid; o < npair; o += kGramThreads) {
                int i, j;
                unpack_index(o, i, j);
                const int dij = sm.D[i] + sm.D[j];
                const unsigned char *e = kids + kGramSlotHead + (size_t)o * 16;
                i128 g = 0;
#pragma unroll 4
                for (int ch = 0; ch < nchild; ++ch)
                    g += shr128(ldcg128(e + ch * a.slot_bytes),
                                dij - kd[32 * ch + i] - kd[32 * ch + j]);
                acc[o] = pack(g);
            }
            __syncthreads();
            off += cnt;
            cidx += next_cnt;
            cnt = next_cnt;
            t = parent;
        }
        if (root) {
            // scale columns, then factor: C at the bottom of shared memory
            Q128 *C = reinterpret_cast<Q128 *>(smem);
            Q128 *rowv = C + n * n;
            bool good = !sm.bad;
            __syncthreads();
            if (tid < n) {
                const i128 d = unpack(acc[tid * (tid + 1) / 2 + tid]);
                const u64 dh = (u64)((u128)d >> 64);
                const int len = dh ? 128 - __clzll((long long)dh) : 64 - __clzll((long long)(u64)d);
                sm.E[tid] = d > 0 ? (122 - len) >> 1 : 1 << 20;  // shift t_j
                if (!(d > 0)) sm.bad = 1;
                sm.Dnew[tid] = 73 - sm.E[tid] + sm.D[tid] - 1086;
            }
            __syncthreads();
            good = good && !sm.bad;
            if (good) {
                for (int o = tid; o < npair; o += kGramThreads) {
                    int i, j;
                    unpack_index(o, i, j);
                    C[i * n + j] = pack(shift128(unpack(acc[o]), sm.E[i] + sm.E[j]));
                }
                __syncthreads();
                good = factor_root(C, rowv, n, sm.Dnew, a.R, a.ldr);
            }
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                atomicExch(a.verdict, good ? 1u : 2u);
            }
            if (good) return;
        }
    }

    // ---- the verdict: 1, done; 2, the Householder reduction
    if (threadIdx.x == 0) {
        unsigned v = 0;
        for (long long it = 0; it < kVerdictPolls; ++it) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.verdict) : "memory");
            if (v) break;
            __nanosleep(200);
        }
        sm.flag = (int)v;
        if (!v) atomicOr(a.status, kStatusTimeoutBit);
    }
    __syncthreads();
    const int v = sm.flag;
    __syncthreads();
    if (v != 2 || c >= a.fold.nleaves || tid >= TSQR_FOLD_THREADS) return;
    fold_job(a.fold, c);
}

typedef void (*GramKernel)(const GramArgs);

struct Variant {
    GramKernel fn;
    size_t smem;
    int kb_round;
};
template <int NB, int S>
Variant variant(int n) {
    return Variant{tsqr_gram_f64_kernel<NB, S>,
                   (size_t)Shape<NB, S>::kStages + Shape<NB, S>::kRaws * Shape<NB, S>::kRaw + sizeof(GramSmem) + (size_t)n * (n + 1) / 2 * 16,
                   Shape<NB, S>::kRoundKb};
}
Variant variant_for(int n) {
    return n <= 8 ? variant<8, 8>(n) : n <= 16 ? variant<16, 8>(n)
           : n <= 24 ? variant<24, 8>(n) : variant<32, 8>(n);
}

}  // namespace

int gram_round_rows(int n) { return 64 * variant_for(n).kb_round; }
size_t gram_smem_bytes(int n) { return variant_for(n).smem; }

cudaError_t gram_prepare(int n, size_t smem_bytes) {
    return set_smem_attrs(variant_for(n).fn, smem_bytes);
}

cudaError_t gram_launch(const GramArgs &a, size_t smem_bytes, cudaStream_t stream) {
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(a.ctas > a.fold.nleaves ? a.ctas : a.fold.nleaves);
    cfg.blockDim = dim3(kGramThreads);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    GramArgs args = a;
    void *params[1] = {&args};
    return cudaLaunchKernelExC(&cfg, (const void *)variant_for(a.n).fn, params);
}

}  // namespace tsqr
