// The exact-Gram reduction past kGramRootMaxN columns: the set sums (tsqr_gram.cu) gathered into
// one matrix of 122-bit fixed-point values in global memory and factored by block rows of 32, on
// many CTAs: per block row one launch factors the diagonal block (every CTA for itself: the serial
// chain of 32 pivots is the launch's time either way) and eliminates the columns right of it, one
// launch takes the block row's product off the rows below.
#include "tsqr_gram.cuh"
#include "tsqr_gram_dev.cuh"

namespace tsqr {

namespace {
using namespace gram;

constexpr int kBw = 32;  // rows of a block

__device__ __forceinline__ const unsigned char *set_top(const GramProblem &p, const int I, const int J) {
    const int per_set = p.nslab + gram_inner_nodes(p.nslab, p.n);
    const int set = I == J ? I : p.nb + J * (J - 1) / 2 + I;
    return p.slots + ((size_t)(set + 1) * per_set - 1) * gram_slot_bytes(kBlock);
}

// The sum (i, j), i <= j, aligned to the column exponents D.
__device__ __forceinline__ i128 wide_entry(const GramProblem &p, const int *D, const int i, const int j) {
    const int I = i / kBlock, J = j / kBlock, li = i % kBlock, lj = j % kBlock;
    const unsigned char *t = set_top(p, I, J);
    const int *h = reinterpret_cast<const int *>(t);
    const int nj = min(kBlock, p.n - J * kBlock);
    const size_t o = I == J ? (size_t)(lj * (lj + 1) / 2 + li) : (size_t)(li * nj + lj);
    return shr128(ldcg128(t + kGramSlotHead + o * 16),
                  D[i] + D[j] - __ldcg(h + li) - __ldcg(h + (I == J ? lj : 64 + lj)));
}

// Column exponents (the largest of a column's sets), shifts and R's powers of two.
__global__ void tsqr_gram_scale_kernel(const GramWideArgs a) {
    const GramProblem &p = a.p;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= p.n) return;
    const int b = j / kBlock, l = j % kBlock;
    int d = 0, bad = 0;
    for (int o = 0; o < p.nb; ++o) {
        const int *h = reinterpret_cast<const int *>(set_top(p, min(o, b), max(o, b)));
        d = max(d, __ldcg(h + (o < b ? 64 : 0) + l));
        bad |= __ldcg(h + kGramSlotHead / 4 - 1);
    }
    a.D[j] = d;
    // the diagonal's set: aligned to d by hand, D being written by other threads
    const int *h = reinterpret_cast<const int *>(set_top(p, b, b));
    const i128 g = shr128(ldcg128(reinterpret_cast<const unsigned char *>(h) + kGramSlotHead +
                                  (size_t)(l * (l + 1) / 2 + l) * 16),
                          2 * (d - __ldcg(h + l)));
    const u64 gh = (u64)((u128)g >> 64);
    const int len = gh ? 128 - __clzll((long long)gh) : 64 - __clzll((long long)(u64)g);
    const int e = g > 0 ? (122 - len) >> 1 : 0;
    a.E[j] = e;
    a.g[j] = 73 - e + d + kUnit + p.guard / 2;
    if (bad || d <= kLeastD || (!(g > 0) && j < p.np)) *a.bad = 1;
}

__global__ void tsqr_gram_fill_kernel(const GramWideArgs a) {
    if (*a.bad) return;
    const int n = a.p.n;
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < (int64_t)n * n;
         o += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(o / n), j = (int)(o - (int64_t)i * n);
        if (i <= j)
            reinterpret_cast<Q128 *>(a.C)[o] =
                pack(shift128(wide_entry(a.p, a.D, i, j), a.E[i] + a.E[j]));
    }
}

__device__ __forceinline__ i128 smul122(const i128 a, const i128 b) {
    const u128 q = mul122((u128)(a < 0 ? -a : a), (u128)(b < 0 ? -b : b));
    return (a < 0) != (b < 0) ? -(i128)q : (i128)q;
}
// c / d for a pivot d in [1/4, 1) with reciprocal r.
__device__ __forceinline__ i128 squotient(const i128 c, const u128 d, const u64 r) {
    const i128 q = (i128)quotient((u128)(c < 0 ? -c : c), d, r);
    return c < 0 ? -q : q;
}
__device__ __forceinline__ i128 shfl128(const i128 x, const int src) {
    const u64 lo = __shfl_sync(0xffffffffu, (u64)x, src);
    const u64 hi = __shfl_sync(0xffffffffu, (u64)((u128)x >> 64), src);
    return (i128)(((u128)hi << 64) | lo);
}

// Block row kb: its diagonal block factored (by every CTA for itself: the root's chain), then the
// columns right of it, one warp a column: lane i holds row i; step k takes row k's multiple off the
// rows below.  Bound by the chain of 32 pivots, 1.7k cycles each of some 45 us.
__global__ void __launch_bounds__(kGramThreads) tsqr_gram_panel_kernel(const GramWideArgs a, const int kb) {
    __shared__ Q128 L[kBw * (kBw + 1) / 2], rowv[3 * kBw];
    __shared__ u64 rec[kBw];
    __shared__ int zs[kBw], low;
    const int n = a.p.n, k0 = kb * kBw, w = min(kBw, n - k0), wp = min(w, a.p.np - k0);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // one thread's read decides for the CTA: another CTA of this launch may be setting the word, and
    // threads that saw it would be missing from the barriers of those that did not
    if (__syncthreads_or(tid == 0 && __ldcg(a.bad) != 0)) return;
    constexpr int kWarps = kGramThreads / 32;
    Q128 *C = reinterpret_cast<Q128 *>(a.C), *P = reinterpret_cast<Q128 *>(a.P);
    for (int o = tid; o < w * w; o += kGramThreads) {
        const int i = o / w, j = o % w;
        if (i <= j) L[rowoff(w, i) - i + j] = C[(int64_t)(k0 + i) * n + k0 + j];
    }
    if (tid == 0) low = 0;
    __syncthreads();
    u128 mine;
    int myz;
    if (!factor_chain(L, rowv, w, wp, &low, mine, myz)) {  // (the same for every thread of every CTA)
        if (tid == 0) *a.bad = 1;
        return;
    }
    Q128 *piv = rowv + 2 * w;
    if (tid < w) {  // (rows past wp go along as they are)
        if (tid >= wp) piv[tid] = pack((i128)1 << 121);
        rec[tid] = recip60(tid < wp ? mine : (u128)1 << 121);
        zs[tid] = tid < wp ? myz : 0;
    }
    __syncthreads();
    if (blockIdx.x == 0) {
        for (int o = tid; o < w * w; o += kGramThreads) {
            const int i = o / w, j = o % w;
            // (mirrored: other CTAs may still be reading the block itself)
            if (i < j) C[(int64_t)(k0 + j) * n + k0 + i] = L[rowoff(w, i) - i + j];
        }
        if (tid < w) {
            reinterpret_cast<Q128 *>(a.d)[k0 + tid] = piv[tid];
            a.z[k0 + tid] = zs[tid];
        }
    }
    for (int j = k0 + kBw + blockIdx.x * kWarps + warp; j < n; j += gridDim.x * kWarps) {  // (w == kBw here)
        i128 c = unpack(C[(int64_t)(k0 + lane) * n + j]);
        for (int k = 0; k < kBw - 1; ++k) {
            i128 ck = shfl128(c, k);
            const int z = zs[k];
            if (z) ck = (i128)((u128)ck << z);
            if (lane > k) c -= smul122(unpack(L[rowoff(kBw, k) - k + lane]), ck);
        }
        const int z = zs[lane];
        if (z) c = (i128)((u128)c << z);
        P[(int64_t)lane * n + j] = pack(c);
        C[(int64_t)(k0 + lane) * n + j] = pack(squotient(c, (u128)unpack(piv[lane]), rec[lane]));
    }
}

// C(I, J) -= sum over block row kb of l(k, i) c(k, j), 32 x 32 a CTA.  Values as x = h 2^62 + l with
// signed h and 0 <= l < 2^62: of a product over 2^122 the high product and the upper words of the
// mixed ones are summed (2^-118 a term is left out).  A thread an output: few tiles, so latency
// counts (17 us a launch at 512 columns, 21 with four outputs a thread).
__global__ void __launch_bounds__(1024) tsqr_gram_update_kernel(const GramWideArgs a, const int kb) {
    __shared__ long long lh[kBw][kBw], ll[kBw][kBw], ch[kBw][kBw], cl[kBw][kBw];
    if (*a.bad) return;
    const int n = a.p.n, k0 = kb * kBw, first = k0 + kBw;
    int J = 0;
    int o = blockIdx.x;  // tile (I, J), I <= J, of the blocks right of the block row
    while (o > J) o -= ++J;
    const int i0 = first + o * kBw, j0 = first + J * kBw;
    const int tid = threadIdx.x;
    Q128 *C = reinterpret_cast<Q128 *>(a.C);
    const Q128 *P = reinterpret_cast<const Q128 *>(a.P);
    constexpr long long kMask = (1ll << 62) - 1;
    {
        const int k = tid / kBw, x = tid % kBw;
        const i128 l = i0 + x < n ? unpack(C[(int64_t)(k0 + k) * n + i0 + x]) : (i128)0;
        const i128 c = j0 + x < n ? unpack(P[(int64_t)k * n + j0 + x]) : (i128)0;
        lh[k][x] = (long long)(l >> 62);
        ll[k][x] = (long long)l & kMask;
        ch[k][x] = (long long)(c >> 62);
        cl[k][x] = (long long)c & kMask;
    }
    __syncthreads();
    const int jx = tid & 31, iy = tid >> 5;
    i128 hh = 0;
    long long mm = 0;
#pragma unroll 4
    for (int k = 0; k < kBw; ++k) {
        const long long ah = lh[k][iy], al = ll[k][iy], bh = ch[k][jx], bl = cl[k][jx];
        hh += (i128)ah * bh;
        mm += __mul64hi(ah, bl) + __mul64hi(al, bh);
    }
    const int i = i0 + iy, j = j0 + jx;
    if (i <= j && j < n) {
        Q128 *e = C + (int64_t)i * n + j;
        *e = pack(unpack(*e) - (hh * 4 + (i128)mm * 16));
    }
}

// R from the factor (or, where the sum cannot serve, only the verdict).
__global__ void tsqr_gram_write_kernel(const GramWideArgs a) {
    const bool bad = *a.bad != 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.p.verdict = bad ? 2u : 1u;
    if (bad) return;
    const int n = a.p.n;
    const Q128 *C = reinterpret_cast<const Q128 *>(a.C), *d = reinterpret_cast<const Q128 *>(a.d);
    // a CTA writes tiles of 32 x 32 (rows of C in, columns of R out)
    __shared__ double t[kBw][kBw + 1];
    __shared__ u64 sq[kBw];
    const int nb = (n + kBw - 1) / kBw;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int tile = blockIdx.x; tile < nb * nb; tile += gridDim.x) {
        const int i0 = tile / nb * kBw, j0 = tile % nb * kBw;
        if (ty == 0) sq[tx] = i0 <= j0 && i0 + tx < a.p.np ? sqrt64((u128)unpack(d[i0 + tx])) : 0;
        __syncthreads();
        for (int u = ty; u < kBw; u += 8) {
            const int i = i0 + u, j = j0 + tx;
            double v = 0.0;
            if (i <= j && j < n && i < a.p.np) {
                // (a diagonal block's l are mirrored, see the panel kernel)
                v = i == j ? round64(sq[u], a.g[j] - 64 - a.z[i], false)
                           : r_entry(unpack(i0 == j0 ? C[(int64_t)j * n + i] : C[(int64_t)i * n + j]),
                                     sq[u], a.g[j]);
            }
            t[u][tx] = v;
        }
        __syncthreads();
        for (int u = ty; u < kBw; u += 8) {
            const int i = i0 + tx, j = j0 + u;
            if (i < n && j < n) a.p.R[i + (int64_t)j * a.p.ldr] = t[tx][u];
        }
        __syncthreads();
    }
}

}  // namespace

int gram_wide_launch(const GramWideArgs &a, cudaStream_t stream) {
    const int n = a.p.n, nb = (n + kBw - 1) / kBw, done = (a.p.np + kBw - 1) / kBw;
    int launches = 0;
    tsqr_gram_scale_kernel<<<(n + 127) / 128, 128, 0, stream>>>(a);
    const int64_t fill = ((int64_t)n * n + 255) / 256;
    tsqr_gram_fill_kernel<<<(int)(fill < 4096 ? fill : 4096), 256, 0, stream>>>(a);
    launches += 2;
    for (int kb = 0; kb < done; ++kb) {
        const int right = n - (kb + 1) * kBw;
        const int ctas = right > 0 ? (right + kGramThreads / 32 - 1) / (kGramThreads / 32) : 1;
        tsqr_gram_panel_kernel<<<ctas < 1024 ? ctas : 1024, kGramThreads, 0, stream>>>(a, kb);
        ++launches;
        if (kb + 1 == done) break;
        const int t = (right + kBw - 1) / kBw;
        tsqr_gram_update_kernel<<<t * (t + 1) / 2, 1024, 0, stream>>>(a, kb);
        ++launches;
    }
    tsqr_gram_write_kernel<<<nb * nb < 1024 ? nb * nb : 1024, 256, 0, stream>>>(a);
    ++launches;
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

}  // namespace tsqr
