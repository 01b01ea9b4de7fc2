// The single launch of the exact-Gram reduction (up to kGramMaxN columns) for tsqr_r and for
// tsqr_qr, which differ in the Householder leaves that stand behind the sum.  Leaves, a type of the
// file that includes this (after it has defined TSQR_FOLD_THREADS, a leaf's threads): kShape, and
// run(), a leaf of the reduction on a group of the CTA's threads.
#pragma once

#include <cstring>

#include "tsqr_gram_dev.cuh"

namespace tsqr {
namespace {
using namespace gram;

constexpr long long kVerdictPolls = 1LL << 27;  // of at least 0.2 us each

// What bounds it: shared memory.  A 128-row round at 32 columns moves some 275 KB through it (A in
// and out 64, its digits 64, the products' operands 147), 2.15k of the 3.2k cycles a round takes;
// cutting alone is 1.2k, the products 0.8k.  Then the flush of every 1,024 rows' sums (7k cycles).
// The Householder leaves it stands before are bound by FP64 arithmetic.  us: 4,194,304 x 32 10,103
// before, 482 now (HBM's share 161); 16,777,216 x 8 2,697 / 395 (161); 10,000 x 16 198 / 38.9,
// latency: the sums 14k cycles, the tree 9k, the root 25k.
//
// One FP64 matrix of at most 32 columns in one launch: CTA c sums slab c, the root factors, every
// CTA waits for its verdict and runs its leaves of the Householder reduction where the Gram cannot
// serve.  One CTA per SM, launched cooperatively.
template <int NB, typename Leaves>
__global__ void __launch_bounds__(kGramThreads, 1)
tsqr_gram_f64_kernel(const __grid_constant__ GramArgs a) {
    extern __shared__ __align__(1024) double smem_d[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(smem_d);
    const int tid = threadIdx.x, b = blockIdx.x;
    const size_t slot_bytes = gram_slot_bytes(NB);
    if (b < a.p.nslab) {
        Cta c;
        cta_begin(c, smem);
        const bool root = item_of<NB, 0>(a.p, Cols{0, a.p.n, 0, 0}, 0, b, slot_bytes, c);
        if (!c.ok && tid == 0) atomicOr(a.status, kStatusTimeoutBit);
        cta_end(c);
        if (root) {
            const bool good = finish(a.p, slot_bytes, c.sm, c.stages);
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                atomicExch(a.p.verdict, good ? 1u : 2u);
            }
            if (good) return;
        }
    }
    // the verdict: 1, done; 2, the Householder reduction (threads past the last group leave)
    Smem &sm = *reinterpret_cast<Smem *>(smem);
    if (tid == 0) {
        unsigned v = 0;
        for (long long it = 0; it < kVerdictPolls; ++it) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.p.verdict) : "memory");
            if (v) break;
            __nanosleep(200);
        }
        sm.flag = (int)v;
        if (!v) atomicOr(a.status, kStatusTimeoutBit);
    }
    __syncthreads();
    const int v = sm.flag;
    __syncthreads();
    const int group = tid / (TSQR_FOLD_THREADS), leaf = b + gridDim.x * group;
    if (v != 2 || leaf >= a.fold.nleaves || group >= Leaves::kShape.groups) return;
    Leaves::run(a.fold, leaf);
}

typedef void (*GramKernel)(const GramArgs);
struct Variant {
    GramKernel fn;
    size_t smem;
    int kb_round;
};
template <int NB, typename Leaves>
Variant variant() {
    using Sh = Shape<NB, 0>;
    return Variant{tsqr_gram_f64_kernel<NB, Leaves>, smem_bytes<Sh>(), Sh::kRoundKb};
}
template <typename Leaves>
Variant variant_for(int n) {
    return n <= 8    ? variant<8, Leaves>()
           : n <= 16 ? variant<16, Leaves>()
           : n <= 24 ? variant<24, Leaves>()
                     : variant<32, Leaves>();
}

template <typename Leaves>
cudaError_t single_prepare(int n, size_t smem_bytes) {
    return set_smem_attrs(variant_for<Leaves>(n).fn, smem_bytes);
}

template <typename Leaves>
cudaError_t single_launch(const GramArgs &a, size_t smem_bytes, cudaStream_t stream) {
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(a.grid);
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
    return cudaLaunchKernelExC(&cfg, (const void *)variant_for<Leaves>(a.p.n).fn, params);
}

}  // namespace
}  // namespace tsqr
