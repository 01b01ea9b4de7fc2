// Exact-Gram reduction on the tensor cores: the kernels (tsqr_gram.cuh has the method,
// tsqr_gram_dev.cuh the device code).
#include "tsqr_gram.cuh"
#define TSQR_FOLD_THREADS (32 * (kGramFoldR.warps + 1))
#include "tsqr_gram_single.cuh"

namespace tsqr {

namespace {

// tsqr_r's leaves: several a CTA hide each other's reflector chains and barriers, as two or three
// CTAs an SM do for that reduction by itself.  Out of line: they run only where the Gram sum cannot
// serve.  (A zero column, us, with one leaf of 12 warps a CTA / so: 10,000 x 16 249 / 180, 1,000,000 x
// 32 3,202 / 2,939.)
struct RLeaves {
    static constexpr GramFold kShape = kGramFoldR;
    template <int B>
    static __device__ __noinline__ void fold(const F64Args &f, const int leaf) {
        leaf_tree_job<double, double, B, 1, false>(f, f.A, f.ldS, f.ldS * f.n, leaf);
    }
    static __device__ __forceinline__ void run(const F64Args &f, const int leaf) {
        if (f.blk == 3)
            fold<3>(f, leaf);
        else if (f.blk == 2)
            fold<2>(f, leaf);
        else
            fold<1>(f, leaf);
    }
};

// A queue of work items (sets of columns over slabs of rows) of one matrix or many: the CTA that
// completes a matrix's last set factors it.  Bound by the two-block sets, 3.9k cycles a 64-row round:
// the digits of 64 columns 1.4k, 64 KB of operands read for each of eight products, the flush 0.9k
// a round (one accumulator set, so every 1,024 rows).  us, Householder / here: 4,194,304 x 128 154,900 /
// 7,115; 1,000,000 x 50 with an odd leading dimension (8-byte copies of every other column) 6,670 / 625;
// 512 problems 27,300 / 1,450.
__global__ void __launch_bounds__(kGramThreads, 1)
tsqr_gram_queue_f64_kernel(const __grid_constant__ GramQueueArgs a) {
    extern __shared__ __align__(1024) double smem_d[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(smem_d);
    const int tid = threadIdx.x;
    constexpr int NB = kBlock;
    Cta c;
    cta_begin(c, smem);
    for (;;) {
        __syncthreads();
        if (tid == 0) c.sm->item = (int)atomicAdd(a.queue, 1u);
        __syncthreads();
        const int it = c.sm->item;
        if (it >= a.nitems) break;
        int which = 0, code = it;
        if (a.probs) {
            const int2 w = __ldg(a.items + it);
            which = w.x;
            code = w.y;
        }
        const GramProblem &p = a.probs ? a.probs[which] : a.one;
        const size_t slot_bytes = gram_slot_bytes(gram_block(p.n));
        const int nset = gram_sets(p.nb);
        int slab = code / nset, set = code - slab * nset;
        if (!a.probs && code >= a.cut) {  // the last slabs set by set
            const int tail = p.nslab - a.cut / nset, q = code - a.cut, o = q / tail;
            slab = p.nslab - tail + q - o * tail;
            set = o < nset - p.nb ? p.nb + o : o - (nset - p.nb);
        }
        Cols cols{0, 0, 0, 0};
        bool root;
        if (set < p.nb) {
            cols.i0 = set * NB;
            cols.ni = min(NB, p.n - cols.i0);
            if (cols.ni <= 8)
                root = item_of<8, 0>(p, cols, set, slab, slot_bytes, c);
            else if (cols.ni <= 16)
                root = item_of<16, 0>(p, cols, set, slab, slot_bytes, c);
            else if (cols.ni <= 24)
                root = item_of<24, 0>(p, cols, set, slab, slot_bytes, c);
            else
                root = item_of<32, 0>(p, cols, set, slab, slot_bytes, c);
        } else {
            int I = 0, J = 1;
            for (int o = set - p.nb; o >= J; ++J) o -= J;
            I = set - p.nb - J * (J - 1) / 2;
            cols = Cols{I * NB, NB, J * NB, min(NB, p.n - J * NB)};
            if (cols.nj <= 8)
                root = item_of<32, 8>(p, cols, set, slab, slot_bytes, c);
            else if (cols.nj <= 16)
                root = item_of<32, 16>(p, cols, set, slab, slot_bytes, c);
            else if (cols.nj <= 24)
                root = item_of<32, 24>(p, cols, set, slab, slot_bytes, c);
            else
                root = item_of<32, 32>(p, cols, set, slab, slot_bytes, c);
        }
        if (!root || p.n > kGramRootMaxN) continue;  // (a wider matrix is factored by its own launches)
        if (nset > 1) {
            if (tid == 0)
                c.sm->flag = atomicAdd(p.counters + (size_t)nset * gram_inner_nodes(p.nslab, p.n), 1u) + 1 ==
                             (unsigned)nset;
            __syncthreads();
            if (!c.sm->flag) continue;
            __threadfence();
        }
        const bool good = finish(p, slot_bytes, c.sm, c.stages);
        __syncthreads();
        if (tid == 0) {
            *p.verdict = good ? 1u : 2u;
            if (!good) atomicAdd(a.failed, 1u);
        }
    }
    if (!c.ok && tid == 0) atomicOr(a.status, kStatusTimeoutBit);
    cta_end(c);
}

constexpr size_t queue_smem() {
    size_t b = smem_bytes<Shape<8, 0>>();
    for (size_t o : {smem_bytes<Shape<16, 0>>(), smem_bytes<Shape<24, 0>>(),
                     smem_bytes<Shape<32, 0>>(), smem_bytes<Shape<32, 8>>(),
                     smem_bytes<Shape<32, 16>>(), smem_bytes<Shape<32, 24>>(),
                     smem_bytes<Shape<32, 32>>()})
        b = o > b ? o : b;
    return b;
}
static_assert(queue_smem() <= 227 * 1024, "one CTA's shared memory");
static_assert(kHead + (kGramRootMaxN * (kGramRootMaxN + 1) / 2 + 3 * kGramRootMaxN) * 16 <= queue_smem(),
              "the root's triangle fits");

}  // namespace

int gram_round_rows(int n) { return 64 * variant_for<RLeaves>(n).kb_round; }
size_t gram_smem_bytes(int n) { return variant_for<RLeaves>(n).smem; }
cudaError_t gram_prepare(int n, size_t smem_bytes) { return single_prepare<RLeaves>(n, smem_bytes); }
cudaError_t gram_launch(const GramArgs &a, size_t smem_bytes, cudaStream_t stream) {
    return single_launch<RLeaves>(a, smem_bytes, stream);
}

cudaError_t gram_queue_launch(const GramQueueArgs &a, int grid, cudaStream_t stream) {
    const cudaError_t e = set_smem_attrs(tsqr_gram_queue_f64_kernel, queue_smem());
    if (e != cudaSuccess) return e;
    tsqr_gram_queue_f64_kernel<<<grid, kGramThreads, queue_smem(), stream>>>(a);
    return cudaGetLastError();
}

}  // namespace tsqr
