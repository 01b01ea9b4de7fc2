// The exact-Gram reduction's single launch for tsqr_qr (tsqr_gram_single.cuh).
#include "tsqr_gram.cuh"
#define TSQR_FOLD_THREADS (32 * (kGramFoldQ.warps + 1))
#include "tsqr_gram_single.cuh"

namespace tsqr {

namespace {

// One leaf a CTA and tall chunks: the passes that apply the reflectors want them (1,000,000 x 32 at
// kappa 1e6, whole call: 6,980 us, with R's leaves 7,540).  The reflectors are kept, or, where only R
// is asked for under tsqr_qr's plan, not.
struct QLeaves {
    static constexpr GramFold kShape = kGramFoldQ;
    template <bool kStore>
    static __device__ __noinline__ void fold(const F64Args &f, const int leaf) {
        leaf_tree_job<double, double, 2, 1, false, kStore>(f, f.A, f.ldS, f.ldS * f.n, leaf);
    }
    static __device__ __forceinline__ void run(const F64Args &f, const int leaf) {
        if (f.q.V)
            fold<true>(f, leaf);
        else
            fold<false>(f, leaf);
    }
};

}  // namespace

cudaError_t gram_qr_prepare(int n, size_t smem_bytes) { return single_prepare<QLeaves>(n, smem_bytes); }
cudaError_t gram_qr_launch(const GramArgs &a, size_t smem_bytes, cudaStream_t stream) {
    return single_launch<QLeaves>(a, smem_bytes, stream);
}

}  // namespace tsqr
