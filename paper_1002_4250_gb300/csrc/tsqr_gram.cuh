// The exact-Gram reduction (TSQR_LEAF_GRAM): arguments shared by the host API and the kernels.
//
// R is the Cholesky factor of A^T A.  In floating point that route loses half the digits, but
// its sums are products of whole numbers once every column is written in fixed point against
// its largest entry, and whole numbers are what the tensor cores add without error: an entry is
// cut into S balanced 8-bit digits (FP16 operands in [-128, 128]), a product of two digits is at
// most 2^14, so an FP32 accumulator holds 1,024 rows of them exactly (2^24).  The digit products
// are put together in 128-bit integers, the row blocks' Grams are added (integer sums: the
// order does not matter), and the root factors the sum in 122-bit fixed point.  What is left of
// rounding is that of the input's fixed-point form and of R's entries.
//
// The tree of Section 2 is the sum over the row blocks.  A matrix this form cannot serve (a
// non-finite or extreme entry, a pivot below 2^-bits of its column's square) is found by the
// root, and the Householder reduction then runs instead.
//
// Columns are taken in blocks of 32: a column set is a block against itself or a block against a
// later one, and a work item is one set over one slab of rows.
#pragma once

#include "tsqr_f64.cuh"

namespace tsqr {

constexpr int kGramSlicers = 16;    // warps that cut entries into digits; one more multiplies
constexpr int kGramThreads = 32 * (kGramSlicers + 1);
// The Householder leaves behind the single launch: `groups` a CTA at a time, of `warps` bulk warps and
// a reducer each.
struct GramFold {
    int warps, groups;
};
constexpr GramFold kGramFoldR{4, 3}, kGramFoldQ{12, 1};
constexpr bool gram_fold_fits(const GramFold f) {
    return 32 * (f.warps + 1) * f.groups <= kGramThreads && f.groups < 16;  // (named barriers)
}
static_assert(gram_fold_fits(kGramFoldR) && gram_fold_fits(kGramFoldQ), "the leaves' threads");
constexpr int kGramMaxN = 32;       // one column block: tsqr_r's single launch
constexpr int kGramRootMaxN = 128;  // widest matrix one CTA factors

// One matrix [A | B] (B: columns na .. n-1, or none) and where its sums go.
struct GramProblem {
    const double *A, *B;
    int64_t lda, ldb, m;
    int n, na;
    int np;                // rows of R that are wanted: n, or na where [A | B] is a least-squares problem's
    int nb;                // column blocks; sets 0 .. nb-1 are a block against itself, then (0, 1),
                           // (0, 2), (1, 2), (0, 3), ...
    int nslab;             // slabs of rows: slab s holds 64-row blocks [s nkb / nslab, ...)
    int64_t nkb;           // ceil(m / 64)
    int guard;             // bits (an even number) by which a slab's sums are shifted down: gram_guard(m)
    unsigned int *counters;  // per set: the tree's inner nodes; then one for the sets; zeroed
    unsigned char *slots;    // per set: one slot per tree node
    unsigned int *verdict;   // 0: not decided; 1: R is written; 2: the Householder reduction runs
    double *R;
    int64_t ldr;
    struct GramQForm *Q;     // where the root leaves R's inverse (at most kGramMaxN columns), or null
};

// What Q = A R^-1 needs (tsqr_gram_q.cuh): A's columns' exponent words, and the columns of the
// scaled inverse in fixed point, 2^62 units to 2^F.
struct GramQForm {
    int D[kGramMaxN], F[kGramMaxN];
    long long w[kGramMaxN * kGramMaxN];  // (i, j) at 32 j + i
};

// A row adds less than 2^100 to a sum (entries below 2^62 units, products in units of 2^24), so a
// slab of up to 2^26 rows stays within 127 bits.  More rows than that in all: the slabs' sums are
// shifted down before they are added (far below the columns' own rounding: the sum is long).
constexpr int64_t kGramSlabRows = (int64_t)1 << 26;
__host__ __device__ inline int gram_guard(int64_t m) {
    int g = 0;
    while ((m >> g) > kGramSlabRows) g += 2;
    return g;
}

struct GramArgs {          // tsqr_r's single launch: one problem of one column block
    GramProblem p;
    int *status;
    int grid;              // CTAs, at least the Householder leaves over the groups of a CTA
    F64Args fold;          // the Householder reduction (its A is FP64)
};

// Q = A R^-1 (tsqr_gram_q.cuh).  Rows of a tile: up to 16 columns, two or four 128-row blocks of A
// stand side by side in it.
__host__ __device__ inline int gram_q_rows(const int n) { return n <= 8 ? 512 : n <= 16 ? 256 : 128; }
struct GramQArgs {
    const double *A;
    double *Q;
    int64_t lda, ldq, m;
    int n;
    int64_t ntiles;               // tiles of gram_q_rows rows
    const GramQForm *form;
    const unsigned int *verdict;  // 1: the Gram factor is there
    int *status;
};

struct GramQueueArgs {     // a queue of work items
    GramProblem one;       // the problem when probs is null
    const GramProblem *probs;
    const int2 *items;     // (problem, set + nsets slab) in the order they are taken; null: item
                           // k of the one problem is set k % nsets of slab k / nsets, so that a
                           // slab's sets find its rows in L2; from item cut on, the two-block
                           // sets (twice the work) of all slabs left, then the others
    int nitems, cut;
    unsigned int *queue;   // next item, zeroed per call
    unsigned int *failed;  // problems left to the Householder reduction, zeroed per call
    int *status;
};

struct GramWideArgs {      // more columns than one CTA factors
    GramProblem p;
    void *C;               // n x n fixed-point values, row-major (upper part)
    void *P;               // 32 x n: the current block row before its division by the pivots
    void *d;               // n scaled pivots
    int *D, *E, *g, *z;    // per column: exponent word, shift, R's power of two; per row: pivot shift
    unsigned int *bad;     // non-zero: the sum cannot serve (zeroed per call)
};

// Children per node of the Gram sum's tree: a level costs some 8,000 cycles (a fence, a counter, the
// children's exponents, their sums), so up to 24 columns, whose sums are small, one level takes
// all the slabs (10,000 x 16, 40 of them: 20,000 cycles in two levels of 16, 9,000 in one); wider,
// one CTA reading them all takes as long as the second level.
__host__ __device__ inline int gram_arity(int n) { return n <= 24 ? 160 : 16; }
// Inner nodes of the tree over `leaves` leaves.
__host__ __device__ inline int gram_inner_nodes(int leaves, int n) {
    int inner = 0;
    const int arity = gram_arity(n);
    for (int c = leaves; c > 1;) {
        c = (c + arity - 1) / arity;
        inner += c;
    }
    return inner;
}
__host__ __device__ inline int gram_sets(int nb) { return nb * (nb + 1) / 2; }

// Slot of a node: 143 column exponents (block I's from 0, block J's from 64), a word that is
// non-zero where a leaf cannot be served, then the sums (128-bit): (i, j) with i <= j at
// j (j + 1) / 2 + i for a block against itself, i nj + j for two blocks.
constexpr int kGramSlotHead = 576;
__host__ __device__ inline size_t gram_slot_bytes(int block) {  // block: columns of a block
    return (size_t)kGramSlotHead + (size_t)block * block * 16;
}

// Columns of a matrix's blocks: a class of 8 for a matrix of one block, else 32.
__host__ __device__ inline int gram_block(int n) { return n <= 24 ? (n + 7) / 8 * 8 : 32; }

}  // namespace tsqr
