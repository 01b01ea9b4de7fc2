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
// non-finite or extreme entry, a pivot below 2^-kGramPivotBits of its column's square) is found
// by the root, and the same launch then runs the Householder reduction instead.
#pragma once

#include "tsqr_f64.cuh"

namespace tsqr {

constexpr int kGramThreads = 512;
constexpr int kGramWarps = kGramThreads / 32;
constexpr int kGramFoldWarps = 12;  // bulk warps of the Householder reduction (and its reducer)
constexpr int kGramArity = 16;      // children per node of the Gram sum's tree
constexpr int kGramMaxN = 32;

struct GramArgs {
    const void *A;         // m x na, leading dimension lda
    const void *B;         // columns na .. n-1 (a second matrix beside A; null when na == n)
    int64_t lda, ldb, m;
    int n, na;
    int ctas;              // leaves: CTA c sums 64-row blocks [c nkb / ctas, (c+1) nkb / ctas)
    int64_t nkb;           // ceil(m / 64)
    unsigned int *counters;  // one per inner tree node, then the verdict word; zeroed per call
    unsigned int *verdict;   // 0: not decided; 1: R is written; 2: run the Householder reduction
    unsigned char *slots;    // one slot per tree node
    size_t slot_bytes;
    double *R;
    int64_t ldr;
    int *status;
    F64Args fold;          // the Householder reduction (its A is FP64; nleaves <= grid)
};

// Slot of a node: 128 column exponents (the last int: non-zero for a leaf that cannot be
// served), then the n (n + 1) / 2 sums (128-bit, (i, j) with i <= j at j (j + 1) / 2 + i).
constexpr int kGramSlotHead = 576;
inline size_t gram_slot_bytes(int n) {
    return ((size_t)kGramSlotHead + (size_t)n * (n + 1) / 2 * 16 + 255) / 256 * 256;
}

}  // namespace tsqr
