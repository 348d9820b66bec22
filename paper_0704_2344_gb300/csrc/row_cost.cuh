// Cost of a block row in a product from its pattern, and the bounds that the
// kernels size their tables by.  Plain C++, so that the arithmetic can be
// checked on the host at mesh sizes that are too large to run in a test.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define FE_HD __host__ __device__ __forceinline__
#else
#define FE_HD inline
#endif

namespace fe {

// Cost in terms: a row's steps and the fixed work of a component (line lookup,
// five inner products, the store), about eight terms; the steps of a pattern
// of real diagonal blocks skip the term codes.
FE_HD int row_cost(int n_re, int n_im, bool diag) { return diag ? 30 : n_re + n_im + 8; }
constexpr int kMaxRowCost = 170;  // 27 blocks x 3 entries, real and imaginary, and the fixed work

// The prefix sums over the rows are 32-bit.  A grid has up to 2^24 elements
// and four times as many nodes (a one-element wide bar), so rows of 170 could
// pass 2^31; the cost unit then grows to 2^shift terms, the smallest that
// keeps every sum below it.  Meshes of up to 12.5 M rows keep shift 0.
inline int cost_shift(int64_t rows) {
    int shift = 0;
    while (rows * ((kMaxRowCost >> shift) + 1) >= ((int64_t)1 << 31)) ++shift;
    return shift;
}
FE_HD int scaled_cost(int cost, int shift) {
    const int c = cost >> shift;
    return c > 0 ? c : 1;
}

// Most rows that a CTA's range can hold when the rows are split at multiples
// of total / n_cta: the costs of all but its last row add up to less than
// total / n_cta + 1.
inline int64_t cta_rows_bound(int64_t n_rows, int64_t total, int n_cta, int cost_min, int cost_max) {
    const int64_t bound = (total / n_cta + cost_max) / cost_min + 2;
    return bound < n_rows ? bound : n_rows;
}

}  // namespace fe
