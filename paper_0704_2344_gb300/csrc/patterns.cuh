// Row patterns: the block rows of a voxel mesh take few distinct values (the
// 29 666 rows of the 3-wavelength cube take 80: the homogeneous interior, the
// faces, edges and corners of the box, of the slab and of the PEC body), and
// in a distinct row only about a fifth of the 18 real numbers per 3x3 block
// are not zero.  A pattern keeps the non-zero real and imaginary parts of one
// such row as a list of terms, and a row keeps the number of its pattern, so a
// product reads no stored block, no column index, and multiplies no zero.
//
// Terms come in triples, one per component alpha of the row, so that three
// neighbouring lanes (the three components) read three neighbouring terms
// and run the same number of steps: term t of component alpha is entry
// 3 t + alpha of the pattern's list; the real parts come first (n_re steps),
// then the imaginary parts (n_im), the row's own node last in each; a
// component with fewer terms is padded with zero weights.  A term names its column by grid line and offset: line m
// (0..8) is the neighbour line (dy, dz) = (m % 3 - 1, m / 3 - 1), whose centre
// node is active whenever any of its three nodes couples to the row (the
// elements shared with the centre node include those shared with either end),
// and along a line the ranks of coupled nodes are consecutive; so the vector
// entry is 3 rank(centre of m) + delta with delta = 3 dx + beta in -3..5.
//
// A pattern whose 27 blocks are real diagonal ones (the homogeneous interior)
// is stored in full, 27 steps in the order of the grid, and read without the
// term codes; the same 27 follow once more with the row's own node last, for
// kernels that read them by their codes.
#pragma once

#include "krylov.cuh"
#include "row_cost.cuh"

namespace fe {

constexpr int kMaxPat = 2048;      // patterns a system may have; above that the products read the stored blocks
// Patterns a grid of `nodes` nodes may have: their term lists (7.8 KB a
// pattern and arithmetic) stay small beside the blocks, and the server's
// memory estimate can count on it.
inline int pat_limit(int64_t nodes) {
    return (int)(nodes / 8 < 128 ? 128 : (nodes / 8 > kMaxPat ? kMaxPat : nodes / 8));
}
constexpr int kPatStride = 162;    // term triples reserved per pattern: 27 blocks x 3 entries x (real, imaginary)
constexpr int kPatHash = 8192;     // hash table entries of the construction

// weight and packed column of a term: DF float4 (hi, lo, code, -), complex64
// float2 (w, code), complex128 double2 (w, code as the low word)
__device__ __forceinline__ int term_code(const float4& t) { return __float_as_int(t.z); }
__device__ __forceinline__ int term_code(const float2& t) { return __float_as_int(t.y); }
__device__ __forceinline__ int term_code(const double2& t) { return __double2loint(t.y); }
__host__ __device__ __forceinline__ int pack_code(int line, int delta) { return line | ((delta + 3) << 4); }
__device__ __forceinline__ int code_line(int c) { return c & 15; }
__device__ __forceinline__ int code_delta(int c) { return (c >> 4) - 3; }

// One component of a row's product: re += w x.re, im += w x.im (real terms)
// or re -= w x.im, im += w x.re (imaginary terms).
template <typename C>
struct TermAcc {
    using T = decltype(C{}.x);
    T re = 0, im = 0;
    __device__ __forceinline__ void add_re(const C& t, const C& x) {
        re += t.x * x.x;
        im += t.x * x.y;
    }
    __device__ __forceinline__ void add_im(const C& t, const C& x) {
        re -= t.x * x.y;
        im += t.x * x.x;
    }
    __device__ __forceinline__ void add(const TermAcc& o) {
        re += o.re;
        im += o.im;
    }
    __device__ __forceinline__ C result_norm() { return mk(re, im); }
};
template <>
struct TermAcc<float4> {
    float a[4] = {0.f, 0.f, 0.f, 0.f};
    __device__ __forceinline__ void add_re(const float4& t, const float4& x) {
        df_mac(a[0], a[1], t.x, t.y, x.x, x.z);
        df_mac(a[2], a[3], t.x, t.y, x.y, x.w);
    }
    __device__ __forceinline__ void add_im(const float4& t, const float4& x) {
        df_mac(a[0], a[1], -t.x, -t.y, x.y, x.w);
        df_mac(a[2], a[3], t.x, t.y, x.x, x.z);
    }
    __device__ __forceinline__ void add(const TermAcc& o) {
        df_add(a[0], a[1], o.a[0], o.a[1]);
        df_add(a[2], a[3], o.a[2], o.a[3]);
    }
    __device__ __forceinline__ float4 result_norm() { return df_result_norm(a); }
};

// Adds the accumulators of the lanes that differ in bit `o` of their number.
template <typename C>
__device__ __forceinline__ void acc_butterfly(TermAcc<C>& acc, int o) {
    if constexpr (std::is_same<C, float4>::value) {
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
            const float h2 = __shfl_xor_sync(0xffffffffu, acc.a[q], o), l2 = __shfl_xor_sync(0xffffffffu, acc.a[q + 1], o);
            df_add(acc.a[q], acc.a[q + 1], h2, l2);
        }
    } else {
        acc.re += __shfl_xor_sync(0xffffffffu, acc.re, o);
        acc.im += __shfl_xor_sync(0xffffffffu, acc.im, o);
    }
}

// Component of a row times column c of a vector [n_dof][R].  terms: the
// pattern's list at the component (terms[3 t] is its step t); base(m):
// 3 x rank of the centre of line m; load(i): vector entry i.
template <typename C, typename Base, typename Load>
__device__ __forceinline__ void pattern_terms(TermAcc<C>& acc, const C* terms, int n_re, int n_im, int R, int c,
                                              Base&& base, Load&& load) {
    auto entry = [&](int code) { return load((size_t)(base(code_line(code)) + code_delta(code)) * R + c); };
    if constexpr (std::is_same<C, float4>::value) {
        // FP32 pairs: two accumulators, every other term each, so that a warp
        // does not wait for one chain of additions (2 to 4 % of an iteration;
        // FP64 and complex64, with one operation per term and part, lose by it)
        TermAcc<C> other;
        int t = 0;
        for (; t + 4 <= n_re; t += 4) {
            C q[4], x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                q[k] = terms[3 * (t + k)];
                x[k] = entry(term_code(q[k]));
            }
            acc.add_re(q[0], x[0]);
            other.add_re(q[1], x[1]);
            acc.add_re(q[2], x[2]);
            other.add_re(q[3], x[3]);
        }
        for (; t < n_re; ++t) {
            const C q = terms[3 * t];
            acc.add_re(q, entry(term_code(q)));
        }
        for (; t < n_re + n_im; ++t) {
            const C q = terms[3 * t];
            other.add_im(q, entry(term_code(q)));
        }
        acc.add(other);
    } else {
#pragma unroll 3
        for (int t = 0; t < n_re; ++t) {
            const C q = terms[3 * t];
            acc.add_re(q, entry(term_code(q)));
        }
        terms += 3 * n_re;
        for (int t = 0; t < n_im; ++t) {
            const C q = terms[3 * t];
            acc.add_im(q, entry(term_code(q)));
        }
    }
}

// The same for a pattern of real diagonal blocks: the three entries of a line
// lie 3 apart, the weights follow in grid order.  kOwnLast takes the row's own
// entry, whose weight is the largest, last: the partial sums of a rough vector
// stay small until then, which rounds to half to a third of the error of the
// grid order (27 interior weights on random entries: FP32 pairs 2.7e-15
// against 8.1e-15, FP32 3.1e-8 against 9.5e-8 of the result).  On smooth
// vectors, where the entry cancels the others' sum, the grid order is the
// better one (2.1e-12 against 2.3e-12), and the Krylov loop uses it.
template <typename C, bool kOwnLast, typename Base, typename Load>
__device__ __forceinline__ void pattern_diag(TermAcc<C>& acc, const C* terms, int al, int R, int c, Base&& base,
                                             Load&& load) {
    auto line = [&](int m, bool own) {
        const size_t i = (size_t)(base(m) + al) * R + c;
        const C x0 = load(i - 3 * R), x1 = load(i), x2 = load(i + 3 * R);
        acc.add_re(terms[9 * m], x0);
        if (!own) acc.add_re(terms[9 * m + 3], x1);
        acc.add_re(terms[9 * m + 6], x2);
        if (own) acc.add_re(terms[9 * m + 3], x1);
    };
    if constexpr (kOwnLast) {
#pragma unroll 2
        for (int k = 0; k < 8; ++k) line(k + (k >= 4), false);
        line(4, true);
    } else if constexpr (!std::is_same<C, float4>::value) {
#pragma unroll 3
        for (int m = 0; m < 9; ++m) line(m, false);
    } else {
        // the lines below the row's plane in one accumulator, those above in
        // another, the row's own plane split between them
        TermAcc<C> other;
        auto both = [&](int m, int k) {
            const size_t i = (size_t)(base(m) + al) * R + c, j = (size_t)(base(k) + al) * R + c;
            const C x0 = load(i - 3 * R), x1 = load(i), x2 = load(i + 3 * R);
            const C z0 = load(j - 3 * R), z1 = load(j), z2 = load(j + 3 * R);
            acc.add_re(terms[9 * m], x0);
            other.add_re(terms[9 * k], z0);
            acc.add_re(terms[9 * m + 3], x1);
            other.add_re(terms[9 * k + 3], z1);
            acc.add_re(terms[9 * m + 6], x2);
            other.add_re(terms[9 * k + 6], z2);
        };
#pragma unroll 2
        for (int m = 0; m < 4; ++m) both(m, 8 - m);
        line(4, false);
        acc.add(other);
    }
}

// Row patterns of a system as the kernels read them (C: one arithmetic).
template <typename C>
struct PatView {
    const uint16_t* id;    // [n_rows] pattern of each row
    const int4* row;       // [n_rows] (first term, n_re | n_im << 10 | real diagonal blocks << 20, grid node, pattern)
    const int4* tab;       // [n_pat] (first term triple, n_re, n_im, 1: real diagonal blocks)
    const C* terms;
    const int* node_id;    // [n_rows] grid node of each row
    const int* node_rank;  // [nodes] row of each grid node
    int sy, sz;            // nodes per grid line and plane
};

// Lines of a row, resolved through the node ranks.
struct LineRanks {
    const int* rank;  // node_rank + node
    int sy, sz;
    __device__ __forceinline__ int operator()(int m) const {
        return 3 * __ldg(rank + (m % 3 - 1) * sy + (m / 3 - 1) * sz);
    }
};

}  // namespace fe
