// Standalone sparse products y = A x (fe_spmv): the Krylov loop's product
// (Section 3.1.5.1) as its own entry point, for one or several vectors.
#include "patterns.cuh"

#include <algorithm>
#include <cstdint>
#include <type_traits>

namespace fe {

template <typename C>
__global__ void __launch_bounds__(256) k_spmv_cols(const C* __restrict__ val, int64_t stride,
                                                   const int* __restrict__ col, const int* __restrict__ rp,
                                                   const C* __restrict__ x, C* __restrict__ y, int n_rows, int nrhs) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n_rows * nrhs) return;
    const int row = (int)(t / nrhs), c = (int)(t - (int64_t)row * nrhs);
    C v[3];
    row_product_colx<C, false>(val, stride, col, __ldg(rp + row), __ldg(rp + row + 1), x, 0, nrhs, c, v[0], v[1],
                               v[2]);
#pragma unroll
    for (int al = 0; al < 3; ++al) y[(size_t)(3 * row + al) * nrhs + c] = v[al];
}

// y = A x for R = 1, 2, 4, ..., 32 columns: one warp per block row, its lanes
// split into 32/R block groups x R columns.  A block's nine entries are read
// once per warp (the R lanes of a group read the same address), the R values
// of one vector entry are contiguous, and the groups' partial sums meet in a
// shuffle reduction (FP32 pairs: error-free pair additions).
template <typename C, int R>
__global__ void __launch_bounds__(256) k_spmv_warp(const C* __restrict__ val, int64_t stride,
                                                   const int* __restrict__ col, const int* __restrict__ rp,
                                                   const C* __restrict__ x, C* __restrict__ y, int n_rows) {
    const int lane = threadIdx.x & 31;
    constexpr int G = 32 / R;
    const int c = lane % R, g = lane / R;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < n_rows; row += nw) {
        const int s0 = __ldg(rp + row), s1 = __ldg(rp + row + 1);
        // the nine entries of a block load before its (dependent) vector entries;
        // the next column index loads one step ahead
        int cb = s0 + g < s1 ? __ldg(col + s0 + g) : 0;
        if constexpr (std::is_same<C, float4>::value) {
            float a[3][4] = {};
            for (int s = s0 + g; s < s1; s += G) {
                const int cb_next = s + G < s1 ? __ldg(col + s + G) : 0;
                float4 m[9];
#pragma unroll
                for (int q = 0; q < 9; ++q) m[q] = __ldg(val + q * stride + s);
                const int xb = 3 * cb * R + c;
                float4 xv[3];
#pragma unroll
                for (int be = 0; be < 3; ++be) xv[be] = __ldg(x + xb + be * R);
#pragma unroll
                for (int al = 0; al < 3; ++al)
#pragma unroll
                    for (int be = 0; be < 3; ++be) dfc_mac(a[al], m[3 * al + be], xv[be]);
                cb = cb_next;
            }
#pragma unroll
            for (int o = 16; o >= R; o >>= 1)
#pragma unroll
                for (int al = 0; al < 3; ++al)
#pragma unroll
                    for (int q = 0; q < 4; q += 2) {
                        const float h2 = __shfl_xor_sync(0xffffffffu, a[al][q], o);
                        const float l2 = __shfl_xor_sync(0xffffffffu, a[al][q + 1], o);
                        df_add(a[al][q], a[al][q + 1], h2, l2);
                    }
            if (g == 0)
#pragma unroll
                for (int al = 0; al < 3; ++al) y[(size_t)(3 * row + al) * R + c] = df_result_norm(a[al]);
        } else {
            using Tr = decltype(C{}.x);
            Tr a[6] = {0, 0, 0, 0, 0, 0};
            for (int s = s0 + g; s < s1; s += G) {
                const int cb_next = s + G < s1 ? __ldg(col + s + G) : 0;
                C m[9];
#pragma unroll
                for (int q = 0; q < 9; ++q) m[q] = __ldg(val + q * stride + s);
                const int xb = 3 * cb * R + c;
                C xv[3];
#pragma unroll
                for (int be = 0; be < 3; ++be) xv[be] = __ldg(x + xb + be * R);
#pragma unroll
                for (int al = 0; al < 3; ++al)
#pragma unroll
                    for (int be = 0; be < 3; ++be) {
                        a[2 * al] += m[3 * al + be].x * xv[be].x - m[3 * al + be].y * xv[be].y;
                        a[2 * al + 1] += m[3 * al + be].x * xv[be].y + m[3 * al + be].y * xv[be].x;
                    }
                cb = cb_next;
            }
#pragma unroll
            for (int o = 16; o >= R; o >>= 1)
#pragma unroll
                for (int k = 0; k < 6; ++k) a[k] += __shfl_xor_sync(0xffffffffu, a[k], o);
            if (g == 0)
#pragma unroll
                for (int al = 0; al < 3; ++al) y[(size_t)(3 * row + al) * R + c] = mk(a[2 * al], a[2 * al + 1]);
        }
    }
}

// y = A x for R = 8, 16 or 32 columns: a warp takes G = 32/R consecutive
// block rows, one group of R lanes (one lane per column) per row.  The warp
// first copies the nine entries and the column index of every block of its
// G rows into shared memory with coalesced loads (lane l takes block l, l +
// 32, ...: the blocks of consecutive rows are consecutive in each plane), so
// that the whole group of rows is in flight at once; then each group walks
// its row from shared memory (the R lanes read the same entry) and multiplies
// by the R contiguous vector values of each block's column.  No reduction
// across lanes is needed.
constexpr int kSpmmWarps = 4;

template <typename C, int R>
__global__ void __launch_bounds__(32 * kSpmmWarps) k_spmm_rows(const C* __restrict__ val, int64_t stride,
                                                               const int* __restrict__ col,
                                                               const int* __restrict__ rp, const C* __restrict__ x,
                                                               C* __restrict__ y, int n_rows) {
    constexpr int G = 32 / R;
    constexpr int kMax = 27 * G;
    __shared__ C s_val[kSpmmWarps][9][kMax];
    __shared__ int s_col[kSpmmWarps][kMax];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = lane % R, g = lane / R;
    const int n_groups = (n_rows + G - 1) / G;
    const int nw = gridDim.x * kSpmmWarps;
    C(*sv)[kMax] = s_val[warp];
    int* sc = s_col[warp];
    for (int grp = blockIdx.x * kSpmmWarps + warp; grp < n_groups; grp += nw) {
        const int r0 = grp * G, r1 = min(r0 + G, n_rows);
        const int b0 = __ldg(rp + r0), nb = __ldg(rp + r1) - b0;
        if (nb > kMax) {  // not a voxel pattern (at most 27 blocks per row): read the blocks directly
            const int row = r0 + g;
            if (row < r1) {
                C v[3];
                row_product_colx<C, false>(val, stride, col, __ldg(rp + row), __ldg(rp + row + 1), x, 0, R, c, v[0],
                                           v[1], v[2]);
#pragma unroll
                for (int al = 0; al < 3; ++al) y[(size_t)(3 * row + al) * R + c] = v[al];
            }
            continue;
        }
        for (int k = lane; k < nb; k += 32) {
            sc[k] = __ldg(col + b0 + k);
#pragma unroll
            for (int q = 0; q < 9; ++q) sv[q][k] = __ldg(val + q * stride + b0 + k);
        }
        __syncwarp();
        const int row = r0 + g;
        if (row < r1) {
            const int k0 = __ldg(rp + row) - b0, k1 = __ldg(rp + row + 1) - b0;
            if constexpr (std::is_same<C, float4>::value) {
                float a[3][4] = {};
                for (int k = k0; k < k1; ++k) {
                    const int xb = 3 * sc[k] * R + c;
                    const float4 x0 = __ldg(x + xb), x1 = __ldg(x + xb + R), x2 = __ldg(x + xb + 2 * R);
#pragma unroll
                    for (int al = 0; al < 3; ++al) {
                        dfc_mac(a[al], sv[3 * al][k], x0);
                        dfc_mac(a[al], sv[3 * al + 1][k], x1);
                        dfc_mac(a[al], sv[3 * al + 2][k], x2);
                    }
                }
#pragma unroll
                for (int al = 0; al < 3; ++al) y[(size_t)(3 * row + al) * R + c] = df_result_norm(a[al]);
            } else {
                using Tr = decltype(C{}.x);
                Tr a[6] = {0, 0, 0, 0, 0, 0};
                for (int k = k0; k < k1; ++k) {
                    const int xb = 3 * sc[k] * R + c;
                    const C xv[3] = {__ldg(x + xb), __ldg(x + xb + R), __ldg(x + xb + 2 * R)};
#pragma unroll
                    for (int al = 0; al < 3; ++al)
#pragma unroll
                        for (int be = 0; be < 3; ++be) {
                            const C m = sv[3 * al + be][k];
                            a[2 * al] += m.x * xv[be].x - m.y * xv[be].y;
                            a[2 * al + 1] += m.x * xv[be].y + m.y * xv[be].x;
                        }
                }
#pragma unroll
                for (int al = 0; al < 3; ++al) y[(size_t)(3 * row + al) * R + c] = mk(a[2 * al], a[2 * al + 1]);
            }
        }
        __syncwarp();
    }
}

// y = A x for R = 8, 16 or 32 complex64 columns, with several columns per
// lane: CPL adjacent columns per lane, L = R / CPL lanes per row and G = 32 /
// L rows per warp.  As in k_spmm_rows the warp first stages its rows' blocks
// (nine planes and the column indices) in shared memory with coalesced
// loads; each entry read from shared memory then serves CPL columns, and a
// lane reads its CPL vector values of a block row with 16-byte loads.  PF
// loads the next block's vector values one step ahead.
template <int CPL>
struct SpmmX;
template <>
struct SpmmX<2> {
    float4 v[1];
};
template <>
struct SpmmX<4> {
    float4 v[2];
};

template <int R, int CPL>
__device__ __forceinline__ void spmm_load_x(const float2* __restrict__ x, int cb, int c0, SpmmX<CPL> (&d)[3]) {
#pragma unroll
    for (int be = 0; be < 3; ++be) {
        const float4* p = (const float4*)(x + (size_t)(3 * cb + be) * R + c0);
#pragma unroll
        for (int v = 0; v < CPL / 2; ++v) d[be].v[v] = __ldg(p + v);
    }
}

template <int R, int CPL, int W, bool PF>
__global__ void __launch_bounds__(32 * W) k_spmm_cpl(const float2* __restrict__ val, int64_t stride,
                                                     const int* __restrict__ col, const int* __restrict__ rp,
                                                     const float2* __restrict__ x, float2* __restrict__ y,
                                                     int n_rows) {
    constexpr int L = R / CPL, G = 32 / L, kMax = 27 * G;
    __shared__ float2 s_val[W][9][kMax];
    __shared__ int s_col[W][kMax];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = (lane % L) * CPL, g = lane / L;
    const int n_groups = (n_rows + G - 1) / G;
    float2(*sv)[kMax] = s_val[warp];
    int* sc = s_col[warp];
    for (int grp = blockIdx.x * W + warp; grp < n_groups; grp += gridDim.x * W) {
        const int r0 = grp * G, r1 = min(r0 + G, n_rows);
        const int b0 = __ldg(rp + r0), nb = __ldg(rp + r1) - b0;
        const int row = r0 + g;
        float a[3][CPL][2] = {};
        if (nb > kMax) {  // not a voxel pattern (at most 27 blocks per row): read the blocks directly
            if (row < r1)
#pragma unroll
                for (int j = 0; j < CPL; ++j) {
                    float2 v[3];
                    row_product_colx<float2, false>(val, stride, col, __ldg(rp + row), __ldg(rp + row + 1), x, 0, R,
                                                    c0 + j, v[0], v[1], v[2]);
#pragma unroll
                    for (int al = 0; al < 3; ++al) {
                        a[al][j][0] = v[al].x;
                        a[al][j][1] = v[al].y;
                    }
                }
        } else {
            for (int k = lane; k < nb; k += 32) {
                sc[k] = __ldg(col + b0 + k);
#pragma unroll
                for (int q = 0; q < 9; ++q) sv[q][k] = __ldg(val + q * stride + b0 + k);
            }
            __syncwarp();
            if (row < r1) {
                const int k0 = __ldg(rp + row) - b0, k1 = __ldg(rp + row + 1) - b0;
                SpmmX<CPL> xn[3];
                if (PF && k0 < k1) spmm_load_x<R, CPL>(x, sc[k0], c0, xn);
                for (int k = k0; k < k1; ++k) {
                    SpmmX<CPL> xv[3];
                    if (PF) {
#pragma unroll
                        for (int be = 0; be < 3; ++be) xv[be] = xn[be];
                        if (k + 1 < k1) spmm_load_x<R, CPL>(x, sc[k + 1], c0, xn);
                    } else {
                        spmm_load_x<R, CPL>(x, sc[k], c0, xv);
                    }
#pragma unroll
                    for (int al = 0; al < 3; ++al)
#pragma unroll
                        for (int be = 0; be < 3; ++be) {
                            const float2 m = sv[3 * al + be][k];
#pragma unroll
                            for (int v = 0; v < CPL / 2; ++v) {
                                const float4 q = xv[be].v[v];
                                a[al][2 * v][0] += m.x * q.x - m.y * q.y;
                                a[al][2 * v][1] += m.x * q.y + m.y * q.x;
                                a[al][2 * v + 1][0] += m.x * q.z - m.y * q.w;
                                a[al][2 * v + 1][1] += m.x * q.w + m.y * q.z;
                            }
                        }
                }
            }
            __syncwarp();
        }
        if (row < r1)
#pragma unroll
            for (int al = 0; al < 3; ++al) {
                float4* p = (float4*)(y + (size_t)(3 * row + al) * R + c0);
#pragma unroll
                for (int v = 0; v < CPL / 2; ++v)
                    p[v] = make_float4(a[al][2 * v][0], a[al][2 * v][1], a[al][2 * v + 1][0], a[al][2 * v + 1][1]);
            }
    }
}

// Columns per lane, warps per CTA and prefetch for each width, chosen by
// timing every combination on a 27-point pattern of 81^3 nodes (14.0 M
// blocks) on GB300: R = 8 2 / 2 / on, R = 16 4 / 2 / off, R = 32 2 / 8 / off.
template <int R, int CPL, int W, bool PF>
static void launch_spmm_cpl_t(cudaStream_t st, int sms, const float2* val, int64_t stride, const int* col,
                              const int* rp, const float2* x, float2* y, int n_rows) {
    constexpr int G = 32 / (R / CPL);
    int per_sm = 0;  // resident CTAs per SM (a host query, no device work)
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spmm_cpl<R, CPL, W, PF>, 32 * W, 0) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    const int64_t groups = ((int64_t)n_rows + G - 1) / G;
    const unsigned blocks =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * per_sm, (groups + W - 1) / W));
    k_spmm_cpl<R, CPL, W, PF><<<blocks, 32 * W, 0, st>>>(val, stride, col, rp, x, y, n_rows);
}

static void launch_spmm_cpl(int R, cudaStream_t st, int sms, const float2* val, int64_t stride, const int* col,
                            const int* rp, const float2* x, float2* y, int n_rows) {
    switch (R) {
        case 8: launch_spmm_cpl_t<8, 2, 2, true>(st, sms, val, stride, col, rp, x, y, n_rows); break;
        case 16: launch_spmm_cpl_t<16, 4, 2, false>(st, sms, val, stride, col, rp, x, y, n_rows); break;
        default: launch_spmm_cpl_t<32, 2, 8, false>(st, sms, val, stride, col, rp, x, y, n_rows); break;
    }
}

template <typename C>
static void launch_spmm_rows(int R, cudaStream_t st, int sms, const C* val, int64_t stride, const int* col,
                             const int* rp, const C* x, C* y, int n_rows) {
    const int G = 32 / R;
    const int64_t groups = ((int64_t)n_rows + G - 1) / G;
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * 16,
                                                                            (groups + kSpmmWarps - 1) / kSpmmWarps));
    switch (R) {
        case 8: k_spmm_rows<C, 8><<<blocks, 32 * kSpmmWarps, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
        case 16: k_spmm_rows<C, 16><<<blocks, 32 * kSpmmWarps, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
        default: k_spmm_rows<C, 32><<<blocks, 32 * kSpmmWarps, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
    }
}

template <typename C>
static void launch_spmv_warp(int R, unsigned blocks, cudaStream_t st, const C* val, int64_t stride, const int* col,
                             const int* rp, const C* x, C* y, int n_rows) {
    switch (R) {
        case 1: k_spmv_warp<C, 1><<<blocks, 256, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
        case 2: k_spmv_warp<C, 2><<<blocks, 256, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
        case 4: k_spmv_warp<C, 4><<<blocks, 256, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
        case 8: k_spmv_warp<C, 8><<<blocks, 256, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
        case 16: k_spmv_warp<C, 16><<<blocks, 256, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
        default: k_spmv_warp<C, 32><<<blocks, 256, 0, st>>>(val, stride, col, rp, x, y, n_rows); break;
    }
}

// ---------------------------------------------------------------------------
// y = A x from the row patterns.  The matrix is a few hundred kilobytes of
// terms that stay in L1 and L2, so a product moves the vectors and the row
// tables only: the 80^3 aircraft's complex64 product reads 25 MB of vectors
// and tables instead of 1.1 GB of blocks.  Work items are (row, component,
// column), consecutive lanes taking consecutive vector entries.  Four forms:
//
//   split   few items: 2 to 8 lanes share one, so that the chip's lanes are used
//           and a lane's chain of dependent loads is short;
//   plain   one lane per item; the first blocks take the explicit rows
//           (collected in a list, so that a warp holds rows of like length),
//           the others sweep all rows for the real diagonal ones.  FP64 and
//           FP32 pairs, which are bound by their arithmetic;
//   keep    complex64, 1, 2 or 4 columns: one CTA per SM walks a range of
//           rows, every thread staying on one component and column, with the
//           27 weights of its pattern in registers;
//   tile    complex64, 8, 16 or 32 columns: the same walk with four
//           consecutive rows per thread, which share two of every three
//           entries along a grid line.  Walking a range keeps a row's lines in
//           L1 for the rows above and beside it.
//
// product_form says which sizes take which form, or the stored blocks.
// Measured per product, from the stored blocks and here (in brackets: all by
// the plain form): FP32 pairs, 9 261 rows 10.1 and 4.1 us (9.1); complex64,
// 80^3 aircraft 196 and 28.9 us (32.4), 60^3 aircraft with 16 columns 306 and
// 128 us (149); complex128, 48^3 nodes with 3 columns 840 and 106 us, 0.8 of
// the FP64 pipe's rate on the non-zero terms.
// ---------------------------------------------------------------------------
template <typename C>
__device__ __forceinline__ void pat_item(const PatView<C>& V, const C* __restrict__ x, C* __restrict__ y, int row,
                                         int al, int R, int c, bool want_diag) {
    const int4 t = __ldg(V.row + row);
    if (((t.y >> 20) & 1) != (int)want_diag) return;
    const LineRanks base{V.node_rank + t.z, V.sy, V.sz};
    const C* terms = V.terms + t.x + al;
    auto load = [&](size_t i) { return __ldg(x + i); };
    TermAcc<C> acc;
    if (want_diag) pattern_diag<C, true>(acc, terms, al, R, c, base, load);
    else pattern_terms<C>(acc, terms, t.y & 0x3ff, (t.y >> 10) & 0x3ff, R, c, base, load);
    y[((size_t)3 * row + al) * R + c] = acc.result_norm();
}

template <typename C, int R_>
__global__ void __launch_bounds__(256) k_spmv_pat(PatView<C> V, int n_rows, const int* __restrict__ list, int n_expl,
                                                  int expl_blocks, int nrhs, const C* __restrict__ x,
                                                  C* __restrict__ y) {
    const int R = R_ ? R_ : nrhs;
    const bool expl = (int)blockIdx.x < expl_blocks;
    const int64_t e = (int64_t)(expl ? blockIdx.x : blockIdx.x - expl_blocks) * blockDim.x + threadIdx.x;
    const int64_t d = e / R;
    const int c = (int)(e - d * R), i = (int)(d / 3), al = (int)(d - 3 * (int64_t)i);
    if (i >= (expl ? n_expl : n_rows)) return;
    if (expl) pat_item<C>(V, x, y, __ldg(list + i), al, R, c, false);
    else pat_item<C>(V, x, y, i, al, R, c, true);
}

// split: K lanes per item, K R columns (a power of two up to 32) per warp part.
// The row's own entry, the last step of its lane, goes last of all: that lane
// adds it to the sum of all lanes and stores the result.  In grid order the
// error of random vectors was up to 1.4 times that of the stored blocks (31^3
// elements, one column, FP32 pairs 5.6e-15, 4.0e-15 now, 4.2e-15 by blocks);
// 9 261 rows take 4.75 us so and 4.1 now; with two lanes an item the step aside
// costs 5 to 7 % (FP32 pairs, two columns of 24^3 elements on three streams 7.3
// and 7.7 us).
template <typename C, int R, int K>
__global__ void __launch_bounds__(256) k_spmv_pat_split(PatView<C> V, int n_rows, const C* __restrict__ x,
                                                        C* __restrict__ y) {
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = (int)(t0 % R), part = (int)(t0 / R) % K;
    const int64_t d = t0 / (R * K);
    const int row = (int)(d / 3), al = (int)(d - 3 * (int64_t)row);
    const bool on = row < n_rows;
    TermAcc<C> acc;
    C own_w{}, own_x{};
    bool last = false;
    if (on) {
        const int4 t = __ldg(V.row + row);
        const LineRanks base{V.node_rank + t.z, V.sy, V.sz};
        const bool diag = (t.y >> 20) & 1;
        const C* terms = V.terms + t.x + al + (diag ? 81 : 0);  // the copy with the own entry last
        const int n_re = t.y & 0x3ff, n_im = (t.y >> 10) & 0x3ff;
        for (int k = n_re + part; k < n_re + n_im; k += K) {
            const C q = terms[3 * k];
            const int code = term_code(q);
            acc.add_im(q, __ldg(x + (size_t)(base(code_line(code)) + code_delta(code)) * R + c));
        }
        int k = part;
#pragma unroll 4
        for (; k + K < n_re; k += K) {
            const C q = terms[3 * k];
            const int code = term_code(q);
            acc.add_re(q, __ldg(x + (size_t)(base(code_line(code)) + code_delta(code)) * R + c));
        }
        last = n_re > 0 ? k == n_re - 1 : part == 0;
        if (k < n_re) {
            own_w = terms[3 * k];
            const int code = term_code(own_w);
            own_x = __ldg(x + (size_t)(base(code_line(code)) + code_delta(code)) * R + c);
            if (!last) acc.add_re(own_w, own_x);
        }
    }
#pragma unroll
    for (int o = R; o < R * K; o <<= 1) acc_butterfly(acc, o);
    if (last) {
        acc.add_re(own_w, own_x);
        y[((size_t)3 * row + al) * R + c] = acc.result_norm();
    }
}

// keep: a thread's component and column do not change along its walk, since
// the block's threads are a multiple of 3 R.
constexpr int kKeepThreads = 768;
template <int R>
__global__ void __launch_bounds__(kKeepThreads, 1) k_spmv_pat_keep(PatView<float2> V, int n_rows,
                                                                  const int* __restrict__ list, int n_expl,
                                                                  const float2* __restrict__ x,
                                                                  float2* __restrict__ y) {
    static_assert(kKeepThreads % (3 * R) == 0, "a thread keeps its component and column");
    const int c = threadIdx.x % R, al = (threadIdx.x / R) % 3, step = kKeepThreads / (3 * R);
    // explicit rows of this block, one walk beside the other
    const int e0 = (int)((int64_t)blockIdx.x * n_expl / gridDim.x), e1 = (int)((int64_t)(blockIdx.x + 1) * n_expl / gridDim.x);
    for (int i = e0 + (int)threadIdx.x / (3 * R); i < e1; i += step)
        pat_item<float2>(V, x, y, __ldg(list + i), al, R, c, false);
    const int r0 = (int)((int64_t)blockIdx.x * n_rows / gridDim.x), r1 = (int)((int64_t)(blockIdx.x + 1) * n_rows / gridDim.x);
    float w[27];
    int held = -1;
    for (int row = r0 + (int)threadIdx.x / (3 * R); row < r1; row += step) {
        const int id = __ldg(V.id + row);
        const int4 t = __ldg(V.tab + id);
        if (!t.w) continue;
        if (id != held) {
#pragma unroll
            for (int k = 0; k < 27; ++k) w[k] = __ldg(&V.terms[(size_t)t.x * 3 + al + 3 * k].x);
            held = id;
        }
        const LineRanks base{V.node_rank + __ldg(V.node_id + row), V.sy, V.sz};
        float re = 0.f, im = 0.f, cr = 0.f, ci = 0.f;
#pragma unroll
        for (int m = 0; m < 9; ++m) {
            const float2* xp = x + (size_t)(base(m) + al) * R + c;
            const float2 x0 = __ldg(xp - 3 * R), x1 = __ldg(xp), x2 = __ldg(xp + 3 * R);
            re += w[3 * m] * x0.x;
            im += w[3 * m] * x0.y;
            if (m == 4) {  // the row's own entry last
                cr = w[13] * x1.x;
                ci = w[13] * x1.y;
            } else {
                re += w[3 * m + 1] * x1.x;
                im += w[3 * m + 1] * x1.y;
            }
            re += w[3 * m + 2] * x2.x;
            im += w[3 * m + 2] * x2.y;
        }
        y[((size_t)3 * row + al) * R + c] = make_float2(re + cr, im + ci);
    }
}

// tile: (four rows, component, column) per thread.
constexpr int kTileThreads = 1024;
template <int R>
__global__ void __launch_bounds__(kTileThreads, 1) k_spmv_pat_tile(PatView<float2> V, int n_rows,
                                                                  const int* __restrict__ list, int n_expl,
                                                                  const float2* __restrict__ x,
                                                                  float2* __restrict__ y) {
    const int e0 = (int)((int64_t)blockIdx.x * n_expl / gridDim.x), e1 = (int)((int64_t)(blockIdx.x + 1) * n_expl / gridDim.x);
    for (int q = threadIdx.x; q < (e1 - e0) * 3 * R; q += kTileThreads) {
        const int c = q % R, d = q / R;
        pat_item<float2>(V, x, y, __ldg(list + e0 + d / 3), d % 3, R, c, false);
    }
    const int n4 = (n_rows + 3) / 4;
    const int q0 = (int)((int64_t)blockIdx.x * n4 / gridDim.x), q1 = (int)((int64_t)(blockIdx.x + 1) * n4 / gridDim.x);
    for (int q = threadIdx.x; q < (q1 - q0) * 3 * R; q += kTileThreads) {
        const int c = q % R, d = q / R, al = d % 3, r0 = 4 * (q0 + d / 3);
        const int id0 = __ldg(V.id + r0);
        bool tile = r0 + 3 < n_rows;
        if (tile)
            tile = __ldg(V.id + r0 + 1) == id0 && __ldg(V.id + r0 + 2) == id0 && __ldg(V.id + r0 + 3) == id0 &&
                   __ldg(V.node_id + r0 + 3) - __ldg(V.node_id + r0) == 3;
        if (!tile) {
            for (int row = r0; row < min(r0 + 4, n_rows); ++row) pat_item<float2>(V, x, y, row, al, R, c, true);
            continue;
        }
        const int4 t = __ldg(V.tab + id0);
        if (!t.w) continue;
        const float2* terms = V.terms + (size_t)t.x * 3 + al;
        const LineRanks base{V.node_rank + __ldg(V.node_id + r0), V.sy, V.sz};
        TermAcc<float2> acc[4];
        float2 own[4];
        auto line = [&](int m, bool centre) {
            const float2* xp = x + ((size_t)(base(m) + al) * R + c) - 3 * R;
            float2 v[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) v[k] = __ldg(xp + 3 * k * R);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                if (centre && k == 1) continue;
                const float2 w = __ldg(terms + 9 * m + 3 * k);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[j].add_re(w, v[j + k]);
            }
            if (centre)
#pragma unroll
                for (int j = 0; j < 4; ++j) own[j] = v[j + 1];
        };
#pragma unroll 2
        for (int k = 0; k < 8; ++k) line(k + (k >= 4), false);
        line(4, true);  // the rows' own entries last
        const float2 w = __ldg(terms + 39);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j].add_re(w, own[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) y[((size_t)3 * (r0 + j) + al) * R + c] = acc[j].result_norm();
    }
}

// Form of a product of `rows` rows and R columns on `lanes` resident lanes
// (2 048 per SM, 311 296), by its items n = 3 rows R.  Lanes share an item while
// that does not take more than the chip's: 8 up to n = lanes / 8, 4 up to
// lanes / 4, 2 up to 0.48 lanes (FP32 pairs of 50 528 rows, just beyond: 11.5 us
// shared and 8.6 plain on three streams; 42 811 rows alone 17 and 19).  FP64 and
// FP32 pairs are plain above; complex64 is plain until the walks pay: from n = lanes with up to 4 columns, from 3.5
// lanes with 8 and 32, from 5 lanes with 16.  A walk takes every SM whole, so that
// products on several streams do not overlap; both ways count.  Times in us
// per product, of systems on three streams in turn / of one alone, on either
// side of a bound (cubes with a slab and a PEC body):
//   1 column    90 909 rows  plain 8.2 / 19, walk 10.6 / 19; 117 306  8.1 / 19, 11.3 / 16
//   2 columns   50 528 rows  plain 8.3 / 21, walk 10.7 / 14; 68 796   9.3 / 21, 11.9 / 16
//   4 columns   24 362 rows  plain 8.2 / 19, walk 10.6 / 14; 35 873  10.2 / 21, 12.0 / 16
//   8 columns   42 811 rows  plain 22.9 / 29, walk 24.4 / 31; 68 796  36.1 / 40, 33.7 / 44
//   16 columns  29 727 rows  plain 31.6 / 37, walk 30.6 / 39; 35 873  39.2 / 43, 35.4 / 43
//   32 columns  10 640 rows  plain 24.2 / 29, walk 24.5 / 37; 15 598  36.2 / 41, 32.5 / 41
// The stored blocks of a small system stay in L2, and a warp reads a row's
// blocks at once, so that their chain of dependent loads is one shorter than a
// pattern's (row, line, term, entry).  They round more (complex64 of 8 columns
// and more 1.0e-7 against 4.6e-8), so they are taken only where the patterns
// are clearly slower, all systems alone:
//   complex64  1 column n <= lanes / 9: 10 640 rows 6.5 stored and 8.2, 12 159 8.2 and 8.2
//              2 columns n <= lanes / 5: 9 253 rows 8.2 and 8.3, 10 640 8.3 and 8.3
//              8 and 16 columns from 0.48 to 0.8 lanes, between the shared
//              items and the others: 8 columns 9 253 rows 12.4 and 16.4; 16 columns
//              4 912 rows 14.4 and 18.5
//   FP32 pairs 1 and 4 columns n <= lanes / 40: 2 196 rows 6.2 and 7.3, 2 743 7.7 and
//              7.4; 4 columns 512 rows 6.3 and 7.2, 1 000 rows 7.3 and 7.3
enum class Form { kStored, kSplit8, kSplit4, kSplit2, kPlain, kWalk };

static Form product_form(int precision, int64_t rows, int R, int sms) {
    const double n = 3.0 * (double)rows * R, lanes = 2048.0 * sms;
    if (R > 32 || (R & (R - 1))) return Form::kPlain;
    const bool c64 = precision == FE_PREC_MIXED;
    if (c64 && ((R == 1 && 9 * n <= lanes) || (R == 2 && 5 * n <= lanes) ||
                ((R == 8 || R == 16) && n > 0.48 * lanes && 5 * n <= 4 * lanes)))
        return Form::kStored;
    if (precision == FE_PREC_DF && (R == 1 || R == 4) && 40 * n <= lanes) return Form::kStored;
    if (8 * R <= 32 && 8 * n <= lanes) return Form::kSplit8;
    if (4 * R <= 32 && 4 * n <= lanes) return Form::kSplit4;
    if (2 * R <= 32 && n <= 0.48 * lanes) return Form::kSplit2;
    const double walk_from = R <= 4 ? lanes : (R == 16 ? 5.0 : 3.5) * lanes;
    return c64 && n > walk_from ? Form::kWalk : Form::kPlain;
}

template <typename C, int R>
static void launch_pat_plain(cudaStream_t st, const PatView<C>& V, const fe_system* s, int nrhs, const C* x, C* y) {
    const int64_t expl = ((int64_t)s->n_expl * 3 * nrhs + 255) / 256, all = ((int64_t)s->mesh->n_act * 3 * nrhs + 255) / 256;
    k_spmv_pat<C, R><<<(unsigned)(expl + all), 256, 0, st>>>(V, s->mesh->n_act, (const int*)s->pat_list.ptr, s->n_expl,
                                                            (int)expl, nrhs, x, y);
}

template <typename C, int R>
static void launch_pat_r(cudaStream_t st, const PatView<C>& V, const fe_system* s, int sms, Form form, const C* x,
                         C* y) {
    const int n = s->mesh->n_act;
    const int64_t items = (int64_t)n * 3 * R;
    auto blocks = [&](int k) { return (unsigned)((items * k + 255) / 256); };
    if constexpr (8 * R <= 32)
        if (form == Form::kSplit8) {
            k_spmv_pat_split<C, R, 8><<<blocks(8), 256, 0, st>>>(V, n, x, y);
            return;
        }
    if constexpr (4 * R <= 32)
        if (form == Form::kSplit4) {
            k_spmv_pat_split<C, R, 4><<<blocks(4), 256, 0, st>>>(V, n, x, y);
            return;
        }
    if constexpr (2 * R <= 32)
        if (form == Form::kSplit2) {
            k_spmv_pat_split<C, R, 2><<<blocks(2), 256, 0, st>>>(V, n, x, y);
            return;
        }
    if constexpr (std::is_same<C, float2>::value)
        if (form == Form::kWalk) {
            if constexpr (R <= 4)
                k_spmv_pat_keep<R><<<sms, kKeepThreads, 0, st>>>(V, n, (const int*)s->pat_list.ptr, s->n_expl, x, y);
            else
                k_spmv_pat_tile<R><<<sms, kTileThreads, 0, st>>>(V, n, (const int*)s->pat_list.ptr, s->n_expl, x, y);
            return;
        }
    launch_pat_plain<C, R>(st, V, s, R, x, y);
}

template <typename C>
static void launch_spmv_pat(cudaStream_t st, const fe_system* s, int sms, const void* terms, int nrhs, Form form,
                            const C* x, C* y) {
    const fe_mesh* m = s->mesh;
    const PatView<C> V{(const uint16_t*)s->pat_id.ptr, (const int4*)s->pat_row.ptr, (const int4*)s->pat_tab.ptr, (const C*)terms,
                       (const int*)m->node_id.ptr,     (const int*)m->node_rank.ptr, m->nx + 1,
                       (m->nx + 1) * (m->ny + 1)};
    switch (nrhs) {
        case 1: launch_pat_r<C, 1>(st, V, s, sms, form, x, y); break;
        case 2: launch_pat_r<C, 2>(st, V, s, sms, form, x, y); break;
        case 4: launch_pat_r<C, 4>(st, V, s, sms, form, x, y); break;
        case 8: launch_pat_r<C, 8>(st, V, s, sms, form, x, y); break;
        case 16: launch_pat_r<C, 16>(st, V, s, sms, form, x, y); break;
        case 32: launch_pat_r<C, 32>(st, V, s, sms, form, x, y); break;
        default: launch_pat_plain<C, 0>(st, V, s, nrhs, x, y); break;
    }
}

}  // namespace fe

using namespace fe;

extern "C" {

fe_status fe_spmv(fe_ctx* ctx, const fe_system* s, int32_t precision, int32_t nrhs, const void* x, void* y) {
    if (!ctx || !s || !x || !y || nrhs < 1) {
        set_error("fe_spmv: NULL argument or nrhs < 1");
        return FE_ERR_INVALID_ARG;
    }
    const fe_mesh* m = s->mesh;
    cudaStream_t st = ctx->stream;
    const int* rp = (const int*)m->row_ptr.ptr;
    const int* col = (const int*)m->col_idx.ptr;
    const bool pow2 = nrhs <= 32 && (nrhs & (nrhs - 1)) == 0;
    const unsigned warp_blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)ctx->num_sms * 8,
                                                                                  ((int64_t)m->n_act + 7) / 8));
    const int64_t n_items = (int64_t)m->n_act * nrhs;
    const unsigned col_blocks = (unsigned)((n_items + 255) / 256);
    const void* terms = precision == FE_PREC_FP64 ? s->pat_t64.ptr
                        : precision == FE_PREC_MIXED ? s->pat_t32.ptr
                        : precision == FE_PREC_DF ? s->pat_tdf.ptr : nullptr;
    const int64_t pat_blocks = ((int64_t)m->n_act + s->n_expl) * 3 * nrhs / 256 + 2;
    const Form form = product_form(precision, m->n_act, nrhs, ctx->num_sms);
    if (s->n_pat && terms && pat_blocks < (1ll << 31) && form != Form::kStored) {
        if (precision == FE_PREC_FP64)
            launch_spmv_pat<double2>(st, s, ctx->num_sms, terms, nrhs, form, (const double2*)x, (double2*)y);
        else if (precision == FE_PREC_MIXED)
            launch_spmv_pat<float2>(st, s, ctx->num_sms, terms, nrhs, form, (const float2*)x, (float2*)y);
        else
            launch_spmv_pat<float4>(st, s, ctx->num_sms, terms, nrhs, form, (const float4*)x, (float4*)y);
    } else if (precision == FE_PREC_FP64) {
        if (pow2 && nrhs >= 8)
            launch_spmm_rows<double2>(nrhs, st, ctx->num_sms, (const double2*)s->val64.ptr, s->stride, col, rp,
                                  (const double2*)x, (double2*)y, m->n_act);
        else if (pow2)
            launch_spmv_warp<double2>(nrhs, warp_blocks, st, (const double2*)s->val64.ptr, s->stride, col, rp,
                                  (const double2*)x, (double2*)y, m->n_act);
        else
            k_spmv_cols<double2><<<col_blocks, 256, 0, st>>>((const double2*)s->val64.ptr, s->stride, col, rp,
                                                             (const double2*)x, (double2*)y, m->n_act, nrhs);
    } else if (precision == FE_PREC_MIXED) {
        if (!s->val32.ptr) {
            set_error("fe_spmv: no complex64 copy (system assembled in FP64)");
            return FE_ERR_INVALID_ARG;
        }
        const bool aligned16 = (((uintptr_t)x | (uintptr_t)y) & 15) == 0;  // the lanes' 16-byte vector accesses
        if (pow2 && nrhs >= 8 && aligned16)
            launch_spmm_cpl(nrhs, st, ctx->num_sms, (const float2*)s->val32.ptr, s->stride, col, rp,
                            (const float2*)x, (float2*)y, m->n_act);
        else if (pow2 && nrhs >= 8)
            launch_spmm_rows<float2>(nrhs, st, ctx->num_sms, (const float2*)s->val32.ptr, s->stride, col, rp,
                                  (const float2*)x, (float2*)y, m->n_act);
        else if (pow2)
            launch_spmv_warp<float2>(nrhs, warp_blocks, st, (const float2*)s->val32.ptr, s->stride, col, rp,
                                  (const float2*)x, (float2*)y, m->n_act);
        else
            k_spmv_cols<float2><<<col_blocks, 256, 0, st>>>((const float2*)s->val32.ptr, s->stride, col, rp,
                                                            (const float2*)x, (float2*)y, m->n_act, nrhs);
    } else if (precision == FE_PREC_DF) {
        if (!s->valdf.ptr) {
            set_error("fe_spmv: no FP32-pair copy (system not assembled with FE_PREC_DF)");
            return FE_ERR_INVALID_ARG;
        }
        if (pow2 && nrhs >= 8)
            launch_spmm_rows<float4>(nrhs, st, ctx->num_sms, (const float4*)s->valdf.ptr, s->stride, col, rp,
                                  (const float4*)x, (float4*)y, m->n_act);
        else if (pow2)
            launch_spmv_warp<float4>(nrhs, warp_blocks, st, (const float4*)s->valdf.ptr, s->stride, col, rp,
                                  (const float4*)x, (float4*)y, m->n_act);
        else
            k_spmv_cols<float4><<<col_blocks, 256, 0, st>>>((const float4*)s->valdf.ptr, s->stride, col, rp,
                                                            (const float4*)x, (float4*)y, m->n_act, nrhs);
    } else {
        set_error("fe_spmv: bad precision");
        return FE_ERR_INVALID_ARG;
    }
    FE_LAUNCHED();
    return FE_OK;
}

}  // extern "C"
