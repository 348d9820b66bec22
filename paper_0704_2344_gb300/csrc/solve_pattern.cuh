// Device code of the persistent solve on the row patterns (patterns.cuh):
// block-Jacobi COCG for R right-hand sides, every arithmetic.  The method and
// its phases are those of solve_kernels.cuh, which serves systems without
// patterns and the block incomplete Cholesky preconditioner; this kernel
// differs in how it is laid out.
//
//   - A CTA owns one range of rows for everything: products, vectors, inner
//     products.  Only u crosses CTAs (the product reads the neighbours' u).
//   - A work item is (row, component, column).  An item's vector entries are
//     kept in shared memory when the CTA's items fit (pat_vec_max), so the
//     update touches global memory only to publish u.  The inner products of
//     r, u, p and s are taken where the update forms them and travel with the
//     next product's u^T w: five values per column and reduction (nine with
//     the expanded recurrence), and the product reads none of r, p and s.
//   - 512 threads with 128 registers instead of 1024 with 64: a CTA of a
//     mid-sized system has some 600 items, so the phases are bound by latency,
//     and registers for loads in flight count more than warps.
//
// Bound by latency: of the 16.2 us an iteration of the 3-wavelength cube takes
// with FP32 pairs, the reduction with its barrier takes 3.8 and the second
// barrier 1.95, and the rest is short phases of dependent operations; FP64 keeps
// its pipe about half busy.  Measured, us per iteration, solve_kernels.cuh and
// here: FP32 pairs 10^3 20.1 and 10.7, 30^3 25.6 and 16.2, 40^3 expanded 90 and
// 26.7, 18^3 with 12 columns 106 and 36; FP64 20^3 48 and 19.6; complex64 20^3
// 14.6 (16.7 before its sums were paired).
#pragma once

#include "solve_kernels.cuh"

namespace fe {

constexpr int kPT = 512;
constexpr int kPW = kPT / 32;
constexpr double kGrown2 = 100.0;  // growth of |r|^2 after which kept directions are given up
constexpr int kPatNV = 15;  // values per column of one reduction: 5, 9 (expanded) or 15 (with a refresh)

// ---------------------------------------------------------------------------
// Grid barrier (bounded, as in solve_kernels.cuh) and reduction.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool pat_barrier(const SolveParams& P, unsigned& passed) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int* verr = &P.sync->err;
        arrive_release(&P.sync->count);
        const unsigned target = (passed + 1u) * (unsigned)P.n_cta;
        int ok = 1;
        if ((int)(load_acquire(&P.sync->count) - target) < 0) {
            const unsigned long long t0 = globaltimer_ns();
            while ((int)(load_acquire(&P.sync->count) - target) < 0) {
                if (*verr) {
                    ok = 0;
                    break;
                }
                if (globaltimer_ns() - t0 > P.timeout_ns) {
                    atomicCAS(&P.sync->err, 0, kDevTimeout);
                    ok = 0;
                    break;
                }
            }
        }
        s_ok = ok && *verr == 0;
    }
    passed += 1u;
    __syncthreads();
    return s_ok != 0;
}

// Sum over the CTAs of NV values (8-byte slots: doubles, or FP32 pairs with
// kPair): every CTA writes its partials, passes the grid barrier and adds all
// CTAs' partials itself, in CTA order (lane-strided, then a fixed butterfly),
// so that all get bitwise the same sums without a second trip.  The partials of
// one value are consecutive, so a warp reads them in whole lines, five
// requests in flight per lane.  Partials alternate between two buffers by
// the barrier's parity: a CTA writes those of barrier e + 2 only after every
// CTA has arrived at barrier e + 1, that is after it has read barrier e's.
// (Words that carry their own number, polled by every CTA instead of a
// counter, were slower: 4.5 us against 2.2 to 2.5 us on 152 CTAs, the polls of all
// CTAs on the same few lines delaying the stores they wait for.)
template <int NV, bool kPair>
__device__ __noinline__ bool pat_reduce(const SolveParams& P, int cta, const double* s_in, double* s_out,
                                        unsigned& passed) {
    constexpr int kAhead = 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_cta = P.n_cta;
    double* part = P.pat_partial + (size_t)(passed & 1u) * (size_t)P.pat_half;
    for (int v = threadIdx.x; v < NV; v += kPT) part[(size_t)v * n_cta + cta] = s_in[v];
    if (!pat_barrier(P, passed)) return false;
    for (int v = warp; v < NV; v += kPW) {
        const double* pv = part + (size_t)v * n_cta;
        float h = 0.f, l = 0.f;
        double acc = 0.0;
        for (int c0 = lane; c0 < n_cta; c0 += 32 * kAhead) {
            double q[kAhead];  // a pair is the bits of one slot
#pragma unroll
            for (int k = 0; k < kAhead; ++k) q[k] = c0 + 32 * k < n_cta ? __ldcg(pv + c0 + 32 * k) : 0.0;
#pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                if (kPair) df_add(h, l, __int_as_float(__double2loint(q[k])), __int_as_float(__double2hiint(q[k])));
                else acc += q[k];
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            if (kPair) {
                const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
                df_add(h, l, h2, l2);
            } else {
                acc += __shfl_xor_sync(0xffffffffu, acc, o);
            }
        }
        if (lane == 0) {
            if (kPair) {
                df_norm(h, l);
                ((float2*)s_out)[v] = make_float2(h, l);
            } else {
                s_out[v] = acc;
            }
        }
    }
    __syncthreads();
    return true;
}

// Warp sums of N doubles over the lanes of one column (lane % R), two values to
// a butterfly step while there are two: a lane hands one of them over and keeps
// the other.  Five values take 8 additions a lane instead of 25; an FP64
// addition holds an SM's FP64 pipe for 16 cycles a warp, so that the 25 of 16
// warps took 3 us of an iteration.  (FP32 pairs, on wider pipes, keep one value
// to a step: 1 us.)  Afterwards a lane's w[k] is the sum of value
// (k << shift) | value, the same in the lanes that differ only in bits `same`.
struct WarpSums {
    int value = 0, same = 0, left = 0, shift = 0;
};
__device__ __forceinline__ double sum_from(double keep, double give, int o) {
    return keep + __shfl_xor_sync(0xffffffffu, give, o);
}
template <int O, int R, int N>
__device__ __forceinline__ void warp_sums(double* w, int lane, WarpSums& m) {
    if constexpr (O < R) {
        m.left = N;
    } else if constexpr (N == 1) {
        w[0] = sum_from(w[0], w[0], O);
        m.same |= O;
        warp_sums<O / 2, R, 1>(w, lane, m);
    } else {
        const bool up = lane & O;
#pragma unroll
        for (int k = 0; k < N / 2; ++k) {
            const double a = w[2 * k], b = w[2 * k + 1];
            w[k] = sum_from(up ? b : a, up ? a : b, O);
        }
        if constexpr (N % 2) w[N / 2] = sum_from(w[N - 1], w[N - 1], O);  // the odd one out; used where !up
        if (up) m.value |= 1 << m.shift;
        ++m.shift;
        warp_sums<O / 2, R, (N + 1) / 2>(w, lane, m);
    }
}

// Sum over the CTA of per-thread values, per column (thread t holds column
// t % R): NV of them, FP32 pairs (f[2k] + f[2k + 1]) or doubles.
template <int R, int NV, bool kPair>
__device__ __forceinline__ void pat_colsum(const float* f, const double* d, double* s_red, double* s_in) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (kPair) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            float h = f[2 * k], l = f[2 * k + 1];
#pragma unroll
            for (int o = 16; o >= R; o >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
                df_add(h, l, h2, l2);
            }
            if (lane < R) ((float2*)s_red)[(k * kPW + warp) * R + lane] = make_float2(h, l);
        }
    } else {
        double w[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) w[k] = d[k];
        WarpSums m;
        warp_sums<16, R, NV>(w, lane, m);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int v = (k << m.shift) | m.value;
            if (k < m.left && v < NV && !(lane & m.same)) s_red[(v * kPW + warp) * R + lane % R] = w[k];
        }
    }
    __syncthreads();
    // kPW = 16 warp totals per value: half a warp adds them, two values at a time
    for (int i0 = 2 * warp; i0 < NV * R; i0 += 2 * kPW) {
        const int i = i0 + (lane >> 4), k = i / R, c = i % R;
        const bool on = i < NV * R;
        if (kPair) {
            const float2 q = on ? ((const float2*)s_red)[(k * kPW + (lane & 15)) * R + c] : make_float2(0.f, 0.f);
            float h = q.x, l = q.y;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
                df_add(h, l, h2, l2);
            }
            if (on && (lane & 15) == 0) {
                df_norm(h, l);
                ((float2*)s_in)[i] = make_float2(h, l);
            }
        } else {
            double a = on ? s_red[(k * kPW + (lane & 15)) * R + c] : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (on && (lane & 15) == 0) s_in[i] = a;
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Tables of a CTA's rows.
// ---------------------------------------------------------------------------
// Rows a CTA's products read: up to three ranges (the planes below, at and
// above its rows), merged where they overlap.
struct PatHalo {
    int lo[3], hi[3];  // centres of the lines per plane, then the merged ranges
    int n;             // merged ranges
    int at[3];         // place of a range's first row in the staged copy, in rows
    unsigned bytes;    // of the staged copy
    int first_diag;    // first slot of the rows with real diagonal blocks (the last in the cost order)
};

constexpr int kPatRowBytes = (int)(sizeof(int4) + 9 * sizeof(int));
constexpr int kPatLocal = 48;       // patterns of a CTA whose diagonal inverses are kept in shared memory
constexpr unsigned kPatNoLoc = 0xffffu;
// info.w of a row: steps of its pattern and where its tables are
constexpr int kInfoDiag = 1 << 20, kInfoShared = 1 << 21, kInfoQuad = 1 << 30;
__device__ __forceinline__ int info_word(const int4& t, unsigned loc, unsigned ord) {
    return t.y | t.z << 10 | (t.w ? kInfoDiag : 0) | (loc != kPatNoLoc ? kInfoShared : 0) |
           (int)min(ord, (unsigned)kPatLocal) << 22;
}

// rows sorted by cost, dearest first (info), their lines (bases), the terms
// and diagonal inverses of the patterns among them; loc and ord give a
// pattern's first term in the shared copy and its number among the CTA's.
// info == nullptr: no row tables (too many rows).
template <typename C, typename VT, int R>
__device__ __noinline__ void build_pat_tables(const SolveParams& P, int pr0, int pr1, int4* info, int* bases, C* terms,
                                              VT* dinv, const VT* dinv_all, uint16_t* loc, uint16_t* ord,
                                              PatHalo* halo) {
    __shared__ unsigned s_bits[kMaxPat / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = pr1 - pr0;
    const bool rows = info != nullptr;
    int* keys = bases;  // scratch until the lines are written
    for (int i = tid; i < kMaxPat / 32; i += kPT) s_bits[i] = 0u;
    if (tid < 3) {
        halo->lo[tid] = 0x3fffffff;
        halo->hi[tid] = -1;
    }
    __syncthreads();
    for (int i = tid; i < n; i += kPT) {
        const int pid = P.pat_id[pr0 + i];
        atomicOr(&s_bits[pid >> 5], 1u << (pid & 31));
        if (rows) {
            const int4 t = P.pat_tab[pid];
            keys[i] = t.w ? 31 : 30 - min(30, (t.y + t.z) / 3);
        }
    }
    __syncthreads();
    if (tid == 0) {  // places of the CTA's patterns, in order of their numbers
        int off = 0;
        unsigned k = 0;
        for (int w = 0; w < kMaxPat / 32; ++w)
            for (unsigned b = s_bits[w]; b; b &= b - 1) {
                const int pid = 32 * w + __ffs(b) - 1;
                const int4 t = P.pat_tab[pid];
                const int cnt = 3 * (t.y + t.z);
                const bool fits = off + cnt <= P.pat_terms_max;
                loc[pid] = (uint16_t)(fits ? (unsigned)off : kPatNoLoc);
                ord[pid] = (uint16_t)min(k, (unsigned)kPatLocal);
                if (fits) off += cnt;
                ++k;
            }
    }
    if (rows && warp == 1) {  // stable counting sort by cost (deterministic)
        int base = 0;
        for (int b = 0; b < 32; ++b) {
            if (b == 31 && lane == 0) halo->first_diag = base;
            for (int c0 = 0; c0 < n; c0 += 32) {
                const int i = c0 + lane;
                const bool m = i < n && keys[i] == b;
                const unsigned bal = __ballot_sync(0xffffffffu, m);
                if (m) info[base + __popc(bal & ((1u << lane) - 1u))].x = pr0 + i;
                base += __popc(bal);
            }
        }
    }
    __syncthreads();
    for (int w = warp; w < kMaxPat / 32; w += kPW)
        for (unsigned b = s_bits[w]; b; b &= b - 1) {
            const int pid = 32 * w + __ffs(b) - 1;
            if (ord[pid] < kPatLocal && lane < 9)
                dinv[9 * ord[pid] + lane] = __ldg(dinv_all + (size_t)9 * P.pat_first[pid] + lane);
            if (loc[pid] == kPatNoLoc) continue;
            const int4 t = P.pat_tab[pid];
            const C* src = (const C*)P.pat_terms + (size_t)3 * t.x;
            for (int j = lane; j < 3 * (t.y + t.z); j += 32) terms[loc[pid] + j] = __ldg(src + j);
        }
    if (rows) {
        for (int i = tid; i < n; i += kPT) {
            const int row = info[i].x, pid = P.pat_id[row];
            const int4 t = P.pat_tab[pid];
            info[i] = make_int4(row, P.node_id[row], loc[pid] != kPatNoLoc ? (int)loc[pid] : 3 * t.x,
                                info_word(t, loc[pid], ord[pid]));
        }
        __syncthreads();
        // four rows in a row of the grid with one pattern: equal places and equal
        // words (a place is in the shared copy or in the global list, as bit
        // kInfoShared says); a row's own word is changed by its four's thread only
        for (int i = halo->first_diag + 4 * tid; i + 3 < n; i += 4 * kPT) {
            bool same = info[i + 3].y - info[i].y == 3;
            for (int k = 1; k < 4; ++k) same = same && info[i + k].z == info[i].z && info[i + k].w == info[i].w;
            if (same) info[i].w |= kInfoQuad;
        }
        // lines of the rows; a line outside the box or with an inactive centre
        // node carries no term and points at the row itself
        const int ny1 = P.pat_sz / P.pat_sy;
        for (int i = tid; i < 9 * n; i += kPT) {
            const int slot = i / 9, m = i - 9 * slot, dy = m % 3 - 1, dz = m / 3 - 1;
            const int node = info[slot].y, y = (node / P.pat_sy) % ny1 + dy, z = node / P.pat_sz + dz;
            int rank = -1;
            if (y >= 0 && y < ny1 && z >= 0 && z < P.pat_nz1) rank = P.node_rank[node + dy * P.pat_sy + dz * P.pat_sz];
            bases[i] = 3 * (rank >= 0 ? rank : info[slot].x);
            if (rank >= 0) {
                atomicMin(&halo->lo[dz + 1], rank);
                atomicMax(&halo->hi[dz + 1], rank);
            }
        }
        __syncthreads();
        if (tid == 0) {
            // ranges in ascending order with the lines' outer nodes; an even
            // first row and an even place keep the copies 16-byte aligned in
            // every arithmetic
            for (int a = 0; a < 2; ++a)
                for (int b = a + 1; b < 3; ++b)
                    if (halo->lo[b] < halo->lo[a]) {
                        const int tl = halo->lo[a], th = halo->hi[a];
                        halo->lo[a] = halo->lo[b];
                        halo->hi[a] = halo->hi[b];
                        halo->lo[b] = tl;
                        halo->hi[b] = th;
                    }
            int k = 0;
            unsigned at = 0;
            for (int g = 0; g < 3; ++g) {
                if (halo->hi[g] < 0) continue;
                const int lo = max(0, halo->lo[g] - 1) & ~1, hi = min(P.n_rows - 1, halo->hi[g] + 1);
                if (k > 0 && lo <= halo->hi[k - 1] + 1) {
                    halo->hi[k - 1] = max(halo->hi[k - 1], hi);
                } else {
                    halo->lo[k] = lo;
                    halo->hi[k] = hi;
                    ++k;
                }
            }
            for (int g = 0; g < k; ++g) {
                halo->at[g] = (int)at;
                at += (unsigned)(halo->hi[g] - halo->lo[g] + 2) & ~1u;
            }
            halo->n = k;
            halo->bytes = at * 3u * R * (unsigned)sizeof(C);
        }
        __syncthreads();
        if (P.stage && (int64_t)halo->bytes <= P.halo_bytes) {  // places in the staged copy instead of rows
            for (int i = tid; i < 9 * n; i += kPT) {
                const int row = bases[i] / 3;
                int g = 0;
                while (g + 1 < halo->n && row > halo->hi[g]) ++g;
                bases[i] = 3 * (row - halo->lo[g] + halo->at[g]);
            }
        }
    }
    __syncthreads();
}

// Copies the ranges of v into the halo buffer with bulk (TMA) copies on one
// mbarrier.  Returns false when the bounded wait expired.
template <typename C, int R>
__device__ __forceinline__ bool stage_pat(const SolveParams& P, const C* v, const PatHalo& h, char* halo_buf,
                                          uint64_t* mbar, unsigned& phase) {
    if (threadIdx.x == 0) {
        fence_proxy_async();
        constexpr unsigned kRow = 3u * R * (unsigned)sizeof(C);
        unsigned total = 0;
        for (int g = 0; g < h.n; ++g) total += ((unsigned)(h.hi[g] - h.lo[g] + 1) * kRow + 15u) & ~15u;
        mbar_expect_tx(mbar, total);
        for (int g = 0; g < h.n; ++g)
            bulk_g2s(halo_buf + (size_t)h.at[g] * kRow, (const char*)v + (size_t)h.lo[g] * kRow,
                     ((unsigned)(h.hi[g] - h.lo[g] + 1) * kRow + 15u) & ~15u, mbar);
    }
    const bool ok = __syncthreads_and(mbar_wait_bounded(mbar, phase & 1u, P.timeout_ns)) != 0;
    if (!ok) {
        atomicCAS(&P.sync->err, 0, kDevTimeout);
        // let the copy land before the CTA leaves (its shared memory is the destination)
        mbar_wait_bounded(mbar, phase & 1u, P.timeout_ns > 2000000000ull ? P.timeout_ns : 2000000000ull);
    }
    phase += 1;
    return ok;
}

// Least groups of fours per warp for a CTA to use them.
constexpr int kQuadGroups = 3;

// A CTA's rows as the phases see them.
template <typename C>
struct PatRows {
    int pr0, n;           // its range of rows
    const int4* info;     // per slot (row, node, first term, info_word); NULL: no row tables
    const int* bases;     // per slot, 3 x row (or place) of the centre of each line
    const C* terms;       // shared copy of the patterns
    const uint16_t* loc;
    const uint16_t* ord;
    int split;            // lanes that share an item (a CTA with few items)
    int first_diag;       // first slot of the rows with real diagonal blocks
    bool quads;           // take those four at a time
};

template <typename C>
__device__ __forceinline__ int4 row_info(const SolveParams& P, const PatRows<C>& pr, int slot) {
    if (pr.info) return pr.info[slot];
    const int row = pr.pr0 + slot, pid = __ldg(P.pat_id + row);
    const int4 t = __ldg(P.pat_tab + pid);
    return make_int4(row, __ldg(P.node_id + row), pr.loc[pid] != kPatNoLoc ? (int)pr.loc[pid] : 3 * t.x,
                     info_word(t, pr.loc[pid], pr.ord[pid]));
}

// Work item e = (3 slot + alpha) R + column.
template <int R>
struct Item {
    int slot, al, c;
    __device__ __forceinline__ explicit Item(int e) {
        c = e % R;
        const int task = e / R;
        slot = task / 3;
        al = task - 3 * slot;
    }
};

template <int R>
__device__ __forceinline__ size_t item_entry(int row, const Item<R>& it) {
    return (size_t)(3 * row + it.al) * R + it.c;
}

// Product of one item with the vector v; part of `split` lanes takes every
// split-th step and the caller adds the parts.
template <typename C, int R, typename Base>
__device__ __forceinline__ void item_product(TermAcc<C>& acc, const SolveParams& P, const PatRows<C>& pr,
                                             const int4& in, const Item<R>& it, int part, int split, const C* v,
                                             Base&& base) {
    const C* terms = ((in.w & kInfoShared) ? pr.terms : (const C*)P.pat_terms) + in.z + it.al;
    const int n_re = in.w & 0x3ff, n_im = (in.w >> 10) & 0x3ff;
    auto load = [&](size_t i) { return v[i]; };
    if (split > 1) {
        for (int t = part; t < n_re + n_im; t += split) {
            const C q = terms[3 * t];
            const int code = term_code(q);
            const C x = load((size_t)(base(code_line(code)) + code_delta(code)) * R + it.c);
            if (t < n_re) acc.add_re(q, x);
            else acc.add_im(q, x);
        }
    } else if (in.w & kInfoDiag) {
        pattern_diag<C, false>(acc, terms, it.al, R, it.c, base, load);
    } else {
        pattern_terms<C>(acc, terms, n_re, n_im, R, it.c, base, load);
    }
}

// Products of one component and column of four rows that follow each other
// along a grid line, all of one pattern of real diagonal blocks: the six
// entries of a line serve all four, so an item reads half the entries, lines
// and weights of four single ones.
template <typename C, int R, typename Base>
__device__ __forceinline__ void quad_product(TermAcc<C> (&acc)[4], const C* terms, int al, int c, const C* v,
                                             Base&& base) {
#pragma unroll 1
    for (int m = 0; m < 9; ++m) {
        const C* xp = v + (size_t)(base(m) + al) * R + c - 3 * R;
        C x[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) x[k] = xp[3 * k * R];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const C w = terms[9 * m + 3 * k];
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j].add_re(w, x[j + k]);
        }
    }
}

// Runs f(e, item, row info, product) over the CTA's items.  Groups of
// 32 consecutive items go to the warps in snake order: the rows are sorted by
// cost, so the lanes of a group run like numbers of steps and the warps end
// together.  With split > 1 every item fits the CTA at once and `split` lanes
// share its steps.
template <typename C, int R, bool kStaged, typename F>
__device__ __forceinline__ void for_products(const SolveParams& P, const PatRows<C>& pr, const C* v, F&& f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int E = 3 * pr.n * R;
    if (pr.split > 1) {
        const int q = threadIdx.x / R, part = q % pr.split, e = (q / pr.split) * R + (int)threadIdx.x % R;
        const bool on = e < E;
        const Item<R> it(on ? e : 0);
        TermAcc<C> acc;
        int4 in = make_int4(0, 0, 0, 0);
        if (on) {
            in = row_info(P, pr, it.slot);
            if (kStaged || pr.info) {
                const int* bs = pr.bases + 9 * it.slot;
                item_product<C, R>(acc, P, pr, in, it, part, pr.split, v, [&](int m) { return bs[m]; });
            } else {
                item_product<C, R>(acc, P, pr, in, it, part, pr.split, v,
                                   LineRanks{P.node_rank + in.y, P.pat_sy, P.pat_sz});
            }
        }
        for (int o = R; o < R * pr.split; o <<= 1) acc_butterfly(acc, o);
        if (on && part == 0) f(e, it, in, acc.result_norm());
        return;
    }
    auto one = [&](int e) {
        const Item<R> it(e);
        const int4 in = row_info(P, pr, it.slot);
        TermAcc<C> acc;
        if (kStaged || pr.info) {
            const int* bs = pr.bases + 9 * it.slot;
            item_product<C, R>(acc, P, pr, in, it, 0, 1, v, [&](int m) { return bs[m]; });
        } else {
            item_product<C, R>(acc, P, pr, in, it, 0, 1, v, LineRanks{P.node_rank + in.y, P.pat_sy, P.pat_sz});
        }
        f(e, it, in, acc.result_norm());
    };
    // groups of the fours first (they are the longest), then of the single items
    const int E1 = pr.quads ? 3 * pr.first_diag * R : E;
    const int n4 = pr.quads ? (pr.n - pr.first_diag + 3) / 4 : 0, E4 = 3 * n4 * R;
    const int groups4 = (E4 + 31) / 32, groups = groups4 + (E1 + 31) / 32;
    for (int k = 0; k * kPW < groups; ++k) {
        const int g = k * kPW + ((k & 1) ? kPW - 1 - warp : warp);
        if (g >= groups) continue;
        if (g < groups4) {
            const int q = 32 * g + lane;
            if (q >= E4) continue;
            const int c = q % R, task = q / R, al = task % 3, slot = pr.first_diag + 4 * (task / 3);
            const int4 in = pr.info[slot];
            const int e0 = (3 * slot + al) * R + c;
            if (in.w & kInfoQuad) {
                const C* terms = ((in.w & kInfoShared) ? pr.terms : (const C*)P.pat_terms) + in.z + al;
                const int* bs = pr.bases + 9 * slot;
                TermAcc<C> acc[4];
                quad_product<C, R>(acc, terms, al, c, v, [&](int m) { return bs[m]; });
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int e = e0 + 3 * j * R;
                    f(e, Item<R>(e), make_int4(in.x + j, in.y + j, in.z, in.w), acc[j].result_norm());
                }
            } else {
                for (int j = 0; j < 4 && slot + j < pr.n; ++j) one(e0 + 3 * j * R);
            }
        } else {
            const int e = 32 * (g - groups4) + lane;
            if (e < E1) one(e);
        }
    }
}

// One product phase: w = A u (and s = A p for columns being refreshed) with
// the fused inner products of w: values 3..4 u^T w, and for a refresh 5..6
// u^T s, 7..8 p^T w, 9..10 p^T s (facc holds pairs, value k at 2k and 2k + 1).
template <typename TM, int R, bool kStaged, bool kRefresh, typename Own>
__device__ __forceinline__ void pat_products(const SolveParams& P, const PatRows<typename CplxT<TM>::type>& pr,
                                             const typename CplxT<TM>::type* xs, const int* s_refresh, const Own& own,
                                             float* facc, double* acc) {
    using C = typename CplxT<TM>::type;
    constexpr bool kDFV = std::is_same<TM, DFloat>::value;
    const bool refresh = kRefresh && s_refresh[threadIdx.x % R] != 0;
    for_products<C, R, kStaged>(P, pr, xs, [&](int e, const Item<R>& it, const int4& in, const C& wy) {
        const size_t i = own.at(e, item_entry<R>(in.x, it));
        ((C*)own.w)[i] = wy;
        if constexpr (kDFV) {
            dfc_mac4(facc + 6, own.u[i], wy);
        } else {
            const double2 uv = own.u[i], wd = to_c128(wy);
            acc[3] += uv.x * wd.x - uv.y * wd.y;
            acc[4] += uv.x * wd.y + uv.y * wd.x;
        }
        if constexpr (kRefresh) {
            if (refresh) {
                TermAcc<C> ta;
                item_product<C, R>(ta, P, pr, in, it, 0, 1, (const C*)P.pM,
                                   LineRanks{P.node_rank + in.y, P.pat_sy, P.pat_sz});
                const C sy = ta.result_norm();
                if constexpr (kDFV) {
                    const float4 uv = own.u[i], pv = own.p[i];
                    dfc_mac4(facc + 10, uv, sy);
                    dfc_mac4(facc + 14, pv, wy);
                    dfc_mac4(facc + 18, pv, sy);
                    own.s[i] = sy;
                } else {
                    const double2 uv = own.u[i], pv = own.p[i], wd = to_c128(wy), sd = to_c128(sy);
                    acc[5] += uv.x * sd.x - uv.y * sd.y;
                    acc[6] += uv.x * sd.y + uv.y * sd.x;
                    acc[7] += pv.x * wd.x - pv.y * wd.y;
                    acc[8] += pv.x * wd.y + pv.y * wd.x;
                    acc[9] += pv.x * sd.x - pv.y * sd.y;
                    acc[10] += pv.x * sd.y + pv.y * sd.x;
                    own.s[i] = sd;
                }
            }
        }
    });
}

// A thread's share of the inner products of r, u, p and s: r^T u (2 values),
// |r|^2 (1), and for the expanded recurrence u^T s and p^T s (2 each), as FP32
// pairs or in FP64.
template <typename VT>
struct Dots;
template <>
struct Dots<float4> {
    float f[14];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int k = 0; k < 14; ++k) f[k] = 0.f;
    }
    __device__ __forceinline__ void add(const float4& r, const float4& u, const float4& p, const float4& s, int expand) {
        dfc_mac4(f + 0, r, u);
        df_mac(f[4], f[5], r.x, r.z, r.x, r.z);
        df_mac(f[4], f[5], r.y, r.w, r.y, r.w);
        if (expand) {
            dfc_mac4(f + 6, u, s);
            dfc_mac4(f + 10, p, s);
        }
    }
    __device__ __forceinline__ void head(float* facc, double*) const {
#pragma unroll
        for (int k = 0; k < 6; ++k) facc[k] = f[k];
    }
    __device__ __forceinline__ void tail(float* facc, double*) const {
#pragma unroll
        for (int k = 0; k < 8; ++k) facc[k] = f[6 + k];
    }
};
template <>
struct Dots<double2> {
    double d[7];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int k = 0; k < 7; ++k) d[k] = 0.0;
    }
    __device__ __forceinline__ void add(const double2& r, const double2& u, const double2& p, const double2& s,
                                        int expand) {
        d[0] += r.x * u.x - r.y * u.y;
        d[1] += r.x * u.y + r.y * u.x;
        d[2] += r.x * r.x + r.y * r.y;
        if (expand) {
            d[3] += u.x * s.x - u.y * s.y;
            d[4] += u.x * s.y + u.y * s.x;
            d[5] += p.x * s.x - p.y * s.y;
            d[6] += p.x * s.y + p.y * s.x;
        }
    }
    __device__ __forceinline__ void head(float*, double* acc) const {
#pragma unroll
        for (int k = 0; k < 3; ++k) acc[k] = d[k];
    }
    __device__ __forceinline__ void tail(float*, double* acc) const {
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] = d[3 + k];
    }
};

// The vectors of a CTA's items: in shared memory at the item's number, or in
// the global vectors at its entry.
template <typename VT>
struct OwnVecs {
    VT *r, *u, *p, *s, *x;
    void* w;       // products, in the product arithmetic
    bool shared;
    __device__ __forceinline__ size_t at(int e, size_t o) const { return shared ? (size_t)e : o; }
};

// The persistent solve of A X = B for R right-hand sides (phases as in
// solve_kernels.cuh: [R] replacement, [A] products, [B] scalars, [C] update).
template <typename TM, int R>
__device__ __forceinline__ void solve_pat_body(const SolveParams& P, const int cta) {
    using C = typename CplxT<TM>::type;
    constexpr bool kDFV = std::is_same<TM, DFloat>::value;  // Krylov vectors of FP32 pairs, else FP64
    using VT = std::conditional_t<kDFV, float4, double2>;
    constexpr bool kSplit = !std::is_same<C, VT>::value;    // the products read copies in their own arithmetic
    C* uM = (C*)P.uM;
    C* pM = (C*)P.pM;
    const VT* dinv_all = kDFV ? (const VT*)(const void*)P.dinvdf : (const VT*)(const void*)P.dinv64;

    // shared memory: [column sums][row tables][terms][inverses][vectors][halo]
    extern __shared__ __align__(128) char dyn[];
    double* s_red = (double*)dyn;
    int4* t_info = (int4*)(dyn + P.red_bytes);
    int* t_bases = (int*)(t_info + P.pat_rows_max);
    C* t_terms = (C*)(dyn + P.red_bytes + (((size_t)P.pat_rows_max * kPatRowBytes + 15) & ~(size_t)15));
    VT* t_dinv = (VT*)(t_terms + P.pat_terms_max);
    VT* t_vecs = t_dinv + 9 * kPatLocal;
    char* halo_buf = dyn + P.red_bytes + P.res_bytes;

    __shared__ __align__(8) uint64_t s_mbar;
    __shared__ double s_in[kPatNV * R], s_out[kPatNV * R];
    __shared__ double s_bn[R], s_rr_ref[R], s_rel[R];
    __shared__ double s_gam_r[R], s_gam_i[R], s_al_r[R], s_al_i[R], s_be_r[R], s_be_i[R];
    __shared__ double s_igam_r[R], s_igam_i[R], s_ial_r[R], s_ial_i[R];  // 1/gamma, 1/alpha of the last iteration
    __shared__ float4 s_a4[R], s_na4[R], s_b4[R];                        // alpha, -alpha, beta as FP32 pairs
    __shared__ float4 s_gam4[kDFV ? R : 1], s_igam4[kDFV ? R : 1], s_ial4[kDFV ? R : 1];
    __shared__ float s_ibn2f[kDFV ? R : 1], s_irrf[kDFV ? R : 1];
    __shared__ int s_scl_ok[kDFV ? R : 1];
    __shared__ int s_active[R], s_done[R], s_status[R], s_iters[R], s_outer[R], s_first[R], s_refresh[R], s_repl[R],
        s_pass_it[R];
    __shared__ int s_kept[R];  // this pass goes on with the directions of the last
    __shared__ int s_any_repl, s_any_refresh;
    __shared__ uint16_t s_loc[kMaxPat], s_ord[kMaxPat];
    __shared__ PatHalo s_halo;
    __shared__ int s_pr[2];
    // FP32 forms of 1/||b||^2 and 1/rr_ref, set whenever those change (rare)
    auto set_scales = [&](int c) {
        if constexpr (kDFV) {
            const double b2 = s_bn[c] * s_bn[c];
            const double ib = b2 > 0.0 ? 1.0 / b2 : 0.0, ir = s_rr_ref[c] > 0.0 ? 1.0 / s_rr_ref[c] : 0.0;
            s_ibn2f[c] = (float)ib;
            s_irrf[c] = (float)ir;
            s_scl_ok[c] = ib > 1.0e-37 && ib < 1.0e37 && ir > 1.0e-37 && ir < 1.0e37;
        }
    };
    const float tol2f = (float)(P.tol * P.tol), rel2f = (float)(P.reliable * P.reliable);
    const int tid = threadIdx.x;

    // the CTA's rows: equal product cost
    if (tid < 2) {
        const int64_t total = P.cost_prefix[P.n_rows];
        const int64_t target = (int64_t)(cta + tid) * total / P.n_cta;
        int lo = 0, hi = P.n_rows;  // first row whose prefix >= target
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((int64_t)P.cost_prefix[mid] < target) lo = mid + 1;
            else hi = mid;
        }
        s_pr[tid] = (cta + tid == P.n_cta) ? P.n_rows : lo;
    }
    __syncthreads();
    const int pr0 = s_pr[0], n = s_pr[1] - pr0;
    const int E = 3 * n * R;  // work items
    const bool rows = n <= P.pat_rows_max;
    build_pat_tables<C, VT, R>(P, pr0, pr0 + n, rows ? t_info : nullptr, t_bases, t_terms, t_dinv, dinv_all, s_loc,
                               s_ord, &s_halo);
    const bool staged = rows && P.stage && (int64_t)s_halo.bytes <= P.halo_bytes;
    PatRows<C> pr{pr0, n, rows ? t_info : nullptr, t_bases, t_terms, s_loc, s_ord, 1, rows ? s_halo.first_diag : n, false};
    while (2 * pr.split * R <= 32 && 2 * pr.split * E <= kPT) pr.split *= 2;
    // fours need a few groups per warp to balance
    pr.quads = 3 * ((n - pr.first_diag) / 4) * R >= kQuadGroups * kPT;
    OwnVecs<VT> own;
    own.shared = rows && E <= P.pat_vec_max;
    if (own.shared) {
        own.r = t_vecs;
        own.u = own.r + P.pat_vec_max;
        own.p = own.u + P.pat_vec_max;
        own.s = own.p + P.pat_vec_max;
        own.x = own.s + P.pat_vec_max;
        own.w = own.x + P.pat_vec_max;
    } else {
        own.r = (VT*)P.r;
        own.u = (VT*)P.u;
        own.p = (VT*)P.p;
        own.s = (VT*)P.s;
        own.x = (VT*)P.x;
        own.w = P.w;
    }
    // runs f(item number, item, row info, entry, place in the own vectors) over the items of this thread
    auto for_items = [&](auto&& f) {
        for (int e = tid; e < E; e += kPT) {
            const Item<R> it(e);
            const int4 in = row_info(P, pr, it.slot);
            const size_t o = item_entry<R>(in.x, it);
            f(e, it, in, o, own.at(e, o));
        }
    };
    if (P.trace && tid == 0) {
        unsigned long long* st = P.trace + (size_t)P.n_cta * kTraceIters * kTracePhases + (size_t)cta * kTraceStats;
        st[0] = (unsigned long long)pr0;
        st[1] = (unsigned long long)(pr0 + n);
    }
    const int my_c = tid % R;  // column of every item this thread handles
    unsigned mbar_phase = 0, passed = 0;
    int trace_it = 0;
    if (tid == 0) mbar_init(&s_mbar, 1);
    int seg_it = 0;
    bool seg_end = false;
    const unsigned long long seg_t0 = (P.state && cta == 0 && tid == 0) ? globaltimer_ns() : 0ull;
    const bool resume = P.state && __ldcg(&P.state->started);
    if (resume) {
        if (tid < R) {
            const ColState& cs = P.state->col[tid];
            s_bn[tid] = cs.bn;
            s_rr_ref[tid] = cs.rr_ref;
            s_rel[tid] = cs.rel;
            s_gam_r[tid] = cs.gam_r;
            s_gam_i[tid] = cs.gam_i;
            s_al_r[tid] = cs.al_r;
            s_al_i[tid] = cs.al_i;
            s_be_r[tid] = cs.be_r;
            s_be_i[tid] = cs.be_i;
            s_igam_r[tid] = cs.igam_r;
            s_igam_i[tid] = cs.igam_i;
            s_ial_r[tid] = cs.ial_r;
            s_ial_i[tid] = cs.ial_i;
            s_a4[tid] = cs.a4;
            s_na4[tid] = cs.na4;
            s_b4[tid] = cs.b4;
            if constexpr (kDFV) {
                s_gam4[tid] = cs.gam4;
                s_igam4[tid] = cs.igam4;
                s_ial4[tid] = cs.ial4;
                set_scales(tid);
            }
            s_active[tid] = cs.active;
            s_done[tid] = cs.done;
            s_status[tid] = cs.status;
            s_iters[tid] = cs.iters;
            s_outer[tid] = cs.outer;
            s_first[tid] = cs.first;
            s_refresh[tid] = cs.refresh;
            s_repl[tid] = cs.repl;
            s_pass_it[tid] = cs.pass_it;
            s_kept[tid] = cs.kept;
        }
        if (tid == 0) {
            s_any_repl = P.state->any_repl;
            s_any_refresh = P.state->any_refresh;
        }
        if (own.shared)
            for_items([&](int, const Item<R>&, const int4&, size_t o, size_t i) {
                own.r[i] = ((const VT*)P.r)[o];
                own.u[i] = ((const VT*)P.u)[o];
                own.p[i] = ((const VT*)P.p)[o];
                own.s[i] = ((const VT*)P.s)[o];
                own.x[i] = ((const VT*)P.x)[o];
            });
    } else {
        if (tid < R) {
            s_done[tid] = 0;
            s_status[tid] = FE_OK;
            s_iters[tid] = 0;
            s_pass_it[tid] = 0;
            s_kept[tid] = 0;
            s_outer[tid] = 0;
            s_active[tid] = 0;
            s_first[tid] = 1;
            s_refresh[tid] = 0;
            s_repl[tid] = 1;  // the first pass computes the initial residual
            s_rel[tid] = 0.0;
            s_bn[tid] = 0.0;
        }
        const double2 zero = make_double2(0.0, 0.0);  // zero bits: also a zero FP32 pair
        for_items([&](int, const Item<R>&, const int4&, size_t o, size_t i) {
            own.x[i] = P.use_x0 ? from_c128<VT>(P.x[o]) : from_c128<VT>(zero);
            own.p[i] = from_c128<VT>(zero);
            own.s[i] = from_c128<VT>(zero);
        });
        if (tid == 0) {
            s_any_repl = 1;
            s_any_refresh = 0;
        }
    }
    // inner products of the vectors as the last update (or replacement) left
    // them, this thread's share: r^T u (2 values), |r|^2 (1), and for the
    // expanded recurrence u^T s and p^T s (2 each); summed with the next
    // product's.  A resumed segment takes them again from the vectors, in the
    // update's order.
    Dots<VT> dots;
    dots.clear();
    // With the vectors in global memory, the FP32-pair update takes whole nodes,
    // three components of a column per thread: r need not be exchanged, and
    // the loads of a thread's 18 entries are in flight together (32 columns on
    // the 3-wavelength cube: 58 us against 90).  From shared memory, and with
    // FP64's long operations, more lanes are worth more (one column on that
    // cube: 1.9 us item by item, 2.5 us by nodes).
    const bool by_node = kDFV && !own.shared;
    // runs f(slot, row info, first entry, place of the first entry) over the thread's (node, column) pairs
    auto for_nodes = [&](auto&& f) {
        for (int q = tid; q < n * R; q += kPT) {
            const int slot = q / R, c = q - slot * R;
            const int4 in = row_info(P, pr, slot);
            const size_t o = (size_t)3 * in.x * R + c;
            f(slot, in, o, own.at(3 * slot * R + c, o));
        }
    };
    __syncthreads();
    if (resume && s_active[my_c] && !s_repl[my_c]) {
        if (by_node)
            for_nodes([&](int, const int4&, size_t, size_t i) {
#pragma unroll
                for (int al = 0; al < 3; ++al)
                    dots.add(own.r[i + al * R], own.u[i + al * R], own.p[i + al * R], own.s[i + al * R], P.expand);
            });
        else
            for_items([&](int, const Item<R>&, const int4&, size_t, size_t i) {
                dots.add(own.r[i], own.u[i], own.p[i], own.s[i], P.expand);
            });
    }

    for (;;) {
        // a segmented solve saves its state here, where every CTA has
        // finished the last iteration (or the replacement request before it)
        if (P.seg_iters > 0 && seg_it >= P.seg_iters) {
            seg_end = true;
            break;
        }
        if (s_any_repl) {
            // ---- [R] FP64 true residual for the columns that ask for it ----
            // x in FP64 for the products (FP32 pairs: in w, free until the
            // next product), and p for the refresh products
            double2* xsrc = kDFV ? (double2*)P.w : P.x;
            for_items([&](int, const Item<R>&, const int4&, size_t o, size_t i) {
                if (kDFV || own.shared) xsrc[o] = to_c128(own.x[i]);
                if (own.shared && !kSplit) ((VT*)P.p)[o] = own.p[i];
            });
            if (!pat_barrier(P, passed)) goto out;
            {
                double acc[2] = {0.0, 0.0};
                if (s_repl[my_c])
                    for_items([&](int, const Item<R>& it, const int4& in, size_t o, size_t i) {
                        const int4 t = __ldg(P.pat_tab + __ldg(P.pat_id + in.x));
                        const LineRanks base{P.node_rank + in.y, P.pat_sy, P.pat_sz};
                        const double2* terms = P.pat_terms64 + (size_t)3 * t.x + it.al;
                        TermAcc<double2> ta;
                        auto load = [&](size_t k) { return xsrc[k]; };
                        if (t.w) pattern_diag<double2, false>(ta, terms, it.al, R, it.c, base, load);
                        else pattern_terms<double2>(ta, terms, t.y, t.z, R, it.c, base, load);
                        const double2 bv = __ldg(P.b + o);
                        const double2 rv = make_double2(bv.x - ta.re, bv.y - ta.im);
                        own.r[i] = from_c128<VT>(rv);
                        acc[0] += rv.x * rv.x + rv.y * rv.y;
                        acc[1] += bv.x * bv.x + bv.y * bv.y;
                    });
                pat_colsum<R, 2, false>(nullptr, acc, s_red, s_in);
                if (!pat_reduce<2 * R, false>(P, cta, s_in, s_out, passed)) goto out;
            }
            if (tid < R) {
                const int c = tid;
                if (s_repl[c] && !s_done[c]) {
                    if (s_first[c] && s_outer[c] == 0) s_bn[c] = sqrt(s_out[R + c]);
                    const double rn = sqrt(s_out[c]), bn = s_bn[c];
                    const double rel = bn > 0.0 ? rn / bn : 0.0;
                    s_rel[c] = rel;
                    s_outer[c] += 1;
                    s_active[c] = 0;
                    if (!(rel == rel)) {
                        s_done[c] = 1;
                        s_status[c] = FE_ERR_NOT_CONVERGED;
                    } else if (rel <= P.tol) {
                        s_done[c] = 1;
                        s_status[c] = FE_OK;
                    } else if (s_iters[c] >= P.max_iter || s_outer[c] > P.max_outer) {
                        s_done[c] = 1;
                        s_status[c] = FE_ERR_NOT_CONVERGED;
                    } else {
                        s_active[c] = 1;
                        s_rr_ref[c] = rn * rn;
                        set_scales(c);
                        s_pass_it[c] = 0;
                        s_refresh[c] = s_first[c] ? 0 : 1;
                        s_kept[c] = s_refresh[c];
                    }
                } else if (s_repl[c]) {
                    s_active[c] = 0;
                }
            }
            __syncthreads();
            // u = Dinv r (FP64) and the product copies for the replaced columns
            if (s_repl[my_c] && s_active[my_c]) {
                dots.clear();
                for_items([&](int, const Item<R>& it, const int4& in, size_t o, size_t i) {
                    const double2* drow = P.dinv64 + (size_t)in.x * 9 + 3 * it.al;
                    double2 uu = make_double2(0.0, 0.0);
#pragma unroll
                    for (int be = 0; be < 3; ++be)
                        uu = cfma(__ldg(drow + be), to_c128(own.r[(int64_t)i + (be - it.al) * R]), uu);
                    const VT uv = from_c128<VT>(uu);
                    own.u[i] = uv;
                    if (own.shared) ((VT*)P.u)[o] = uv;
                    if constexpr (kSplit) {
                        uM[o] = from_c128<C>(uu);
                        pM[o] = from_c128<C>(to_c128(own.p[i]));
                    }
                    dots.add(own.r[i], uv, own.p[i], own.s[i], P.expand);
                });
            }
            __syncthreads();
            if (tid == 0) {
                int refr = 0;
                for (int c = 0; c < R; ++c) {
                    s_repl[c] = 0;
                    refr |= s_refresh[c];
                }
                s_any_refresh = refr;
                s_any_repl = 0;
            }
            if (!pat_barrier(P, passed)) goto out;
            {
                int any = 0;
                for (int c = 0; c < R; ++c) any |= !s_done[c];
                if (!any) break;
            }
        }

        // ---- [A] products and fused inner products ----
        // The last warp takes the reciprocals the next scalars need, 1/gamma
        // and 1/alpha of the last iteration, while the others begin.
        if (tid >= kPT - R) {
            const int c = kPT - 1 - tid;
            if constexpr (kDFV) {
                if (s_active[c] && !s_first[c]) {
                    const DZ one = {make_float2(1.f, 0.f), make_float2(0.f, 0.f)};
                    s_igam4[c] = dz_f4(dz_div(one, dz_of(s_gam4[c])));
                    s_ial4[c] = dz_f4(dz_div(one, dz_of(s_a4[c])));
                }
            } else if (s_active[c] && !s_first[c]) {
                const double ig = rcp64(s_gam_r[c] * s_gam_r[c] + s_gam_i[c] * s_gam_i[c]);
                const double ia = rcp64(s_al_r[c] * s_al_r[c] + s_al_i[c] * s_al_i[c]);
                s_igam_r[c] = s_gam_r[c] * ig;
                s_igam_i[c] = -s_gam_i[c] * ig;
                s_ial_r[c] = s_al_r[c] * ia;
                s_ial_i[c] = -s_al_i[c] * ia;
            }
        }
        FE_TRACE_MARK(0);
        if (staged && !stage_pat<C, R>(P, uM, s_halo, halo_buf, &s_mbar, mbar_phase)) goto out;
        FE_TRACE_MARK(1);
        // values: 0..1 r^T u, 2 |r|^2, 3..4 u^T w, with a refresh 5..10, then
        // u^T s and p^T s of the last update (expanded recurrence)
#define FE_PAT_PRODUCTS(NV, REFRESH)                                                                             \
    float facc[2 * (NV)] = {};                                                                                  \
    double acc[NV] = {};                                                                                        \
    dots.head(facc, acc);                                                                                       \
    if (staged) pat_products<TM, R, true, REFRESH>(P, pr, (const C*)halo_buf, s_refresh, own, facc, acc);       \
    else pat_products<TM, R, false, REFRESH>(P, pr, uM, s_refresh, own, facc, acc);                             \
    FE_TRACE_MARK(2);                                                                                           \
    if ((NV) > 5) dots.tail(facc + 2 * ((NV) - 4), acc + ((NV) - 4));                                           \
    pat_colsum<R, NV, kDFV>(facc, acc, s_red, s_in);                                                            \
    FE_TRACE_MARK(3);                                                                                           \
    if (!pat_reduce<(NV) * R, kDFV>(P, cta, s_in, s_out, passed)) goto out
        if (s_any_refresh) {
            FE_PAT_PRODUCTS(15, true);
        } else if (P.expand) {
            FE_PAT_PRODUCTS(9, false);
        } else {
            FE_PAT_PRODUCTS(5, false);
        }
#undef FE_PAT_PRODUCTS
        FE_TRACE_MARK(4);
        // ---- [B] scalars ----
        // B1: does any column need its true residual first?  (No state of the
        // other columns changes in a replacement round: they redo the same
        // products next round.)
        int ask = 0;
        if (tid < R) {
            const int c = tid;
            if (s_active[c]) {
                bool small, nan, grown;
                if constexpr (kDFV) {  // |r|^2 as an FP32 pair; the tests scaled into FP32 range
                    const float2 q = ((const float2*)s_out)[2 * R + c];
                    const float rr = __fadd_rn(q.x, q.y);
                    nan = !(rr == rr);
                    if (s_scl_ok[c]) {
                        small = rr * s_ibn2f[c] <= tol2f || rr * s_irrf[c] < rel2f;
                        grown = rr * s_irrf[c] > (float)kGrown2;
                    } else {
                        const double rd = (double)q.x + (double)q.y, tb = P.tol * s_bn[c];
                        small = rd <= tb * tb || rd < P.reliable * P.reliable * s_rr_ref[c];
                        grown = rd > kGrown2 * s_rr_ref[c];
                    }
                } else {
                    const double rr = s_out[2 * R + c];
                    const double tb = P.tol * s_bn[c];
                    small = rr <= tb * tb || rr < P.reliable * P.reliable * s_rr_ref[c];
                    grown = rr > kGrown2 * s_rr_ref[c];
                    nan = !(rr == rr);
                }
                const bool stalled = P.restart && P.max_pass > 0 && s_pass_it[c] >= P.max_pass;
                // Directions kept across a replacement near the attainable accuracy
                // are not conjugate to a residual that the replacement has
                // changed by as much as itself.  As a rule it falls again within a
                // few hundred iterations; where it has grown tenfold, or has not
                // fallen in a quarter of the iterations before, the directions
                // are dropped.  Measured on 24 cubes each of 10^3, 30^3 (FP32
                // pairs to 5e-11), 20^3 (FP64 to 1e-11) and 18^3 with 12 columns
                // (to 1e-10), and all of them to 1e-8: the rule fires once, on a
                // 30^3 cube that ends unconverged after 20 000 iterations without
                // it and converges after 7 000 with it; every other column has
                // the same iterations with and without.
                const bool lost = s_kept[c] && !s_first[c] &&
                                  (grown || s_pass_it[c] >= max(500, (s_iters[c] - s_pass_it[c]) / 4));
                if (nan || s_iters[c] >= P.max_iter || (!s_first[c] && (small || stalled)) || lost) {
                    s_repl[c] = 1;
                    if (P.restart || lost) s_first[c] = 1;
                    ask = 1;
                }
            }
        }
        // (only warp 0 holds columns; its vote decides for the CTA)
        bool replace = false;
        if (tid < 32) {
            replace = __any_sync(0xffffffffu, ask) != 0;
            if (tid == 0) s_any_repl = replace;
        }
        // B2: Chronopoulos-Gear scalars (exact p^T A p after a replacement),
        // with 1/gamma_old and 1/alpha_old taken during the products.
        int bad = 0, refr = 0;
        if (tid < R && !replace) {
            const int c = tid;
            if (s_active[c]) {
                const bool refresh = s_refresh[c] != 0;
                // slots of u^T s and p^T s behind the other values
                const int xo = s_any_refresh ? 11 : 5;
                if constexpr (kDFV) {  // FP32-pair arithmetic
                    const float2* so = (const float2*)s_out;
                    const float2 zero = make_float2(0.f, 0.f);
                    const DZ g = {so[c], so[R + c]}, d = {so[3 * R + c], so[4 * R + c]};
                    DZ b = {zero, zero}, e = d;
                    if (!s_first[c]) {
                        b = dz_mul(g, dz_of(s_igam4[c]));  // beta = gamma / gamma_old
                        if (refresh) {
                            // p^T A p for p = u + beta p_old: u^T w + beta (u^T s + p^T w) + beta^2 p^T s
                            const DZ e12 = {dd_add(so[5 * R + c], so[7 * R + c]), dd_add(so[6 * R + c], so[8 * R + c])};
                            const DZ e3 = {so[9 * R + c], so[10 * R + c]};
                            e = dz_add(dz_add(d, dz_mul(b, e12)), dz_mul(dz_mul(b, b), e3));
                        } else if (P.expand) {
                            // u^T w + 2 beta u^T s + beta^2 p^T s
                            const DZ us = {so[xo * R + c], so[(xo + 1) * R + c]};
                            const DZ ps = {so[(xo + 2) * R + c], so[(xo + 3) * R + c]};
                            e = dz_add(dz_add(d, dz_mul(dz_add(b, b), us)), dz_mul(dz_mul(b, b), ps));
                        } else {
                            e = dz_sub(d, dz_mul(dz_mul(b, g), dz_of(s_ial4[c])));  // delta - beta gamma / alpha_old
                        }
                    }
                    s_b4[c] = dz_f4(b);
                    if (!dz_usable(e) || !dz_usable(g)) {
                        bad = 1;
                    } else {
                        const float4 a4 = dz_f4(dz_div(g, e));
                        s_a4[c] = a4;
                        s_na4[c] = make_float4(-a4.x, -a4.y, -a4.z, -a4.w);
                        s_gam4[c] = dz_f4(g);
                    }
                } else {
                    const double gr = s_out[c], gi = s_out[R + c];
                    const double dr = s_out[3 * R + c], di = s_out[4 * R + c];
                    double br = 0.0, bi = 0.0, er = dr, ei = di;
                    if (!s_first[c]) {
                        br = gr * s_igam_r[c] - gi * s_igam_i[c];  // beta = gamma / gamma_old
                        bi = gr * s_igam_i[c] + gi * s_igam_r[c];
                        const double b2r = br * br - bi * bi, b2i = br * bi + bi * br;
                        if (refresh) {
                            const double e12r = s_out[5 * R + c] + s_out[7 * R + c];
                            const double e12i = s_out[6 * R + c] + s_out[8 * R + c];
                            const double e3r = s_out[9 * R + c], e3i = s_out[10 * R + c];
                            er = dr + (br * e12r - bi * e12i) + (b2r * e3r - b2i * e3i);
                            ei = di + (br * e12i + bi * e12r) + (b2r * e3i + b2i * e3r);
                        } else if (P.expand) {
                            const double usr = s_out[xo * R + c], usi = s_out[(xo + 1) * R + c];
                            const double psr = s_out[(xo + 2) * R + c], psi = s_out[(xo + 3) * R + c];
                            er = dr + 2.0 * (br * usr - bi * usi) + (b2r * psr - b2i * psi);
                            ei = di + 2.0 * (br * usi + bi * usr) + (b2r * psi + b2i * psr);
                        } else {
                            // delta - beta gamma / alpha_old
                            const double tr = br * gr - bi * gi, ti = br * gi + bi * gr;
                            er = dr - (tr * s_ial_r[c] - ti * s_ial_i[c]);
                            ei = di - (tr * s_ial_i[c] + ti * s_ial_r[c]);
                        }
                    }
                    const double ed = er * er + ei * ei, gg = gr * gr + gi * gi;
                    if (!(ed > 0.0) || !(ed < 1e300) || !(gg > 0.0) || !(gg < 1e300)) {
                        bad = 1;
                    } else {
                        const double ie = rcp64(ed);
                        s_al_r[c] = (gr * er + gi * ei) * ie;
                        s_al_i[c] = (gi * er - gr * ei) * ie;
                        s_be_r[c] = br;
                        s_be_i[c] = bi;
                        s_gam_r[c] = gr;
                        s_gam_i[c] = gi;
                    }
                }
                if (bad) {
                    if (s_first[c]) {  // breakdown right after a (re)start
                        s_active[c] = 0;
                        s_done[c] = 1;
                        s_status[c] = FE_ERR_BREAKDOWN;
                        bad = 0;
                    } else {  // restart from the true residual next round
                        s_repl[c] = 1;
                        s_first[c] = 1;
                    }
                } else {
                    s_iters[c] += 1;
                    s_pass_it[c] += 1;
                    s_first[c] = 0;
                    s_refresh[c] = 0;
                }
            }
            refr = s_refresh[c];
        }
        if (tid < 32 && !replace) {
            const bool any_bad = __any_sync(0xffffffffu, bad) != 0, any_refr = __any_sync(0xffffffffu, refr) != 0;
            if (tid == 0) {
                s_any_repl = any_bad;  // a breakdown restarts at the top of the next round
                s_any_refresh = any_refr;
            }
        }
        if (tid == 0) s_pr[0] = replace ? 1 : 0;  // (s_pr is free after the setup)
        __syncthreads();
        if (s_pr[0]) {  // a replacement round: the directions of restarting columns are dropped
            if (s_repl[my_c] && s_first[my_c])
                for_items([&](int, const Item<R>&, const int4&, size_t, size_t i) {
                    own.p[i] = from_c128<VT>(make_double2(0.0, 0.0));
                    own.s[i] = from_c128<VT>(make_double2(0.0, 0.0));
                });
            __syncthreads();
            continue;
        }
        FE_TRACE_MARK(5);
        // ---- [C] update ----
        // The inner products of the new vectors travel with the next reduction
        // (expanded recurrence: u^T w of the next product, u^T s and p^T s give
        // the next p^T A p = u^T w + 2 beta u^T s + beta^2 p^T s; A symmetric,
        // so p^T A u = u^T A p, here u^T s).
        {
            const bool act = s_active[my_c] != 0 && !s_repl[my_c];
            const float4 a4 = s_a4[my_c], na4 = s_na4[my_c], b4 = s_b4[my_c];
            const double2 alpha = make_double2(s_al_r[my_c], s_al_i[my_c]);
            const double2 nalpha = make_double2(-s_al_r[my_c], -s_al_i[my_c]);
            const double2 beta = make_double2(s_be_r[my_c], s_be_i[my_c]);
            // p = u + beta p, s = w + beta s, x += alpha p, r -= alpha s
            auto step = [&](const VT& uu, const C& ww, VT& pp, VT& ss, VT& xx, VT& rr) {
                if constexpr (kDFV) {
                    pp = dfc_axpy(uu, b4, pp);
                    ss = dfc_axpy(ww, b4, ss);
                    xx = dfc_axpy(xx, a4, pp);
                    rr = dfc_axpy(rr, na4, ss);
                } else {
                    pp = cfma(beta, pp, uu);
                    ss = cfma(beta, ss, to_c128(ww));
                    xx = cfma(alpha, pp, xx);
                    rr = cfma(nalpha, ss, rr);
                }
            };
            auto inverse_row = [&](const int4& in) {
                const int ord = (in.w >> 22) & 0xff;
                return ord < kPatLocal ? (const VT*)t_dinv + 9 * ord : dinv_all + (size_t)9 * in.x;
            };
            // u = row al of Dinv times r (a real diagonal block has a real diagonal inverse)
            auto precond = [&](const int4& in, const VT* drow, int al, const VT& r0, const VT& r1, const VT& r2) {
                VT uu;
                if constexpr (kDFV) {
                    float acc[4] = {0.f, 0.f, 0.f, 0.f};
                    if (in.w & kInfoDiag) {
                        const VT d = drow[al], rr = al == 0 ? r0 : (al == 1 ? r1 : r2);
                        df_mac(acc[0], acc[1], d.x, d.z, rr.x, rr.z);
                        df_mac(acc[2], acc[3], d.x, d.z, rr.y, rr.w);
                    } else {
                        dfc_mac(acc, drow[0], r0);
                        dfc_mac(acc, drow[1], r1);
                        dfc_mac(acc, drow[2], r2);
                    }
                    uu = df_result_norm(acc);
                } else {
                    uu = cfma(drow[2], r2, cfma(drow[1], r1, cfma(drow[0], r0, make_double2(0.0, 0.0))));
                }
                return uu;
            };
            auto publish = [&](const VT& uu, size_t o) {
                if (own.shared) ((VT*)P.u)[o] = uu;
                if constexpr (kSplit) uM[o] = from_c128<C>(uu);
            };
            if (!act && s_active[my_c] && s_repl[my_c])
                for_items([&](int, const Item<R>&, const int4&, size_t, size_t i) {
                    own.p[i] = from_c128<VT>(make_double2(0.0, 0.0));
                    own.s[i] = from_c128<VT>(make_double2(0.0, 0.0));
                });
            dots.clear();
            if (by_node) {
                if (act)
                    for_nodes([&](int, const int4& in, size_t o, size_t i) {
                        VT uu[3], pp[3], ss[3], xx[3], rr[3];
                        C ww[3];
#pragma unroll
                        for (int al = 0; al < 3; ++al) {
                            uu[al] = own.u[i + al * R];
                            ww[al] = ((const C*)own.w)[i + al * R];
                            pp[al] = own.p[i + al * R];
                            ss[al] = own.s[i + al * R];
                            xx[al] = own.x[i + al * R];
                            rr[al] = own.r[i + al * R];
                        }
                        const VT* drow = inverse_row(in);
#pragma unroll
                        for (int al = 0; al < 3; ++al) {
                            step(uu[al], ww[al], pp[al], ss[al], xx[al], rr[al]);
                            own.p[i + al * R] = pp[al];
                            own.s[i + al * R] = ss[al];
                            own.x[i + al * R] = xx[al];
                            own.r[i + al * R] = rr[al];
                        }
#pragma unroll
                        for (int al = 0; al < 3; ++al) {
                            const VT un = precond(in, drow + 3 * al, al, rr[0], rr[1], rr[2]);
                            own.u[i + al * R] = un;
                            publish(un, o + al * R);
                            dots.add(rr[al], un, pp[al], ss[al], P.expand);
                        }
                    });
            } else {
                if (act)
                    for_items([&](int, const Item<R>&, const int4&, size_t, size_t i) {
                        VT pp = own.p[i], ss = own.s[i], xx = own.x[i], rr = own.r[i];
                        step(own.u[i], ((const C*)own.w)[i], pp, ss, xx, rr);
                        own.p[i] = pp;
                        own.s[i] = ss;
                        own.x[i] = xx;
                        own.r[i] = rr;
                    });
                __syncthreads();
                if (act)
                    for_items([&](int, const Item<R>& it, const int4& in, size_t o, size_t i) {
                        const VT* r0 = own.r + (int64_t)i - it.al * R;
                        const VT un = precond(in, inverse_row(in) + 3 * it.al, it.al, r0[0], r0[R], r0[2 * R]);
                        own.u[i] = un;
                        publish(un, o);
                        // p and s are read again only for the expanded form: without it 32 complex64
                        // columns of the 30^3 cube take 360 us an iteration instead of 428
                        if (P.expand) dots.add(own.r[i], un, own.p[i], own.s[i], 1);
                        else dots.add(own.r[i], un, un, un, 0);
                    });
            }
        }
        FE_TRACE_MARK(6);
        if (!pat_barrier(P, passed)) goto out;
        FE_TRACE_MARK(7);
        ++trace_it;
        ++seg_it;
    }
out:
    __syncthreads();
    if (seg_end) {  // the job goes on in a later launch: keep x in its working form, save the scalars
        if (own.shared)
            for_items([&](int, const Item<R>&, const int4&, size_t o, size_t i) {
                ((VT*)P.r)[o] = own.r[i];
                ((VT*)P.u)[o] = own.u[i];
                ((VT*)P.p)[o] = own.p[i];
                ((VT*)P.s)[o] = own.s[i];
                ((VT*)P.x)[o] = own.x[i];
            });
        if (cta == 0) {
            if (tid < R) {
                ColState& cs = P.state->col[tid];
                cs.bn = s_bn[tid];
                cs.rr_ref = s_rr_ref[tid];
                cs.rel = s_rel[tid];
                cs.gam_r = s_gam_r[tid];
                cs.gam_i = s_gam_i[tid];
                cs.al_r = s_al_r[tid];
                cs.al_i = s_al_i[tid];
                cs.be_r = s_be_r[tid];
                cs.be_i = s_be_i[tid];
                cs.igam_r = s_igam_r[tid];
                cs.igam_i = s_igam_i[tid];
                cs.ial_r = s_ial_r[tid];
                cs.ial_i = s_ial_i[tid];
                cs.a4 = s_a4[tid];
                cs.na4 = s_na4[tid];
                cs.b4 = s_b4[tid];
                if constexpr (kDFV) {
                    cs.gam4 = s_gam4[tid];
                    cs.igam4 = s_igam4[tid];
                    cs.ial4 = s_ial4[tid];
                }
                cs.active = s_active[tid];
                cs.done = s_done[tid];
                cs.status = s_status[tid];
                cs.iters = s_iters[tid];
                cs.outer = s_outer[tid];
                cs.first = s_first[tid];
                cs.refresh = s_refresh[tid];
                cs.repl = s_repl[tid];
                cs.pass_it = s_pass_it[tid];
                cs.kept = s_kept[tid];
                P.rep_status[tid] = FE_PENDING;
                P.rep_iters[tid] = s_iters[tid];
                P.rep_outer[tid] = s_outer[tid];
                P.rep_rel[tid] = s_rel[tid];
            }
            if (tid == 0) {
                P.state->any_repl = s_any_repl;
                P.state->any_refresh = s_any_refresh;
                P.state->seg_done = seg_it;
                P.state->seg_ns = globaltimer_ns() - seg_t0;
                P.state->started = 1;
                P.state->finished = 0;
            }
        }
        return;
    }
    for_items([&](int, const Item<R>&, const int4&, size_t o, size_t i) { P.x[o] = to_c128(own.x[i]); });
    if (cta == 0 && tid < R) {
        P.rep_status[tid] = s_status[tid];
        P.rep_iters[tid] = s_iters[tid];
        P.rep_outer[tid] = s_outer[tid];
        P.rep_rel[tid] = s_rel[tid];
    }
    if (cta == 0 && tid == 0 && P.state) {
        P.state->seg_done = seg_it;
        P.state->seg_ns = globaltimer_ns() - seg_t0;
        P.state->started = 1;
        P.state->finished = 1;
    }
}

// One system: CTA b of the grid is CTA b of the system.
template <typename TM, int R>
__global__ void __launch_bounds__(kPT, 1) k_solve_pat(SolveParams P) {
    solve_pat_body<TM, R>(P, blockIdx.x);
}

// Several independent systems in one cooperative launch (see k_solve_jobs).
template <typename TM, int R>
__global__ void __launch_bounds__(kPT, 1)
    k_solve_pat_jobs(const SolveParams* __restrict__ jobs, const int* __restrict__ cta0, int n_jobs) {
    __shared__ __align__(16) SolveParams sP;
    __shared__ int s_job;
    if (threadIdx.x == 0) {
        int lo = 0, hi = n_jobs - 1;  // last job whose first CTA is <= blockIdx.x
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cta0[mid] <= (int)blockIdx.x) lo = mid;
            else hi = mid - 1;
        }
        s_job = lo;
    }
    __syncthreads();
    const int j = s_job;
    const int* src = (const int*)(jobs + j);
    int* dst = (int*)&sP;
    for (int i = threadIdx.x; i < (int)(sizeof(SolveParams) / sizeof(int)); i += kPT) dst[i] = src[i];
    __syncthreads();
    solve_pat_body<TM, R>(sP, (int)blockIdx.x - cta0[j]);
}

// Shared memory of a launch: the column sums, the row tables when they take at
// most kPatRowsBytes, kPatTermBytes of terms (the 10 to 20 patterns of a CTA's
// rows take about 25 KB in FP32 pairs), their diagonal inverses, and as far as
// the budget goes the staged neighbourhood of the rows (three ranges of about
// the CTA's rows and two grid lines each; a CTA whose ranges turn out longer
// reads the vector through L1) and the CTA's own vectors.
constexpr int64_t kPatRowsBytes = 64 * 1024;
constexpr int kPatTermBytes = 32 * 1024;
constexpr int64_t kPatSmem = 196 * 1024;  // dynamic; static shared memory adds up to 30 KB

template <typename T, int R>
void size_pat(SolveParams& P, int n_cta, size_t& dyn) {
    using C = typename CplxT<T>::type;
    P.n_cta = n_cta;
    P.pat_half = (int64_t)n_cta * kPatNV * R;
    P.red_bytes = (int)(kPatNV * kPW * R * sizeof(double));
    const int64_t rows = (cta_rows_bound(P.n_rows, P.cost_total, n_cta, P.cost_min, P.cost_max) + 3) & ~3ll;
    P.pat_rows_max = rows * kPatRowBytes <= kPatRowsBytes ? (int)rows : 0;
    P.pat_terms_max = kPatTermBytes / (int)sizeof(C);
    int64_t used = P.red_bytes + (((int64_t)P.pat_rows_max * kPatRowBytes + 15) & ~15ll) + kPatTermBytes +
                   9 * kPatLocal * 16;
    const int64_t vecs = rows * 3 * R;
    const int64_t halo = (3 * (rows + 2 * (int64_t)P.res_tmid + 8) * 3 * R * (int64_t)sizeof(C) + 15) & ~15ll;
    P.stage = P.pat_rows_max > 0 && used + halo <= kPatSmem ? 1 : 0;
    P.halo_bytes = P.stage ? halo : 0;
    used += P.halo_bytes;
    P.pat_vec_max = P.pat_rows_max > 0 && used + vecs * 96 <= kPatSmem ? (int)vecs : 0;
    used += (int64_t)P.pat_vec_max * 96;
    P.res_bytes = (int)(used - P.halo_bytes - P.red_bytes);
    P.res = 0;
    P.col_bytes = 0;
    dyn = (size_t)used;
}

template <typename T, int R>
fe_status launch_pat(fe_ctx* ctx, SolveParams& P) {
    const int n_cta = std::min(P.n_cta_req > 0 ? std::min(P.n_cta_req, ctx->num_sms) : ctx->num_sms, std::max(1, P.n_rows));
    size_t dyn = 0;
    size_pat<T, R>(P, n_cta, dyn);
    FE_CUDA(cudaFuncSetAttribute((const void*)k_solve_pat<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
    int per_sm = 0;
    FE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve_pat<T, R>, kPT, dyn));
    if (per_sm < 1) {
        set_error("solve kernel does not fit on an SM");
        return FE_ERR_CUDA;
    }
    void* args[] = {&P};
    FE_CUDA(cudaEventRecord(ctx->ev0, ctx->stream));
    FE_CUDA(cudaLaunchCooperativeKernel((void*)k_solve_pat<T, R>, dim3(n_cta), dim3(kPT), args, dyn, ctx->stream));
    FE_CUDA(cudaEventRecord(ctx->ev1, ctx->stream));
    count_launches(1);
    ctx->last_solve.launches += 1;
    ctx->last_solve.tile_width = R;
    ctx->last_solve.grid_ctas = n_cta;
    return FE_OK;
}

template <typename T>
fe_status dispatch_pat(fe_ctx* ctx, int R, SolveParams& P) {
    switch (R) {
        case 1: return launch_pat<T, 1>(ctx, P);
        case 2: return launch_pat<T, 2>(ctx, P);
        case 4: return launch_pat<T, 4>(ctx, P);
        case 8: return launch_pat<T, 8>(ctx, P);
        case 16: return launch_pat<T, 16>(ctx, P);
        case 32: return launch_pat<T, 32>(ctx, P);
        default: set_error("unsupported tile width %d", R); return FE_ERR_UNSUPPORTED;
    }
}

template <typename T, int R>
fe_status launch_pat_jobs_t(fe_ctx* ctx, SolveJob* const* jobs, const int* n_cta, int n, cudaStream_t stream,
                            const int* seg_iters) {
    std::vector<SolveParams> Ps(n);
    std::vector<int> cta0(n + 1, 0);
    size_t dyn = 0;
    for (int i = 0; i < n; ++i) {
        SolveParams& P = Ps[i];
        P = jobs[i]->P;
        size_t d = 0;
        size_pat<T, R>(P, n_cta[i], d);
        dyn = std::max(dyn, d);
        P.seg_iters = seg_iters ? seg_iters[i] : 0;
        cta0[i + 1] = cta0[i] + n_cta[i];
        FE_CUDA(cudaMemsetAsync(P.sync, 0, sync_bytes(P.n_cta), stream));
    }
    const int grid = cta0[n];
    DevBuf dparams, dcta;
    FE_TRY(dev_alloc(stream, dparams, (size_t)n * sizeof(SolveParams)));
    fe_status e = dev_alloc(stream, dcta, (size_t)(n + 1) * sizeof(int));
    if (e != FE_OK) {
        dev_free(stream, dparams);
        return e;
    }
    auto done = [&](fe_status st) {
        dev_free(stream, dparams);
        dev_free(stream, dcta);
        return st;
    };
    if (cudaMemcpyAsync(dparams.ptr, Ps.data(), (size_t)n * sizeof(SolveParams), cudaMemcpyHostToDevice,
                        stream) != cudaSuccess ||
        cudaMemcpyAsync(dcta.ptr, cta0.data(), (size_t)(n + 1) * sizeof(int), cudaMemcpyHostToDevice,
                        stream) != cudaSuccess) {
        set_error("jobs: parameter upload failed");
        return done(FE_ERR_CUDA);
    }
    if (cudaFuncSetAttribute((const void*)k_solve_pat_jobs<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)dyn) != cudaSuccess) {
        set_error("jobs: shared-memory attribute rejected");
        return done(FE_ERR_CUDA);
    }
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve_pat_jobs<T, R>, kPT, dyn);
    if (per_sm < 1 || grid > per_sm * ctx->num_sms) {
        set_error("jobs: %d CTAs do not fit on the device at once", grid);
        return done(FE_ERR_INVALID_ARG);
    }
    const SolveParams* pp = (const SolveParams*)dparams.ptr;
    const int* pc = (const int*)dcta.ptr;
    void* args[] = {(void*)&pp, (void*)&pc, (void*)&n};
    const cudaError_t le = cudaLaunchCooperativeKernel((void*)k_solve_pat_jobs<T, R>, dim3(grid), dim3(kPT), args, dyn,
                                                       stream);
    if (le != cudaSuccess) {
        set_error("jobs: launch failed: %s", cudaGetErrorString(le));
        return done(FE_ERR_CUDA);
    }
    count_launches(1);
    return done(FE_OK);
}

template <typename T>
fe_status launch_pat_jobs(fe_ctx* ctx, int R, SolveJob* const* jobs, const int* n_cta, int n, cudaStream_t stream,
                          const int* seg_iters) {
    switch (R) {
        case 1: return launch_pat_jobs_t<T, 1>(ctx, jobs, n_cta, n, stream, seg_iters);
        case 2: return launch_pat_jobs_t<T, 2>(ctx, jobs, n_cta, n, stream, seg_iters);
        case 4: return launch_pat_jobs_t<T, 4>(ctx, jobs, n_cta, n, stream, seg_iters);
        case 8: return launch_pat_jobs_t<T, 8>(ctx, jobs, n_cta, n, stream, seg_iters);
        case 16: return launch_pat_jobs_t<T, 16>(ctx, jobs, n_cta, n, stream, seg_iters);
        case 32: return launch_pat_jobs_t<T, 32>(ctx, jobs, n_cta, n, stream, seg_iters);
        default: set_error("jobs: unsupported tile width %d", R); return FE_ERR_UNSUPPORTED;
    }
}

}  // namespace fe
