// Construction of the row patterns (patterns.cuh) of a system.
//
// The blocks of a row follow from its surroundings alone: the materials of
// the eight elements around the node, whether the node (and, where held
// components or the penalty surface term reach further, its neighbours) lies
// on a face of the box, and then also which of the 4 x 4 x 4 elements around
// it are PEC.  Those are at most 140 bits, a row's key; the gather assembly
// sums in a fixed order, so rows of equal keys get bitwise equal blocks.
// Rows are grouped by a hash of the key in an open-addressing table (one
// insertion per distinct hash and warp), the groups numbered by their first
// row (deterministic), every row's key compared with its group's first row's,
// the first rows assembled, and the others copy them.  A table overflow, more
// than pat_limit groups or a key that differs from its group's leaves the system
// without patterns: every row is then assembled by itself and the products
// read the stored blocks.  Bound by launches and dependent loads, but for the
// copies (k_pat_spread: two stored forms of 51^3 rows, 1 GB).  Mesh, assembly,
// four right-hand sides and a product of 51^3 nodes: 7.5 ms with every row
// assembled, 1.6 ms with the first rows only, 0.75 ms with the right-hand side
// and the other set-up kernels shortened.
#include "patterns.cuh"

#include <algorithm>

namespace fe {

namespace {

constexpr int kPatProbes = 64;

// What the values of a row depend on (variant S of the H formulation without
// symmetry planes: `far` = 0, only the eight elements and the faces the node
// lies on; else the wider surroundings).
struct RowKey {
    unsigned long long mat;  // material byte of the eight elements (255 PEC, 254 outside the box)
    unsigned long long pec;  // far: which of the 4 x 4 x 4 elements around are PEC
    unsigned pos;            // per axis, distance to either end of the box, capped at 1 (far: 2)
};

__device__ __forceinline__ RowKey row_key(const uint8_t* __restrict__ mat, int nx, int ny, int nz, int id, int far) {
    const int i = id % (nx + 1), j = (id / (nx + 1)) % (ny + 1), k = id / ((nx + 1) * (ny + 1));
    RowKey key{0, 0, 0};
    auto at = [&](int a, int b, int c) -> unsigned {
        if (a < 0 || a >= nx || b < 0 || b >= ny || c < 0 || c >= nz) return 254u;
        return mat[a + (int64_t)nx * (b + (int64_t)ny * c)];
    };
#pragma unroll
    for (int e = 0; e < 8; ++e)
        key.mat |= (unsigned long long)at(i - 1 + (e & 1), j - 1 + ((e >> 1) & 1), k - 1 + (e >> 2)) << (8 * e);
    const int cap = far ? 2 : 1;
    key.pos = min(i, cap) | min(nx - i, cap) << 2 | min(j, cap) << 4 | min(ny - j, cap) << 6 | min(k, cap) << 8 |
              min(nz - k, cap) << 10;
    if (far)
        for (int e = 0; e < 64; ++e)
            key.pec |= (unsigned long long)(at(i - 2 + (e & 3), j - 2 + ((e >> 2) & 3), k - 2 + (e >> 4)) == kPEC) << e;
    return key;
}

// Writes the rows' keys and groups them by key hash: keys/first are the table,
// slot_of[r] the row's entry.  flags[0] counts groups, flags[1] reports an
// overflow.  Once there are more than `limit` groups no row need insert, and a
// warp counts its new groups in one addition: a mesh without patterns makes a
// group of nearly every row, and 68 921 of them took 60 us one by one (set-up
// of 40^3 random materials in FP64 1.71 ms so, 1.67 ms now, 1.69 ms with every
// row assembled and no grouping).
__global__ void k_pat_insert(const uint8_t* __restrict__ mat, int nx, int ny, int nz, const int* __restrict__ node_id,
                             int n, int far, int limit, RowKey* __restrict__ row_keys,
                             unsigned long long* __restrict__ keys, int* __restrict__ first,
                             int* __restrict__ slot_of, int* __restrict__ flags) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned live = __ballot_sync(0xffffffffu, r < n);
    if (r >= n) return;
    const RowKey rk = row_key(mat, nx, ny, nz, node_id[r], far);
    row_keys[r] = rk;
    const unsigned long long h = mix64(mix64(rk.mat + 0x9e3779b97f4a7c15ull * (rk.pos + 1u)) ^ rk.pec) | 1ull;  // 0: empty
    const unsigned same = __match_any_sync(live, h);
    const int lane = threadIdx.x & 31, leader = __ffs(same) - 1;  // lowest lane, lowest row
    int slot = -1;
    bool created = false, full = false;
    if (lane == leader) {
        unsigned t = (unsigned)(h >> 51);
        full = true;
        for (int probe = 0; probe < kPatProbes; ++probe, t = (t + 1) & (kPatHash - 1)) {
            if (probe % 8 == 0 && __ldcg(flags) > limit) {
                full = false;  // (too many groups anyway)
                break;
            }
            unsigned long long k = __ldcg(keys + t);
            if (k == 0ull) {
                k = atomicCAS(keys + t, 0ull, h);
                if (k == 0ull) {
                    created = true;
                    k = h;
                }
            }
            if (k == h) {
                if (__ldcg(first + t) > r) atomicMin(first + t, r);
                slot = (int)t;
                full = false;
                break;
            }
        }
    }
    const unsigned made = __ballot_sync(live, created), over = __ballot_sync(live, full);
    if (lane == 0) {
        if (made) atomicAdd(flags, __popc(made));
        if (over) atomicExch(flags + 1, 1);
    }
    slot_of[r] = __shfl_sync(same, slot, leader);
}

// Numbers the occupied entries by their first row (one block).  More than
// `limit` of them are marked in flags[1] like an overflow.
__global__ void __launch_bounds__(1024) k_pat_number(const unsigned long long* __restrict__ keys,
                                                     const int* __restrict__ first, int limit,
                                                     int* __restrict__ id_of_slot, int* __restrict__ first_of_id,
                                                     int* __restrict__ flags) {
    __shared__ int s_first[kMaxPat], s_slot[kMaxPat], s_n;
    if (flags[1] || flags[0] > limit) {
        if (threadIdx.x == 0) flags[1] = 1;
        return;
    }
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < kPatHash; t += blockDim.x)
        if (keys[t]) {
            const int i = atomicAdd(&s_n, 1);  // below limit <= kMaxPat
            s_first[i] = first[t];
            s_slot[i] = t;
        }
    __syncthreads();
    const int n = s_n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        int id = 0;
        const int f = s_first[i];
        for (int j = 0; j < n; ++j) id += s_first[j] < f;
        id_of_slot[s_slot[i]] = id;
        first_of_id[id] = f;
    }
}

__device__ __forceinline__ void put_term(double2* p, double v, int code) {
    *p = make_double2(v, __hiloint2double(0, code));
}
__device__ __forceinline__ void put_term(float2* p, double v, int code) {
    *p = make_float2(__double2float_rn(v), __int_as_float(code));
}
__device__ __forceinline__ void put_term(float4* p, double v, int code) {
    const float h = __double2float_rn(v);
    *p = make_float4(h, __double2float_rn(v - (double)h), __int_as_float(code), 0.f);
}

// Term lists of one pattern per block, one warp per component: lane k < nb
// holds the component's three entries of block k.  A part is left out only
// where the stored one is zero: the contributions of a uniform material that
// cancel do so exactly (they are the same table entries with opposite signs),
// and any other part is data however small it is beside the row's largest (a
// loss tangent of 1e-17 alone makes the imaginary parts).  NaN is not zero.
__global__ void __launch_bounds__(96) k_pat_terms(const int* __restrict__ first_of_id, const int* __restrict__ row_ptr,
                                                  const int* __restrict__ col, const int* __restrict__ node_id,
                                                  const double2* __restrict__ val, int64_t stride, int sy, int sz,
                                                  int4* __restrict__ tab, double2* __restrict__ t64,
                                                  float2* __restrict__ t32, float4* __restrict__ tdf, int cost_shift,
                                                  int* __restrict__ flags) {
    __shared__ int s_nre[3], s_nim[3], s_diag[3];
    const int p = blockIdx.x, al = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = first_of_id[p], s0 = row_ptr[row], nb = row_ptr[row + 1] - s0;
    double2 v[3];
    int line = 0, dx = 0;
#pragma unroll
    for (int be = 0; be < 3; ++be) v[be] = make_double2(0.0, 0.0);
    if (lane < nb) {
#pragma unroll
        for (int be = 0; be < 3; ++be) v[be] = val[(3 * al + be) * stride + s0 + lane];
        // grid offset of the column, split into (dx, dy, dz) by the extents
        const int id = node_id[row], o = node_id[col[s0 + lane]];
        dx = o % sy - id % sy;
        line = ((o / sy) % (sz / sy) - (id / sy) % (sz / sy) + 1) + 3 * (o / sz - id / sz + 1);
    }
    bool re[3], im[3], offdiag = false;
    int cre = 0, cim = 0;
#pragma unroll
    for (int be = 0; be < 3; ++be) {
        re[be] = !(v[be].x == 0.0);
        im[be] = !(v[be].y == 0.0);
        cre += re[be];
        cim += im[be];
        offdiag = offdiag || im[be] || (be != al && re[be]);
    }
    const bool diag_row = !__any_sync(0xffffffffu, offdiag) && nb == 27;
    // exclusive prefix of the counts over the lanes (blocks in grid order)
    int pre = cre, pim = cim;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, pre, o), b = __shfl_up_sync(0xffffffffu, pim, o);
        if (lane >= o) {
            pre += a;
            pim += b;
        }
    }
    const int nre = __shfl_sync(0xffffffffu, pre, 31), nim = __shfl_sync(0xffffffffu, pim, 31);
    pre -= cre;
    pim -= cim;
    // the row's own block goes last, its own component last of all
    const bool own = lane < nb && line == 4 && dx == 0;
    const int own_lane = __ffs(__ballot_sync(0xffffffffu, own)) - 1;
    const int own_re = __shfl_sync(0xffffffffu, cre, own_lane), own_im = __shfl_sync(0xffffffffu, cim, own_lane);
    if (own) {
        pre = nre - cre;
        pim = nim - cim;
    } else if (lane > own_lane) {
        pre -= own_re;
        pim -= own_im;
    }
    if (lane == 0) {
        s_nre[al] = nre;
        s_nim[al] = nim;
        s_diag[al] = diag_row;
    }
    __syncthreads();
    const bool diag = s_diag[0] && s_diag[1] && s_diag[2];
    const int n_re = diag ? 27 : max(s_nre[0], max(s_nre[1], s_nre[2]));
    const int n_im = diag ? 0 : max(s_nim[0], max(s_nim[1], s_nim[2]));
    const size_t base = (size_t)p * kPatStride * 3 + al;
    auto put = [&](int t, double w, int code) {
        put_term(t64 + base + 3 * t, w, code);
        if (t32) put_term(t32 + base + 3 * t, w, code);
        if (tdf) put_term(tdf + base + 3 * t, w, code);
    };
    if (diag) {
        if (lane < 27) {
            const double w = al == 0 ? v[0].x : (al == 1 ? v[1].x : v[2].x);
            put(lane, w, pack_code(line, 3 * dx + al));
            put(27 + (lane == 13 ? 26 : lane - (lane > 13)), w, pack_code(line, 3 * dx + al));  // own entry last
        }
    } else {
        if (lane < nb) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {  // beta = 0, 1, 2 but alpha, then alpha
                const int be = q < 3 ? q : al;
                if (q < 3 && q == al) continue;
                const bool r = be == 0 ? re[0] : (be == 1 ? re[1] : re[2]), i = be == 0 ? im[0] : (be == 1 ? im[1] : im[2]);
                const double2 e = be == 0 ? v[0] : (be == 1 ? v[1] : v[2]);
                if (r) put(pre++, e.x, pack_code(line, 3 * dx + be));
                if (i) put(n_re + pim++, e.y, pack_code(line, 3 * dx + be));
            }
        }
        // padding: zero weights on the row's own node
        for (int t = nre + lane; t < n_re; t += 32) put(t, 0.0, pack_code(4, 0));
        for (int t = nim + lane; t < n_im; t += 32) put(n_re + t, 0.0, pack_code(4, 0));
    }
    if (threadIdx.x == 0) {
        tab[p] = make_int4(p * kPatStride, n_re, n_im, diag ? 1 : 0);
        const int cost = scaled_cost(row_cost(n_re, n_im, diag), cost_shift);
        atomicMin(flags + 3, cost);
        atomicMax(flags + 4, cost);
    }
}

// Group of every row; a key that differs from its group's first row's (a hash
// collision) is reported in flags[2].
__global__ void k_pat_group(const RowKey* __restrict__ keys, const int* __restrict__ slot_of,
                            const int* __restrict__ id_of_slot, const int* __restrict__ first_of_id, int n,
                            int* __restrict__ group, int* __restrict__ flags) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n || flags[1]) return;
    const int id = id_of_slot[slot_of[r]];
    const RowKey a = keys[r], b = keys[first_of_id[id]];
    if (a.mat != b.mat || a.pec != b.pec || a.pos != b.pos) atomicExch(flags + 2, 1);
    group[r] = id;
}

template <typename C>
__device__ __forceinline__ void copy_block(C* val, int64_t stride, int64_t from, int64_t to) {
    C v[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q] = val[q * stride + from];
#pragma unroll
    for (int q = 0; q < 9; ++q) val[q * stride + to] = v[q];
}

// One warp per row: copies the blocks of its pattern's first row (planes in
// every arithmetic, and the diagonal inverse) and writes its pattern, cost and
// whether it is explicit (not of real diagonal blocks).  Bound by the stores,
// 288 bytes a block with two arithmetics.
__global__ void __launch_bounds__(256) k_pat_spread(const int* __restrict__ group, const int* __restrict__ first_of_id,
                                                    const int4* __restrict__ tab, const int* __restrict__ row_ptr,
                                                    int64_t stride, int n, double2* __restrict__ val64,
                                                    float2* __restrict__ val32, float4* __restrict__ valdf,
                                                    double2* __restrict__ dinv64, float2* __restrict__ dinv32,
                                                    float4* __restrict__ dinvdf, const int* __restrict__ node_id,
                                                    uint16_t* __restrict__ pat_id, int4* __restrict__ pat_row,
                                                    int cost_shift, int* __restrict__ cost, int* __restrict__ expl) {
    const int r = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (r >= n) return;
    const int id = __ldg(group + r);
    const int f = __ldg(first_of_id + id);
    if (f != r) {
        const int s0 = __ldg(row_ptr + r), nb = __ldg(row_ptr + r + 1) - s0, f0 = __ldg(row_ptr + f);
        if (lane < nb) {
            copy_block(val64, stride, f0 + lane, s0 + lane);
            if (val32) copy_block(val32, stride, f0 + lane, s0 + lane);
            if (valdf) copy_block(valdf, stride, f0 + lane, s0 + lane);
        }
        if (lane < 9) {
            dinv64[(size_t)9 * r + lane] = dinv64[(size_t)9 * f + lane];
            if (dinv32) dinv32[(size_t)9 * r + lane] = dinv32[(size_t)9 * f + lane];
            if (dinvdf) dinvdf[(size_t)9 * r + lane] = dinvdf[(size_t)9 * f + lane];
        }
    }
    if (lane == 0) {
        const int4 t = __ldg(tab + id);
        pat_id[r] = (uint16_t)id;
        pat_row[r] = make_int4(3 * t.x, t.y | t.z << 10 | t.w << 20, __ldg(node_id + r), id);
        cost[r] = scaled_cost(row_cost(t.y, t.z, t.w != 0), cost_shift);
        expl[r] = t.w ? 0 : 1;
    }
}

// List of the explicit rows, ascending, from the scanned flags (pos[n] = total).
__global__ void k_pat_list(const uint16_t* __restrict__ pat_id, const int4* __restrict__ tab,
                           const int* __restrict__ pos, int n, int* __restrict__ list) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n && !__ldg(&tab[pat_id[r]].w)) list[pos[r]] = r;
}

}  // namespace

// Groups the rows of a system by their surroundings.  With few enough groups
// n_pat is set, pat_first lists the groups' first rows and row_group (device)
// has every row's group; else n_pat stays 0.
fe_status group_rows(fe_ctx* ctx, fe_system* s, DevBuf& row_group, int* d_flags) {
    const fe_mesh* m = s->mesh;
    cudaStream_t st = ctx->stream;
    const int n = m->n_act;
    DevBuf keys, first, slot_of, id_of_slot, row_keys;
    auto done = [&](fe_status e) {
        for (DevBuf* b : {&keys, &first, &slot_of, &id_of_slot, &row_keys}) dev_free(st, *b);
        return e;
    };
    fe_status e;
    if ((e = dev_alloc(st, keys, kPatHash * sizeof(unsigned long long))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, first, kPatHash * sizeof(int))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, slot_of, (size_t)n * sizeof(int))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, id_of_slot, kPatHash * sizeof(int))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, row_keys, (size_t)n * sizeof(RowKey))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, row_group, (size_t)n * sizeof(int))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, s->pat_first, kMaxPat * sizeof(int))) != FE_OK) return done(e);
    cudaMemsetAsync(keys.ptr, 0, kPatHash * sizeof(unsigned long long), st);
    cudaMemsetAsync(first.ptr, 0x7f, kPatHash * sizeof(int), st);
    cudaMemsetAsync(d_flags, 0, 3 * sizeof(int), st);
    // variant S adds nothing on PEC faces and its boundary form couples nodes
    // of one face only; the other variants, symmetry planes and the E
    // formulation's held components look one element further
    const int far = s->variant != FE_VARIANT_S || s->formulation == FE_FORMULATION_E || pack_planes(m->boundary) != 0;
    const unsigned grid = (unsigned)((n + 255) / 256);
    const int limit = pat_limit(m->n_nodes_total);
    k_pat_insert<<<grid, 256, 0, st>>>((const uint8_t*)m->material.ptr, m->nx, m->ny, m->nz,
                                       (const int*)m->node_id.ptr, n, far, limit, (RowKey*)row_keys.ptr,
                                       (unsigned long long*)keys.ptr, (int*)first.ptr, (int*)slot_of.ptr, d_flags);
    k_pat_number<<<1, 1024, 0, st>>>((const unsigned long long*)keys.ptr, (const int*)first.ptr, limit,
                                     (int*)id_of_slot.ptr, (int*)s->pat_first.ptr, d_flags);
    k_pat_group<<<grid, 256, 0, st>>>((const RowKey*)row_keys.ptr, (const int*)slot_of.ptr,
                                      (const int*)id_of_slot.ptr, (const int*)s->pat_first.ptr, n,
                                      (int*)row_group.ptr, d_flags);
    count_launches(3);
    int* h = ctx->h_small + 40;
    cudaMemcpyAsync(h, d_flags, 3 * sizeof(int), cudaMemcpyDeviceToHost, st);
    cudaError_t ce = cudaStreamSynchronize(st);
    if (ce == cudaSuccess) ce = cudaGetLastError();
    if (ce != cudaSuccess) {
        set_error("row patterns (grouping): %s", cudaGetErrorString(ce));
        return done(FE_ERR_CUDA);
    }
    if (!h[1] && !h[2] && h[0] >= 1 && h[0] <= limit) s->n_pat = h[0];
    return done(FE_OK);
}

// Term lists and row tables of a grouped system whose groups' first rows are
// assembled.  Least and largest cost are left in d_flags[3] and [4], the
// sums over the rows (cost, explicit rows) in d_totals, for the caller's next
// synchronisation.
fe_status build_patterns(fe_ctx* ctx, fe_system* s, const DevBuf& row_group, int* d_flags, int* d_totals) {
    const fe_mesh* m = s->mesh;
    cudaStream_t st = ctx->stream;
    const int n = m->n_act, n_pat = s->n_pat;
    DevBuf expl;
    auto done = [&](fe_status e) {
        dev_free(st, expl);
        return e;
    };
    fe_status e;
    const size_t triples = (size_t)n_pat * kPatStride;
    if ((e = dev_alloc(st, s->pat_id, (size_t)n * sizeof(uint16_t))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, s->pat_row, (size_t)n * sizeof(int4))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, s->pat_tab, (size_t)n_pat * sizeof(int4))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, s->pat_t64, triples * 3 * sizeof(double2))) != FE_OK) return done(e);
    if (s->val32.ptr && (e = dev_alloc(st, s->pat_t32, triples * 3 * sizeof(float2))) != FE_OK) return done(e);
    if (s->valdf.ptr && (e = dev_alloc(st, s->pat_tdf, triples * 3 * sizeof(float4))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, s->pat_cost, (size_t)(n + 1) * sizeof(int))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, s->pat_list, (size_t)n * sizeof(int))) != FE_OK) return done(e);
    if ((e = dev_alloc(st, expl, (size_t)n * sizeof(int))) != FE_OK) return done(e);
    const int sy = m->nx + 1, sz = (m->nx + 1) * (m->ny + 1);
    const int shift = cost_shift(n);
    const int* rp = (const int*)m->row_ptr.ptr;
    const int* first = (const int*)s->pat_first.ptr;
    int* cost = (int*)s->pat_cost.ptr;
    cudaMemsetAsync(d_flags + 3, 0x7f, sizeof(int), st);
    cudaMemsetAsync(d_flags + 4, 0, sizeof(int), st);
    k_pat_terms<<<n_pat, 96, 0, st>>>(first, rp, (const int*)m->col_idx.ptr, (const int*)m->node_id.ptr,
                                      (const double2*)s->val64.ptr, s->stride, sy, sz, (int4*)s->pat_tab.ptr,
                                      (double2*)s->pat_t64.ptr, (float2*)s->pat_t32.ptr, (float4*)s->pat_tdf.ptr,
                                      shift, d_flags);
    k_pat_spread<<<(unsigned)(((int64_t)n * 32 + 255) / 256), 256, 0, st>>>(
        (const int*)row_group.ptr, first, (const int4*)s->pat_tab.ptr, rp, s->stride, n, (double2*)s->val64.ptr,
        (float2*)s->val32.ptr, (float4*)s->valdf.ptr, (double2*)s->dinv64.ptr, (float2*)s->dinv32.ptr,
        (float4*)s->dinvdf.ptr, (const int*)m->node_id.ptr, (uint16_t*)s->pat_id.ptr,
        (int4*)s->pat_row.ptr, shift, cost, (int*)expl.ptr);
    count_launches(2);
    if ((e = scan_exclusive(st, cost, cost, n, d_totals, ctx->scan_tmp)) != FE_OK) return done(e);
    cudaMemcpyAsync(cost + n, d_totals, sizeof(int), cudaMemcpyDeviceToDevice, st);
    if ((e = scan_exclusive(st, (const int*)expl.ptr, (int*)expl.ptr, n, d_totals + 1, ctx->scan_tmp)) != FE_OK)
        return done(e);
    k_pat_list<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const uint16_t*)s->pat_id.ptr,
                                                            (const int4*)s->pat_tab.ptr, (const int*)expl.ptr, n,
                                                            (int*)s->pat_list.ptr);
    count_launches(1);
    const cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) {
        set_error("row patterns (terms): %s", cudaGetErrorString(ce));
        return done(FE_ERR_CUDA);
    }
    return done(FE_OK);
}

void drop_patterns(fe_system* s) {
    cudaStream_t st = s->ctx->stream;
    for (DevBuf* b : {&s->pat_first, &s->pat_id, &s->pat_row, &s->pat_tab, &s->pat_t64, &s->pat_t32, &s->pat_tdf, &s->pat_cost,
                      &s->pat_list})
        dev_free(st, *b);
    s->n_pat = 0;
}

}  // namespace fe
