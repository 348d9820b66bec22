// Right-hand side of Eq. 4 for incident plane waves:
//   b(W) = G(W, H_i) - int_Sext W . (n x curl H_i) ds,
// with G the weak Engquist-Majda form of Eq. 3 (the same integrated-by-parts
// form as the left-hand side) and H_i = p_hat H0 exp(-j k0 k_hat . r),
// curl H_i = -j k0 k_hat x H_i.  On an axis-aligned face the 2 x 2 Gauss sums
// of a node's hat (or of its tangential gradient) times the wave's phase are
// products of one-dimensional sums, so a first kernel tabulates those per
// wave, axis and grid position (k_rhs_axis: eight phases each), and one thread
// per (active node, wave) multiplies three table entries per face: a sine and
// cosine in FP64 take this GPU some two hundred operations at a sixty-fourth
// of the FP32 rate, and the direct sums needed sixteen pairs per face node
// (719 us for 4 waves on 51^3 nodes).  The sums are deterministic and
// atomic-free.
#include "fe_internal.cuh"

namespace fe {

struct Wave {
    double k[3], p[3];
    double ar, ai;
};

// One-dimensional sums of wave w at position i of an axis: over the (up to)
// two elements beside it and two Gauss points each,
//     val = sum (h/2) N e^{-j k0 k x},  grad = sum (h/2) N' e^{-j k0 k x},
// and the phase at the position itself.
struct AxisSum {
    double2 val, grad, at;
};

// cos and sin of -k0 k (org + (e + xi) h), the angle carried as an unevaluated
// pair of doubles (Dekker's and Knuth's error-free product and sum).  A product
// of three such phases would otherwise hold three rounded angles where the
// direct sum held one; with the pairs it holds none, and the right-hand side of
// 50^3 elements is off by 1.9e-16 to 2.6e-16 of its norm (plain angles 6.8e-16 to 1.5e-15, the
// direct sums 6.4e-16 to 1.1e-15), at any distance from the origin.
__device__ double2 phase(double k0, double k, double org, double e, double xi, double h) {
    auto mul = [](double a, double b, double& lo) {
        const double p = __dmul_rn(a, b);
        lo = __fma_rn(a, b, -p);
        return p;
    };
    auto add = [](double a, double b, double& lo) {
        const double s = __dadd_rn(a, b), t = __dsub_rn(s, a);
        lo = __dadd_rn(__dsub_rn(a, __dsub_rn(s, t)), __dsub_rn(b, t));
        return s;
    };
    double l0, l1, l2, l3, cl, al;
    const double eh = mul(e, h, l0), xh = mul(xi, h, l1), ch = mul(-k0, k, cl);
    const double x = add(add(eh, org, l2), xh, l3), xl = (l0 + l1) + (l2 + l3);
    const double a = mul(ch, x, al);
    al += ch * xl + cl * x;
    double sn, cs;
    sincos(a, &sn, &cs);
    return make_double2(cs - al * sn, sn + al * cs);
}

__global__ void k_rhs_axis(int nx, int ny, int nz, double hx, double hy, double hz, double ox, double oy, double oz,
                           double k0, const Wave* __restrict__ waves, int nrhs, AxisSum* __restrict__ tab) {
    const int len = nx + ny + nz + 3;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)len * nrhs) return;
    const int w = (int)(t / len);
    int i = (int)(t - (int64_t)w * len), axis = 0, n = nx;
    double h = hx, org = ox;
    if (i > nx) {
        i -= nx + 1;
        axis = 1;
        n = ny;
        h = hy;
        org = oy;
        if (i > ny) {
            i -= ny + 1;
            axis = 2;
            n = nz;
            h = hz;
            org = oz;
        }
    }
    const double k = waves[w].k[axis];
    const double g0 = 0.5 - 0.5 / sqrt(3.0), g1 = 0.5 + 0.5 / sqrt(3.0);
    AxisSum s;
    s.val = s.grad = make_double2(0.0, 0.0);
    for (int e = i - 1; e <= i; ++e) {
        if (e < 0 || e >= n) continue;
        const bool up = e == i - 1;  // the node is the element's upper end
        for (int q = 0; q < 2; ++q) {
            const double xi = q ? g1 : g0;
            const double2 p = phase(k0, k, org, e, xi, h);
            const double f = 0.5 * h * (up ? xi : 1.0 - xi), g = up ? 0.5 : -0.5;
            s.val.x += f * p.x;
            s.val.y += f * p.y;
            s.grad.x += g * p.x;
            s.grad.y += g * p.y;
        }
    }
    s.at = phase(k0, k, org, i, 0.0, h);
    tab[t] = s;
}

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__global__ void k_rhs(int nx, int ny, int nz, double k0, double sigma, const int* __restrict__ node_id, int n_act,
                      const Wave* __restrict__ waves, const AxisSum* __restrict__ tab, int nrhs, unsigned abc,
                      unsigned planes, const uint8_t* __restrict__ mat, int form_e, double2* __restrict__ B) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n_act * nrhs) return;
    const int r = (int)(t / nrhs), w = (int)(t - (int64_t)r * nrhs);
    const int id = node_id[r];
    const int c[3] = {id % (nx + 1), (id / (nx + 1)) % (ny + 1), id / ((nx + 1) * (ny + 1))};
    const int dim[3] = {nx, ny, nz};
    double br[3] = {0, 0, 0}, bi[3] = {0, 0, 0};
    if (c[0] == 0 || c[0] == nx || c[1] == 0 || c[1] == ny || c[2] == 0 || c[2] == nz) {
        const Wave wv = waves[w];
        const AxisSum* tw = tab + (size_t)w * (nx + ny + nz + 3);
        const int first[3] = {0, nx + 1, nx + ny + 2};
#pragma unroll
        for (int f = 0; f < 6; ++f) {
            const int nu = f >> 1, side = f & 1;
            if (c[nu] != (side ? dim[nu] : 0) || !((abc >> f) & 1u)) continue;  // absorbing faces only
            const int t1 = nu == 0 ? 1 : 0, t2 = nu == 2 ? 1 : 2;
            const AxisSum& a1 = tw[first[t1] + c[t1]];
            const AxisSum& a2 = tw[first[t2] + c[t2]];
            const double2 e = zmul(make_double2(wv.ar, wv.ai), tw[first[nu] + c[nu]].at);
            const double2 v1 = zmul(a1.val, e);
            const double2 val = zmul(v1, a2.val);                    // int N e^{-j k0 k.r}
            const double2 d1 = zmul(zmul(a1.grad, e), a2.val), d2 = zmul(v1, a2.grad);
            const double gr = wv.k[t1] * d1.x + wv.k[t2] * d2.x;     // int (grad_t N . k_hat) e^{-j k0 k.r}
            const double gi = wv.k[t1] * d1.y + wv.k[t2] * d2.y;
            const double nsgn = side ? 1.0 : -1.0;
            const double nk = nsgn * wv.k[nu], np = nsgn * wv.p[nu];  // n . k_hat, n . p_hat
#pragma unroll
            for (int al = 0; al < 3; ++al) {
                // -N (n x curl H_i) = j k0 N (k_hat (n.H_i) - H_i (n.k_hat)), and for the tangential
                // components j k0 N H_al + sigma (j / 2k0)(grad_t N . (-j k0 k_t)) H_al
                double u = wv.k[al] * np - wv.p[al] * nk;
                if (al != nu) {
                    u += wv.p[al];
                    br[al] += 0.5 * sigma * wv.p[al] * gr;
                    bi[al] += 0.5 * sigma * wv.p[al] * gi;
                }
                br[al] -= k0 * u * val.y;
                bi[al] += k0 * u * val.x;
            }
        }
    }
    // held by symmetry planes (and, for E, on conductor surfaces)
    unsigned fix = fixed_components(c[0], c[1], c[2], nx, ny, nz, planes);
    if (form_e) fix |= pec_held(mat, nx, ny, nz, c[0], c[1], c[2]);
    for (int al = 0; al < 3; ++al)
        B[((int64_t)3 * r + al) * nrhs + w] = (fix >> al) & 1u ? make_double2(0.0, 0.0) : make_double2(br[al], bi[al]);
}

fe_status build_rhs(fe_ctx* ctx, const fe_system* s, int nrhs, const fe_planewave* waves, double2* d_B,
                    DevBuf& wave_buf) {
    const fe_mesh* m = s->mesh;
    cudaStream_t st = ctx->stream;
    std::vector<Wave> hw(nrhs);
    for (int w = 0; w < nrhs; ++w) {
        for (int d = 0; d < 3; ++d) {
            hw[w].k[d] = waves[w].k_hat[d];
            hw[w].p[d] = waves[w].p_hat[d];
        }
        hw[w].ar = waves[w].amplitude.re;
        hw[w].ai = waves[w].amplitude.im;
    }
    // the waves, then the axis tables (16-byte aligned behind them)
    const int len = m->nx + m->ny + m->nz + 3;
    const size_t tab_at = ((size_t)nrhs * sizeof(Wave) + 15) & ~(size_t)15;
    FE_TRY(dev_alloc(st, wave_buf, tab_at + (size_t)nrhs * len * sizeof(AxisSum)));
    FE_CUDA(cudaMemcpyAsync(wave_buf.ptr, hw.data(), (size_t)nrhs * sizeof(Wave), cudaMemcpyHostToDevice, st));
    AxisSum* tab = (AxisSum*)((char*)wave_buf.ptr + tab_at);
    k_rhs_axis<<<(unsigned)(((int64_t)len * nrhs + 63) / 64), 64, 0, st>>>(
        m->nx, m->ny, m->nz, m->h[0], m->h[1], m->h[2], m->origin[0], m->origin[1], m->origin[2], s->k0,
        (const Wave*)wave_buf.ptr, nrhs, tab);
    FE_LAUNCHED();
    const int64_t n = (int64_t)m->n_act * nrhs;
    k_rhs<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(m->nx, m->ny, m->nz, s->k0, s->sigma,
                                                       (const int*)m->node_id.ptr, m->n_act,
                                                       (const Wave*)wave_buf.ptr, tab, nrhs, abc_faces(m->boundary),
                                                       pack_planes(m->boundary), (const uint8_t*)m->material.ptr,
                                                       s->formulation == FE_FORMULATION_E ? 1 : 0, d_B);
    FE_LAUNCHED();
    // the host staging vector must outlive the copy
    FE_CUDA(cudaStreamSynchronize(st));
    return FE_OK;
}

}  // namespace fe

using namespace fe;

extern "C" fe_status fe_rhs(fe_ctx* ctx, const fe_system* s, int32_t nrhs, const fe_planewave* waves, void* b_out,
                            int32_t on_device) {
    if (!ctx || !s || !waves || !b_out || nrhs < 1) {
        set_error("fe_rhs: NULL argument or nrhs < 1");
        return FE_ERR_INVALID_ARG;
    }
    cudaSetDevice(ctx->device);
    cudaStream_t st = ctx->stream;
    const size_t bytes = (size_t)3 * s->mesh->n_act * nrhs * sizeof(double2);
    DevBuf wb, tmp;
    double2* dB = (double2*)b_out;
    if (!on_device) {
        fe_status e = dev_alloc(st, tmp, bytes);
        if (e != FE_OK) return e;
        dB = (double2*)tmp.ptr;
    }
    fe_status e = build_rhs(ctx, s, nrhs, waves, dB, wb);
    if (e == FE_OK && !on_device) {
        cudaError_t ce = cudaMemcpyAsync(b_out, dB, bytes, cudaMemcpyDeviceToHost, st);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
        if (ce != cudaSuccess) {
            set_error("fe_rhs copy: %s", cudaGetErrorString(ce));
            e = FE_ERR_CUDA;
        }
    }
    dev_free(st, wb);
    dev_free(st, tmp);
    return e;
}
