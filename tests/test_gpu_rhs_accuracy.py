"""The right-hand side against the same 2 x 2 Gauss sums in extended precision,
near the origin and many wavelengths away from it.

Bound on the norm of the error, in units of u = 2^-53: a one-dimensional sum
holds at most four phases (3 u of sine and cosine, 3 u of weight and product,
3 u of addition, the angle itself being carried to about 2^-100), three of them
make a node's value (27 u), with three complex products (7 u) and the sums over
components and faces (6 u): below 45 u = 5e-15 wherever the box lies."""
import numpy as np
import pytest

from paper_0704_2344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LD, CLD = np.longdouble, np.clongdouble


def _direct(prob, waves):
    """b [n_dof, R] of a box without conductors, face by face in extended precision (absorbing faces, sigma = 1)."""
    dim = (prob.nx, prob.ny, prob.nz)
    h, org = [LD(v) for v in prob.h], [LD(v) for v in prob.origin]
    k0 = LD(2.0 * np.pi * prob.freq_hz / W.C0)
    gauss = [LD(0.5) - LD(0.5) / np.sqrt(LD(3)), LD(0.5) + LD(0.5) / np.sqrt(LD(3))]
    b = np.zeros((dim[2] + 1, dim[1] + 1, dim[0] + 1, 3, waves.count), CLD)
    for r in range(waves.count):
        k, p = [LD(v) for v in waves.k_hat[r]], [LD(v) for v in waves.p_hat[r]]
        amp = CLD(waves.amplitude[r])
        for f in range(6):
            nu, side = f >> 1, f & 1
            t1, t2 = [a for a in range(3) if a != nu]
            sign = LD(1 if side else -1)
            n1, n2 = dim[t1] + 1, dim[t2] + 1
            val, grad = np.zeros((n1, n2), CLD), np.zeros((n1, n2), CLD)
            for s1 in range(2):
                for s2 in range(2):
                    e1, e2 = np.arange(n1) - 1 + s1, np.arange(n2) - 1 + s2
                    on = ((e1 >= 0) & (e1 < dim[t1]))[:, None] & ((e2 >= 0) & (e2 < dim[t2]))[None, :]
                    for q in range(4):
                        x1, x2 = gauss[q & 1], gauss[q >> 1]
                        f1, f2 = (1 - x1 if s1 else x1), (1 - x2 if s2 else x2)
                        gk = (-1 if s1 else 1) / h[t1] * f2 * k[t1] + (-1 if s2 else 1) / h[t2] * f1 * k[t2]
                        pos = [None] * 3
                        pos[nu] = org[nu] + (dim[nu] if side else 0) * h[nu]
                        pos[t1] = (org[t1] + (e1.astype(LD) + x1) * h[t1])[:, None]
                        pos[t2] = (org[t2] + (e2.astype(LD) + x2) * h[t2])[None, :]
                        ph = -k0 * (k[0] * pos[0] + k[1] * pos[1] + k[2] * pos[2])
                        e = amp * h[t1] * h[t2] / 4 * (np.cos(ph) + 1j * np.sin(ph))
                        val += np.where(on, f1 * f2 * e, 0)
                        grad += np.where(on, gk * e, 0)
            at = [slice(None)] * 3
            at[2 - nu] = dim[nu] if side else 0
            for al in range(3):
                c = 1j * k0 * sign * (k[al] * p[nu] - p[al] * k[nu]) * val
                if al != nu:
                    c = c + 1j * k0 * p[al] * val + p[al] / 2 * grad
                b[tuple(at) + (al, r)] += c.T  # grid order: the lower axis runs fastest
    return b.reshape(-1, waves.count)


@pytest.mark.parametrize("shape", [7, (3, 9, 5)])
@pytest.mark.parametrize("origin", [(0.0, 0.0, 0.0), (41.3, -25.7, 60.1), (-5.25, 0.5, 7.75)])
def test_rhs_error(fe, ctx, shape, origin):
    prob = W.empty_box(shape, 3e9)
    prob.origin = np.asarray(prob.origin) + np.array(origin)
    waves = W.random_waves(3, np.random.default_rng(8))
    m = fe.fe_mesh_create_from(ctx, prob)
    s = fe.fe_assemble(ctx, m, prob.freq_hz, fe.FE_PREC_FP64)
    try:
        b = fe.fe_rhs(ctx, s, waves, fe.fe_mesh_info(m)["n_dof"])
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)
    ref = _direct(prob, waves)
    err = np.sqrt((np.abs(b - ref) ** 2).sum(axis=0) / (np.abs(ref) ** 2).sum(axis=0))
    assert np.all(err <= 5e-15), err.astype(float)
