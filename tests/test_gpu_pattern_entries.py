"""Products keep every entry of the assembled matrix, however small beside the
row's largest, and what is not finite in it.

A real vector times the matrix has an imaginary part that only the matrix's
imaginary parts make, so that a loss tangent of 1e-17 is visible on its own.
Bounds per entry in units of sum |Im a_ij x_j|, as for whole products: FP64
1e-13, complex64 5e-6, FP32 pairs 1e-12 (81 terms and the assembly's own
rounding).  The widths take the stored blocks, the shared items, the plain form
and, at 30^3 elements, the walks."""
import numpy as np
import pytest

from oracle import fem
from paper_0704_2344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"FP64": 1e-13, "MIXED": 5e-6, "DF": 1e-12}


def _product(fe, ctx, prob, precision, x):
    """y = A x in complex128 from complex128 x whose entries the precision holds exactly; and the system's blocks."""
    import torch

    prec = getattr(fe, f"FE_PREC_{precision}")
    v = {"FP64": x, "MIXED": x.astype(np.complex64),
         "DF": np.stack([x.real, x.imag, 0 * x.real, 0 * x.real], axis=-1).astype(np.float32)}[precision]
    m = fe.fe_mesh_create_from(ctx, prob)
    s = fe.fe_assemble(ctx, m, prob.freq_hz, prec)
    try:
        xd = torch.from_numpy(np.ascontiguousarray(v)).cuda()
        yd = torch.empty_like(xd)
        torch.cuda.synchronize()
        fe.fe_spmv(ctx, s, prec, x.shape[1], xd, yd)
        fe.fe_ctx_synchronize(ctx)
        y = yd.cpu().numpy()
        blocks, maps = fe.fe_system_export(ctx, s, m)["c128"], fe.fe_mesh_export_maps(ctx, m)
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)
    if precision == "DF":
        y = y.astype(np.float64)
        y = (y[..., 0] + y[..., 2]) + 1j * (y[..., 1] + y[..., 3])
    return y, blocks, maps


def _slab(n, eps, mu):
    prob = W.empty_box(n)
    prob.material[3:n // 2, 3:n - 3, 2:n - 2] = 1
    prob.material[n - 4:n - 2, 3:6, 3:6] = W.PEC
    prob.eps_r, prob.mu_r = np.array([1, eps]), np.array([1, mu])
    return prob


@pytest.mark.parametrize("precision", ["FP64", "MIXED", "DF"])
@pytest.mark.parametrize("n,nrhs", [(11, 1), (11, 2), (11, 5), (11, 8), (11, 16), (31, 4), (31, 8)])
@pytest.mark.parametrize("eps,mu", [(2.5 - 1e-17j, 1.0 + 0j), (1.0 + 0j, 1.5 - 1e-18j)])
def test_small_losses_reach_the_product(fe, ctx, eps, mu, n, nrhs, precision):
    prob = _slab(n, eps, mu)
    A = fem.assemble(prob, maps=fem.mesh_maps(prob))
    x = np.random.default_rng(nrhs).standard_normal((A.shape[0], nrhs)).astype(np.float32).astype(np.float64)
    y, _, _ = _product(fe, ctx, prob, precision, x + 0j)
    bound = abs(A.imag) @ np.abs(x)
    assert np.all(np.abs(y.imag - A.imag @ x) <= TOL[precision] * bound)


@pytest.mark.parametrize("precision", ["FP64", "MIXED", "DF"])
@pytest.mark.parametrize("nrhs", [1, 5, 8])
@pytest.mark.parametrize("eps,mu", [(complex(np.nan, 0), 1.0), (complex(np.inf, 0), 1.0), (2.0, complex(0, np.nan)),
                                    (2.0, complex(np.inf, 0))])
def test_non_finite_materials_are_seen_in_every_row(fe, ctx, eps, mu, nrhs, precision):
    prob = _slab(11, eps, mu)
    n_dof = 3 * int(np.count_nonzero(fem.mesh_maps(prob).node_active))
    x = np.random.default_rng(1).standard_normal((n_dof, nrhs)).astype(np.float32).astype(np.float64) + 0.25j
    y, blocks, maps = _product(fe, ctx, prob, precision, x)
    rp = maps["row_ptr"]
    bad = np.concatenate([~np.isfinite(blocks[rp[r]:rp[r + 1]]).all(axis=(0, 2)) for r in range(len(rp) - 1)])
    assert bad.any() and not bad.all()
    np.testing.assert_array_equal(~np.isfinite(y), np.repeat(bad[:, None], nrhs, axis=1))
