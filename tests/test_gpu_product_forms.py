"""Products on either side of the bounds between their forms (stored blocks,
shared items, one lane an item, walks), on meshes where patterns of real
diagonal blocks lie side by side (a permeable block in air: eps 1, mu 2), and
solves whose rows are taken four at a time on such a mesh.  Bounds per entry as
for products elsewhere: FP64 1e-13, complex64 5e-6, FP32 pairs 1e-12 of
sum |a x|; solves to a true residual of 1e-8."""
import numpy as np
import pytest

from oracle import fem
from paper_0704_2344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"FP64": 1e-13, "MIXED": 5e-6, "DF": 1e-12}


def _permeable(n):
    prob = W.empty_box(n)
    a = max(1, n // 5)
    prob.material[a:n - a, a:n // 2, 1:n - 1] = 1  # lines along x enter and leave it near the outer faces
    prob.material[n // 2:n // 2 + a, n // 2:n - a, a:n - a] = 2
    prob.material[n - 1 - a:n - 1, n - 1 - a:n - 1, n - 1 - a:n - 1] = W.PEC
    prob.eps_r = np.array([1.0, 1.0, 2.5 - 0.4j])
    prob.mu_r = np.array([1.0, 2.0, 1.0])
    return prob


def _check(fe, ctx, prob, A, absA, precision, widths):
    import torch

    prec = getattr(fe, f"FE_PREC_{precision}")
    m = fe.fe_mesh_create_from(ctx, prob)
    s = fe.fe_assemble(ctx, m, prob.freq_hz, prec)
    try:
        for nrhs in widths:
            rng = np.random.default_rng(nrhs)
            x = rng.standard_normal((A.shape[0], nrhs, 2)).astype(np.float32).astype(np.float64)
            z = x[..., 0] + 1j * x[..., 1]
            v = {"FP64": z, "MIXED": z.astype(np.complex64),
                 "DF": np.concatenate([x, 0 * x], axis=-1).astype(np.float32)}[precision]
            xd = torch.from_numpy(np.ascontiguousarray(v)).cuda()
            yd = torch.empty_like(xd)
            torch.cuda.synchronize()
            fe.fe_spmv(ctx, s, prec, nrhs, xd, yd)
            fe.fe_ctx_synchronize(ctx)
            y = yd.cpu().numpy()
            if precision == "DF":
                y = y.astype(float)
                y = (y[..., 0] + y[..., 2]) + 1j * (y[..., 1] + y[..., 3])
            assert np.all(np.abs(y - A @ z) <= TOL[precision] * (absA @ np.abs(z))), nrhs
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)


@pytest.mark.parametrize("n", [4, 8, 13, 14, 20, 22, 25])
@pytest.mark.parametrize("precision", ["FP64", "MIXED", "DF"])
def test_products_around_the_bounds(fe, ctx, n, precision):
    prob = _permeable(n)
    A = fem.assemble(prob, maps=fem.mesh_maps(prob))
    _check(fe, ctx, prob, A, abs(A), precision, (1, 2, 3, 4, 8, 16, 32))


@pytest.fixture(scope="module")
def large():
    """48^3 nodes: the walks of one column, and of eight and sixteen in tiles."""
    prob = _permeable(47)
    A = fem.assemble(prob, maps=fem.mesh_maps(prob))
    return prob, A, abs(A)


@pytest.mark.parametrize("precision,widths", [("MIXED", (1, 2, 4, 8, 16)), ("DF", (1, 8)), ("FP64", (1, 2))])
def test_products_of_the_walks(fe, ctx, large, precision, widths):
    _check(fe, ctx, *large, precision, widths)


@pytest.mark.parametrize("precision,nrhs", [("DF", 32), ("FP64", 32), ("MIXED", 32), ("DF", 1)])
def test_solves_on_adjacent_diagonal_patterns(fe, ctx, precision, nrhs):
    prob = _permeable(20)
    maps = fem.mesh_maps(prob)
    A = fem.assemble(prob, maps=maps)
    waves = W.random_waves(nrhs, np.random.default_rng(nrhs))
    prec = getattr(fe, f"FE_PREC_{precision}")
    m = fe.fe_mesh_create_from(ctx, prob)
    s = fe.fe_assemble(ctx, m, prob.freq_hz, prec)
    try:
        _, x, rep = fe.fe_solve_batch(ctx, s, waves, maps.n_dof, fe.solve_opts(precision=prec, rhs_tile=nrhs))
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)
    assert all(r["status"] == 0 for r in rep)
    assert fem.true_relative_residual(A, x, fem.rhs(prob, waves, maps=maps)).max() <= 1e-8
