"""Products and solves with and without row patterns against the oracle.

A voxel mesh whose rows take few distinct values is multiplied through its row
patterns (patterns.cuh); a mesh of random materials has more patterns than its
size allows and is multiplied from the stored blocks.  Both are compared with
the oracle's matrix at widths on and off the powers of two.  Bounds per entry,
in units of sum |a_ij x_j| over at most 81 terms: FP64 81 x 2^-53 plus the
assembly's own rounding, below 1e-13; complex64 2 x 2^-24 for the rounded
inputs plus 81 x 2^-24 at worst, below 5e-6; FP32 pairs a few 81 x 2^-48,
below 1e-12."""
import numpy as np
import pytest

from oracle import fem
from paper_0704_2344_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _random_materials(n=9, kinds=6, seed=11):
    """n^3 elements, each inner one of `kinds` materials at random: nearly every inner row is its own pattern."""
    rng = np.random.default_rng(seed)
    prob = W.empty_box(n, name="random_materials")
    prob.material[1:-1, 1:-1, 1:-1] = rng.integers(0, kinds, (n - 2,) * 3)
    prob.eps_r = 1.0 + np.arange(kinds) * (0.4 - 0.05j)
    prob.mu_r = np.ones(kinds, complex)
    return prob


def _lossy_slab():
    prob = W.pec_box_problem(13, 3e9, np.random.default_rng(4))
    prob.material[2:4, 2:9, 3:11][prob.material[2:4, 2:9, 3:11] != W.PEC] = 1
    prob.eps_r = np.array([1.0, 2.5 - 0.4j])
    prob.mu_r = np.array([1.0, 1.2 - 0.1j])
    return prob


MESHES = {
    "lossy": _lossy_slab,
    "thin": lambda: W.empty_box((3, 5, 17)),
    "pec": lambda: W.pec_box_problem(11, 3e9, np.random.default_rng(6)),
    "random": _random_materials,  # stored blocks
}


def _pairs(v):
    hi = v.astype(np.float32)
    return hi, (v - hi).astype(np.float32)


@pytest.mark.parametrize("nrhs", [1, 2, 5, 8, 16, 32, 33])
@pytest.mark.parametrize("name", list(MESHES))
def test_product_matches_the_oracle(fe, ctx, name, nrhs):
    import torch

    prob = MESHES[name]()
    maps = fem.mesh_maps(prob)
    A = fem.assemble(prob, maps=maps)
    rng = np.random.default_rng(nrhs)
    x = rng.standard_normal((maps.n_dof, nrhs)) + 1j * rng.standard_normal((maps.n_dof, nrhs))
    (rh, rl), (ih, il) = _pairs(x.real), _pairs(x.imag)
    ins = {fe.FE_PREC_FP64: x, fe.FE_PREC_MIXED: x.astype(np.complex64),
           fe.FE_PREC_DF: np.ascontiguousarray(np.stack([rh, ih, rl, il], axis=-1))}
    ref, bound = A @ x, abs(A) @ np.abs(x)
    m = fe.fe_mesh_create_from(ctx, prob)
    try:
        for prec, tol in ((fe.FE_PREC_FP64, 1e-13), (fe.FE_PREC_MIXED, 5e-6), (fe.FE_PREC_DF, 1e-12)):
            s = fe.fe_assemble(ctx, m, prob.freq_hz, prec)
            try:
                xd = torch.from_numpy(ins[prec]).cuda()
                yd = torch.empty_like(xd)
                torch.cuda.synchronize()
                fe.fe_spmv(ctx, s, prec, nrhs, xd, yd)
                fe.fe_ctx_synchronize(ctx)
                y = yd.cpu().numpy()
            finally:
                fe.fe_system_destroy(s)
            if prec == fe.FE_PREC_DF:
                y = y.astype(np.float64)
                y = (y[..., 0] + y[..., 2]) + 1j * (y[..., 1] + y[..., 3])
            assert np.all(np.abs(y - ref) <= tol * bound + 1e-300), (name, nrhs, prec)
    finally:
        fe.fe_mesh_destroy(m)


@pytest.mark.parametrize("nrhs", [1, 3, 17])
@pytest.mark.parametrize("precision", ["DF", "FP64", "MIXED"])
@pytest.mark.parametrize("name", ["lossy", "random"])
def test_solve_matches_the_oracle(fe, ctx, name, precision, nrhs):
    prob = MESHES[name]()
    waves = W.random_waves(nrhs, np.random.default_rng(nrhs))
    prec = getattr(fe, f"FE_PREC_{precision}")
    maps = fem.mesh_maps(prob)
    A = fem.assemble(prob, maps=maps)
    B = fem.rhs(prob, waves, maps=maps)
    m = fe.fe_mesh_create_from(ctx, prob)
    s = fe.fe_assemble(ctx, m, prob.freq_hz, prec)
    try:
        for rec in (fe.FE_RECURRENCE_CG, fe.FE_RECURRENCE_EXPANDED):
            _, x, rep = fe.fe_solve_batch(ctx, s, waves, maps.n_dof, fe.solve_opts(precision=prec, recurrence=rec))
            assert all(r["status"] == 0 for r in rep)
            assert fem.true_relative_residual(A, x, B).max() <= 1e-8
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)


@pytest.fixture(scope="module")
def walk_case():
    """31 x 34 x 30 nodes with a PEC block and a lossy slab: enough rows for the walks from 4 columns on."""
    prob = W.empty_box((30, 33, 29))
    prob.material[10:17, 12:19, 8:15] = W.PEC
    prob.material[3:6, 4:30, 5:20] = 1
    prob.eps_r = np.array([1.0, 2.5 - 0.4j])
    prob.mu_r = np.array([1.0, 1.2 - 0.1j])
    maps = fem.mesh_maps(prob)
    return prob, maps, fem.assemble(prob, maps=maps)


@pytest.mark.parametrize("nrhs", [1, 2, 4, 8, 32])
def test_walk_product_matches_the_oracle(fe, ctx, walk_case, nrhs):
    import torch

    prob, maps, A = walk_case
    rng = np.random.default_rng(nrhs)
    x = (rng.standard_normal((maps.n_dof, nrhs)) + 1j * rng.standard_normal((maps.n_dof, nrhs))).astype(np.complex64)
    m = fe.fe_mesh_create_from(ctx, prob)
    s = fe.fe_assemble(ctx, m, prob.freq_hz, fe.FE_PREC_MIXED)
    try:
        xd = torch.from_numpy(x).cuda()
        yd = torch.empty_like(xd)
        torch.cuda.synchronize()
        fe.fe_spmv(ctx, s, fe.FE_PREC_MIXED, nrhs, xd, yd)
        fe.fe_ctx_synchronize(ctx)
        err = np.abs(yd.cpu().numpy() - A @ x.astype(complex))
        assert np.all(err <= 5e-6 * (abs(A) @ np.abs(x)) + 1e-300)
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)
