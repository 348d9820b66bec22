"""Meshes with more distinct rows than row patterns may have: the grouping
gives up (more groups than the limit, or than its hash table holds) and every
row is assembled, multiplied and solved from the stored blocks.  Bounds as for
the products elsewhere: FP64 1e-13 and FP32 pairs 1e-12 of sum |a x|."""
import numpy as np
import pytest

from oracle import fem
from paper_0704_2344_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def random_core(n, core, kinds=6, seed=3):
    """n^3 elements of vacuum around core^3 elements of random materials: about (core + 1)^3 distinct rows."""
    rng = np.random.default_rng(seed)
    prob = W.empty_box(n, name=f"core{core}")
    a = (n - core) // 2
    prob.material[a:a + core, a:a + core, a:a + core] = rng.integers(0, kinds, (core,) * 3)
    prob.eps_r = 1.0 + np.arange(kinds) * (0.4 - 0.05j)
    prob.mu_r = np.ones(kinds, complex)
    return prob


# limit 2 048 at 27^3 nodes, 8 192 entries in the table; limit 128 at 10^3 nodes
@pytest.mark.parametrize("n,core", [(26, 14), (26, 24), (9, 5)])
@pytest.mark.parametrize("nrhs", [1, 3, 8])
def test_products_beyond_the_limits(fe, ctx, n, core, nrhs):
    import torch

    prob = random_core(n, core)
    A = fem.assemble(prob, maps=fem.mesh_maps(prob))
    rng = np.random.default_rng(nrhs)
    x = (rng.standard_normal((A.shape[0], nrhs)) + 1j * rng.standard_normal((A.shape[0], nrhs))).astype(np.complex64)
    x = x.astype(complex)
    ins = {fe.FE_PREC_FP64: x, fe.FE_PREC_DF: np.stack([x.real, x.imag, 0 * x.real, 0 * x.real], -1).astype(np.float32)}
    m = fe.fe_mesh_create_from(ctx, prob)
    try:
        for prec, tol in ((fe.FE_PREC_FP64, 1e-13), (fe.FE_PREC_DF, 1e-12)):
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
                y = y.astype(float)
                y = (y[..., 0] + y[..., 2]) + 1j * (y[..., 1] + y[..., 3])
            assert np.all(np.abs(y - A @ x) <= tol * (abs(A) @ np.abs(x)))
    finally:
        fe.fe_mesh_destroy(m)
