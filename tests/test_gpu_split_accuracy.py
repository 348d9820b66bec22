"""Rounding of the products in which several lanes share a row's component.

A product rounds most where its largest term, the row's own entry, is added;
every form adds that entry last, so that a sum over lanes holds no more large
roundings than the sum of one lane: its rms error on random vectors, against
extended precision, is at most that of the same columns multiplied among five
(one lane each), with a fifth allowed for chance (12 167 rows, three
components: the rms of either is known to one percent)."""
import numpy as np
import pytest

from paper_0704_2344_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 22  # one, two and four columns are shared by eight, four and two lanes


def _problem(loss):
    prob = W.empty_box(N, 3e9)
    prob.material[3:6, 4:18, 4:18] = 1
    prob.material[9:13, 9:13, 9:13] = W.PEC
    prob.eps_r = np.array([1.0, 2.5 - 0.4j if loss else 4.0])
    prob.mu_r = np.array([1.0, 1.2 - 0.1j if loss else 1.0])
    return prob


@pytest.mark.parametrize("loss", [False, True])
@pytest.mark.parametrize("precision", ["FP64", "MIXED", "DF"])
def test_shared_items_round_as_little(fe, ctx, precision, loss):
    import torch

    prob, prec = _problem(loss), getattr(fe, f"FE_PREC_{precision}")
    m = fe.fe_mesh_create_from(ctx, prob)
    s = fe.fe_assemble(ctx, m, prob.freq_hz, prec)
    try:
        blocks, maps = fe.fe_system_export(ctx, s, m)["c128"], fe.fe_mesh_export_maps(ctx, m)
        rp, col = maps["row_ptr"], maps["col_idx"]
        n = len(rp) - 1
        v = np.random.default_rng(5).standard_normal((3 * n, 5, 2))
        hi = v.astype(np.float32)
        lo = (v - hi).astype(np.float32)
        held = {"FP64": v, "MIXED": hi.astype(float), "DF": hi.astype(float) + lo}[precision]
        x = held[..., 0] + 1j * held[..., 1]
        ins = {"FP64": x, "MIXED": x.astype(np.complex64), "DF": np.concatenate([hi, lo], axis=-1)}[precision]

        def product(cols):
            xd = torch.from_numpy(np.ascontiguousarray(ins[:, :cols])).cuda()
            yd = torch.empty_like(xd)
            torch.cuda.synchronize()
            fe.fe_spmv(ctx, s, prec, cols, xd, yd)
            fe.fe_ctx_synchronize(ctx)
            y = yd.cpu().numpy()
            if precision == "DF":
                y = y.astype(np.longdouble)
                y = (y[..., 0] + y[..., 2]) + 1j * (y[..., 1] + y[..., 3])
            return y

        ref = np.empty((3 * n, 4), np.clongdouble)
        for c in range(4):
            xb = x[:, c].reshape(n, 3)[col].astype(np.clongdouble)
            ref[:, c] = np.add.reduceat((blocks.astype(np.clongdouble) * xb[:, None, :]).sum(axis=2), rp[:-1],
                                        axis=0).reshape(-1)

        def rms(cols, upto):
            return float(np.sqrt((np.abs(product(cols)[:, :upto] - ref[:, :upto]) ** 2).mean()))

        for cols in (1, 2, 4):
            assert rms(cols, cols) <= 1.2 * rms(5, cols), cols
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)
