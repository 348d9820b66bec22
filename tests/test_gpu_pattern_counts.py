"""Which systems have row patterns, and what runs without them: the count that
fe_system_patterns reports on either side of the limit (an eighth of the nodes,
at least 128 and at most 2 048), the terms against the matrix's non-zero parts,
and solves, batched and served, of a mesh without patterns whose distinct
blocks fit the resident dictionary, also beside requests with patterns."""
import numpy as np
import pytest

from oracle import fem
from paper_0704_2344_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _core(n, core, kinds=6, seed=3):
    rng = np.random.default_rng(seed)
    prob = W.empty_box(n, name=f"core{core}")
    a = (n - core) // 2
    prob.material[a:a + core, a:a + core, a:a + core] = rng.integers(0, kinds, (core,) * 3)
    prob.eps_r = 1.0 + np.arange(kinds) * (0.4 - 0.05j)
    prob.mu_r = np.ones(kinds, complex)
    return prob


def _speckle(seed=1):
    """8^3 elements, each inner one vacuum or one lossy material at random: more distinct rows than the limit of 128,
    few distinct blocks."""
    rng = np.random.default_rng(seed)
    prob = W.empty_box(8, name="speckle")
    prob.material[1:-1, 1:-1, 1:-1] = rng.integers(0, 2, (6, 6, 6))
    prob.eps_r = np.array([1.0, 2.5 - 0.4j])
    prob.mu_r = np.array([1.0, 1.0])
    return prob


def _system(fe, ctx, prob, prec):
    m = fe.fe_mesh_create_from(ctx, prob)
    return m, fe.fe_assemble(ctx, m, prob.freq_hz, prec)


@pytest.mark.parametrize("make,has", [(lambda: W.empty_box((3, 5, 17)), True),
                                      (lambda: W.pec_box_problem(11, 3e9, np.random.default_rng(6)), True),
                                      (lambda: _core(9, 3), True), (lambda: _core(9, 5), False),
                                      (lambda: _core(26, 10), True), (lambda: _core(26, 14), False),
                                      (lambda: _core(26, 24), False), (_speckle, False)])
@pytest.mark.parametrize("precision", ["FP64", "DF"])
def test_pattern_count(fe, ctx, make, has, precision):
    prob = make()
    m, s = _system(fe, ctx, prob, getattr(fe, f"FE_PREC_{precision}"))
    try:
        n, terms = fe.fe_system_patterns(ctx, s)
        blocks, maps = fe.fe_system_export(ctx, s, m)["c128"], fe.fe_mesh_export_maps(ctx, m)
        assert (n > 0) == has
        if not has:
            assert terms == 0
            return
        rp = maps["row_ptr"]
        rows = [blocks[rp[r]:rp[r + 1]] for r in range(len(rp) - 1)]
        assert n >= len({(len(b), b.tobytes()) for b in rows})  # equal rows may differ in their surroundings
        want = 0
        for b in rows:  # every component as long as the longest; rows of 27 real diagonal blocks in full
            re, im = (b.real != 0).sum(axis=(0, 2)).max(), (b.imag != 0).sum(axis=(0, 2)).max()
            diag = len(b) == 27 and im == 0 and not b[:, ~np.eye(3, dtype=bool)].any()
            want += 3 * (27 if diag else int(re + im))
        assert terms == want
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)


@pytest.mark.parametrize("precision", ["MIXED", "DF"])
@pytest.mark.parametrize("nrhs", [1, 4])
@pytest.mark.parametrize("expanded", [False, True])
def test_solve_through_the_dictionary(fe, ctx, precision, nrhs, expanded):
    prob = _speckle()
    waves = W.random_waves(nrhs, np.random.default_rng(nrhs))
    maps = fem.mesh_maps(prob)
    A, B = fem.assemble(prob, maps=maps), fem.rhs(prob, waves, maps=maps)
    prec = getattr(fe, f"FE_PREC_{precision}")
    m, s = _system(fe, ctx, prob, prec)
    try:
        assert fe.fe_system_patterns(ctx, s) == (0, 0)
        assert 0 < fe.fe_system_info(s)["dict_blocks"] <= 455  # its blocks fit 64 KiB in either arithmetic
        rec = fe.FE_RECURRENCE_EXPANDED if expanded else fe.FE_RECURRENCE_CG
        _, x, rep = fe.fe_solve_batch(ctx, s, waves, maps.n_dof, fe.solve_opts(precision=prec, recurrence=rec))
    finally:
        fe.fe_system_destroy(s)
        fe.fe_mesh_destroy(m)
    assert all(r["status"] == 0 for r in rep)
    assert fem.true_relative_residual(A, x, B).max() <= 1e-8


@pytest.mark.parametrize("precision", ["DF", "MIXED"])
def test_served_batch_of_both_kinds(fe, ctx, precision):
    """Requests of one tile width with and without patterns share segments; each gives the field it gives alone."""
    reqs = []
    for q in range(6):
        prob = _speckle(seed=q) if q % 2 else W.pec_box_problem(9, 2.5e9, np.random.default_rng(q))
        reqs.append((prob, W.random_waves(2, np.random.default_rng(q))))
    opts = fe.serve_opts(precision=getattr(fe, f"FE_PREC_{precision}"))

    def serve(some):
        srv = fe.fe_serve_create(ctx, opts)
        try:
            tickets = [fe.fe_serve_submit(srv, p, w) for p, w in some]
            return [fe.fe_serve_wait(srv, t, timeout_s=120.0) for t in tickets]
        finally:
            fe.fe_serve_destroy(srv)

    together = serve(reqs)
    assert max(r["batch_jobs"] for r in together) >= 2
    for (prob, waves), r in zip(reqs, together):
        assert r["status"] == 0, r["message"]
        np.testing.assert_array_equal(r["x"], serve([(prob, waves)])[0]["x"])
        maps = fem.mesh_maps(prob)
        A, B = fem.assemble(prob, maps=maps), fem.rhs(prob, waves, maps=maps)
        assert fem.true_relative_residual(A, r["x"], B).max() <= 1e-8


def test_both_kinds_run_side_by_side(fe, ctx):
    """Requests of one tile width with and without patterns are launched separately in a segment, not one after the
    other in one launch's turn: two requests that share every segment make two launches of it."""
    srv = fe.fe_serve_create(ctx, fe.serve_opts(seg_iters=16))
    try:
        probs = [_speckle(), W.pec_box_problem(9, 2.5e9, np.random.default_rng(0))]
        waves = [W.random_waves(1, np.random.default_rng(q)) for q in range(2)]
        tickets = [fe.fe_serve_submit(srv, p, w) for p, w in zip(probs, waves)]
        results = [fe.fe_serve_wait(srv, t, timeout_s=60.0) for t in tickets]
        info = fe.fe_serve_info(srv)
    finally:
        fe.fe_serve_destroy(srv)
    assert all(r["status"] == 0 for r in results) and max(r["batch_jobs"] for r in results) == 2
    assert info["launches"] == info["jobs_launched"]


def test_tuned_choice_is_kept_per_kind_of_kernel(fe, ctx):
    """Two systems of one shape, one with patterns and one without, run different kernels: each is tuned itself."""
    rng = np.random.default_rng(8)
    prob = _core(9, 7, seed=8)
    flat = W.empty_box(9)
    waves = W.random_waves(13, rng)
    how = []
    for p, has in ((flat, True), (prob, False), (flat, True), (prob, False)):
        m, s = _system(fe, ctx, p, fe.FE_PREC_DF)
        try:
            assert (fe.fe_system_patterns(ctx, s)[0] > 0) == has
            fe.fe_solve_batch(ctx, s, waves, fe.fe_mesh_info(m)["n_dof"], fe.solve_opts(max_iter=40),
                              raise_on_fail=False)
            how.append(fe.fe_last_solve_stats(ctx)["tuned"])
        finally:
            fe.fe_system_destroy(s)
            fe.fe_mesh_destroy(m)
    assert how == [1, 1, 2, 2]


# a request's device memory without patterns (8^3 elements, two waves), by precision
@pytest.mark.parametrize("precision,budget", [("DF", 8483037), ("FP64", 5360656), ("MIXED", 6960337)])
def test_serve_budget_without_room_for_patterns(fe, ctx, precision, budget):
    """A budget that holds a request without its row patterns serves it, and one byte less refuses it."""
    prob = W.pec_box_problem(8, 3e9, np.random.default_rng(8))
    waves = W.random_waves(2, np.random.default_rng(1))
    out = []
    for b in (budget, budget - 1, 0):
        srv = fe.fe_serve_create(ctx, fe.serve_opts(precision=getattr(fe, f"FE_PREC_{precision}"), hbm_budget=b))
        try:
            out.append(fe.fe_serve_wait(srv, fe.fe_serve_submit(srv, prob, waves), timeout_s=60.0))
            assert fe.fe_serve_info(srv)["peak_admitted_bytes"] <= (b or 1 << 62)
        finally:
            fe.fe_serve_destroy(srv)
    assert out[0]["status"] == 0, out[0]["message"]
    assert out[1]["status"] == fe.FE_ERR_OOM and "budget" in out[1]["message"]
    maps = fem.mesh_maps(prob)
    A, B = fem.assemble(prob, maps=maps), fem.rhs(prob, waves, maps=maps)
    for r in (out[0], out[2]):
        assert fem.true_relative_residual(A, r["x"], B).max() <= 1e-8
