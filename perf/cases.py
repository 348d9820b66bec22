"""The work a user of this library has it do, as cases that can be timed.

Four kinds of call, all through the public binding (paper_0704_2344_gb300.fe):

  product  y = A x (fe_spmv) on an assembled system the program keeps, as an
           outer iteration of the caller's own calls it;
  setup    a new scatterer: fe_mesh_create, fe_assemble, the right-hand sides
           (fe_rhs) and the first product on a given field;
  solve    fe_solve_batch on a system the program keeps, for new incident
           waves, to a true residual well below the default 1e-8, as fields
           are asked for whose differences are then taken;
  serve    a burst of requests of different sizes submitted to the server and
           waited for.

Geometries are this repository's own: a cube with a centred PEC cube and a
dielectric slab at a seeded height (the 3-wavelength cube at any size), the
voxel aircraft, and the serving stream's cubes with a random PEC box.
"""
import math

import numpy as np
import torch

from paper_0704_2344_gb300 import fe, workloads as W

PRECISION = {"fp64": fe.FE_PREC_FP64, "mixed": fe.FE_PREC_MIXED, "df": fe.FE_PREC_DF}
RECURRENCE = {"cg": fe.FE_RECURRENCE_CG, "expanded": fe.FE_RECURRENCE_EXPANDED}
FREQ = 3.0e9


# --------------------------------------------------------------------------
# The cases.
# --------------------------------------------------------------------------
def listed():
    return [
        # The caller's own iteration on a cube of two wavelengths: a few hundred
        # kilobytes a vector, so launch and call latency count.
        {"name": "product_small_df", "kind": "product", "shape": "cube", "n": 20, "loss": False, "nrhs": 1,
         "precision": "df"},
        # One vector through the 1.6 M-unknown aircraft system in complex64, the
        # largest product a program does.
        {"name": "product_large_c64", "kind": "product", "shape": "aircraft", "n": 80, "loss": False, "nrhs": 1,
         "precision": "mixed"},
        # Sixteen incidence angles at once on a mid-sized aircraft.
        {"name": "product_16_c64", "kind": "product", "shape": "aircraft", "n": 60, "loss": False, "nrhs": 16,
         "precision": "mixed"},
        # A count of vectors that is no power of two, odd sizes and a lossy slab,
        # in full FP64: the residual check of the caller's own loop.
        {"name": "product_ragged_fp64", "kind": "product", "shape": "cube", "n": 47, "loss": True, "nrhs": 3,
         "precision": "fp64"},
        # A new scatterer from voxels to the first residual: what every new
        # geometry pays before its solve.
        {"name": "setup_df", "kind": "setup", "shape": "cube", "n": 50, "loss": False, "nrhs": 4,
         "precision": "df"},
        # One wave on a cube of one wavelength: the smallest solve in use.
        {"name": "solve_small_df", "kind": "solve", "shape": "cube", "n": 10, "loss": False, "nrhs": 1,
         "precision": "df", "recurrence": "cg", "tol": 5e-11},
        # The 3-wavelength cube with a PEC cube and a slab, one wave: the
        # library's default solve at the paper's own size.
        {"name": "solve_cube_df", "kind": "solve", "shape": "cube", "n": 30, "loss": False, "nrhs": 1,
         "precision": "df", "recurrence": "cg", "tol": 5e-11},
        # The plain complex128 method, used where every operation has to be FP64.
        {"name": "solve_cube_fp64", "kind": "solve", "shape": "cube", "n": 20, "loss": False, "nrhs": 1,
         "precision": "fp64", "recurrence": "cg", "tol": 1e-11},
        # Complex64 products inside FP64 refinement, on a small lossy scatterer.
        {"name": "solve_cube_mixed", "kind": "solve", "shape": "cube", "n": 13, "loss": True, "nrhs": 1,
         "precision": "mixed", "recurrence": "cg", "tol": 1e-11},
        # A dozen incidence angles in one call (padded to a tile of sixteen).
        {"name": "solve_batch_df", "kind": "solve", "shape": "cube", "n": 18, "loss": False, "nrhs": 12,
         "precision": "df", "recurrence": "cg", "tol": 1e-10},
        # The same scatterer on a mesh twice as fine, 205 000 unknowns: the
        # largest single solve, with the expanded recurrence that the library's
        # documentation advises for hard systems.
        {"name": "solve_fine_df", "kind": "solve", "shape": "cube", "n": 40, "per_wavelength": 20, "loss": False,
         "nrhs": 1, "precision": "df", "recurrence": "expanded", "tol": 1e-10},
        # A burst of small and middling requests at the server, 1 to 8 waves each.
        {"name": "serve_burst", "kind": "serve", "requests": 12, "stream": 1, "n_min": 7, "n_max": 14, "nrhs_max": 6,
         "precision": "df", "tol": 5e-11},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["product", "product", "setup", "solve", "solve", "solve", "serve"])
    if kind == "product":
        precision = rng.choice(["fp64", "mixed", "df"])
        shape = rng.choice(["cube", "cube", "aircraft"])
        n = _log_int(rng, 24, 70) if shape == "aircraft" else _log_int(rng, 15, 70)
        nrhs = rng.choice([1, 1, 2, 3, 4, 5, 8, 12, 16, 32])
        while nrhs > 1 and (n + 1) ** 3 * nrhs > 61 ** 3 * 16:
            nrhs //= 2
        return {"kind": kind, "shape": shape, "n": n, "loss": rng.random() < 0.3, "nrhs": nrhs,
                "precision": precision}
    if kind == "setup":
        return {"kind": kind, "shape": "cube", "n": _log_int(rng, 9, 50), "loss": rng.random() < 0.3,
                "nrhs": rng.choice([1, 2, 3, 4]), "precision": rng.choice(["fp64", "mixed", "df"])}
    if kind == "solve":
        precision = rng.choice(["df", "df", "df", "fp64", "mixed"])
        n = _log_int(rng, 8, {"df": 31, "fp64": 21, "mixed": 13}[precision])
        nrhs = rng.choice([1, 1, 1, 2, 3, 6, 8, 12, 16]) if precision == "df" else 1
        while nrhs > 1 and (n + 1) ** 3 * nrhs > 21 ** 3 * 16:
            nrhs //= 2
        # complex64 products go with the default recurrence; the larger systems with the expanded one
        recurrence = "cg" if precision == "mixed" else "expanded" if n > 18 else rng.choice(["cg", "expanded"])
        return {"kind": kind, "shape": "cube", "n": n, "loss": precision == "mixed" or rng.random() < 0.3,
                "nrhs": nrhs, "precision": precision, "recurrence": recurrence,
                "tol": 1e-10 if precision == "df" else 1e-11}
    return {"kind": kind, "requests": rng.randint(3, 12), "stream": rng.randrange(1000), "n_min": 7,
            "n_max": rng.randint(11, 14), "nrhs_max": rng.randint(1, 6), "precision": "df", "tol": 5e-11}


# --------------------------------------------------------------------------
# Inputs.
# --------------------------------------------------------------------------
def _problem(case, seed):
    """The voxel problem of a case: the seed moves the slab (the aircraft is one body at every seed)."""
    n = case["n"]
    rng = np.random.default_rng([20070704, int(seed), n])
    if case["shape"] == "aircraft":
        return W.aircraft_mesh(n, 4, FREQ)
    prob = W.empty_box(n, FREQ, float(case.get("per_wavelength", 10)), name=f"cube{n}")
    c0, c1, thick = round(0.4 * n), round(0.6 * n), max(1, n // 10)
    heights = list(range(2, c0 - thick + 1)) + list(range(c1, n - 2 - thick + 1))
    kz = int(rng.choice(heights))
    lo, hi = max(2, round(0.2 * n)), min(n - 2, round(0.8 * n))
    prob.material[kz:kz + thick, lo:hi, lo:hi] = 1
    prob.material[c0:c1, c0:c1, c0:c1] = W.PEC
    prob.eps_r = np.array([1.0 + 0j, 2.5 - 0.4j if case["loss"] else 4.0 + 0j])
    prob.mu_r = np.array([1.0 + 0j, 1.2 - 0.1j if case["loss"] else 1.0 + 0j])
    return prob


def _requests(case, seed):
    """The burst: cubes of log-uniform size and random frequency with a random PEC box (by the case's stream), and
    each one's waves by the seed."""
    rng = np.random.default_rng([20070704, case["stream"]])
    wave = np.random.default_rng([20070704, int(seed), 5])
    out = []
    for q in range(case["requests"]):
        n = int(round(np.exp(rng.uniform(np.log(case["n_min"]), np.log(case["n_max"])))))
        prob = W.pec_box_problem(n, float(rng.uniform(1e9, 6e9)), rng, name=f"req{q}")
        out.append((prob, W.random_waves(int(rng.integers(1, case["nrhs_max"] + 1)), wave)))
    return out


def _waves(case, seed):
    return W.random_waves(case["nrhs"], np.random.default_rng([20070704, int(seed), 7]))


def _active(prob):
    """Grid node ids of the active nodes, ascending."""
    act = np.zeros((prob.nz + 1, prob.ny + 1, prob.nx + 1), bool)
    on = np.asarray(prob.material) != W.PEC
    for c in range(8):
        act[c >> 2:prob.nz + (c >> 2), (c >> 1) & 1:prob.ny + ((c >> 1) & 1), c & 1:prob.nx + (c & 1)] |= on
    return np.flatnonzero(act.ravel())


def _field(prob, nrhs, seed):
    """complex128 [n_dof, nrhs] on the GPU: a field of order one, as a caller's iterate has."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 11)
    n_dof = 3 * _active(prob).size
    return torch.view_as_complex(torch.randn(n_dof, nrhs, 2, generator=g, device="cuda", dtype=torch.float64))


def _stored(x, precision):
    """A field as the products of a precision take it."""
    if precision == "fp64":
        return x
    if precision == "mixed":
        return x.to(torch.complex64)
    v = torch.view_as_real(x)
    hi = v.float()
    return torch.cat([hi, (v - hi.double()).float()], dim=-1).contiguous()  # (re_hi, im_hi, re_lo, im_lo)


class _State:
    """What the program keeps; the handles go with it."""

    def __init__(self):
        self.ctx = fe.fe_ctx_create(0)
        self.mesh = self.system = self.server = None

    def __del__(self):
        if self.server is not None:
            fe.fe_serve_destroy(self.server)
        if self.system is not None:
            fe.fe_system_destroy(self.system)
        if self.mesh is not None:
            fe.fe_mesh_destroy(self.mesh)
        fe.fe_ctx_destroy(self.ctx)


def prepare(case, seed):
    s = _State()
    s.case = case
    s.prec = PRECISION[case["precision"]]
    if case["kind"] == "serve":
        s.server = fe.fe_serve_create(s.ctx, fe.serve_opts(precision=s.prec, tol=case["tol"]))
        s.requests = _requests(case, seed)
        return s
    s.problem = _problem(case, seed)
    if case["kind"] != "setup":
        s.mesh = fe.fe_mesh_create_from(s.ctx, s.problem)
        s.system = fe.fe_assemble(s.ctx, s.mesh, s.problem.freq_hz, s.prec)
        s.n_dof = fe.fe_mesh_info(s.mesh)["n_dof"]
    if case["kind"] == "solve":
        s.waves = _waves(case, seed)
        s.opts = fe.solve_opts(precision=s.prec, tol=case["tol"], recurrence=RECURRENCE[case["recurrence"]])
    elif case["kind"] == "product":
        s.x = _stored(_field(s.problem, case["nrhs"], seed), case["precision"])
        s.y = torch.empty_like(s.x)
    else:
        s.waves = _waves(case, seed)
        s.x = _field(s.problem, case["nrhs"], seed)
        s.b, s.y = torch.empty_like(s.x), torch.empty_like(s.x)
    torch.cuda.synchronize()
    return s


# --------------------------------------------------------------------------
# One pass.
# --------------------------------------------------------------------------
def run(s):
    kind, nrhs = s.case["kind"], s.case.get("nrhs")
    if kind == "product":
        fe.fe_spmv(s.ctx, s.system, s.prec, nrhs, s.x, s.y)
        return s.y
    if kind == "solve":
        _, x, _ = fe.fe_solve_batch(s.ctx, s.system, s.waves, s.n_dof, s.opts)
        return x
    if kind == "setup":
        mesh = fe.fe_mesh_create_from(s.ctx, s.problem)
        system = fe.fe_assemble(s.ctx, mesh, s.problem.freq_hz, s.prec)
        info = fe.fe_mesh_info(mesh)
        fe.fe_rhs(s.ctx, system, s.waves, info["n_dof"], out=s.b, on_device=True)
        fe.fe_spmv(s.ctx, system, fe.FE_PREC_FP64, nrhs, s.x, s.y)
        fe.fe_system_destroy(system)
        fe.fe_mesh_destroy(mesh)
        return {"b": s.b, "y": s.y, "n_dof": info["n_dof"], "nnzb": info["nnzb"],
                "n_faces_ext": info["n_faces_ext"], "n_faces_pec": info["n_faces_pec"]}
    tickets = [fe.fe_serve_submit(s.server, p, w) for p, w in s.requests]
    out = []
    for t in tickets:
        out.append(fe.fe_serve_wait(s.server, t, timeout_s=600)["x"])
        fe.fe_serve_release(s.server, t)
    return out


# --------------------------------------------------------------------------
# What a pass cannot do without.
# --------------------------------------------------------------------------
def _entry_bytes(precision):
    return 8 if precision == "mixed" else 16


def _counts(n):
    """Unknowns and 3x3 blocks of a full cube of n^3 elements (the PEC body takes a few percent of it)."""
    return 3 * (n + 1) ** 3, (3 * n + 1) ** 3


def _solve_work(n, nrhs, tol):
    """A Krylov solve on a cube of n^3 elements: of the order of 20 iterations per element along an edge at
    1e-8, each with one product (12 flops a block: three real weights on complex values) and five vector updates
    and the preconditioner (64 flops an unknown); the fields come back once."""
    dof, blocks = _counts(n)
    its = 20.0 * n * math.log10(1.0 / tol) / 8.0
    return {"bytes": 16.0 * dof * nrhs + n ** 3, "flops": its * nrhs * (12.0 * blocks + 64.0 * dof)}


def work(case):
    if case["kind"] == "serve":
        n, r = math.sqrt(case["n_min"] * case["n_max"]), 0.5 * (1 + case["nrhs_max"])
        w = _solve_work(n, r, case["tol"])
        return {k: v * case["requests"] for k, v in w.items()}
    n, nrhs = case["n"], case["nrhs"]
    dof, blocks = _counts(n)
    if case["kind"] == "solve":
        return _solve_work(n, nrhs, case["tol"])
    # the vectors in and out and the voxels that determine the matrix; 12 flops a block as above
    product = {"bytes": 2.0 * dof * nrhs * _entry_bytes(case["precision"]) + n ** 3, "flops": 12.0 * blocks * nrhs}
    if case["kind"] == "product":
        return product
    # the matrix the program asks for, each block once, and the right-hand sides
    return {"bytes": product["bytes"] + 16.0 * dof * nrhs + 16.0 * 9 * blocks +
            (0.0 if case["precision"] == "fp64" else _entry_bytes(case["precision"]) * 9.0 * blocks),
            "flops": product["flops"] + 8.0 * 18 * blocks}


# --------------------------------------------------------------------------
# The same in plain 64-bit torch: quadrature element matrices applied element
# by element, and COCG with refinement on that operator.
# --------------------------------------------------------------------------
_CORNER = np.array([[a & 1, (a >> 1) & 1, (a >> 2) & 1] for a in range(8)])
_G = (0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0))


def _shape(h, xi):
    """Trilinear values [8] and gradients [8, 3] at reference point xi in [0, 1]^3."""
    f = np.where(_CORNER == 1, xi, 1.0 - np.asarray(xi))
    d = np.where(_CORNER == 1, 1.0, -1.0) / np.asarray(h)
    val = f.prod(1)
    grad = np.stack([d[:, 0] * f[:, 1] * f[:, 2], f[:, 0] * d[:, 1] * f[:, 2], f[:, 0] * f[:, 1] * d[:, 2]], 1)
    return val, grad


def _volume(h, eps, mu, k0):
    """24 x 24: (1/eps) curl.curl + div.div - k0^2 mu, dof 3 a + component."""
    out = np.zeros((8, 3, 8, 3), complex)
    eye = np.eye(3)
    for q in range(8):
        val, g = _shape(h, [_G[q & 1], _G[(q >> 1) & 1], _G[(q >> 2) & 1]])
        w = np.prod(h) / 8.0
        gg = np.einsum("ak,bk->ab", g, g)
        curl = np.einsum("ab,ij->aibj", gg, eye) - np.einsum("aj,bi->aibj", g, g)
        out += w * (curl / eps + np.einsum("ai,bj->aibj", g, g) -
                    k0 * k0 * mu * np.einsum("ab,ij->aibj", np.outer(val, val), eye))
    return out.reshape(24, 24)


def _faces(h, f, k0):
    """Quadrature points of face f with values, tangential gradients and weights; and its 24 x 24 absorbing form."""
    nu, side = f >> 1, f & 1
    t = [a for a in range(3) if a != nu]
    pts, form = [], np.zeros((8, 3, 8, 3), complex)
    for q in range(4):
        xi = np.zeros(3)
        xi[nu], xi[t[0]], xi[t[1]] = side, _G[q & 1], _G[q >> 1]
        val, g = _shape(h, xi)
        val = np.where(_CORNER[:, nu] == side, val, 0.0)
        g = np.where((_CORNER[:, nu] == side)[:, None], g, 0.0)
        g[:, nu] = 0.0
        w = h[t[0]] * h[t[1]] / 4.0
        m = 1j * k0 * np.outer(val, val) + 1j / (2.0 * k0) * (g @ g.T)
        for c in t:
            form[:, c, :, c] += w * m
        pts.append((xi, val, g, w))
    return pts, form.reshape(24, 24)


class _Exact:
    """The matrix of a voxel problem, applied element by element in complex128 (absorbing faces all round)."""

    def __init__(self, prob, dev):
        self.dev, self.prob, h = dev, prob, prob.h
        self.k0 = 2.0 * math.pi * prob.freq_hz / W.C0
        ids = _active(prob)
        rank = np.full((prob.nx + 1) * (prob.ny + 1) * (prob.nz + 1), -1, np.int64)
        rank[ids] = np.arange(ids.size)
        self.n_dof = 3 * ids.size
        k, j, i = np.meshgrid(np.arange(prob.nz), np.arange(prob.ny), np.arange(prob.nx), indexing="ij")
        self.ijk = np.stack([i.ravel(), j.ravel(), k.ravel()], 1)
        node = [(self.ijk[:, 0] + c[0]) + (prob.nx + 1) * ((self.ijk[:, 1] + c[1]) + (prob.ny + 1) *
                                                           (self.ijk[:, 2] + c[2])) for c in _CORNER]
        self.dofs = (3 * rank[np.stack(node, 1)][:, :, None] + np.arange(3)).reshape(-1, 24)
        mat = np.asarray(prob.material).ravel()
        self.parts = []
        for m in np.unique(mat):
            if m != W.PEC:
                self._part(np.flatnonzero(mat == m), _volume(h, prob.eps_r[m], prob.mu_r[m], self.k0))
        self.face = []
        dim = (prob.nx, prob.ny, prob.nz)
        for f in range(6):
            el = np.flatnonzero(self.ijk[:, f >> 1] == (dim[f >> 1] - 1 if f & 1 else 0))
            pts, form = _faces(h, f, self.k0)
            self._part(el, form)
            self.face.append((f, el, pts))

    def _part(self, el, a):
        self.parts.append((torch.as_tensor(self.dofs[el], device=self.dev), torch.as_tensor(a, device=self.dev)))

    def __call__(self, x):
        y = torch.zeros_like(x)
        step = max(1, (1 << 24) // (24 * x.shape[1]))
        for dofs, a in self.parts:
            for c in range(0, dofs.shape[0], step):
                d = dofs[c:c + step]
                z = torch.einsum("ij,ejr->eir", a, x[d]) if x.shape[1] > 1 else (x[d][..., 0] @ a.T)[..., None]
                y.index_add_(0, d.reshape(-1), z.reshape(-1, x.shape[1]))
        return y

    def diagonal(self):
        d = torch.zeros(self.n_dof, dtype=torch.complex128, device=self.dev)
        for dofs, a in self.parts:
            d.index_add_(0, dofs.reshape(-1), a.diagonal().repeat(dofs.shape[0]))
        return d[:, None]

    def rhs(self, waves):
        """b(W) = G(W, H_i) - int W . (n x curl H_i) over the outer faces, 2 x 2 Gauss points a face."""
        k0, h, org = self.k0, np.asarray(self.prob.h), np.asarray(self.prob.origin)
        b = np.zeros((self.n_dof, waves.count), complex)
        for f, el, pts in self.face:
            nu, n = f >> 1, np.zeros(3)
            n[nu] = 1.0 if f & 1 else -1.0
            for xi, val, g, w in pts:
                pos = org + (self.ijk[el] + xi) * h
                for r in range(waves.count):
                    k, p = waves.k_hat[r], waves.p_hat[r]
                    e = waves.amplitude[r] * np.exp(-1j * k0 * (pos @ k))
                    u = k * (n @ p) - p * (n @ k)
                    for c in range(3):
                        v = 1j * k0 * val * u[c]
                        if c != nu:
                            v = v + 1j * k0 * val * p[c] + 0.5 * (g @ k) * p[c]
                        for a in range(8):
                            if v[a] != 0:
                                np.add.at(b[:, r], self.dofs[el, 3 * a + c], w * v[a] * e)
        return torch.as_tensor(b, device=self.dev)

    def solve(self, b, tol=1e-13, limit=60000):
        """COCG with diagonal preconditioning on all columns, restarted from the true residual until it is below tol."""
        minv = 1.0 / self.diagonal()
        bn = torch.linalg.vector_norm(b, dim=0)
        x, its = torch.zeros_like(b), 0
        r = b.clone()
        while its < limit:
            stop = 0.2 * tol * bn
            z = minv * r
            p, rho = z.clone(), (r * z).sum(0)
            live = torch.ones_like(bn)
            while its < limit:
                q = self(p)
                alpha = live * rho / (p * q).sum(0)
                x += alpha * p
                r -= alpha * q
                its += 1
                if its % 40 == 0:
                    norm = torch.linalg.vector_norm(r, dim=0)
                    if bool((norm <= stop).all()):
                        break
                z = minv * r
                new = (r * z).sum(0)
                p = z + (new / rho) * p
                rho = new
            r = b - self(x)
            if bool((torch.linalg.vector_norm(r, dim=0) <= tol * bn).all()):
                break
        return x


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "serve":
        out = []
        for prob, waves in _requests(case, seed):
            a = _Exact(prob, dev)
            out.append(a.solve(a.rhs(waves)).cpu().numpy())
        return out
    prob = _problem(case, seed)
    a = _Exact(prob, dev)
    if case["kind"] == "solve":
        return a.solve(a.rhs(_waves(case, seed))).cpu().numpy()
    x = _field(prob, case["nrhs"], seed)
    if case["kind"] == "setup":
        return {"b": a.rhs(_waves(case, seed)), "y": a(x), "n_dof": None, "nnzb": None, "n_faces_ext": None,
                "n_faces_pec": None}
    if case["precision"] == "mixed":
        x = x.to(torch.complex64).to(torch.complex128)
    y = a(x)
    if case["precision"] != "df":
        return y
    v = torch.view_as_real(y)
    hi = v.float().double()
    return torch.cat([hi, v - hi], dim=-1)
