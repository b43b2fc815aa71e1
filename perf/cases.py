"""The work that this library is timed on, through its public entry points.

A user uploads a tetrahedral mesh, assembles the Riesz operator (or one of the other
operators) on it and solves for one or more right-hand sides; keeps a handle and solves
again; differentiates a loss through the solve; or hands over a batch of meshes.  The
listed cases are one or two sizes of each; ``draw`` spreads the same kinds over their ranges.

Every mesh is a Kuhn-split cube (six tetrahedra a cell), its interior vertices jittered and,
for ``skew``, mapped to the parallelepiped of the largest configuration.  ``exact`` solves the
same problem in FP64 with plain torch: every Gauss-point line is cut with every tetrahedron
near it, without walking from one to the next.
"""
import math

import numpy as np
import torch

from paper_1811_03339_gb300 import fem3, inputs

AFFINE = inputs.PARALLELEPIPED24["affine"]


# ---------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------
def _step(name, n, precision, nrhs=1, jitter=0.2, skew=False, alpha=(1.3, 1.6, 1.8),
          K=(1.0, 2.0, 0.5), matrix=False, kind="step"):
    c = dict(kind=kind, n=n, jitter=jitter, skew=skew, precision=precision, nrhs=nrhs,
             matrix=matrix)
    c.update({f"alpha{i}": alpha[i] for i in range(3)})
    c.update({f"K{i}": K[i] for i in range(3)})
    return dict(name=name, **c) if name else c


def listed():
    return [
        # a first look at a problem, or one of many tiny ones: all launches and host work
        _step("step_cube4_fp64", 4, "fp64", jitter=0.1, alpha=(1.5, 1.5, 1.5),
              K=(1.0, 1.0, 1.0)),
        # an ordinary solve in the tensor-core form: upload, assemble, factor, refine
        _step("step_cube16_tf32x3", 16, "tf32x3"),
        # the largest configuration: many right-hand sides on a skew domain
        _step("step_skew24_bf16x3_17rhs", 24, "bf16x3", nrhs=17, jitter=0.15, skew=True,
              alpha=(1.2, 1.5, 1.9), K=(1.0, 1.0, 1.0)),
        # FP64 throughout with the matrix handed out (spectra, conditioning, other solvers);
        # a size that no tile divides
        _step("step_skew11_fp64_matrix", 11, "fp64", nrhs=3, jitter=0.15, skew=True,
              alpha=(1.2, 1.5, 1.9), matrix=True),
        # FP32 contraction on the CUDA cores, for users who want no split products
        _step("step_cube13_fp32", 13, "fp32", nrhs=2),
        # time stepping and parameter studies: a factored handle, new sources each call
        _step("resolve_skew20_bf16x3_8rhs", 20, "bf16x3", nrhs=8, jitter=0.15, skew=True,
              alpha=(1.2, 1.5, 1.9), kind="resolve"),
        # one iteration of an inverse problem: assemble and solve forward, then the gradient
        # of a loss in K and f
        _step("gradient_cube16_tf32x3", 16, "tf32x3", kind="gradient"),
        # many uneven meshes at once, 16 right-hand sides each
        dict(name="batch12_tf32x3_16rhs", kind="batch", meshes=12, nmin=6, nmax=20,
             sizes_seed=3, precision="tf32x3", nrhs=16),
        # the divergence form with variable coefficients: six general-form terms, GMRES
        dict(name="divergence_skew8_fp64", kind="divergence", n=8, jitter=0.15, skew=True,
             precision="fp64", nrhs=2, beta0=0.6, beta1=0.7, beta2=0.8),
        # one term of the general form, for operators that a user composes
        dict(name="form_cube13_fp64", kind="form", n=13, jitter=0.2, skew=False,
             precision="fp64", axis=1, alpha=0.7, beta=0.4, trial_left=True, coef=True),
        # the integer-order comparison: P1 stiffness, dense FP64 solve
        dict(name="integer_cube15", kind="integer", n=15, jitter=0.2, skew=False, nrhs=1,
             K0=1.0, K1=2.0, K2=0.5),
        # a small dense system inside a loop that must not allocate
        dict(name="static_384", kind="static", n=384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "resolve", "gradient", "batch", "divergence",
                       "form", "integer", "static"])
    skew = rng.random() < 0.5
    jitter = round(rng.uniform(0.05, 0.2), 3)
    mesh = dict(jitter=jitter, skew=skew)
    if kind in ("step", "resolve", "gradient"):
        precision = rng.choice(["tf32x3", "bf16x3", "tf32x3", "bf16x3", "fp64", "fp32"])
        n = _log_int(rng, 4, 13 if precision in ("fp64", "fp32") else 23)
        return _step(None, n, precision, kind=kind, **mesh,
                     nrhs=1 if kind == "gradient" else rng.choice([1, 1, 2, 5, 8, 16, 17]),
                     matrix=kind == "step" and precision == "fp64" and rng.random() < 0.5,
                     alpha=tuple(round(rng.uniform(1.1, 1.95), 3) for _ in range(3)),
                     K=tuple(round(rng.uniform(0.5, 2.0), 3) for _ in range(3)))
    if kind == "batch":
        nmin = rng.randint(4, 8)
        return dict(kind=kind, meshes=rng.randint(3, 10), nmin=nmin, nmax=nmin + rng.randint(2, 9),
                    sizes_seed=rng.randint(0, 999), precision=rng.choice(["tf32x3", "bf16x3"]),
                    nrhs=rng.choice([1, 4, 9, 16]))
    if kind == "divergence":
        return dict(kind=kind, n=_log_int(rng, 4, 10), **mesh, precision="fp64",
                    nrhs=rng.randint(1, 2),
                    **{f"beta{i}": round(rng.uniform(0.4, 0.9), 3) for i in range(3)})
    if kind == "form":
        return dict(kind=kind, n=_log_int(rng, 4, 14), **mesh, precision="fp64",
                    axis=rng.randint(0, 2), alpha=round(rng.uniform(0.1, 0.9), 3),
                    beta=round(rng.uniform(0.1, 0.9), 3), trial_left=rng.random() < 0.5,
                    coef=rng.random() < 0.5)
    if kind == "integer":
        return dict(kind=kind, n=_log_int(rng, 4, 16), **mesh, nrhs=rng.randint(1, 3),
                    **{f"K{i}": round(rng.uniform(0.5, 2.0), 3) for i in range(3)})
    return dict(kind=kind, n=_log_int(rng, 16, 512))


# ---------------------------------------------------------------------------------
# inputs (seeded)
# ---------------------------------------------------------------------------------
def _triple(case, key):
    return tuple(case[f"{key}{i}"] for i in range(3))


def _mesh(case, seed):
    return inputs.cube_mesh(case["n"], case["jitter"], seed, AFFINE if case["skew"] else None)


def _sources(n_nodes, nrhs, seed):
    """nodal sources: a constant one first where there are several, then N(0, 1) columns"""
    f = np.random.default_rng([seed, 7]).standard_normal((n_nodes, nrhs))
    if nrhs > 1:
        f[:, 0] = 1.0
    return f if nrhs > 1 else f[:, 0].copy()


def _gauss_points(verts, tets):
    a, b = (5 + 3 * math.sqrt(5)) / 20, (5 - math.sqrt(5)) / 20
    bary = np.full((4, 4), b) + (a - b) * np.eye(4)
    return np.einsum("qk,tkd->tqd", bary, verts[tets]).reshape(-1, 3)


def _coefficients(mesh):
    """Section 3's p_i = cos x_i, q_i = 1 - cos x_i at the Gauss points"""
    x = _gauss_points(mesh.verts, mesh.tets)
    p = np.ascontiguousarray(np.cos(x).T)
    return p, 1.0 - p


def _batch_inputs(case, seed):
    ns = np.random.default_rng(case["sizes_seed"]).integers(case["nmin"], case["nmax"] + 1,
                                                            size=case["meshes"])
    rng = np.random.default_rng([seed, 5])
    meshes = [inputs.cube_mesh(int(n)) for n in ns]
    alpha = rng.uniform(1.1, 1.9, size=(len(ns), 3))
    fs = [rng.standard_normal((m.n_nodes, case["nrhs"])) for m in meshes]
    return meshes, alpha, np.ones((len(ns), 3)), fs


def _spd(n, seed):
    rng = np.random.default_rng([seed, 9])
    B = rng.standard_normal((n, n))
    return B @ B.T + n * np.eye(n), rng.standard_normal(n)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "static":
        A, b = _spd(case["n"], seed)
        return dict(case=case, A=_gpu(A), b=_gpu(b), x=torch.empty(case["n"], dtype=torch.float64,
                                                                  device="cuda"))
    if kind == "batch":
        meshes, alpha, K, fs = _batch_inputs(case, seed)
        return dict(case=case, batch=fem3.Batch([(m.verts, m.tets) for m in meshes]),
                    alpha=alpha, K=K, fs=[_gpu(f) for f in fs])
    mesh = _mesh(case, seed)
    st = dict(case=case, verts=_gpu(mesh.verts), tets=_gpu(mesh.tets))
    if "nrhs" in case:
        st["f"] = _gpu(_sources(mesh.n_nodes, case["nrhs"], seed))
    if kind == "resolve":
        st["mesh"] = fem3.Mesh(st["verts"], st["tets"])
        st["mesh"].assemble(_triple(case, "alpha"), _triple(case, "K"), case["precision"])
        st["mesh"].solve(torch.ones_like(st["f"]))
    elif kind == "gradient":
        st["mesh"] = fem3.Mesh(st["verts"], st["tets"])
        st["K"] = torch.tensor(_triple(case, "K"), dtype=torch.float64, device="cuda",
                               requires_grad=True)
        st["f"].requires_grad_(True)
        st["grad_u"] = _gpu(_upstream(st["mesh"].n_dof, seed))
    elif kind == "divergence":
        p, q = _coefficients(mesh)
        st.update(p=_gpu(p), q=_gpu(q))
    elif kind == "form":
        st["mesh"] = fem3.Mesh(st["verts"], st["tets"])
        st["c"] = _gpu(_coefficients(mesh)[0][case["axis"]]) if case["coef"] else None
    return st


def _upstream(n_dof, seed):
    return np.random.default_rng([seed, 8]).standard_normal(n_dof)


# ---------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "static":
        fem3.spd_solve_static(state["A"], state["b"], state["x"])
        return state["x"]
    if kind == "batch":
        return state["batch"].run(state["alpha"], state["K"], state["fs"], case["precision"])
    if kind == "resolve":
        return state["mesh"].solve(state["f"])
    if kind == "gradient":
        u = fem3.frac_solve(state["mesh"], _triple(case, "alpha"), state["K"], state["f"],
                            case["precision"])
        gK, gf = torch.autograd.grad(u, (state["K"], state["f"]), state["grad_u"])
        return dict(u=u.detach(), K=gK, f=gf)
    if kind == "form":
        return state["mesh"].assemble_form(case["axis"], case["alpha"], case["beta"],
                                           case["trial_left"], state["c"], case["precision"])
    mesh = fem3.Mesh(state["verts"], state["tets"])
    if kind == "divergence":
        mesh.assemble_divergence(_triple(case, "beta"), state["p"], state["q"],
                                 case["precision"])
        A = None
    elif kind == "integer":
        mesh.assemble_integer(_triple(case, "K"))
        A = None
    else:
        A = mesh.assemble(_triple(case, "alpha"), _triple(case, "K"), case["precision"],
                          return_matrix=case["matrix"])
    u = mesh.solve(state["f"])
    mesh.free()
    return (u, A) if A is not None else u


# ---------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------
def _solve_flops(n, factor=True):
    """flops(n_dof, nrhs) of a dense symmetric factorisation and its solves"""
    return lambda nrhs: (n ** 3 / 3 if factor else 0) + 2.0 * n * n * nrhs


def _element_flops(n, axes=3):
    """Sum over Gauss points of the outer products of a row of L and one of R.  A path that
    crosses all n cells touches about 3 n vertices, so the two sides of a point at the fraction
    t of its chord have 3 n t and 3 n (1 - t) nonzeros: 1.5 n^2 pairs on average."""
    return axes * 24 * n ** 3 * 4 * 1.5 * n * n


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "static":
        return dict(bytes=8 * (n * n / 2 + 2 * n), flops=_solve_flops(n)(1))
    if kind == "batch":
        ns = np.random.default_rng(case["sizes_seed"]).integers(case["nmin"], case["nmax"] + 1,
                                                                size=case["meshes"])
        parts = [(int(k), int((k - 1) ** 3)) for k in ns]
        return dict(bytes=sum(8 * case["nrhs"] * ((k + 1) ** 3 + d) + 24 * (k + 1) ** 3 + 96 * k ** 3
                              for k, d in parts),
                    flops=sum(_solve_flops(d)(case["nrhs"]) + _element_flops(k) for k, d in parts))
    nodes, tets, dofs = (n + 1) ** 3, 6 * n ** 3, (n - 1) ** 3
    nrhs = case.get("nrhs", 0)
    mesh_bytes = 24 * nodes + 16 * tets
    io = 8 * nrhs * (nodes + dofs)
    if kind == "resolve":
        return dict(bytes=io + 2 * dofs * dofs, flops=_solve_flops(dofs, factor=False)(nrhs))
    if kind == "form":
        return dict(bytes=mesh_bytes + 8 * dofs * dofs + (32 * tets if case["coef"] else 0),
                    flops=_element_flops(n, 1) / 2)
    if kind == "integer":
        return dict(bytes=mesh_bytes + io, flops=_solve_flops(dofs)(nrhs))
    if kind == "divergence":
        return dict(bytes=mesh_bytes + io + 6 * 32 * tets,
                    flops=_solve_flops(dofs)(nrhs) + 6 * 24 * n ** 3 * 2 * 4 * 1.5 * n)
    flops = _solve_flops(dofs)(nrhs if kind == "step" else 2) + _element_flops(n)
    bytes_ = mesh_bytes + (2 if kind == "gradient" else 1) * io
    return dict(bytes=bytes_ + (8 * dofs * dofs if case.get("matrix") else 0), flops=flops)


# ---------------------------------------------------------------------------------
# the same problems in FP64 with plain torch
# ---------------------------------------------------------------------------------
class _Exact:
    def __init__(self, mesh, n):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.n = n
        self.v = torch.as_tensor(mesh.verts, device=dev)
        self.t = torch.as_tensor(mesh.tets, device=dev).long()
        T = self.t.shape[0]
        corners = self.v[self.t]                                   # [T, 4, 3]
        self.box = corners.amin(1), corners.amax(1)
        B = torch.cat([torch.ones(T, 1, 4, device=dev, dtype=torch.float64),
                       corners.transpose(1, 2)], 1)
        self.M = torch.linalg.inv(B)                               # lambda_k = M[k] . (1, x)
        self.vol = torch.linalg.det(B).abs() / 6
        self.x = torch.as_tensor(_gauss_points(mesh.verts, mesh.tets), device=dev)
        self.w = (self.vol / 4).repeat_interleave(4)
        g = torch.arange(n + 1, device=dev)
        inside = (g > 0) & (g < n)
        self.interior = (inside[:, None, None] & inside[None, :, None] & inside).reshape(-1)
        self.dof = torch.where(self.interior, self.interior.cumsum(0) - 1, -1)
        self.n_dof = int(self.interior.sum())
        self.span = float((self.v.amax(0) - self.v.amin(0)).max())

    def chunks(self, axis, size=1024):
        """Gauss points in groups that lie close together across the axis, each with the
        tetrahedra whose boxes meet the group's box there"""
        c = [i for i in range(3) if i != axis]
        lo, hi = self.v.amin(0), self.v.amax(0)
        cell = ((self.x - lo) / (hi - lo) * self.n).floor().clamp(0, self.n - 1).long()
        order = torch.argsort(cell[:, c[0]] * self.n + cell[:, c[1]], stable=True)
        for s in range(0, len(order), size):
            g = order[s:s + size]
            a, b = self.x[g].amin(0), self.x[g].amax(0)
            near = ((self.box[0][:, c] <= b[c]) & (self.box[1][:, c] >= a[c])).all(1)
            yield g, near.nonzero()[:, 0]

    def rows(self, g, near, axis, direction, order):
        """Rows g of the left (direction -1) or right (+1) table as padded lists: dof [C, P]
        (-1: none) and value [C, P]"""
        M = self.M[near]
        lam = M[None, :, :, 0] + torch.einsum("cd,tkd->ctk", self.x[g], M[:, :, 1:])
        slope = direction * M[None, :, :, 1 + axis]
        r = -lam / slope
        inf = math.inf
        r0 = torch.where(slope > 0, r, -inf).amax(2).clamp(min=0.0)
        r1 = torch.where(slope < 0, r, inf).amin(2)
        hit = (r1 - r0 > 1e-12 * self.span) & ~((slope == 0) & (lam < 0)).any(2)
        c, t = hit.nonzero(as_tuple=True)
        p = 1.0 - order

        def power(s):
            return torch.where(s > 0, s ** p, torch.zeros_like(s))
        val = (power(r1[c, t]) - power(r0[c, t])) * (-direction / math.gamma(2 - order))
        val = (val[:, None] * M[t, :, 1 + axis]).reshape(-1)
        j = self.dof[self.t[near[t]]].reshape(-1)
        key = (c.repeat_interleave(4) * (self.n_dof + 1) + j)[j >= 0]
        key, inv = torch.unique(key, return_inverse=True)
        tot = torch.zeros(len(key), dtype=torch.float64, device=val.device)
        tot.index_add_(0, inv, val[j >= 0])
        row = key // (self.n_dof + 1)
        count = torch.bincount(row, minlength=len(g))
        at = torch.arange(len(key), device=key.device) - (count.cumsum(0) - count)[row]
        P = max(1, int(count.max()))
        J = torch.full((len(g), P), -1, dtype=torch.int64, device=key.device)
        V = torch.zeros((len(g), P), dtype=torch.float64, device=key.device)
        J[row, at] = key % (self.n_dof + 1)
        V[row, at] = tot
        return J, V

    def form(self, axis, order_left, order_right, coef=None):
        """F[j, k] = sum_g w_g c_g L[g, j] R[g, k]"""
        F = torch.zeros(self.n_dof * self.n_dof, dtype=torch.float64, device=self.x.device)
        w = self.w if coef is None else self.w * coef
        for g, near in self.chunks(axis):
            jl, vl = self.rows(g, near, axis, -1, order_left)
            jr, vr = self.rows(g, near, axis, +1, order_right)
            pairs = jl[:, :, None] * self.n_dof + jr[:, None, :]
            ok = (jl >= 0)[:, :, None] & (jr >= 0)[:, None, :]
            val = (vl * w[g][:, None])[:, :, None] * vr[:, None, :]
            F.index_add_(0, pairs[ok], val[ok])
        return F.view(self.n_dof, self.n_dof)

    def axis_matrix(self, axis, alpha):
        """dA/dK_axis of the Riesz operator"""
        F = self.form(axis, alpha / 2, alpha / 2)
        return (F + F.T) / (2.0 * math.cos(math.pi * alpha / 2.0))

    def stiffness(self, axis, coef=1.0):
        """sum_T |T| c_T (d phi_j / dx_axis)(d phi_k / dx_axis) over the dofs"""
        d = self.M[:, :, 1 + axis]
        val = (self.vol * coef)[:, None, None] * d[:, :, None] * d[:, None, :]
        j = self.dof[self.t]
        ok = (j >= 0)[:, :, None] & (j >= 0)[:, None, :]
        pairs = j[:, :, None] * self.n_dof + j[:, None, :]
        S = torch.zeros(self.n_dof * self.n_dof, dtype=torch.float64, device=self.x.device)
        S.index_add_(0, pairs[ok], val[ok])
        return S.view(self.n_dof, self.n_dof)

    def mass(self, f):
        """P1 mass matrix (all nodes) times f [n_nodes, r]"""
        ft = f[self.t]                                             # [T, 4, r]
        e = (ft.sum(1, keepdim=True) + ft) * (self.vol / 20)[:, None, None]
        b = torch.zeros_like(f)
        return b.index_add_(0, self.t.reshape(-1), e.reshape(-1, f.shape[1]))

    def load(self, f):
        f = torch.as_tensor(f, device=self.x.device)
        return self.mass(f.reshape(f.shape[0], -1))[self.interior]


def exact(case, seed):
    kind = case["kind"]
    if kind == "static":
        A, b = _spd(case["n"], seed)
        return torch.linalg.solve(torch.from_numpy(A), torch.from_numpy(b))
    if kind == "batch":
        meshes, alpha, K, fs = _batch_inputs(case, seed)
        out = []
        for m, a, f in zip(meshes, alpha, fs):
            e = _Exact(m, m.n)
            A = sum(e.axis_matrix(i, float(a[i])) for i in range(3))
            out.append(torch.linalg.solve(A, e.load(f)))
        return out
    mesh = _mesh(case, seed)
    e = _Exact(mesh, mesh.n)
    if kind == "form":
        left = case["trial_left"]
        c = e.x[:, case["axis"]].cos() if case["coef"] else None
        F = e.form(case["axis"], case["alpha"] if left else case["beta"],
                   case["beta"] if left else case["alpha"], c)
        return F.T.contiguous() if left else F      # row: test function, column: trial function
    f = _sources(mesh.n_nodes, case["nrhs"], seed)
    b = e.load(f)
    if kind == "divergence":
        # -(p D_L u, D v) + (q D_R u, D v): D the first derivative (order 1 of either table is
        # the slope on the point's own tetrahedron, with a minus sign on the right)
        A = 0
        for i in range(3):
            p = e.x[:, i].cos()
            A = A + e.form(i, case[f"beta{i}"], 1.0, p).T
            A = A + e.form(i, 1.0, case[f"beta{i}"], 1.0 - p)
        u = torch.linalg.solve(A, b)
    elif kind == "integer":
        A = sum(case[f"K{i}"] * e.stiffness(i) for i in range(3))
        u = torch.linalg.solve(A, b)
    else:
        parts = [e.axis_matrix(i, case[f"alpha{i}"]) for i in range(3)]
        A = sum(case[f"K{i}"] * parts[i] for i in range(3))
        u = torch.linalg.solve(A, b)
    if kind == "gradient":
        g = torch.as_tensor(_upstream(e.n_dof, seed), device=u.device)
        lam = torch.linalg.solve(A, g)
        full = torch.zeros(len(e.v), 1, dtype=torch.float64, device=u.device)
        full[e.interior, 0] = lam
        gK = torch.stack([-(lam @ (P @ u[:, 0])) for P in parts])
        return dict(u=u[:, 0], K=gK, f=e.mass(full)[:, 0])
    u = u[:, 0] if case["nrhs"] == 1 else u
    return (u, A) if case.get("matrix") else u
