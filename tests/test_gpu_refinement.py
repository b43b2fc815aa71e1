"""What the refinement (csrc/solve.cu, csrc/batch.cu) reports and accepts: residuals against
b - A u formed from the FP64 form's matrix, tolerances that FP64 solutions cannot reach, and
coefficients of any scale."""
import numpy as np
import pytest

from test_gpu_contract_rows import _bar_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1811_03339_gb300 import fem3  # noqa: E402

ALPHA, K = (1.3, 1.6, 1.8), (1.0, 2.0, 0.5)
MIXED = ("tf32x3", "bf16x3", "fp32")


def _dense(mesh, f, alpha=ALPHA, k=K):
    """the FP64 form's matrix and load vectors [n_dof, nrhs]"""
    m = fem3.Mesh(mesh.verts, mesh.tets)
    A = m.assemble(alpha, k, "fp64", return_matrix=True)
    b = m.load(f).reshape(m.n_dof, -1)
    m.free()
    return A, b


def _residual(A, b, u):
    r = b - A @ u.reshape(b.shape)
    return float((r.norm(dim=0) / b.norm(dim=0)).max())


def _source(mesh, nrhs, seed=1):
    return torch.from_numpy(np.random.default_rng(seed).standard_normal((mesh.n_nodes, nrhs))).cuda()


@pytest.mark.parametrize("precision", MIXED)
def test_batch_residual_is_double_float(precision):
    """The residual that a run reports is b - A u to what double-float products and the evaluation
    here (FP64, a matrix that differs by 2^-48 of its terms) leave open: with |A| |u| near 10 |b|, as
    on these meshes, below 1e-14 of b.  Updates in plain FP32 are off by 2^-24 of |A| |d| with d of
    1e-6 of u, a few 1e-14."""
    meshes = [_bar_mesh(c) for c in ((9, 8, 10), (14, 11, 9), (13, 13, 13))]
    fs = [_source(m, 3, i) for i, m in enumerate(meshes)]
    dense = [_dense(m, f) for m, f in zip(meshes, fs)]
    b = fem3.Batch([(m.verts, m.tets) for m in meshes])
    n = len(meshes)
    for tol in (1e-6, 1e-7, 1e-8, 1e-9, 1e-10, 1e-12):
        us = b.run(np.tile(ALPHA, (n, 1)), np.tile(K, (n, 1)), fs, precision, tol=tol)
        for (A, rhs), u, res in zip(dense, us, b.resid):
            true = _residual(A, rhs, u)
            assert res <= tol
            assert abs(res - true) <= 1e-14, (tol, res, true)
    b.free()


@pytest.mark.parametrize("precision", MIXED)
def test_unreachable_tolerance_is_refused(precision):
    """FP64 u leaves a residual of 2^-53 of |A| |u| or so, above 1e-17 of b whatever the matrix."""
    mesh = _bar_mesh((9, 8, 10))
    f = _source(mesh, 2)
    m = fem3.Mesh(mesh.verts, mesh.tets)
    m.assemble(ALPHA, K, precision)
    with pytest.raises(fem3.Fem3Error) as e:
        m.solve(f, tol=1e-22, max_iter=12)
    assert e.value.code == fem3.FEM3_E_NO_CONVERGE
    m.solve(f, tol=1e-12)   # the handle is still good
    m.free()
    b = fem3.Batch([(mesh.verts, mesh.tets)] * 2)
    with pytest.raises(fem3.Fem3Error) as e:
        b.run(np.tile(ALPHA, (2, 1)), np.tile(K, (2, 1)), [f, f], precision, tol=1e-17, max_iter=12)
    assert e.value.code == fem3.FEM3_E_NO_CONVERGE
    b.free()


@pytest.mark.parametrize("nrhs", [1, 5, 17])
@pytest.mark.parametrize("precision", MIXED)
def test_reported_residual_has_the_rounding_of_u(precision, nrhs):
    """At tolerances below it the residual is that of u's rounding to FP64: the norm of A c for c
    uniform within half a unit of u's entries, a sum of some 1e5 independent terms, here within a factor of
    four.  A residual that leaves the rounding out shrinks on with tol."""
    mesh = _bar_mesh((13, 13, 13))
    f = _source(mesh, nrhs)
    A, b = _dense(mesh, f)
    m = fem3.Mesh(mesh.verts, mesh.tets)
    m.assemble(ALPHA, K, precision)
    for tol in (1e-15, 1e-17):
        u = m.solve(f, tol=tol).reshape(b.shape)
        ulp = torch.ldexp(torch.ones_like(u), torch.frexp(u).exponent - 53)
        c = ulp * (torch.rand(u.shape, dtype=u.dtype, device="cuda",
                              generator=torch.Generator("cuda").manual_seed(3)) - 0.5)
        floor = float(((A @ c).norm(dim=0) / b.norm(dim=0)).max())
        assert floor / 4 <= m.resid <= 4 * floor, (tol, m.resid, floor)
    m.free()


@pytest.mark.parametrize("precision", MIXED)
def test_coefficients_of_any_scale(precision):
    """K times a power of two divides the solution by it: to the refinement's tolerance, for
    scales at which s K w is no FP32 pair (below 2^-74 such a pair has 24 bits)."""
    mesh = _bar_mesh((6, 8, 7), h=(0.2, 0.1, 0.15))
    f = _source(mesh, 3)
    A, b = _dense(mesh, f)
    ref = torch.linalg.solve(A, b)
    for e in (-90, -75, -60, 0, 60):
        m = fem3.Mesh(mesh.verts, mesh.tets)
        m.assemble(ALPHA, [k * 2.0 ** e for k in K], precision)
        u = m.solve(f, tol=1e-12).reshape(ref.shape) * 2.0 ** e
        m.free()
        assert float((u - ref).norm() / ref.norm()) <= 1e-10, e


@pytest.mark.parametrize("precision", ["tf32x3", "fp64"])
def test_batch_replay_after_another_scale(precision):
    """A replayed graph writes the operator of the run it was captured from, whatever operator the
    mesh's handle was used with since."""
    import ctypes as C
    mesh = _bar_mesh((6, 8, 7), h=(0.2, 0.1, 0.15))
    f = _source(mesh, 2)
    A, b = _dense(mesh, f)
    ref = torch.linalg.solve(A, b)
    batch = fem3.Batch([(mesh.verts, mesh.tets)])
    h = C.c_void_p()
    fem3._check(fem3._lib.fem3_batch_mesh(batch.h, 0, C.byref(h)))
    fc, u1 = f.T.contiguous(), torch.empty((2, batch.n_dof[0]), dtype=torch.float64, device="cuda")
    for _ in range(4):   # eager, captured, replayed twice
        u = batch.run([ALPHA], [K], [f], precision)[0]
        assert float((u - ref).norm() / ref.norm()) <= 1e-8
        fem3.solve(h, fc, 2, u1)   # the run's factor and operator
        assert float((u1.T - ref).norm() / ref.norm()) <= 1e-8
        fem3.assemble(h, (1.7, 1.2, 1.5), [k * 2.0 ** 40 for k in K], "tf32x3")
        fem3.solve(h, fc, 2, u1)
    batch.free()
