"""The gradient's per-axis forms (k_axis_form, csrc/solve.cu): dK is bilinear in the solution and the
adjoint solution and is evaluated in FP64, so it keeps its digits under factors of two over the FP64
range and equals lambda^T (dA/dK_a) u formed densely.  Bins of one dof, of a few, and of more
rows and points than one round of a CTA takes."""
import numpy as np
import pytest

from test_gpu_contract_rows import SHAPES, _bar_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1811_03339_gb300 import fem3  # noqa: E402

ALPHA, K = (1.3, 1.6, 1.8), (1.0, 2.0, 0.5)


def _case(cells, scale):
    mesh = _bar_mesh(cells)
    m = fem3.Mesh(mesh.verts, mesh.tets, bin_scale=scale)
    rng = np.random.default_rng(5)
    u, g = (torch.from_numpy(rng.standard_normal(m.n_dof)).cuda() for _ in range(2))
    return mesh, m, u, g, torch.from_numpy(rng.standard_normal(mesh.n_nodes)).cuda()


def _dk(m, u, g):
    return np.asarray(m.vjp(u, g)[0])


@pytest.mark.parametrize("cells,scale", [s[:2] for s in SHAPES])
def test_forms_match_dense(cells, scale):
    mesh, m, u, g, f = _case(cells, scale)
    A = m.assemble(ALPHA, K, "fp64", return_matrix=True)
    parts = []
    for a in range(3):
        Ka = list(K)
        Ka[a] *= 2.0
        parts.append((m.assemble(ALPHA, Ka, "fp64", return_matrix=True) - A) / K[a])
    lam = torch.linalg.solve(A, g)
    ref = np.array([-float(lam @ (P @ u)) for P in parts])
    # rounding errors are relative to the sum of magnitudes; lambda is off by at most the condition
    # number (below 1e3) times 2^-53 (some) or the solve's 1e-12
    mag = max(float(lam.abs() @ (P.abs() @ u.abs())) for P in parts)
    for precision, bar in (("fp64", 1e-12), ("tf32x3", 1e-9)):
        m.assemble(ALPHA, K, precision)
        m.solve(f)
        assert np.abs(_dk(m, u, g) - ref).max() <= bar * mag
    m.free()


@pytest.mark.parametrize("precision,shifts_g", [("fp64", (-200, -140, -80, 80, 200)), ("tf32x3", (-60, 60))])
def test_forms_keep_digits_under_scaling(precision, shifts_g):
    """Powers of two are exact in every step of an FP64 evaluation; the sums over the bins are added
    in no fixed order (1e-12 of the largest)."""
    mesh, m, u, g, f = _case((5, 6, 4), 0.5)
    m.assemble(ALPHA, K, precision)
    m.solve(f)
    ref = _dk(m, u, g)
    bar = (1e-12 if precision == "fp64" else 1e-9) * np.abs(ref).max()
    for su in (-200, -80, 0, 140, 200):
        for sg in (0,) + shifts_g:
            dk = _dk(m, u * 2.0 ** su, g * 2.0 ** sg) * 2.0 ** -(su + sg)
            assert np.abs(dk - ref).max() <= bar, (su, sg, dk, ref)
    m.free()


def test_forms_pass_on_nan():
    mesh, m, u, g, f = _case((5, 3, 4), 0.5)
    m.assemble(ALPHA, K, "fp64")
    m.solve(f)
    u[3] = float("nan")
    assert np.isnan(_dk(m, u, g)).all()
    m.free()
