"""The CUDA-core contraction over the nonzeros (csrc/contract.cu, k_contract_rows) where its
windows and groups end: bins of more columns than one window, bins whose entries need several
groups of Gauss points, and bins of a few dofs; matrices against the oracle."""
import itertools

import numpy as np
import pytest

import oracle
from paper_1811_03339_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1811_03339_gb300 import fem3  # noqa: E402

# relative to the largest entry of the oracle's matrix: the FP64 form keeps 48-bit tables and
# FP64 sums; the FP32 form rounds each of up to a few thousand products to 24 bits
BAR = {"fp64": 1e-10, "fp32": 1e-5}


def _bar_mesh(cells, h=(1.0, 1.0, 1.0)):
    """Kuhn-split box of cells[0] x cells[1] x cells[2] cells of size h"""
    nx, ny, nz = (c + 1 for c in cells)
    idx = np.arange(nx * ny * nz).reshape(nz, ny, nx)
    z, y, x = np.meshgrid(*(np.arange(k) for k in (nz, ny, nx)), indexing="ij")
    verts = np.stack([x.ravel() * h[0], y.ravel() * h[1], z.ravel() * h[2]], 1).astype(np.float64)
    inner = ((x > 0) & (x < nx - 1) & (y > 0) & (y < ny - 1) & (z > 0) & (z < nz - 1)).ravel()
    rng = np.random.default_rng(12)
    verts[inner] += rng.uniform(-0.15, 0.15, (int(inner.sum()), 3)) * np.asarray(h)
    c = idx[:-1, :-1, :-1].ravel()
    step = (1, nx, nx * ny)
    tets = []
    for p in itertools.permutations(range(3)):
        a = c + step[p[0]]
        tets.append(np.stack([c, a, a + step[p[1]], c + sum(step)], 1))
    return inputs.Mesh(verts=verts, tets=np.ascontiguousarray(
        np.stack(tets, 1).reshape(-1, 4).astype(np.int32)))


# cells, bin_scale, least columns of the widest bin: one dof; a bin of a few dofs; one over 512
# columns (three windows of 256, more entries than shared memory holds: several groups)
SHAPES = [((2, 2, 2), 0.5, 1), ((5, 3, 4), 0.5, 4), ((45, 4, 5), 1.5, 513)]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("cells,scale,least", SHAPES)
def test_rows_contraction_matches_oracle(cells, scale, least, precision):
    mesh = _bar_mesh(cells)
    o = oracle.Oracle.from_mesh(mesh)
    alpha, K = (1.3, 1.6, 1.8), (1.0, 2.0, 0.5)
    m = fem3.Mesh(mesh.verts, mesh.tets, bin_scale=scale)
    assert max(m.bin_stats(a)["max_dof"] for a in range(3)) >= least
    A = m.assemble(alpha, K, precision, return_matrix=True).cpu().numpy()
    m.sync()
    A_ref = o.assemble(alpha, K)
    assert np.abs(A - A_ref).max() <= BAR[precision] * np.abs(A_ref).max()
    assert np.array_equal(A, A.T)
    # general form: the axis with the widest bins, both trial sides, with and without c
    c = np.cos(o.gp[:, 0])
    for left, coef in ((True, c), (False, None)):
        F = m.assemble_form(0, 0.7, 0.4, left, coef, precision).cpu().numpy()
        m.sync()
        F_ref = o.assemble_form(0, 0.7, 0.4, left, coef)
        assert np.abs(F - F_ref).max() <= BAR[precision] * np.abs(F_ref).max()
    m.free()


@pytest.mark.parametrize("precision", ["fp32", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("cells,scale", [(SHAPES[0][0], SHAPES[0][1]), (SHAPES[1][0], SHAPES[1][1]),
                                         (SHAPES[2][0], SHAPES[2][1])])
def test_operator_of_the_refinement(cells, scale, precision):
    """The refinement's operator from the same meshes (its contraction is the double-float one):
    1, 3 and 21 columns (one-, four- and 17-wide passes) refined to 1e-13 equal the oracle's
    solutions to 1e-10, and the mixed form's residual is that of the oracle's matrix."""
    mesh = _bar_mesh(cells)
    o = oracle.Oracle.from_mesh(mesh)
    alpha, K = (1.3, 1.6, 1.8), (1.0, 2.0, 0.5)
    A = o.assemble(alpha, K)
    m = fem3.Mesh(mesh.verts, mesh.tets, bin_scale=scale)
    m.assemble(alpha, K, precision)
    for nrhs in (1, 3, 21):
        f = np.random.default_rng(nrhs).standard_normal((mesh.n_nodes, nrhs))
        b = o.load(f)
        u = m.solve(f, tol=1e-13).cpu().numpy().reshape(o.n_dof, nrhs)
        ref = np.linalg.solve(A, b)
        assert np.linalg.norm(u - ref) <= 1e-10 * np.linalg.norm(ref)
        res = np.linalg.norm(b - A @ u, axis=0) / np.linalg.norm(b, axis=0)
        assert res.max() <= 1e-12, res
    m.free()
