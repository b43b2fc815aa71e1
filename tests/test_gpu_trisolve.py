"""The blocked triangular solves (csrc/trisolve.cu) at the edges of their diagonal blocks and
column groups: integer-order problems (FP64 factor) and FP32-form problems with the refinement
cut to one sweep, so that the FP32 solve itself shows."""
import numpy as np
import pytest

import oracle
from test_gpu_contract_rows import _bar_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1811_03339_gb300 import fem3  # noqa: E402

# orders n around the block widths: one block (64, 128, 512), ragged last blocks of the 256-wide
# FP64 and 512-wide FP32 doubling (513, 576, 605, 1,040)
SIZES = {64: (5, 5, 5), 128: (9, 9, 3), 130: (14, 11, 2), 256: (9, 9, 5), 260: (14, 11, 3),
         512: (9, 9, 9), 513: (20, 28, 2), 576: (9, 9, 10), 605: (12, 12, 6), 1040: (14, 11, 9)}


@pytest.mark.parametrize("n", sorted(SIZES))
@pytest.mark.parametrize("nrhs", [1, 3, 8, 17, 26])
def test_f64_solve_sizes(n, nrhs):
    mesh = _bar_mesh(SIZES[n])
    m = fem3.Mesh(mesh.verts, mesh.tets)
    assert m.n_dof == n
    A = m.assemble_integer((1.0, 2.0, 0.5), return_matrix=True).cpu().numpy()
    f = np.random.default_rng(n + nrhs).standard_normal((mesh.n_nodes, nrhs))
    u = m.solve(f).cpu().numpy().reshape(n, nrhs)
    b = m.load(torch.from_numpy(f).cuda()).cpu().numpy().reshape(n, nrhs)
    res = np.linalg.norm(b - A @ u, axis=0) / np.linalg.norm(b, axis=0)
    assert res.max() <= 1e-12, res
    m.free()


@pytest.mark.parametrize("n", [64, 130, 512, 605, 1040])
@pytest.mark.parametrize("nrhs", [1, 4, 17, 24])
def test_f32_solve_sizes(n, nrhs):
    """One sweep is the FP32 solve alone: its residual is that of an FP32 factorisation and
    substitution, far below 1e-3 (the iteration would need many sweeps otherwise)."""
    mesh = _bar_mesh(SIZES[n])
    o = oracle.Oracle.from_mesh(mesh)
    assert o.n_dof == n
    alpha, K = (1.3, 1.6, 1.8), (1.0, 2.0, 0.5)
    m = fem3.Mesh(mesh.verts, mesh.tets)
    m.assemble(alpha, K, "fp32")
    f = np.random.default_rng(n + nrhs).standard_normal((mesh.n_nodes, nrhs))
    u = m.solve(f, tol=1e-3, max_iter=1).cpu().numpy().reshape(n, nrhs)
    assert m.iters == 1
    A, b = o.assemble(alpha, K), o.load(f).reshape(n, nrhs)
    res = np.linalg.norm(b - A @ u, axis=0) / np.linalg.norm(b, axis=0)
    assert res.max() <= 1e-3, res
    m.free()


@pytest.mark.parametrize("chol_tc", [-1, 1])
@pytest.mark.parametrize("nrhs", [1, 8, 17])
def test_f32_solve_of_wide_blocks(nrhs, chol_tc):
    """Above 4,096 unknowns the FP32 blocks are 1,024 wide, and one column's updates of more than 4,864
    rows take four rows a warp: 6,156 unknowns, a ragged last block.  One sweep's residual is formed in
    FP64; a backward-stable FP32 solve leaves 2^-24 sqrt(n) of |A| |u| (tens of b): below 1e-4."""
    mesh = _bar_mesh((19, 19, 20))
    m = fem3.Mesh(mesh.verts, mesh.tets, chol_tc=chol_tc)
    assert m.n_dof == 6156
    m.assemble((1.3, 1.6, 1.8), (1.0, 2.0, 0.5), "fp32")
    f = np.random.default_rng(nrhs).standard_normal((mesh.n_nodes, nrhs))
    m.solve(f, tol=1e-4, max_iter=1)
    assert m.iters == 1 and m.resid <= 1e-4
    m.free()
