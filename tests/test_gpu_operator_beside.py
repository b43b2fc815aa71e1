"""The refinement's operator built beside the factorisation (csrc/operator.cu, factor() in
csrc/solve.cu): orders on both sides of the small block patterns (32
block rows) and of the blocked factorisation (4,096), a handle assembled again, and a batch whose
precision changes between eager runs, captures and replays.  Reference: a dense FP64 solve
(torch) with the FP64 form's matrix; the mixed forms' bound is 1e-8."""
import numpy as np
import pytest

from test_gpu_contract_rows import _bar_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1811_03339_gb300 import fem3  # noqa: E402

SIZES = {504: (9, 8, 10), 512: (9, 9, 9), 1024: (9, 9, 17), 1040: (14, 11, 9), 4104: (20, 13, 19)}
ALPHA, K = ((1.3, 1.6, 1.8), (1.7, 1.2, 1.5)), (1.0, 2.0, 0.5)


def _reference(mesh, alpha, f):
    m = fem3.Mesh(mesh.verts, mesh.tets)
    A = m.assemble(alpha, K, "fp64", return_matrix=True)
    b = m.load(f).reshape(m.n_dof, -1)
    m.free()
    return torch.linalg.solve(A, b)


def _near(u, ref):
    u = u.reshape(ref.shape)
    return float((u - ref).norm() / ref.norm()) <= 1e-8


@pytest.mark.parametrize("n", sorted(SIZES))
def test_handle_assembled_again(n):
    mesh = _bar_mesh(SIZES[n])
    f = torch.from_numpy(np.random.default_rng(n).standard_normal((mesh.n_nodes, 3))).cuda()
    refs = [_reference(mesh, a, f) for a in ALPHA]
    for precision in ("tf32x3", "fp32"):
        m = fem3.Mesh(mesh.verts, mesh.tets)
        assert m.n_dof == n
        for a, ref in list(zip(ALPHA, refs)) * 2:
            m.assemble(a, K, precision)
            assert _near(m.solve(f), ref)
        m.free()


def test_batch_precision_changes():
    meshes = [_bar_mesh(SIZES[n]) for n in (504, 1040, 512, 4104)]
    fs = [torch.from_numpy(np.random.default_rng(i).standard_normal((m.n_nodes, 2))).cuda()
          for i, m in enumerate(meshes)]
    refs = [[_reference(m, a, f) for m, f in zip(meshes, fs)] for a in ALPHA]
    b = fem3.Batch([(m.verts, m.tets) for m in meshes])
    Ks = np.tile(K, (len(meshes), 1))
    # an eager run, then per line a capture with its first launch and a replay
    for j, precision in [(0, "tf32x3"), (0, "tf32x3"), (0, "tf32x3"), (1, "fp64"), (1, "fp64"),
                         (1, "bf16x3"), (1, "bf16x3"), (0, "fp32"), (0, "fp32")]:
        us = b.run(np.tile(ALPHA[j], (len(meshes), 1)), Ks, fs, precision)
        for u, ref in zip(us, refs[j]):
            assert _near(u, ref), (j, precision)
    b.free()
