"""The FP64 tile factorisation (csrc/chol_f64.cu) at the edges of its 32-column tiles and of
the 64-column diagonal inverses that the solves use: integer-order problems of chosen order
against the oracle's matrix, solved by numpy; and the allocation-free solve, which shares it, on dense
systems of the same kind of sizes."""
import ctypes as C
import os
import subprocess
import time
from fractions import Fraction

import numpy as np
import pytest

import oracle
from test_gpu_contract_rows import _bar_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1811_03339_gb300 import _build_lib, fem3  # noqa: E402

# interior dofs of a box of cells: (a - 1)(b - 1)(c - 1)
SIZES = {1: (2, 2, 2), 8: (3, 3, 3), 9: (10, 2, 2), 31: (32, 2, 2), 32: (3, 5, 5), 33: (4, 12, 2),
         63: (8, 10, 2), 64: (5, 5, 5), 65: (6, 14, 2), 96: (4, 5, 9), 98: (8, 15, 2),
         130: (14, 11, 2)}


@pytest.mark.parametrize("n", sorted(SIZES))
def test_f64_factor_sizes(n):
    mesh = _bar_mesh(SIZES[n])
    o = oracle.Oracle.from_mesh(mesh)
    assert o.n_dof == n
    K = (1.0, 2.0, 0.5)
    A = o.assemble((2.0, 2.0, 2.0), K)
    f = np.random.default_rng(n).standard_normal((mesh.n_nodes, 3))
    m = fem3.Mesh(mesh.verts, mesh.tets)
    m.assemble_integer(K)
    u = m.solve(f).cpu().numpy().reshape(n, 3)
    ref = np.linalg.solve(A, o.load(f))
    assert np.linalg.norm(u - ref) <= 1e-10 * np.linalg.norm(ref)
    m.free()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 127, 160, 384, 511, 512])
def test_static_solve_sizes(n):
    """B B^T + n I has a condition number below about 5 (Gaussian B), so numpy's and the
    library's solutions agree to n u 5 < 3e-13"""
    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, n))
    A, b = B @ B.T + n * np.eye(n), rng.standard_normal(n)
    x = torch.empty(n, dtype=torch.float64, device="cuda")
    fem3.spd_solve_static(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), x)
    ref = np.linalg.solve(A, b)
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    y = torch.from_numpy(b).cuda()        # in place
    fem3.spd_solve_static(torch.from_numpy(A).cuda(), y, y)
    assert torch.equal(x, y)


# cells of a long box: 1,416 dofs, band 29 (every ticket below the chain's tiles is skipped);
# 1,536, band 73; 2,760, band 93: two and three tiles of a column are left
@pytest.mark.parametrize("cells", [(5, 7, 60), (9, 9, 25), (9, 11, 35)])
def test_f64_factor_band(cells):
    """The integer order's profile: most tickets are skipped, several by one CTA in a row.  Repeats
    differ by the element sum's order only (a few rounding errors of a matrix of condition below
    1e3), and every one is the dense solution."""
    mesh = _bar_mesh(cells)
    m = fem3.Mesh(mesh.verts, mesh.tets)
    f = np.random.default_rng(3).standard_normal(mesh.n_nodes)
    A = m.assemble_integer((1.0, 2.0, 0.5), return_matrix=True)
    b = m.load(torch.from_numpy(f).cuda())
    first = m.solve(f)
    ref = torch.linalg.solve(A, b)
    assert float((first - ref).norm() / ref.norm()) <= 1e-10
    for _ in range(20):
        m.assemble_integer((1.0, 2.0, 0.5))
        u = m.solve(f)
        assert float((u - first).norm() / first.norm()) <= 1e-11
    m.free()


def _pairs(d, c):
    """block-diagonal matrix of [[d, c], [c, d]] for arrays d, c"""
    n = 2 * len(d)
    A = np.zeros((n, n))
    i = np.arange(0, n, 2)
    A[i, i] = A[i + 1, i + 1] = d
    A[i, i + 1] = A[i + 1, i] = c
    return A


def _static(A, b):
    x = torch.empty(len(b), dtype=torch.float64, device="cuda")
    fem3.spd_solve_static(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), x)
    return x.cpu().numpy()


# exponents of the pivots: subnormal, the ends of the range in which a reciprocal is normal (biased 8
# and 2,038: -1,015 and 1,015), one and the largest
@pytest.mark.parametrize("e", [-1074, -1060, -1030, -1025, -1024, -1023, -1022, -1017, -1016, -1015,
                               -1014, -500, 0, 500, 1013, 1014, 1015, 1016, 1017, 1020])
def test_pivots_of_any_exponent(e):
    """[[d, d/2], [d/2, d]] x = d (2, 2.5) and, for the smallest numbers, diag(d, d) x = d (1, 2):
    every step is exact in binary but the square roots, so 64 of them give (1, 2) to a few 2^-53"""
    d = np.ldexp(np.ones(32), e)
    tiny = e < -1060
    A = _pairs(d, 0.0 * d if tiny else d / 2)
    x = _static(A, np.ldexp(np.tile((1.0, 2.0) if tiny else (2.0, 2.5), 32), e))
    assert np.abs(x - np.tile((1.0, 2.0), 32)).max() <= 16 * 2.0 ** -53


def test_pivot_reciprocals():
    """x / d to a unit or two in the last place for pivots of random significands, against exact
    fractions: 256 systems [[d, c], [c, d]] of condition 3 at most per call"""
    rng = np.random.default_rng(11)
    for e in (-900, -1, 0, 1, 900):
        d = np.ldexp(1.0 + rng.random(256), e)
        c = d * rng.uniform(-0.5, 0.5, 256)
        b = np.ldexp(rng.standard_normal(512), e)
        x = _static(_pairs(d, c), b)
        for i in range(256):
            D, Cc, p, q = (Fraction(float(v)) for v in (d[i], c[i], b[2 * i], b[2 * i + 1]))
            det = D * D - Cc * Cc
            ref = np.array([float((D * p - Cc * q) / det), float((D * q - Cc * p) / det)])
            assert np.abs(x[2 * i:2 * i + 2] - ref).max() <= 32 * 2.0 ** -53 * np.abs(ref).max()


def test_rows_of_any_scale():
    """D M D x = D c for a diagonal D of powers of two from 2^-500 to 2^500: x is D^{-1} M^{-1} c, row by
    row to the accuracy of M (condition below 5)"""
    n = 130
    rng = np.random.default_rng(4)
    B = rng.standard_normal((n, n))
    M, c, e = B @ B.T + n * np.eye(n), rng.standard_normal(n), rng.integers(-500, 501, n)
    x = np.ldexp(_static(np.ldexp(np.ldexp(M, e[:, None]), e[None, :]), np.ldexp(c, e)), e)
    ref = np.linalg.solve(M, c)
    assert np.linalg.norm(x - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("e", [-1013, -1008, 1008, 1013])
def test_integer_order_at_the_range_ends(e):
    """K times 2^e: pivots on both sides of the exponents from which their reciprocal is taken by
    division"""
    mesh = _bar_mesh((5, 6, 7))
    f = np.random.default_rng(2).standard_normal(mesh.n_nodes)
    m = fem3.Mesh(mesh.verts, mesh.tets)
    m.assemble_integer((1.0, 2.0, 0.5))
    ref = m.solve(f)
    m.assemble_integer([k * 2.0 ** e for k in (1.0, 2.0, 0.5)])
    u = m.solve(f) * 2.0 ** (e // 2) * 2.0 ** (e - e // 2)
    assert float((u - ref).norm() / ref.norm()) <= 1e-11
    m.free()


HOLD = r"""
#include <cuda_runtime.h>
__global__ void k_hold(long long ns) {
    long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (int i = 0; i < 1 << 27; i++) {
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        if (t - t0 >= ns) break;
        __nanosleep(1000);
    }
}
extern "C" int hold(int ctas, int smem, long long ns, void *stream) {
    cudaFuncSetAttribute(k_hold, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    k_hold<<<ctas, 1, smem, (cudaStream_t)stream>>>(ns);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def hold(tmp_path_factory):
    d = tmp_path_factory.mktemp("hold")
    (d / "hold.cu").write_text(HOLD)
    subprocess.run([os.environ.get("NVCC", "nvcc"), *_build_lib.ARCH, "-shared", "-Xcompiler", "-fPIC",
                    str(d / "hold.cu"), "-o", str(d / "hold.so")], check=True)
    f = C.CDLL(str(d / "hold.so")).hold
    f.argtypes = [C.c_int, C.c_int, C.c_longlong, C.c_void_p]
    return f


@pytest.mark.parametrize("n,free", [(384, 1), (512, 1), (384, 2)])
def test_static_solve_beside_other_work(hold, n, free):
    """All SMs but `free` are held for a second by blocks that leave no room for one of the
    factorisation's: it finishes there, before they do."""
    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, n))
    A, b = torch.from_numpy(B @ B.T + n * np.eye(n)).cuda(), torch.from_numpy(rng.standard_normal(n)).cuda()
    x, ref = torch.empty_like(b), torch.empty_like(b)
    fem3.spd_solve_static(A, b, ref)
    assert hold(1, 1 << 17, 1000, None) == 0   # loads the kernel
    torch.cuda.synchronize()
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert hold(sms - free, 200 << 10, 1_000_000_000, side.cuda_stream) == 0
    done.record(side)
    time.sleep(0.05)
    fem3.spd_solve_static(A, b, x)
    assert not done.query()
    assert torch.equal(x, ref)
    torch.cuda.synchronize()
