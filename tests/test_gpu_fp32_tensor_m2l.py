"""The single-precision M2L on the tensor cores (four exact 8-bit digits, csrc/m2l_oz.cu) against the same
handle's double-precision product.

Tolerance.  A single-precision product rounds the densities, the tables and every pair scalar to 24 bits
(6e-8 each) and sums some hundreds of terms per row; rounding errors of mixed signs leave about 3e-7 of the
norm, and the bound is 2e-6.  The digits add 2^-31 of the largest terms of a pair result."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402

TOL = 2e-6


def handle(mesh, p, k0=1.5, **opt):
    V, F, D = fi.torus(1.0, 0.25, 97, 31) if mesh == "torus" else fi.torus_and_sphere(nu=60, nv=18, sphere_subdiv=2)[0]
    eps, mu = [1.0, -8.5 + 0.3j, 2.25][: D.max() + 1], [1.0] * (D.max() + 1)
    return fm.FMBEM(V, F, D, eps, mu, k0, p=p, **opt)


def rel(a, b):
    return float((a - b).norm() / b.norm())


# one and several tiles of 128 columns, several windows; BF16x3 with 9 to 15 right-hand sides takes it too
@pytest.mark.parametrize("p", [4, 6, 8, 10])
@pytest.mark.parametrize("n_rhs,precision", [(1, fm.FP32), (2, fm.FP32), (5, fm.FP32), (17, fm.FP32), (33, fm.FP32),
                                             (9, fm.BF16X3), (15, fm.BF16X3)])
def test_matches_double(p, n_rhs, precision):
    a = handle("torus", p, leaf_size=16)  # levels 2 to 4
    x = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=p + n_rhs)).cuda()
    assert rel(a.matvec(x, precision=precision), a.matvec(x)) < TOL
    assert rel(a.adjoint_matvec(x, precision=precision), a.adjoint_matvec(x)) < TOL


@pytest.mark.parametrize("opt", [{}, dict(adaptive=1, leaf_size=12), dict(boundary=fm.IMPEDANCE)])
def test_sizes_of_columns(opt):
    """Zero, very small and ordinary right-hand sides beside each other."""
    a = handle("two", 8, **opt)
    x = torch.from_numpy(fi.random_complex((3, a.N, 6), seed=2)).cuda()
    x[1] = 0
    x[2] *= 2.0 ** -30
    y, z = a.matvec(x, precision=fm.FP32), a.matvec(x)
    for r in range(3):
        assert float((y[r] - z[r]).norm()) <= TOL * float(z[r].norm())


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_inputs_show(bad):
    a = handle("torus", 8)
    x = torch.from_numpy(fi.random_complex((2, a.N, 6), seed=4)).cuda()
    y0 = a.matvec(x, precision=fm.FP32)
    x[0, 77, 1] = bad
    y, z = a.matvec(x, precision=fm.FP32), a.matvec(x)
    fin = [torch.isfinite(v.real) & torch.isfinite(v.imag) for v in (y, z)]
    assert not bool((fin[0] & ~fin[1]).any())  # nothing finite that is not so in double precision
    assert torch.equal(y[1], y0[1])


def test_captured_and_repeated():
    """In a CUDA graph and after calls with other column counts: the same bits."""
    a = handle("torus", 10)
    x = torch.from_numpy(fi.random_complex((4, a.N, 6), seed=5)).cuda()
    y = a.matvec(x, precision=fm.FP32)
    a.matvec(x.repeat(9, 1, 1), precision=fm.FP32)
    a.matvec(x)
    out = torch.zeros_like(x)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        a.matvec(x, out, precision=fm.FP32)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, out)
