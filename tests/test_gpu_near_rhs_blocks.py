"""Single-precision products of four and more right-hand sides (the near field by slabs of 4, 8 and 32
right-hand sides, P2M from the node-major densities) against the double-precision product.

Tolerance: as for every single-precision product here, 24-bit roundings of the densities, tables and pair
scalars in rows of some hundreds of terms of mixed signs, about 3e-7 of the norm; 2e-6.  BF16x3 translations
keep 16 + 8 bits of each operand and drop the product of the low parts (2^-18 a term): 2e-5."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402

MESHES = {
    "torus": lambda: fi.torus(1.0, 0.25, 61, 19),
    "two": lambda: fi.torus_and_sphere(nu=60, nv=18, sphere_subdiv=2)[0],  # targets of several scatterers
}


def handle(mesh, **opt):
    V, F, D = MESHES[mesh]()
    eps, mu = [1.0, -8.5 + 0.3j, 2.25][: D.max() + 1], [1.0] * (D.max() + 1)
    return fm.FMBEM(V, F, D, eps, mu, 1.5, p=8, **opt)


def check(y, z, tol):
    for r in range(len(z)):
        assert float((y[r] - z[r]).norm()) < tol * float(z[r].norm()), r


# slabs of four, eight (full and ragged) and whole blocks of 32 with each kind of rest
@pytest.mark.parametrize("mesh,opt", [("torus", {}), ("two", dict(leaf_size=20)), ("two", dict(boundary=fm.IMPEDANCE)),
                                      ("torus", dict(adaptive=1, leaf_size=12))])
@pytest.mark.parametrize("n_rhs", [4, 5, 8, 9, 15, 16, 31, 32, 33, 36, 45, 64])
def test_blocks(mesh, opt, n_rhs):
    a = handle(mesh, **opt)
    x = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=n_rhs)).cuda()
    x[1] *= 1e-3
    z = a.matvec(x)
    check(a.matvec(x, precision=fm.FP32), z, 2e-6)
    check(a.matvec(x, precision=fm.BF16X3), z, 2e-5)


@pytest.mark.parametrize("n_rhs", [4, 5, 8, 21, 32, 35])
def test_static_scratch(n_rhs):
    """The allocation-free product: below 32 right-hand sides in two parts."""
    a = handle("torus")
    x = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=n_rhs)).cuda()
    y = fm.fmbem_matvec_noalloc(a.h, x, torch.empty_like(x), fm.FP32)
    check(y, a.matvec(x), 2e-6)


@pytest.mark.parametrize("n_rhs", [1, 3, 4, 5, 8, 9, 12, 20, 31])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_unknowns_of_another_scatterer(bad, n_rhs):
    """The scatterer rows (3 to 5) of a node sum over its own scatterer: non-finite unknowns of the other one
    leave them as they are, in every form of the near field below 32 right-hand sides."""
    V, F, D = fi.merge_meshes(fi.torus(1.0, 0.25, 60, 18, domain=1), fi.icosphere(2, 0.1, (1.0, 0.0, 0.37), domain=2))
    a = fm.FMBEM(V, F, D, [1.0, -8.5 + 0.3j, 2.25], [1.0] * 3, 1.5, p=8, leaf_size=40)
    other = torch.zeros(a.N, dtype=torch.bool, device="cuda")
    other[torch.from_numpy(F[D == 2].ravel()).long().cuda()] = True
    x = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=n_rhs)).cuda()
    x[:, other] = 0
    z = a.matvec(x, precision=fm.FP32)
    x[:, other] = bad
    y = a.matvec(x, precision=fm.FP32)
    assert torch.equal(y[:, ~other, 3:], z[:, ~other, 3:])
