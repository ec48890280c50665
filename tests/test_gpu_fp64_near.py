"""The double-precision near field by warps (k_near_d, k_near_finish) against the allocation-free product,
which keeps the block-per-leaf kernels, and the dense oracle.

Tolerance.  Both sum the same FP64 terms in another order; a row adds at most ~1000 near terms, so their
rounding differs by at most about 1000 x 2^-53 = 1e-13 of the terms' sum and by 1e-15 in the mean; 1e-12 of
the result's norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402


def mesh(name):
    if name == "ring":
        return fi.split_ring(1.0, 0.2, 10.0, 60, 3, grading=2.0)
    if name == "two":
        return fi.torus_and_sphere(nu=48, nv=12, sphere_subdiv=2)[0]
    return fi.icosphere(int(name))


# leaves of one to several hundred nodes (one target group of 32 and remainders), one to many splits
@pytest.mark.parametrize("name,opt", [("1", {}), ("3", {}), ("2", dict(leaf_size=1, max_level=3)), ("3", dict(max_level=2)),
                                      ("3", dict(near_cache=0)), ("two", {}), ("two", dict(near_cache=0)),
                                      ("ring", dict(adaptive=1, leaf_size=20)), ("2", dict(node_mode=fm.NODES_CENTROID)),
                                      ("3", dict(boundary=fm.IMPEDANCE))])
@pytest.mark.parametrize("n_rhs", [1, 3, 6])
def test_matches_block_kernels(name, opt, n_rhs):
    V, F, D = mesh(name)
    h = fm.FMBEM(V, F, D, [1.0, -5 + 0.2j, 2.25][: D.max() + 1], [1.0, 1.3, 1.0][: D.max() + 1], 1.7, p=4, m2l_rotation=0,
                 **opt)
    x = torch.from_numpy(fi.random_complex((n_rhs, h.N, 6), seed=n_rhs)).cuda()
    y = h.matvec(x)
    z = torch.cat([fm.fmbem_matvec_noalloc(h.h, c.contiguous(), torch.empty_like(c)) for c in (x.split(1) if n_rhs < 4 else [x])])
    for r in range(n_rhs):
        assert float((y[r] - z[r]).norm()) <= 1e-12 * float(z[r].norm())
    assert torch.equal(y, h.matvec(x))  # the same bits again: fixed orders


def test_oracle_near_only():
    """One level with few boxes: most pairs are near (p = 12 for the rest)."""
    import oracle
    V, F, D = mesh("two")
    eps, mu = [1.0, -5 + 0.2j, 2.25], [1.0, 1.3, 1.0]
    h = fm.FMBEM(V, F, D, eps, mu, 1.7, p=12, leaf_size=500)
    o = oracle.Oracle(V, F, D, eps, mu, 1.7)
    x = fi.random_complex((2, h.N, 6), seed=9)
    y = h.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    yo = o.matvec(x)
    assert np.linalg.norm(y - yo) < 1e-5 * np.linalg.norm(yo)


# the transposed near field by warps (k_near_adj): b . (A x) = x . (A^T b) with the forward product, in double
# precision to the rounding of their sums (as above, over the terms' sum), in single to 2^-24 of ~1000 terms
@pytest.mark.parametrize("name,opt", [("1", {}), ("3", {}), ("2", dict(leaf_size=1, max_level=3)), ("3", dict(near_cache=0)),
                                      ("two", {}), ("two", dict(near_cache=0)), ("ring", dict(adaptive=1, leaf_size=20)),
                                      ("2", dict(node_mode=fm.NODES_CENTROID)), ("3", dict(boundary=fm.IMPEDANCE))])
@pytest.mark.parametrize("n_rhs", [1, 2, 3, 4])
@pytest.mark.parametrize("precision,tol", [(fm.FP64, 1e-12), (fm.FP32, 1e-5)])
def test_adjoint_identity(name, opt, n_rhs, precision, tol):
    V, F, D = mesh(name)
    h = fm.FMBEM(V, F, D, [1.0, -5 + 0.2j, 2.25][: D.max() + 1], [1.0, 1.3, 1.0][: D.max() + 1], 1.7, p=4, m2l_rotation=0,
                 **opt)
    x, b = (torch.from_numpy(fi.random_complex((n_rhs, h.N, 6), seed=s)).cuda() for s in (1, 2))
    y, z = h.matvec(x, precision=precision), h.adjoint_matvec(b, precision=precision)
    for r in range(n_rhs):
        assert abs(complex((b[r] * y[r]).sum() - (x[r] * z[r]).sum())) <= tol * float((b[r] * y[r]).abs().sum())
    assert torch.equal(z, h.adjoint_matvec(b, precision=precision))
