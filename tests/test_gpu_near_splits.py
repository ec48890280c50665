"""The single-precision near field for few right-hand sides with its sources split over several units
(k_near_ws, k_near_sum) against the allocation-free product, which keeps whole items.

Tolerance.  The same FP32 terms in another order: at most ~1000 of them a row, 2^-24 each, 1e-6 in the mean
square of the result's norm."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402


@pytest.mark.parametrize("mesh,opt", [(lambda: fi.icosphere(1), {}), (lambda: fi.icosphere(3), {}), (lambda: fi.icosphere(4), {}),
                                      (lambda: fi.icosphere(2), dict(leaf_size=1, max_level=3)),
                                      (lambda: fi.torus_and_sphere(nu=48, nv=12, sphere_subdiv=2)[0], {}),
                                      (lambda: fi.split_ring(1.0, 0.2, 10.0, 60, 3, grading=2.0), dict(adaptive=1, leaf_size=20)),
                                      (lambda: fi.icosphere(3), dict(boundary=fm.IMPEDANCE))])
@pytest.mark.parametrize("n_rhs", [1, 3])
def test_splits_match_whole_items(mesh, opt, n_rhs):
    V, F, D = mesh()
    h = fm.FMBEM(V, F, D, [1.0, -5 + 0.2j, 2.25][: D.max() + 1], [1.0, 1.3, 1.0][: D.max() + 1], 1.7, p=4, m2l_rotation=0,
                 **opt)
    x = torch.from_numpy(fi.random_complex((n_rhs, h.N, 6), seed=n_rhs)).cuda()
    y = h.matvec(x, precision=fm.FP32)
    for r in range(n_rhs):
        c = x[r:r + 1].contiguous()
        z = fm.fmbem_matvec_noalloc(h.h, c, torch.empty_like(c), precision=fm.FP32)
        assert float((y[r] - z[0]).norm()) <= 1e-6 * float(z[0].norm())
    assert torch.equal(y, h.matvec(x, precision=fm.FP32))
