"""The Krylov reductions whose groups of basis vectors are split over blocks (csrc/solver.cu, dot_splits):
restart lengths around whole groups of four and eight vectors, one and several right-hand sides.

A wrong or missing inner product leaves a basis that is not orthogonal: the recurrence's residual then
departs from the true one, which is taken here with a separate product."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402


@pytest.mark.parametrize("restart", [8, 9, 12, 40])
@pytest.mark.parametrize("n_rhs", [1, 3])
def test_true_residual(restart, n_rhs):
    V, F, D = fi.icosphere(3)
    a = fm.FMBEM(V, F, D, [1.0, 2.25], [1.0, 1.0], 1.0, p=6, gmres_restart=restart)
    b = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=restart)).cuda()
    x = a.solve(b, tol=1e-8, max_iter=600)[0]
    res = (b - a.matvec(x)).flatten(1).norm(dim=1) / b.flatten(1).norm(dim=1)
    assert float(res.max()) < 2e-8  # the tolerance, and as much again for the recurrence's own rounding
