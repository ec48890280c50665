"""The FP64 M2L on the tensor cores (exact 8-bit digits, csrc/m2l_oz.cu) against the dense FP64 S|R sums
(m2l_rotation=0) and, for a whole product, against the dense oracle.

Tolerance.  Both forms translate with the same matrices; a pair result differs by the rounding of the
dense form's sum of K = 2 p^2 <= 200 terms, at most about K 2^-53 of the terms' sum and 1e-15 of the
result in the mean, and by the digits that are not multiplied, below 2^-62 of the largest terms.  A product adds
the near field, which is the same, and up to 189 pairs per box: 1e-13 leaves two orders.  M2M and L2L
between levels 2 to 4 are further such translations, at most four in a row."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402

MESHES = {
    "sphere": lambda: fi.icosphere(4),
    "torus": lambda: fi.torus(1.0, 0.25, 97, 31),
    "two": lambda: fi.torus_and_sphere(nu=60, nv=18, sphere_subdiv=2)[0],
}


def handles(mesh, p, k0=1.5, **opt):
    V, F, D = MESHES[mesh]()
    eps, mu = [1.0, -8.5 + 0.3j, 2.25][: D.max() + 1], [1.0] * (D.max() + 1)
    return [fm.FMBEM(V, F, D, eps, mu, k0, p=p, m2l_rotation=m, **opt) for m in (-1, 0)]


def rel(a, b):
    return float((a - b).norm() / b.norm())


# one and several tiles of 80 columns, windows of unequal width, ragged column counts
@pytest.mark.parametrize("p", [4, 6, 8, 10])
@pytest.mark.parametrize("n_rhs", [1, 2, 5, 16, 17, 33])
def test_matches_dense_form(p, n_rhs):
    a, d = handles("torus", p, leaf_size=16)  # levels 2 to 4
    x = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=p + n_rhs)).cuda()
    assert rel(a.matvec(x), d.matvec(x)) < 1e-13
    assert rel(a.adjoint_matvec(x), d.adjoint_matvec(x)) < 1e-13


@pytest.mark.parametrize("mesh,opt", [("two", {}), ("two", dict(adaptive=1, leaf_size=12)),
                                      ("sphere", dict(node_mode=fm.NODES_CENTROID)), ("sphere", dict(leaf_size=1000)),
                                      ("sphere", dict(boundary=fm.IMPEDANCE)), ("torus", dict(near_cache=0, k0=6.0))])
def test_forms_of_handle(mesh, opt):
    a, d = handles(mesh, 8, **opt)
    x = torch.from_numpy(fi.random_complex((3, a.N, 6), seed=2)).cuda()
    x[1] = 0  # a zero right-hand side, and very different sizes
    x[2] *= 1e-200
    y, z = a.matvec(x), d.matvec(x)
    for r in range(3):
        assert float((y[r] - z[r]).norm()) <= 1e-13 * float(z[r].norm())


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_inputs_show(bad):
    """One non-finite unknown: the rows that it reaches are non-finite in both forms, the other
    right-hand sides stay as they are."""
    a, d = handles("torus", 8)
    x = torch.from_numpy(fi.random_complex((2, a.N, 6), seed=4)).cuda()
    y0 = a.matvec(x)
    x[0, 77, 1] = bad
    y, z = a.matvec(x), d.matvec(x)
    assert torch.equal(torch.isfinite(y.real) & torch.isfinite(y.imag), torch.isfinite(z.real) & torch.isfinite(z.imag))
    assert torch.equal(y[1], y0[1])


def test_captured_and_repeated():
    """In a CUDA graph, on another stream, and after calls with other column counts: the same bits."""
    a, _ = handles("torus", 8)
    x = torch.from_numpy(fi.random_complex((4, a.N, 6), seed=5)).cuda()
    y = a.matvec(x)
    a.matvec(x.repeat(9, 1, 1))
    a.matvec(x[:1].contiguous())
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        y1 = a.matvec(x, stream=st)
    st.synchronize()
    assert torch.equal(y, y1)
    out = torch.zeros_like(x)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        a.matvec(x, out)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, out)
    y2 = torch.empty_like(x[:1])
    assert rel(fm.fmbem_matvec_noalloc(a.h, x[:1].contiguous(), y2), y[:1]) < 1e-13  # the FP64 pipe's kernels


def test_oracle_rows():
    import oracle
    V, F, D = fi.icosphere(3)
    a = fm.FMBEM(V, F, D, [1.0, 2.25], [1.0, 1.0], 1.0, p=10)
    o = oracle.Oracle(V, F, D, [1.0, 2.25], [1.0, 1.0], 1.0)
    x = fi.random_complex((2, a.N, 6), seed=6)
    y = a.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    yo = o.matvec(x)
    assert np.linalg.norm(y - yo) < 2e-5 * np.linalg.norm(yo)  # the truncation at p = 10
