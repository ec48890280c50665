"""CUDA graphs captured from products, replayed after other products of the handle: scratch that those outgrow
stays allocated for the graph, and a product can be captured after one of another kind.

Tolerances: a replay gives the bits of the product it recorded; a product recorded without its optional scratch
differs from the usual one by the rounding of sums of some hundreds of terms, 1e-13 in FP64 and 2e-6 in FP32."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402

CALLS = {"fp64": ("matvec", fm.FP64), "fp32": ("matvec", fm.FP32), "fp64 T": ("adjoint_matvec", fm.FP64),
         "fp32 T": ("adjoint_matvec", fm.FP32)}


def handle(p=8):
    V, F, D = fi.torus(1.0, 0.25, 61, 19)
    return fm.FMBEM(V, F, D, [1.0, -8.5 + 0.3j], [1.0, 1.0], 1.5, p=p, leaf_size=16)


def call(h, kind, x, y=None):
    name, precision = CALLS[kind]
    return getattr(h, name)(x, y, precision=precision)


def capture(h, kind, x):
    y = torch.zeros_like(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call(h, kind, x, y)
    return g, y


def others(h, x):
    """Products of every kind with no more right-hand sides, and memory of the freed sizes written over."""
    for n in (1, len(x), max(1, len(x) // 2)):
        for kind in CALLS:
            call(h, kind, x[:n].contiguous())
        h.matvec(x[:n].contiguous(), precision=fm.BF16X3)
    junk = [torch.full((1 << 18,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(64)]
    torch.cuda.synchronize()
    del junk


@pytest.mark.parametrize("p", [8, 9, 10])
@pytest.mark.parametrize("n_rhs", [1, 3, 8])
@pytest.mark.parametrize("kind", list(CALLS))
def test_replay_after_other_products(kind, n_rhs, p):
    h = handle(p)
    x = torch.from_numpy(fi.random_complex((n_rhs, h.N, 6), seed=n_rhs)).cuda()
    y = call(h, kind, x)
    g, out = capture(h, kind, x)
    g.replay()
    assert torch.equal(out, y)
    others(h, x)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, y)
    assert torch.equal(call(h, kind, x), y)


@pytest.mark.parametrize("n_rhs", [1, 3, 8])
@pytest.mark.parametrize("first", list(CALLS))
@pytest.mark.parametrize("kind", list(CALLS))
def test_capture_after_another_kind(first, kind, n_rhs):
    h = handle()
    x = torch.from_numpy(fi.random_complex((n_rhs, h.N, 6), seed=n_rhs)).cuda()
    call(h, first, x)
    g, out = capture(h, kind, x)
    g.replay()
    y = call(h, kind, x)
    assert float((out - y).norm()) < (1e-13 if CALLS[kind][1] == fm.FP64 else 2e-6) * float(y.norm())
    others(h, x)
    z = out.clone()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, z)


def test_capture_needs_a_product_before():
    h = handle()
    x = torch.from_numpy(fi.random_complex((2, h.N, 6), seed=1)).cuda()
    h.matvec(x[:1].contiguous())
    y = torch.zeros_like(x)
    g = torch.cuda.CUDAGraph()
    with pytest.raises(fm.FMBEMError, match="capture"):
        with torch.cuda.graph(g):
            h.matvec(x, y)
    assert torch.isfinite(torch.view_as_real(h.matvec(x))).all()
