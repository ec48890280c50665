"""Waits of the tensor-core kernels that run out (raised by the library's fault injection, so that the kernels
give up as soon as they start): the product's rows are not finite, exactly one call reports it, and the
handle's next products are what they were."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402

TIMEOUT = 7


def handle(**opt):
    V, F, D = fi.torus(1.0, 0.25, 61, 19)
    return fm.FMBEM(V, F, D, [1.0, -8.5 + 0.3j], [1.0, 1.0], 1.5, p=8, leaf_size=16, **opt)


def raise_timeout(h):
    assert fm.load_library().fmbem_debug_raise_wait_timeout(h.h) == 0


@pytest.mark.parametrize("call", ["matvec", "adjoint_matvec"])
@pytest.mark.parametrize("precision,n_rhs", [(fm.FP64, 1), (fm.FP64, 17), (fm.FP32, 2), (fm.BF16X3, 9), (fm.TF32, 9)])
def test_reported_once(call, precision, n_rhs):
    h = handle()
    x = torch.from_numpy(fi.random_complex((n_rhs, h.N, 6), seed=n_rhs)).cuda()
    product = lambda: getattr(h, call)(x, precision=precision)  # noqa: E731
    y = product()
    raise_timeout(h)
    if precision in (fm.FP64, fm.FP32):  # these products do not wait for the device: the next call reports it
        bad = product()
        torch.cuda.synchronize()
        assert torch.isnan(bad.real).all()
    with pytest.raises(fm.FMBEMError) as e:
        product()
    assert e.value.status == TIMEOUT
    for _ in range(2):
        assert torch.equal(product(), y)


@pytest.mark.parametrize("opt", [{}, dict(solve_precision=fm.FP32)])
def test_solve(opt):
    h = handle(**opt)
    b = h.plane_wave_rhs([[0.0, 0.0, 1.0]], [[1.0, 0.0, 0.0]])
    x = h.solve(b, tol=1e-4)[0]
    raise_timeout(h)
    with pytest.raises(fm.FMBEMError) as e:
        h.solve(b, tol=1e-4)
    assert e.value.status == TIMEOUT
    assert torch.equal(h.solve(b, tol=1e-4)[0], x)


def test_calls_that_return_host_results():
    """They wait for their products and report what happened to them."""
    h = handle()
    x = torch.from_numpy(fi.random_complex((1, h.N, 6), seed=1)).cuda()
    pts = [[0.0, 0.0, 2.0], [2.0, 0.5, 0.0]]
    calls = [lambda: h.near_field(x, pts, fmm=True), lambda: h.eps_sensitivity(1, x, x)]
    for call in calls:
        want = torch.as_tensor(call())
        raise_timeout(h)
        with pytest.raises(fm.FMBEMError) as e:
            call()
        assert e.value.status == TIMEOUT
        assert torch.equal(torch.as_tensor(call()), want)
        # (the flag that the other call's handles had: theirs is not this one's)
        for other in calls:
            try:
                other()
            except fm.FMBEMError as e2:
                assert other is not call and e2.status == TIMEOUT
