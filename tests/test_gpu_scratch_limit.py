"""Products whose optional scratch (digits and pair results of the tensor-core M2L, the near field's partial
sums) the device has no room for: the forms without it give the result, and nothing fails that needs no more
than the densities and expansions.

Tolerance: the two forms differ by the rounding of FP64 sums of some hundreds of terms, 1e-15 to 1e-14 (the
tensor-core M2L against the dense one: 1e-13 is two orders above); FP32 2e-6 as for every such product."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import fmbem_inputs as fi  # noqa: E402
import paper_1211_7177_gb300 as fm  # noqa: E402


@pytest.mark.parametrize("n_rhs", [1, 9])
@pytest.mark.parametrize("precision,tol", [(fm.FP64, 1e-13), (fm.FP32, 2e-6)])
def test_without_room(n_rhs, precision, tol):
    V, F, D = fi.torus(1.0, 0.25, 61, 19)
    lib = fm.load_library()
    a, b = [fm.FMBEM(V, F, D, [1.0, -8.5 + 0.3j], [1.0, 1.0], 1.5, p=8, leaf_size=16) for _ in range(2)]
    x = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=n_rhs)).cuda()
    b.matvec(x[:1], precision=fm.BF16X3)  # densities, expansions and pair results of one right-hand side
    if n_rhs > 1:
        b.matvec(x.repeat(2, 1, 1), precision=fm.BF16X3)  # and, without pair results, of eighteen
    lib.fmbem_debug_set_device_budget(0)
    try:
        y = b.matvec(x, precision=precision)
    finally:
        lib.fmbem_debug_set_device_budget(-1)
    z = a.matvec(x)
    assert float((y - z).norm()) < tol * float(z.norm())
    assert float((b.matvec(x, precision=precision) - z).norm()) < tol * float(z.norm())


@pytest.mark.parametrize("room", [0, 1 << 18, 1 << 20, 1 << 22, 1 << 24])
def test_without_room_after_fewer_right_hand_sides(room):
    """A handle whose near-field scratch was sized by a product of one right-hand side, then one of nine with
    no room, or room for a part, of what they want: each buffer holds the call's size or is not used."""
    V, F, D = fi.torus(1.0, 0.25, 61, 19)
    lib = fm.load_library()
    a, b = [fm.FMBEM(V, F, D, [1.0, -8.5 + 0.3j], [1.0, 1.0], 1.5, p=8, leaf_size=16) for _ in range(2)]
    x = torch.from_numpy(fi.random_complex((9, a.N, 6), seed=room)).cuda()
    z = a.matvec(x)
    b.matvec(x[:1])
    b.matvec(x.repeat(2, 1, 1), precision=fm.BF16X3)  # densities and expansions of eighteen
    lib.fmbem_debug_set_device_budget(room)
    try:
        y = b.matvec(x)
    finally:
        lib.fmbem_debug_set_device_budget(-1)
    assert float((y - z).norm()) < 1e-13 * float(z.norm())
    assert float((b.matvec(x, precision=fm.FP32) - z).norm()) < 2e-6 * float(z.norm())


@pytest.mark.parametrize("call", ["matvec", "adjoint_matvec"])
@pytest.mark.parametrize("room", [0, 9 * 1159 * 192, 9 * 1159 * 192 + (1 << 20)])
def test_refused_product_leaves_the_handle_usable(call, room):
    """No room (or room for the densities alone) for the expansions of more right-hand sides: that product is
    refused, and the handle's next products, smaller and the same, give what they gave."""
    V, F, D = fi.torus(1.0, 0.25, 61, 19)
    lib = fm.load_library()
    b = fm.FMBEM(V, F, D, [1.0, -8.5 + 0.3j], [1.0, 1.0], 1.5, p=8, leaf_size=16)
    x = torch.from_numpy(fi.random_complex((9, b.N, 6), seed=3)).cuda()
    y1 = getattr(b, call)(x[:1])
    lib.fmbem_debug_set_device_budget(room)
    try:
        with pytest.raises(fm.FMBEMError):
            getattr(b, call)(x)
    finally:
        lib.fmbem_debug_set_device_budget(-1)
    assert torch.equal(getattr(b, call)(x[:1]), y1)
    assert float((getattr(b, call)(x)[0] - y1[0]).norm()) < 1e-13 * float(y1.norm())


@pytest.mark.parametrize("mesh,opt", [("torus", {}), ("two", {}), ("two", dict(boundary=fm.IMPEDANCE)),
                                      ("torus", dict(near_cache=0)), ("torus", dict(adaptive=1, leaf_size=12))])
@pytest.mark.parametrize("n_rhs", [1, 2, 4, 9])
@pytest.mark.parametrize("precision,tol", [(fm.FP64, 1e-13), (fm.FP32, 2e-6)])
def test_transposed_without_room(mesh, opt, n_rhs, precision, tol):
    """The transposed product without its partial sums: they go to the result and the densities' unused
    components."""
    if mesh == "torus":
        V, F, D = fi.torus(1.0, 0.25, 61, 19)
    else:
        V, F, D = fi.torus_and_sphere(nu=60, nv=18, sphere_subdiv=2)[0]
    eps, mu = [1.0, -8.5 + 0.3j, 2.25][: D.max() + 1], [1.0] * (D.max() + 1)
    lib = fm.load_library()
    a, b = [fm.FMBEM(V, F, D, eps, mu, 1.5, p=8, **opt) for _ in range(2)]
    x = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=n_rhs)).cuda()
    x[0] *= 1e-3
    z = a.adjoint_matvec(x)
    b.matvec(x, precision=fm.FP32)  # densities and expansions
    if 4 <= n_rhs <= 8:
        b.matvec(x)  # and FP64 pair results
    y = torch.full_like(x, float("nan"))
    lib.fmbem_debug_set_device_budget(0)
    try:
        b.adjoint_matvec(x, y, precision=precision)
    finally:
        lib.fmbem_debug_set_device_budget(-1)
    for r in range(n_rhs):
        assert float((y[r] - z[r]).norm()) < tol * float(z[r].norm())


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("n_rhs", [1, 3, 9])
@pytest.mark.parametrize("call", ["matvec", "adjoint_matvec"])
def test_part_of_the_room(call, n_rhs, captured):
    """Room for some of the optional scratch only, in steps of two: every product runs, in some form, and once
    there is room again in its usual one (the same bits as a handle that never lacked it)."""
    V, F, D = fi.torus(1.0, 0.25, 61, 19)
    lib = fm.load_library()
    a = fm.FMBEM(V, F, D, [1.0, -8.5 + 0.3j], [1.0, 1.0], 1.5, p=8, leaf_size=16)
    x = torch.from_numpy(fi.random_complex((n_rhs, a.N, 6), seed=n_rhs)).cuda()
    z = getattr(a, call)(x)
    for k in range(14, 29, 2):
        b = fm.FMBEM(V, F, D, [1.0, -8.5 + 0.3j], [1.0, 1.0], 1.5, p=8, leaf_size=16)
        y32 = b.matvec(x, precision=fm.FP32)
        if captured:
            out = torch.zeros_like(x)
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                b.matvec(x, out, precision=fm.FP32)
        lib.fmbem_debug_set_device_budget(1 << k)
        try:
            y, again = getattr(b, call)(x), getattr(b, call)(x)
            short = b.matvec(x, precision=fm.FP32)
        finally:
            lib.fmbem_debug_set_device_budget(-1)
        assert torch.equal(short, y32)
        for v in (y, again):
            assert float((v - z).norm()) < 1e-13 * float(z.norm())
        assert torch.equal(getattr(b, call)(x), z)
        if captured:
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, y32)
        b.close()
