"""Performance cases of the FMM-BEM library: what its users run, through its public entry points.

A user solves scattering problems.  That is one handle per scatterer and frequency, and then many
products y = A x inside a Krylov solve (the library's own, ``FMBEM.solve``, or theirs around
``FMBEM.matvec``), their transposes for gradients, or the products of many small particles in one
launch (``PersistentBatch``).  The listed cases are these calls from 642 to 163842 nodes and from 1 to
128 right-hand sides, in every precision that is used in earnest.

A case is a dict of plain values:
  call       "product", "adjoint" (transposed product), "solve" or "batch"
  shape      "sphere" (icosphere of ``subdiv``), "torus" (``nu`` x ``nv`` grid) or "torus_sphere"
             (a torus and a small sphere above it: two scatterers); a batch draws its particles
  precision  "fp64", "fp32" or "bf16x3"; for a solve, of its Krylov iterations
  n_rhs, p   right-hand sides and truncation number
  eps_re, eps_im, k0   the scatterer's permittivity and the vacuum wavenumber

Products asked for in single precision (fp32, bf16x3) are kept in complex64, as the library's own
refined solve keeps their Krylov basis: their last digits beyond that carry nothing.
"""
import math

import numpy as np
import torch

import paper_1211_7177_gb300 as fm
from paper_1211_7177_gb300.batch import PersistentBatch

PRECISION = {"fp64": fm.FP64, "fp32": fm.FP32, "bf16x3": fm.BF16X3}
SPHERE = {"shape": "sphere", "eps_re": -8.5, "eps_im": 0.3, "k0": 0.5}  # silver-like, a = 1
TORUS = {"shape": "torus", "eps_re": -10.0, "eps_im": 0.4, "k0": 1.5}  # silver-like, R = 1, r = 0.25
GLASS = {"shape": "sphere", "eps_re": 2.25, "eps_im": 0.0, "k0": 1.0}  # the dielectric sphere


def listed():
    return [
        # the smallest product: one wave on a particle far below the wavelength; launches count
        dict(GLASS, name="product fp64 642x1", call="product", subdiv=3, precision="fp64", n_rhs=1, p=8),
        # the plain method, a whole call: the dielectric sphere solved to 1e-6
        dict(GLASS, name="solve fp64 2562x1", call="solve", subdiv=4, precision="fp64", n_rhs=1, p=8, tol=1e-6),
        # the true residual of a batched solve of ordinary size (16 waves at once, FP64)
        dict(TORUS, name="product fp64 9216x16", call="product", nu=192, nv=48, precision="fp64", n_rhs=16, p=8),
        # the plain method at scale: every iteration of an FP64 solve, every true residual
        dict(SPHERE, name="product fp64 163842x1", call="product", subdiv=7, precision="fp64", n_rhs=1, p=10),
        # the inner iteration of the refined solve at scale
        dict(SPHERE, name="product bf16x3 163842x1", call="product", subdiv=7, precision="bf16x3", n_rhs=1, p=10),
        # the same in plain single precision, ordinary size
        dict(SPHERE, name="product fp32 40962x1", call="product", subdiv=6, precision="fp32", n_rhs=1, p=10),
        # many directions and polarisations at once: the inner iteration of the batched solve
        dict(TORUS, name="product bf16x3 65536x128", call="product", nu=512, nv=128, precision="bf16x3", n_rhs=128, p=8),
        # the same on an ordinary mesh, with a count of waves that fills no whole blocks and odd grid sizes
        dict(TORUS, name="product bf16x3 21973x40", call="product", nu=301, nv=73, precision="bf16x3", n_rhs=40, p=8),
        # gradients: the three adjoints of an optical force on a particle above a torus
        dict(TORUS, name="adjoint bf16x3 17026x3", call="adjoint", shape="torus_sphere", nu=256, nv=64, precision="bf16x3",
             n_rhs=3, p=8),
        # gradients: the true residual of an adjoint solve
        dict(SPHERE, name="adjoint fp64 10242x1", call="adjoint", subdiv=5, precision="fp64", n_rhs=1, p=10),
        # a whole refined solve: BF16x3 Krylov iterations, FP64 residuals, to the accuracy that
        # gradients and their finite-difference checks ask for
        dict(SPHERE, name="solve bf16x3 10242x1", call="solve", subdiv=5, precision="bf16x3", n_rhs=1, p=10, tol=1e-12),
        # particles of uneven sizes, every product in one launch
        dict(name="batch fp32 12 particles", call="batch", particles=12, smallest=1000, largest=8000, precision="fp32",
             n_rhs=4, p=8, k0=1.0),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["product"] * 6 + ["adjoint"] * 2 + ["solve", "batch"])
    if call == "batch":
        smallest = int(_log_uniform(rng, 400, 2000))
        return {"call": "batch", "particles": rng.randint(3, 16), "smallest": smallest,
                "largest": int(smallest * _log_uniform(rng, 1.5, 6)), "precision": "fp32", "n_rhs": rng.randint(1, 4),
                "p": rng.choice([6, 8]), "k0": round(rng.uniform(0.3, 3.0), 3)}
    precision = rng.choice(["fp64", "fp64", "fp32", "bf16x3", "bf16x3"])
    if call == "solve":
        precision = rng.choice(["fp64", "bf16x3"])
    # nodes x right-hand sides, kept below the largest listed case of the same precision
    most, most_nodes, most_rhs = {"fp64": (163000, 163000, 24), "fp32": (400000, 100000, 24), "bf16x3": (4000000, 163000, 128)}[
        precision]
    if call == "adjoint":
        most, most_rhs = most // 8, min(most_rhs, 32)
    if call == "solve":
        most, most_nodes, most_rhs = 10000, 10000, 2
    nodes = _log_uniform(rng, 600, most_nodes)
    n_rhs = max(1, min(most_rhs, int(_log_uniform(rng, 1, max(1.0, most / nodes)))))
    nodes = min(nodes, most / n_rhs)
    ratio = rng.uniform(2.0, 6.0)
    nv = max(8, int(math.sqrt(nodes / ratio)))
    nu = max(16, int(nodes / nv))
    case = dict(TORUS, call=call, nu=nu, nv=nv, precision=precision, n_rhs=n_rhs, p=rng.choice([8, 10]) if n_rhs <= 8 else 8,
                k0=round(rng.uniform(0.3, 2.0), 3))
    case["eps_re"], case["eps_im"] = rng.choice([(2.25, 0.0), (-5.0, 0.2), (-10.0, 0.4)])
    if call == "solve":  # the plain solve to the usual residual, the refined one to a gradient's
        case["eps_re"], case["eps_im"] = 2.25, 0.0
        case["tol"] = 1e-6 if precision == "fp64" else 1e-12
    return case


# ------------------------------------------------------------------------------------------- meshes
def _torus(R, r, nu, nv):
    u, w = np.meshgrid(2 * np.pi * np.arange(nu) / nu, 2 * np.pi * np.arange(nv) / nv, indexing="ij")
    V = np.stack([(R + r * np.cos(w)) * np.cos(u), (R + r * np.cos(w)) * np.sin(u), r * np.sin(w)], -1).reshape(-1, 3)
    i, j = (a.ravel() for a in np.meshgrid(np.arange(nu), np.arange(nv), indexing="ij"))
    ip, jp = (i + 1) % nu, (j + 1) % nv
    a, b, c, d = i * nv + j, ip * nv + j, ip * nv + jp, i * nv + jp
    return V, np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)]).astype(np.int32)


def _icosphere(subdiv):
    t = (1 + math.sqrt(5)) / 2
    V = np.array([(-1, t, 0), (1, t, 0), (-1, -t, 0), (1, -t, 0), (0, -1, t), (0, 1, t), (0, -1, -t), (0, 1, -t), (t, 0, -1),
                  (t, 0, 1), (-t, 0, -1), (-t, 0, 1)], dtype=np.float64)
    F = np.array([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2), (10, 7, 6),
                  (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5), (2, 4, 11), (6, 2, 10),
                  (8, 6, 7), (9, 8, 1)])
    V /= np.linalg.norm(V, axis=1, keepdims=True)
    for _ in range(subdiv):
        e = np.sort(np.concatenate([F[:, [0, 1]], F[:, [1, 2]], F[:, [2, 0]]]), axis=1)
        e, at = np.unique(e, axis=0, return_inverse=True)
        m = V[e[:, 0]] + V[e[:, 1]]
        ab, bc, ca = (len(V) + at.reshape(3, -1)).astype(np.int64)
        V = np.concatenate([V, m / np.linalg.norm(m, axis=1, keepdims=True)])
        a, b, c = F.T
        F = np.concatenate([np.stack(q, 1) for q in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    return V, F.astype(np.int32)


def _mesh(case):
    """(vertices, triangles, scatterer of each triangle, number of scatterers) of a case."""
    if case["shape"] == "sphere":
        V, F = _icosphere(case["subdiv"])
    else:
        V, F = _torus(1.0, 0.25, case["nu"], case["nv"])
    D = np.ones(len(F), dtype=np.int32)
    if case["shape"] != "torus_sphere":
        return V, F, D, 1
    Vs, Fs = _icosphere(3)
    Vs = 0.1 * Vs + np.array([1.0, 0.0, 0.5])
    return (np.concatenate([V, Vs]), np.concatenate([F, Fs + len(V)]).astype(np.int32),
            np.concatenate([D, np.full(len(Fs), 2, dtype=np.int32)]), 2)


def _media(case, scatterers):
    """eps and mu of the background and the scatterers (the second scatterer is a dielectric)."""
    return [1.0, complex(case["eps_re"], case["eps_im"]), 2.5][: scatterers + 1], [1.0] * (scatterers + 1)


def _nodes(V, F):
    """Vertex nodes: normals (sum of the incident triangles' area vectors) and weights (a third of
    their areas)."""
    c = np.cross(V[F[:, 1]] - V[F[:, 0]], V[F[:, 2]] - V[F[:, 0]])
    n, w = np.zeros_like(V), np.zeros(len(V))
    for k in range(3):
        for q in range(3):
            n[:, q] += np.bincount(F[:, k], c[:, q], len(V))
        w += np.bincount(F[:, k], np.linalg.norm(c, axis=1) / 6, len(V))
    return n / np.linalg.norm(n, axis=1, keepdims=True), w


# ------------------------------------------------------------------------------------------- inputs
def _waves(n, seed):
    """n plane waves: unit directions and unit polarisations across them."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    e = np.cross(d, rng.normal(size=(n, 3)))
    return d, (e / np.linalg.norm(e, axis=1, keepdims=True)).astype(np.complex128)


def _surface_data(V, F, k0, n_rhs, seed):
    """What a Krylov iteration multiplies: the surface data (E, n x curl E) of plane waves, which
    vary smoothly, and a tenth of complex noise."""
    d, e = _waves(n_rhs, seed)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    s, n = (torch.as_tensor(a, device="cuda") for a in (V, _nodes(V, F)[0]))
    d, e = torch.as_tensor(d, device="cuda"), torch.as_tensor(e, device="cuda")
    E = torch.exp(1j * k0 * (d @ s.T))[:, :, None] * e[:, None, :]  # [n_rhs, N, 3]
    curl = 1j * k0 * torch.linalg.cross(d.to(E.dtype)[:, None, :].expand_as(E), E)
    x = torch.cat([E, torch.linalg.cross(n.to(E.dtype)[None].expand_as(E), curl)], dim=2)
    noise = torch.randn(tuple(x.shape) + (2,), generator=g, device="cuda", dtype=torch.float64)
    return (x + 0.1 * torch.view_as_complex(noise)).contiguous()


def _particles(case):
    """The particles of a batch: spheroids and tori of log-uniform sizes, scaled to a largest
    dimension of 1; the same ones for every seed (the fields differ)."""
    rng = np.random.default_rng(case["particles"] * 100003 + case["smallest"] + case["largest"])
    out = []
    for i in range(case["particles"]):
        nodes = math.exp(rng.uniform(math.log(case["smallest"]), math.log(case["largest"])))
        if i % 4 == 3:
            V, F = _icosphere(3 if nodes < 1500 else 4)
            V = V * np.array([1.0, 1.0, rng.uniform(1.0, 3.0)])
        else:
            ratio = rng.uniform(2.0, 5.0)
            nv = max(8, int(math.sqrt(nodes / ratio)))
            V, F = _torus(1.0, 1.0 / ratio, max(16, int(nodes / nv)), nv)
        out.append((V / np.ptp(V, axis=0).max(), F, [1.0, [2.25, -5 + 0.2j, -12 + 0.5j][int(rng.integers(3))]]))
    return out


def prepare(case, seed):
    n, p = case["n_rhs"], case["p"]
    if case["call"] == "batch":
        parts = _particles(case)
        handles = [fm.FMBEM(V, F, np.ones(len(F), np.int32), eps, [1.0, 1.0], case["k0"], p=p, fp32_only=1)
                   for V, F, eps in parts]
        xs = [_surface_data(V, F, case["k0"], n, seed * 1009 + i) for i, (V, F, _) in enumerate(parts)]
        return {"call": "batch", "batch": PersistentBatch(handles, n), "xs": xs}
    V, F, D, J = _mesh(case)
    eps, mu = _media(case, J)
    options = {"p": p}
    if case["call"] == "solve" and case["precision"] != "fp64":
        options.update(solve_precision=PRECISION[case["precision"]], inner_tol=1e-4)
    h = fm.FMBEM(V, F, D, eps, mu, case["k0"], **options)
    state = {"call": case["call"], "handle": h, "precision": PRECISION[case["precision"]]}
    if case["call"] == "solve":
        state.update(b=h.plane_wave_rhs(*_waves(n, seed)), tol=case["tol"])
    else:
        state["x"] = _surface_data(V, F, case["k0"], n, seed)
    return state


def run(state):
    if state["call"] == "batch":
        return [y.to(torch.complex64) for y in state["batch"].matvec(state["xs"])]
    h = state["handle"]
    if state["call"] == "solve":
        x, _, _, status = h.solve(state["b"], tol=state["tol"])
        if status != 0:
            raise RuntimeError("the solve did not converge")
        return x
    product = h.matvec if state["call"] == "product" else h.adjoint_matvec
    y = product(state["x"], precision=state["precision"])
    return y if state["precision"] == fm.FP64 else y.to(torch.complex64)


# --------------------------------------------------------------------------------------------- work
# Counts of the method on a surface mesh at its default leaf size: a node has about 450 near
# sources per domain, and there are about 1.7 far-field translations per node and domain.
NEAR_PAIRS, FAR_PAIRS = 450, 1.7


def work(case):
    n_rhs, p = case["n_rhs"], case["p"]
    if case["call"] == "batch":
        nodes = sum(len(V) for V, _, _ in _particles(case))
    elif case["shape"] == "sphere":
        nodes = 10 * 4 ** case["subdiv"] + 2
    else:
        nodes = case["nu"] * case["nv"] + (642 if case["shape"] == "torus_sphere" else 0)
    # two domains; per near pair the Green's function and its gradient (52 operations) and their use
    # on a right-hand side (78); per translation three components of about 12.3 p^3 operations
    flops = 2.0 * nodes * (NEAR_PAIRS * (52 + 78 * n_rhs) + FAR_PAIRS * 3 * n_rhs * 12.3 * p ** 3)
    # x read, y written (six complex128 each, complex64 where the result is kept so), node data
    out = 16 if case["precision"] == "fp64" or case["call"] == "solve" else 8
    size = nodes * (6.0 * n_rhs * (16 + out) + 64)
    if case["call"] != "solve":
        return {"bytes": size, "flops": flops}
    steps = {1e-6: 20, 1e-12: 60}.get(case["tol"], 40)  # Krylov steps; each reads its basis twice
    return {"bytes": size * steps + nodes * 96.0 * n_rhs * steps * steps, "flops": flops * steps}


# -------------------------------------------------------------------------------------------- exact
def _self_blocks(V, F, eps, mu, k0, dom):
    """The 6 x 6 blocks of a node with itself: Eq. (2.12)'s delta terms and the integrals of Appendix B
    over the node's dual cell projected on its tangent plane (Eqs. B.2-B.9), edge by edge."""
    n, _ = _nodes(V, F)
    N = len(V)
    I1, S, V1, V3 = np.zeros(N), np.zeros(N), np.zeros((N, 3)), np.zeros((N, 3))
    add = lambda a, v, x: np.add.at(a, v, x)  # noqa: E731
    for k in range(3):
        v = F[:, k]
        A, B, C, nv = V[v], V[F[:, (k + 1) % 3]], V[F[:, (k + 2) % 3]], n[v]
        flat = lambda P: (P - A) - np.sum((P - A) * nv, 1, keepdims=True) * nv  # noqa: E731
        corner = [flat((A + B) / 2), flat((A + B + C) / 3), flat((A + C) / 2)]
        for P, Q in zip(corner[:2], corner[1:]):
            e = Q - P
            foot = P - (np.sum(P * e, 1) / np.sum(e * e, 1))[:, None] * e
            h = np.linalg.norm(foot, axis=1)
            i = foot / h[:, None]
            j = np.cross(nv, i)
            fP, fQ = (np.arctan2(np.sum(x * j, 1), np.sum(x * i, 1)) for x in (P, Q))
            L = np.arcsinh(np.tan(fQ)) - np.arcsinh(np.tan(fP))  # ln tan(pi/4 + f/2) = asinh(tan f)
            add(I1, v, h * L)
            add(S, v, 0.5 * h * h * (np.tan(fQ) - np.tan(fP)))
            add(V1, v, 0.5 * (h * h)[:, None] * (L[:, None] * i + (1 / np.cos(fQ) - 1 / np.cos(fP))[:, None] * j))
            add(V3, v, -L[:, None] * i)
    k = k0 * np.sqrt(np.asarray(eps, np.complex128) * np.asarray(mu, np.complex128))
    k = np.where(k.imag < 0, -k, k)
    M = np.zeros((N, 6, 6), np.complex128)
    for side in (0, 1):
        d = np.zeros(N, int) if side == 0 else dom
        kd, e = k[d][:, None], np.asarray(eps, np.complex128)[d]
        sg = (I1 + 1j * kd[:, 0] * S) / (4 * np.pi)
        a = -kd ** 2 / (8 * np.pi) * V1 - V3 / (4 * np.pi)
        nd = (-1 if side == 0 else 1) * n
        T = np.eye(3)[None] + ((eps[0] - e) / e)[:, None, None] * n[:, :, None] * n[:, None, :]
        na = np.sum(nd * a, 1)[:, None, None]
        bracket = nd[:, :, None] * a[:, None, :] - na * np.eye(3)[None] - a[:, :, None] * nd[:, None, :]
        M[:, 3 * side:3 * side + 3, :3] = 0.5 * T - bracket @ T
        gamma = np.asarray(mu, np.complex128)[d] / mu[0] * (-1 if side == 0 else 1)
        M[:, 3 * side:3 * side + 3, 3:] = (gamma * sg)[:, None, None] * np.eye(3)[None]
    return M


def _dense(V, F, eps, mu, k0, dom, x, transpose):
    """y = A x (or A^T x) of Eq. (2.12) by direct sums over all nodes, in 64 bits."""
    cd = torch.complex128
    n, w = _nodes(V, F)
    s, nt, wt, dt = (torch.as_tensor(a, device="cuda") for a in (V, n, w, dom))
    k = np.sqrt(np.asarray(eps, np.complex128) * np.asarray(mu, np.complex128)) * k0
    k = np.where(k.imag < 0, -k, k)
    N, R = len(V), x.shape[0]
    M = torch.as_tensor(_self_blocks(V, F, eps, mu, k0, dom), device="cuda")
    y = torch.einsum("nji,rnj->rni" if transpose else "nij,rnj->rni", M, x)
    for d in range(len(eps)):
        of = torch.arange(N, device="cuda") if d == 0 else torch.nonzero(dt == d)[:, 0]
        side = 0 if d == 0 else 1
        sd, nd, wd, jump = s[of], nt[of], wt[of], 0.0 if d == 0 else (eps[0] - eps[d]) / eps[d]
        sign, gamma = (-1.0, -1.0) if d == 0 else (1.0, mu[d] / mu[0])
        nn = nd.to(cd)
        T = lambda v: v + jump * nn * torch.sum(nn * v, -1, keepdim=True)  # noqa: E731
        if transpose:  # sources: this side's rows of x; targets get the transposed bracket
            src = [x[:, of, 3 * side + c].T.contiguous() for c in range(3)]  # [N_d, R]
        else:
            v, q = T(x[:, of, :3]), gamma * x[:, of, 3:]
            nv = torch.sum(nn * v, -1)
            # -bracket(n', a) v summed over sources: columns that multiply a_x, a_y, a_z and g
            W = torch.zeros(4, 3, len(of), R, dtype=cd, device="cuda")
            for c in range(3):
                for m in range(3):
                    t = sign * (nd[:, m] * v[:, :, c] - nd[:, c] * v[:, :, m])
                    W[m, c] = (wd * (t + (sign * nv if m == c else 0))).T
                W[3, c] = (wd * q[:, :, c]).T
            W = [W[m].permute(1, 0, 2).reshape(len(of), 3 * R) for m in range(4)]
        step = max(1, int(3e7 // len(of)))
        for b in range(0, len(of), step):
            at = of[b:b + step]
            r = sd[None, :, :] - s[at][:, None, :]  # source minus target
            if transpose:
                r = -r  # the gathering node is the source of the forward product
            dist = torch.linalg.norm(r, dim=-1)
            dist.masked_fill_(at[:, None] == of[None, :], math.inf)
            ph = torch.exp(1j * complex(k[d]) * torch.where(torch.isinf(dist), torch.zeros_like(dist), dist))
            g = ph / (4 * math.pi * dist)
            c = g * (1j * complex(k[d]) - 1 / dist) / dist
            del ph, dist
            if transpose:
                G = [torch.stack([(c * r[..., m]) @ src[i] for i in range(3)]) for m in range(3)]  # [m][i, at, R]
                n1, w1 = sign * nn[b:b + step][:, :, None], wd[b:b + step][:, None]
                grad = torch.stack(G, 0)  # [m, i, at, R] = sum a_m u_i
                div = grad[0, 0] + grad[1, 1] + grad[2, 2]
                out = []
                for q_ in range(3):
                    # -Bk^T u: -(a_q (n.u) - (n.a) u_q - n_q (a.u))
                    t = -sum(n1[:, i] * grad[q_, i] for i in range(3)) + sum(n1[:, m] * grad[m, q_] for m in range(3)) + n1[:, q_] * div
                    out.append(w1 * t)
                phi = torch.stack(out, -1).permute(1, 0, 2)  # [R, at, 3]
                nb = nn[b:b + step]
                y[:, at, :3] += phi + jump * nb * torch.sum(nb * phi, -1, keepdim=True)
                for i in range(3):
                    y[:, at, 3 + i] += (gamma * w1 * (g @ src[i])).T
            else:
                t = g @ W[3]
                for m in range(3):
                    t = t + (c * r[..., m]) @ W[m]
                y[:, at, 3 * side:3 * side + 3] += t.reshape(len(at), 3, R).permute(2, 0, 1)
    return y


def exact(case, seed):
    """The dense operator in 64 bits (no multipole expansion), where it takes seconds; a solve has no
    such value."""
    n = case["n_rhs"]
    if case["call"] == "solve":
        return None
    if case["call"] == "batch":
        return [_dense(V, F, eps, [1.0, 1.0], case["k0"], np.ones(len(V), int),
                       _surface_data(V, F, case["k0"], n, seed * 1009 + i), False) for i, (V, F, eps) in enumerate(_particles(case))]
    V, F, D, J = _mesh(case)
    if float(len(V)) ** 2 * (2000 + 100 * n) > 4e12:
        return None
    eps, mu = _media(case, J)
    dom = np.zeros(len(V), int)
    dom[F.ravel()] = np.repeat(D, 3)
    return _dense(V, F, eps, mu, case["k0"], dom, _surface_data(V, F, case["k0"], n, seed), case["call"] == "adjoint")
