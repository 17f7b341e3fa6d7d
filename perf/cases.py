"""Performance cases of the shifted boundary method operator.

Each case is one call a program makes once its problem is set up: an operator
apply (one problem on device vectors, one on host vectors, a batch of
problems with several right-hand sides) or a Krylov solve.  The sizes come
from the five workloads of ``synthetic.py`` and their neighbourhood.

``exact`` restates the operator in plain torch/numpy FP64 straight from the
weak form (dense cell matrix, Gauss quadrature on every face, closest points
by bisection); it uses none of this repository's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_17053_gb300 as G

# ---------------------------------------------------------------------------
# The cases
#
# call       "apply"  y = A x on device vectors
#            "host"   y = A x on page-locked host vectors (copies included)
#            "batch"  y_k = A_k x_k, nprob problems x nrhs right-hand sides
#            "cg" / "gmres"  a solve to a relative residual of 1e-10
# dtype      "f64" or "f32"; faces: the FP32 apply's face arithmetic
# values     "uniform" U(-1,1), "normal" N(0,1), or "graded" U(-1,1) with
#            magnitudes over six decades (a residual late in a solve)
# tuned      the problem's or batch's autotuner has run (long-lived handles)
# ---------------------------------------------------------------------------

_APPLY = dict(call="apply", dim=3, dg=False, domain="ball", gseed=0, dtype="f64", faces="fp32",
              extension="exact", values="uniform", tuned=True)


def _case(name=None, **kw):
    c = dict(_APPLY)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest use: a 2D study on 1 801 DoFs, where launches are all there is
        _case("f64_disk_q2_n32", dim=2, degree=2, cells=32, tuned=False),
        # the headline apply: 10.8 M DoFs in FP64, and as the inner operator of a
        # mixed-precision solve in FP32
        _case("f64_sphere_q4_n96", degree=4, cells=96),
        _case("f32_sphere_q4_n96", degree=4, cells=96, dtype="f32"),
        # the highest degree (Newton-projected ellipsoid), on a late residual in FP64 and
        # with tensor-core faces in FP32
        _case("f64_ellipsoid_q6_n48", degree=6, cells=48, domain="ellipsoid", values="graded"),
        _case("tf32_ellipsoid_q6_n48", degree=6, cells=48, domain="ellipsoid", dtype="f32",
              faces="tf32"),
        # discontinuous Galerkin on the torus, FP64 and FP32 cells with BF16 faces
        _case("f64_torus_dg_q3_n64", degree=3, cells=64, domain="torus", dg=True,
              values="normal"),
        _case("bf16_torus_dg_q3_n64", degree=3, cells=64, domain="torus", dg=True, dtype="f32",
              faces="bf16", values="normal"),
        # many small uneven problems at once: rotated ellipsoids of mixed degree and size
        dict(name="f64_batch_9x3", call="batch", nprob=9, nrhs=3, nmin=16, nmax=48, pmin=2,
             pmax=6, gseed=4, dtype="f64", values="uniform", tuned=True),
        dict(name="f32_batch_16x8", call="batch", nprob=16, nrhs=8, nmin=16, nmax=48, pmin=2,
             pmax=6, gseed=4, dtype="f32", values="uniform", tuned=True),
        # a host program without device buffers
        _case("host_sphere_q4_n96", call="host", degree=4, cells=96),
        # solves to 1e-10: CG where the operator is symmetric (a box on mesh planes), GMRES
        # on the nonsymmetric disk
        _case("cg_box_q3_n24", call="cg", degree=3, cells=24, domain="box", tuned=True),
        _case("gmres_disk_q2_n32", call="gmres", dim=2, degree=2, cells=32, tuned=False),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.random()
    if kind < 0.2:
        nmin = rng.randint(12, 24)
        return dict(call="batch", nprob=rng.randint(2, 16), nrhs=rng.randint(1, 8), nmin=nmin,
                    nmax=rng.randint(nmin, 40), pmin=rng.randint(1, 3), pmax=rng.randint(3, 6),
                    gseed=rng.randint(5, 10 ** 6), dtype=rng.choice(["f64", "f32"]),
                    values=rng.choice(["uniform", "normal", "graded"]),
                    tuned=rng.random() < 0.7)
    if kind < 0.27:
        p = rng.randint(1, 3)
        return _case(call="cg", degree=p, cells=2 * _log_int(rng, 4, 72 // (2 * p)),
                     domain="box", gseed=rng.randint(0, 10 ** 6))
    dim = 2 if rng.random() < 0.2 else 3
    p = rng.randint(1, 6)
    span = _log_int(rng, 20, 1500) if dim == 2 else _log_int(rng, 20, 300)     # p * cells
    domain = rng.choice(["ball", "ellipsoid"] if dim == 2 else ["ball", "ellipsoid", "torus"])
    cells = max(12 if domain == "torus" else 8, span // p)
    dtype = rng.choice(["f64", "f64", "f32"])
    extension = "taylor1" if rng.random() < 0.15 else "exact"
    faces = "fp32"
    if dtype == "f32" and dim == 3 and extension == "exact":
        faces = rng.choice(["fp32", "fp32", "tf32", "bf16"])
    dg = rng.random() < 0.25
    call = "host" if dtype == "f64" and rng.random() < 0.15 else "apply"
    return _case(call=call, dim=dim, degree=p, cells=cells, domain=domain,
                 gseed=rng.randint(1, 10 ** 6), dg=dg, dtype=dtype, faces=faces,
                 extension=extension,
                 values=rng.choice(["uniform", "normal", "graded"]),
                 tuned=rng.random() < 0.6)


# ---------------------------------------------------------------------------
# Domains: kind and parameters of the level set, from the case alone
# ---------------------------------------------------------------------------

def _rotation(rng, d):
    q = rng.standard_normal((d, d))
    q, r = np.linalg.qr(q)
    return q * np.sign(np.diag(r))


def _domain(case):
    """(kind, geometry parameters) as the problem description takes them."""
    d, s = case["dim"], case["gseed"]
    rng = np.random.default_rng(s)
    if case["domain"] == "ball":
        if s == 0:
            return "ball", [0.05, -0.03, 0.73] if d == 2 else [0.02, 0.01, -0.03, 0.71]
        return "ball", list(rng.uniform(-0.06, 0.06, d)) + [rng.uniform(0.6, 0.85)]
    if case["domain"] == "ellipsoid":
        if s == 0:
            return "ellipsoid", [0.8, 0.6, 0.5][:d] + list(np.eye(d).ravel()) + [0.0] * d
        return "ellipsoid", (list(rng.uniform(0.4, 0.85, d)) + list(_rotation(rng, d).ravel())
                             + list(rng.uniform(-0.05, 0.05, d)))
    if case["domain"] == "torus":
        return "torus", [0.6, 0.25] if s == 0 else [rng.uniform(0.5, 0.62),
                                                     rng.uniform(0.2, 0.3)]
    # a box whose faces are mesh planes: no shift, a symmetric positive definite operator
    h = 2.0 / case["cells"]
    lo = h * max(1, case["cells"] // 12)
    return "box", [0.0] * d + [1.0 - lo] * d


def _members(case):
    """The single problems of a batch, as apply cases."""
    rng = np.random.default_rng(case["gseed"])
    out = []
    for k in range(case["nprob"]):
        n = int(rng.integers(case["nmin"], case["nmax"] + 1))
        p = int(rng.integers(case["pmin"], case["pmax"] + 1))
        # high degrees on the finer meshes would hide the small problems
        n = max(min(case["nmin"], n), min(n, 168 // p))
        out.append(_case(degree=p, cells=n, domain="ellipsoid",
                         gseed=int(rng.integers(1, 2 ** 31)), dtype=case["dtype"],
                         values=case["values"], tuned=False))
    return out


# ---------------------------------------------------------------------------
# What a program has in hand, and one pass
# ---------------------------------------------------------------------------

def _problem(case):
    kind, geom = _domain(case)
    return G.Problem(case["dim"], case["degree"], case["cells"], kind, geom, dg=case["dg"],
                     extension=case["extension"], gpu_setup=True)


def _vector(case, n, seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    if case["values"] == "normal":
        x = torch.randn(n, generator=g, device=device, dtype=torch.float64)
    else:
        x = 2.0 * torch.rand(n, generator=g, device=device, dtype=torch.float64) - 1.0
        if case["values"] == "graded":
            x *= 10.0 ** (-6.0 * torch.rand(n, generator=g, device=device, dtype=torch.float64))
    return x.to(torch.float32) if case["dtype"] == "f32" else x


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        members = _members(case)
        problems = [_problem(m) for m in members]
        batch = G.Batch(problems, case["nrhs"], autotune=case["tuned"])
        xs = [_vector(m, p.n_dofs * case["nrhs"], seed * 64 + k)
              for k, (m, p) in enumerate(zip(members, problems))]
        return dict(call=call, batch=batch, problems=problems, xs=xs,
                    ys=[torch.empty_like(x) for x in xs])
    P = _problem(case)
    if case["tuned"]:
        G.sbm_autotune(P.handle)
    if call in ("cg", "gmres"):
        # the manufactured problem's right-hand side, perturbed from case to case
        b = P.rhs_device(0)
        b = b * (1.0 + 0.1 * _vector(case, P.n_dofs, seed))
        return dict(call=call, P=P, b=b, x=torch.zeros_like(b))
    x = _vector(case, P.n_dofs, seed)
    if call == "host":
        x = x.cpu().pin_memory()
        return dict(call=call, P=P, x=x, y=torch.empty_like(x).pin_memory())
    return dict(call=call, P=P, x=x, y=torch.empty_like(x), f32=case["dtype"] == "f32",
                faces=case["faces"])


def run(state):
    call = state["call"]
    if call == "apply":
        if state["f32"]:
            return state["P"].apply_f32(state["x"], state["y"], face_mode=state["faces"])
        return state["P"].apply_f64(state["x"], state["y"])
    if call == "host":
        return state["P"].apply_f64_host(state["x"], state["y"])
    if call == "batch":
        return state["batch"].apply(state["xs"], state["ys"])
    state["x"].zero_()
    if call == "cg":
        G.sbm_cg(state["P"].handle, state["b"], state["x"], rtol=1e-10, maxit=5000,
                 raise_not_converged=True)
    else:
        G.sbm_gmres(state["P"].handle, state["b"], state["x"], rtol=1e-10, maxit=5000,
                    restart=100, raise_not_converged=True)
    return state["x"]


# ---------------------------------------------------------------------------
# Work and tolerance
# ---------------------------------------------------------------------------

def _counts(case):
    """(DoFs, active cells, surrogate faces, interior faces)."""
    d, p = case["dim"], case["degree"]
    act = _active(case)                              # axis order (d-1, ..., 0)
    nc = int(act.sum())
    sur = inner = 0
    for ax in range(d):
        both = int((act & np.roll(act, 1, ax)).sum())
        first = act.take(0, ax) & act.take(-1, ax)   # not neighbours: opposite ends
        both -= int(first.sum())
        inner += both
        sur += 2 * (nc - both)
    if case["dg"]:
        return nc * (p + 1) ** d, nc, sur, inner
    # nodes by entity: every lattice entity (vertex .. cell) of an active cell, once
    total = 0
    for ext in range(2 ** d):                        # axes along which the entity extends
        e = np.pad(act, 1)
        span = 0
        for ax in range(d):
            if ext >> ax & 1:
                e = e.take(range(1, e.shape[ax] - 1), ax)
                span += 1
            else:
                e = e.take(range(0, e.shape[ax] - 1), ax) | e.take(range(1, e.shape[ax]), ax)
        total += int(e.sum()) * (p - 1) ** span
    return total, nc, sur, inner


def _apply_flops(case, counts):
    """Sum-factorised operator: the cell term's even/odd line products and
    folds, n^(2d-1) products per surrogate face, the traces and mass products
    of the interior faces."""
    d, n = case["dim"], case["degree"] + 1
    _, nc, sur, inner = counts
    lines = n ** (d - 1)
    prod = 2 * ((n // 2) ** 2 + ((n + 1) // 2) ** 2) + 4 * (n // 2)
    cell = lines * prod * (5 if d == 3 else 4)
    face = 2 * n ** (2 * d - 1) + 8 * d * n ** d
    return nc * cell + sur * face + inner * 2 * lines * (2 * n + 4 * (d - 1) * n)


def work(case):
    size = 4 if case.get("dtype") == "f32" else 8
    if case["call"] == "batch":
        total = dict(bytes=0, flops=0)
        for m in _members(case):
            c = _counts(m)
            total["bytes"] += case["nrhs"] * 2 * size * c[0]
            total["flops"] += case["nrhs"] * _apply_flops(m, c)
        return total
    c = _counts(case)
    if case["call"] in ("cg", "gmres"):
        # the right-hand side in, the solution out, and at the least as many applies as
        # there are cells across the mesh (information travels one cell per apply)
        k = case["cells"]
        return dict(bytes=16 * c[0], flops=k * _apply_flops(case, c))
    return dict(bytes=2 * size * c[0], flops=_apply_flops(case, c))


def tolerance(case):
    if case["call"] in ("cg", "gmres"):
        # two solves stopped at a relative residual of 1e-10 differ by up to the condition
        # number times that
        return {"rel": 1e-7, "max": 1e-6}
    # four times the distance measured between the path and exact() (FP64: 1.4e-14, most of
    # it the shifted points' rounding over h; FP32: 1.2e-7; tensor-core faces: 2.4e-4 to 4e-4
    # in TF32, 2e-3 to 2.6e-3 in BF16)
    if case["dtype"] == "f64":
        return {"rel": 6e-14, "max": 3e-12}
    if case.get("faces") == "tf32":
        return {"rel": 1.6e-3, "max": 6e-2}
    if case.get("faces") == "bf16":
        return {"rel": 1e-2, "max": 4e-1}
    return {"rel": 5e-7, "max": 2e-5}


# ---------------------------------------------------------------------------
# The operator in plain FP64
# ---------------------------------------------------------------------------

def _phi(kind, g, x):
    d = x.shape[-1]
    g = np.asarray(g, dtype=np.float64)
    if kind == "ball":
        s = np.zeros(x.shape[:-1])
        for i in range(d):
            s = s + (x[..., i] - g[i]) * (x[..., i] - g[i])
        return np.sqrt(s) - g[d]
    if kind == "ellipsoid":
        R, c = g[d:d + d * d].reshape(d, d), g[d + d * d:]
        s = np.zeros(x.shape[:-1])
        for i in range(d):
            y = np.zeros(x.shape[:-1])
            for j in range(d):
                y = y + R[j, i] * (x[..., j] - c[j])
            s = s + (y / g[i]) * (y / g[i])
        return s - 1.0
    if kind == "torus":
        rho = np.sqrt(x[..., 0] * x[..., 0] + x[..., 1] * x[..., 1])
        return (rho - g[0]) * (rho - g[0]) + x[..., 2] * x[..., 2] - g[1] * g[1]
    m = np.abs(x[..., 0] - g[0]) - g[d]
    for i in range(1, d):
        m = np.maximum(m, np.abs(x[..., i] - g[i]) - g[d + i])
    return m


def _active(case):
    """Cells whose centre lies strictly inside, as a bool array over axes
    (d-1, ..., 0)."""
    d, N = case["dim"], case["cells"]
    kind, geom = _domain(case)
    c = -1.0 + (2.0 / N) * (np.arange(N) + 0.5)
    grid = np.stack(np.meshgrid(*([c] * d), indexing="ij")[::-1], axis=-1)
    return _phi(kind, geom, grid) < 0.0


def _closest(kind, g, x):
    """Closest points on the boundary (torch, [..., d])."""
    d = x.shape[-1]
    g = torch.tensor(np.asarray(g, dtype=np.float64), device=x.device)
    if kind == "ball":
        v = x - g[:d]
        return g[:d] + g[d] * v / v.norm(dim=-1, keepdim=True)
    if kind == "torus":
        q = x.clone()
        q[..., 2] = 0.0
        q = g[0] * q / q.norm(dim=-1, keepdim=True)
        v = x - q
        return q + g[1] * v / v.norm(dim=-1, keepdim=True)
    if kind == "ellipsoid":
        a, R, c = g[:d], g[d:d + d * d].reshape(d, d), g[d + d * d:]
        y = (x - c) @ R
        a2 = a * a
        inside = ((y / a) ** 2).sum(-1) <= 1.0
        lo = torch.where(inside, -a2.min(), torch.zeros_like(a[0]))
        hi = torch.where(inside, torch.zeros_like(a[0]), a.max() * y.norm(dim=-1))
        for _ in range(120):
            mid = 0.5 * (lo + hi)
            up = ((a * y / (a2 + mid[..., None])) ** 2).sum(-1) > 1.0
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        z = a2 * y / (a2 + (0.5 * (lo + hi))[..., None])
        return c + z @ R.T
    v, half = x - g[:d], g[d:2 * d]
    near = (half - v.abs()).argmin(-1, keepdim=True)
    on = g[:d] + torch.where(v >= 0, half, -half)
    return x.scatter(-1, near, on.expand_as(x).gather(-1, near))


def _lagrange(nodes, x):
    """Values and derivatives of the Lagrange basis at x: [..., n] each."""
    n = len(nodes)
    val = torch.ones(x.shape + (n,), dtype=x.dtype, device=x.device)
    der = torch.zeros_like(val)
    for j in range(n):
        for m in range(n):
            if m == j:
                continue
            f = 1.0 / (nodes[j] - nodes[m])
            der[..., j] = der[..., j] * (x - nodes[m]) * f + val[..., j] * f
            val[..., j] = val[..., j] * (x - nodes[m]) * f
    return val, der


def _tables(p, dev):
    inner = np.polynomial.legendre.Legendre.basis(p).deriv().roots() if p > 1 else []
    for _ in range(3):                       # polish the Gauss-Lobatto points
        if len(inner):
            L1 = np.polynomial.legendre.Legendre.basis(p).deriv()
            inner = inner - L1(inner) / L1.deriv()(inner)
    nodes = 0.5 + 0.5 * np.concatenate([[-1.0], np.sort(np.real(inner)), [1.0]])
    gq, gw = np.polynomial.legendre.leggauss(p + 1)
    nodes = torch.tensor(nodes, device=dev)
    gq, gw = torch.tensor(0.5 + 0.5 * gq, device=dev), torch.tensor(0.5 * gw, device=dev)
    S, D = _lagrange(nodes, gq)
    M = torch.einsum("q,qi,qj->ij", gw, S, S)
    K = torch.einsum("q,qi,qj->ij", gw, D, D)
    ends = _lagrange(nodes, torch.tensor([0.0, 1.0], device=dev, dtype=torch.float64))[1]
    return dict(nodes=nodes, gq=gq, gw=gw, S=S, D=D, M=M, K=K, ends=ends)


def _operator(case, xs):
    """A x for each vector of xs (torch FP64), in the problem's DoF order."""
    d, p, N = case["dim"], case["degree"], case["cells"]
    n, h = p + 1, 2.0 / case["cells"]
    dev = xs[0].device
    t = _tables(p, dev)
    kind, geom = _domain(case)
    mask = torch.tensor(_active(case), device=dev)
    cells = mask.nonzero()                                   # [Nc, d], axes d-1 .. 0
    nc = len(cells)
    if case["dg"]:
        idx = torch.arange(nc * n ** d, device=dev).reshape((nc,) + (n,) * d)
    else:
        m = p * N + 1
        lat = torch.zeros((nc,) + (1,) * d, dtype=torch.int64, device=dev)
        for a in range(d):                                   # array axis a is mesh axis d-1-a
            shape = [1] * (d + 1)
            shape[a + 1] = n
            pos = (p * cells[:, a])[:, None] + torch.arange(n, device=dev)
            view = [nc] + shape[1:]
            lat = lat * m + pos.reshape(view)
        seen = torch.zeros(m ** d, dtype=torch.bool, device=dev)
        seen[lat.reshape(-1)] = True
        number = torch.cumsum(seen, 0) - 1
        idx = number[lat.reshape(-1)].reshape(lat.shape)
        del seen, number, lat
    M, K, S, D, ends = t["M"], t["K"], t["S"], t["D"], t["ends"]
    AK = None
    for k in range(d):
        term = torch.ones(1, 1, device=dev, dtype=torch.float64)
        for a in range(d):
            term = torch.kron(term, K if d - 1 - a == k else M)
        AK = term if AK is None else AK + term
    AK = AK * h ** (d - 2)
    pen = 10.0 * (p + 1) ** 2 / h if case["dg"] else 10.0 * p ** 2 / h
    pen_in = (p + 1) ** 2 / h
    look = torch.full((N + 2,) * d, -1, dtype=torch.int64, device=dev)
    look[tuple((cells + 1).T)] = torch.arange(nc, device=dev)
    W = t["gw"] if d == 2 else torch.outer(t["gw"], t["gw"])  # [second, first] tangential axis
    W = W.reshape(-1) * h ** (d - 1)

    def trace(U, k, s):
        """Value and outward-axis derivative of U [F, n..n] on face (k, s) at
        its tangential nodes, [F, n^(d-1)] (first tangential axis fastest)."""
        V = U.movedim(d - k, -1)                             # the normal axis last
        return (V[..., p if s else 0].reshape(len(U), -1),
                (V @ ends[s] / h).reshape(len(U), -1))

    def embed(rv, rg, k, s):
        """Transpose of trace."""
        V = rg[..., None] * (ends[s] / h)
        V[..., p if s else 0] += rv
        return V.reshape((len(rv),) + (n,) * d).movedim(-1, d - k)

    SS = S if d == 2 else torch.kron(S, S)                   # tangential nodes -> Gauss points
    out = []
    blocks = [slice(i, i + 1024) for i in range(0, nc, 1024)]
    surf = []
    for k in range(d):
        for s in (0, 1):
            step = torch.zeros(d, dtype=torch.int64, device=dev)
            step[d - 1 - k] = 1 if s else -1
            nb = look[tuple((cells + 1 + step).T)]
            own = (nb < 0).nonzero()[:, 0]
            for i in range(0, len(own), 2048):
                c = own[i:i + 2048]
                lo = -1.0 + h * cells[c].flip(-1).to(torch.float64)          # axes 0 .. d-1
                ref = torch.zeros((len(c), n ** (d - 1), d), dtype=torch.float64, device=dev)
                ref[..., k] = float(s)
                tang = [l for l in range(d) if l != k]
                ref[..., tang[0]] = t["gq"].repeat(n ** (d - 2))
                if d == 3:
                    ref[..., tang[1]] = t["gq"].repeat_interleave(n)
                xt = lo[:, None, :] + h * ref
                xg = _closest(kind, geom, xt)
                if case["extension"] == "exact":
                    aux = _lagrange(t["nodes"], (xg - lo[:, None, :]) / h)[0]  # [F, Q, d, n]
                else:
                    aux = xg - xt
                surf.append((k, s, c, aux))
            if case["dg"] and s == 1:
                low = (nb >= 0).nonzero()[:, 0]
                for i in range(0, len(low), 8192):
                    surf.append((k, 2, low[i:i + 8192], nb[low[i:i + 8192]]))
    for x in xs:
        y = torch.zeros_like(x)

        def add(c, V):
            y.index_add_(0, idx[c].reshape(-1), V.reshape(-1))

        for b in blocks:
            c = torch.arange(nc, device=dev)[b]
            add(c, x[idx[c]].reshape(len(c), -1) @ AK)
        for k, s, c, aux in surf:
            U = x[idx[c]]
            if s == 2:                                       # interior face, Algorithm 2
                U2 = x[idx[aux]]
                u1, d1 = trace(U, k, 1)
                u2, d2 = trace(U2, k, 0)
                jump, avg = (u1 - u2) @ SS.T, 0.5 * (d1 + d2) @ SS.T
                tv = (W * (pen_in * jump - avg)) @ SS
                tg = (-0.5 * W * jump) @ SS
                add(c, embed(tv, tg, k, 1))
                add(aux, embed(-tv, tg, k, 0))
                continue
            sg = 1.0 if s else -1.0
            uv, dn = trace(U, k, s)
            dn = sg * (dn @ SS.T)
            if case["extension"] == "exact":
                E = torch.einsum("f...i,fqi->fq...", U, aux[:, :, 0])
                for l in range(1, d):
                    E = torch.einsum("fq...i,fqi->fq...", E, aux[:, :, l])
            else:
                tang = [l for l in range(d) if l != k]
                E = uv @ SS.T + aux[..., k] * sg * dn
                if d == 2:
                    E = E + aux[..., tang[0]] * (uv @ D.T) / h
                else:
                    E = E + aux[..., tang[0]] * (uv @ torch.kron(S, D).T) / h
                    E = E + aux[..., tang[1]] * (uv @ torch.kron(D, S).T) / h
            add(c, embed((W * (pen * E - dn)) @ SS, (-sg * W * E) @ SS, k, s))
        out.append(y)
    return out


def exact(case, seed):
    if case["call"] in ("cg", "gmres"):
        return None                                          # defined by its residual only
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["call"] != "batch":
        n = _counts(case)[0]
        return _operator(case, [_vector(case, n, seed, dev).to(torch.float64)])[0]
    out = []
    for k, m in enumerate(_members(case)):
        n = _counts(m)[0]
        x = _vector(m, n * case["nrhs"], seed * 64 + k, dev).to(torch.float64)
        out.append(torch.cat(_operator(m, list(x.reshape(case["nrhs"], n)))))
    return out
