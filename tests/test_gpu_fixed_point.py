"""The fixed-point FP64 cell term on the GPU: exponent range and non-finite
values (the arithmetic itself: test_fixed_point.py, and every FP64 apply test)."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2507_17053_gb300 as G
import synthetic as S
from oracle import local
from oracle.operator import Problem as OracleProblem

pytestmark = pytest.mark.gpu

CASES = [S.SPHERE_3D_Q4.resized(8, degree=p) for p in range(1, 7)]


@pytest.mark.parametrize("shape", [0, 1, 3])
@pytest.mark.parametrize("w", CASES, ids=lambda w: f"q{w.degree}")
def test_power_of_two_scaling_is_exact(w, shape):
    """A (2^k x) = 2^k (A x) bitwise, also where the careful conversions run
    (biased exponents below 128 and above 1900); all-zero input gives zeros."""
    P = G.Problem.from_workload(w)
    G.sbm_set_tile_shape(P.handle, shape, 0)
    x = torch.from_numpy(S.random_vector(w.seed, P.n_dofs, w.dist)).cuda()
    y = P.apply_f64(x)
    for k in (-950, -900, -300, 300, 870, 900):
        assert torch.equal(P.apply_f64(x * 2.0 ** k) * 2.0 ** -k, y), k
    assert not P.apply_f64(torch.zeros_like(x)).any()


@pytest.mark.parametrize("w", CASES, ids=lambda w: f"q{w.degree}")
def test_subnormal_input(w):
    """Inputs of a few subnormal units against the scaled problem, to the
    units the result can hold (the face term rounds there as well)."""
    P = G.Problem.from_workload(w)
    x = torch.from_numpy(np.rint(1e3 * S.random_vector(w.seed, P.n_dofs, w.dist))).cuda()
    y = P.apply_f64(x)
    tiny = 2.0 ** -1074
    yt = P.apply_f64(x * tiny).cpu().numpy() / tiny
    # h < 1 scales the products down: intermediate values of the face kernel and the
    # result are rounded to units of 2^-1074, the face results then multiplied by sigma,
    # 1/h and phi' (each below 10 p^2 / h)
    bound = 64.0 * (10.0 * w.degree ** 2 * w.cells / 2.0) ** 2
    assert np.abs(yt - y.cpu().numpy()).max() <= bound


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("w", CASES, ids=lambda w: f"q{w.degree}")
def test_non_finite_input_stays_in_its_cells(w, value):
    """One non-finite entry: the DoFs of the cells that hold it are not
    finite, every other one is bitwise unchanged."""
    P = G.Problem.from_workload(w)
    x = torch.from_numpy(S.random_vector(w.seed, P.n_dofs, w.dist)).cuda()
    i = P.n_dofs // 2
    e = torch.zeros_like(x)
    e[i] = 1.0
    for shape in (0, 1, 3):
        G.sbm_set_tile_shape(P.handle, shape, 0)
        y = P.apply_f64(x)
        near = P.apply_f64(e) != 0           # the rows that see x_i
        xb = x.clone()
        xb[i] = value
        yb = P.apply_f64(xb)
        assert not torch.isfinite(yb[near]).any()
        fin = torch.isfinite(yb)
        assert torch.equal(yb[fin], y[fin])
        assert int((~fin).sum()) <= 8 * (w.degree + 1) ** 3


# ---- discontinuous Galerkin: exponents of a cell and its neighbours ----------------

DG_CASES = [dataclasses.replace(w, dg=True) for w in CASES]


@pytest.mark.parametrize("w", DG_CASES, ids=lambda w: f"q{w.degree}")
def test_dg_power_of_two_scaling_is_exact(w):
    test_power_of_two_scaling_is_exact(w, 0)


@pytest.mark.parametrize("w", DG_CASES, ids=lambda w: f"q{w.degree}")
def test_dg_subnormal_input(w):
    test_subnormal_input(w)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("w", DG_CASES, ids=lambda w: f"q{w.degree}")
def test_dg_non_finite_input_stays_near(w, value):
    """One non-finite entry: its cell and that cell's neighbours are not finite,
    every other one is bitwise unchanged."""
    P = G.Problem.from_workload(w)
    nd = (w.degree + 1) ** 3
    O = OracleProblem.from_workload(w)
    x = torch.from_numpy(S.random_vector(w.seed, P.n_dofs, w.dist)).cuda()
    y = P.apply_f64(x).view(-1, nd)
    c = len(O.mesh.cells) // 2
    xb = x.clone()
    xb[c * nd + nd // 3] = value
    yb = P.apply_f64(xb).view(-1, nd)
    near = {c} | {int(b) for a, _, b in O.mesh.ifaces if a == c} \
        | {int(a) for a, _, b in O.mesh.ifaces if b == c}
    far = torch.ones(len(O.mesh.cells), dtype=torch.bool)
    far[sorted(near)] = False
    assert not torch.isfinite(yb[~far]).any()
    assert torch.equal(yb[far], y[far])


@pytest.mark.parametrize("w", DG_CASES, ids=lambda w: f"q{w.degree}")
def test_dg_neighbours_of_other_magnitudes(w):
    """Cells scaled by 2^-60 .. 2^60, neighbours at random: every cell against
    the oracle, relative to the largest values the double form sums for it --
    test_gpu_apply's bound times |A| |x| over the cell and its neighbours."""
    O = OracleProblem.from_workload(w)
    P = G.Problem.from_workload(w)
    nd, nc = (w.degree + 1) ** 3, len(O.mesh.cells)
    k = np.random.default_rng(5).integers(-60, 61, nc)
    x = (S.random_vector(w.seed, O.n_dofs, w.dist).reshape(nc, nd) * 2.0 ** k[:, None])
    y = P.apply_f64(torch.from_numpy(x.ravel()).cuda()).cpu().numpy().reshape(nc, nd)
    ref = O.apply(x.ravel()).reshape(nc, nd)
    big = np.abs(x).max(axis=1)
    for a, _, b in O.mesh.ifaces:
        m = max(np.abs(x[a]).max(), np.abs(x[b]).max())
        big[a], big[b] = max(big[a], m), max(big[b], m)
    one = np.abs(O.apply(np.ones(O.n_dofs) * S.random_vector(9, O.n_dofs, "uniform"))).max()
    assert (np.abs(y - ref).max(axis=1) <= 1e-12 * one * big).all()


# ---- discontinuous Galerkin: interior-face penalties of every size -----------------

DG_BOX = S._wl("box", 3, 2, 5, S.box((0.0,) * 3, (1.5,) * 3), dg=True, seed=5)
PENALTIES = [1.0, 2.0, 30.0, 1e3, 1e6, 1e9]    # in the line operators up to 1.2 .. 2.2


def _dg(p, pen=1.0):
    w = dataclasses.replace(DG_BOX.resized(5, degree=p), pen_interior=pen)
    return w, G.Problem.from_workload(w)


def _inner_cells(O):
    """Rows of the cells without surrogate faces."""
    rows = np.ones(len(O.mesh.cells), bool)
    rows[O.mesh.sfaces[:, 0]] = False
    return O.dofmap[rows].ravel()


@pytest.mark.parametrize("p", range(1, 7))
def test_dg_penalty_costs_conforming_data_nothing(p):
    """Data with equal traces: the penalty multiplies zeros, so the apply at
    any penalty is the one at pen_interior = 1, to test_gpu_apply's bound and
    on the cells without surrogate faces relative to their own values."""
    O = OracleProblem.from_workload(_dg(p)[0])
    X = np.sin(np.arange(5 * p + 1) * 0.37 + 0.2)      # by lattice index: traces equal bitwise
    lat = p * O.mesh.cells[:, None, :] + local.tensor_index(p + 1, 3)
    x = np.empty(O.n_dofs)
    x[O.dofmap] = X[lat[..., 0]] + 0.5 * X[lat[..., 1]] * X[lat[..., 2]]
    ref, rows = O.apply(x), _inner_cells(O)
    xd = torch.from_numpy(x).cuda()
    for pen in PENALTIES:
        y = _dg(p, pen)[1].apply_f64(xd).cpu().numpy()
        assert np.abs(y - ref).max() <= 1e-12 * np.abs(ref).max(), pen
        assert np.abs(y - ref)[rows].max() <= 1e-12 * np.abs(ref[rows]).max(), pen


@pytest.mark.parametrize("p", range(1, 7))
def test_dg_penalty_on_jumps(p):
    """Random data against the oracle; a node inside a cell does not see the
    penalty (its test function vanishes on the faces): to the same bound
    relative to such nodes' own values."""
    O1 = OracleProblem.from_workload(_dg(p)[0])
    x = S.random_vector(5, O1.n_dofs, "uniform")
    xd = torch.from_numpy(x).cuda()
    ref1 = O1.apply(x)
    mi = local.tensor_index(p + 1, 3)
    inside = O1.dofmap[:, np.all((mi > 0) & (mi < p), axis=1)].ravel()
    for pen in PENALTIES:
        w, P = _dg(p, pen)
        y = P.apply_f64(xd).cpu().numpy()
        ref = OracleProblem.from_workload(w).apply(x)
        assert np.abs(y - ref).max() <= 1e-12 * np.abs(ref).max(), pen
        if inside.size:
            assert np.abs(y - ref1)[inside].max() <= 1e-12 * np.abs(ref1[inside]).max(), pen


@pytest.mark.parametrize("p", range(1, 7))
def test_dg_penalty_not_finite(p):
    """An infinite penalty (or one that overflows in (p+1)^2 / h) shows on the
    nodes of interior faces; the others are those of pen_interior = 1."""
    w, P = _dg(p)
    O = OracleProblem.from_workload(w)
    xd = torch.from_numpy(S.random_vector(5, O.n_dofs, "uniform")).cuda()
    y1 = P.apply_f64(xd).cpu().numpy()
    mi = local.tensor_index(p + 1, 3)
    seen = np.zeros(O.n_dofs, bool)
    for c1, k, c2 in O.mesh.ifaces:
        seen[O.dofmap[c1][mi[:, k] == p]] = True
        seen[O.dofmap[c2][mi[:, k] == 0]] = True
    for pen in (float("inf"), 1.7e308):
        y = _dg(p, pen)[1].apply_f64(xd).cpu().numpy()
        assert not np.isfinite(y[seen]).any()
        assert np.abs(y - y1)[~seen].max(initial=0.0) <= 1e-12 * np.abs(y1[~seen]).max(initial=1.0)
