"""The fixed-point FP64 cell term on the GPU: exponent range and non-finite
values (the arithmetic itself: test_fixed_point.py, and every FP64 apply test)."""
import numpy as np
import pytest
import torch

import paper_2507_17053_gb300 as G
import synthetic as S

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
