"""GPU parity of the DG apply, the diagonal and the FP32 apply with the oracle."""
import numpy as np
import pytest
import torch

import paper_2507_17053_gb300 as G
import synthetic as S
from oracle.operator import Problem as OracleProblem

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


DG_CASES = [
    S.TORUS_3D_DG_Q3.resized(16),
    S.TORUS_3D_DG_Q3.resized(11),
] + [S._wl(f"dg2d_q{p}", 2, p, 9, S.ball(2, (0.05, -0.03), 0.73), dg=True, seed=3,
           dist="normal") for p in range(1, 7)] \
  + [S._wl(f"dg3d_q{p}", 3, p, 6, S.ball(3, (0.02, 0.01, -0.03), 0.71), dg=True, seed=3,
           dist="normal") for p in range(1, 7)]


@pytest.mark.parametrize("w", DG_CASES, ids=lambda w: w.name)
def test_dg_apply_matches_oracle(w):
    O = OracleProblem.from_workload(w)
    P = G.Problem.from_workload(w)
    assert P.n_dofs == O.n_dofs and P.n_ifaces == len(O.mesh.ifaces)
    x = S.random_vector(w.seed, O.n_dofs, w.dist)
    xd = torch.from_numpy(x).cuda()
    y = P.apply_f64(xd)
    y2 = P.apply_f64(xd)
    assert torch.equal(y, y2)
    assert _rel(y.cpu().numpy(), O.apply(x)) <= TOL


def test_dg_full_size_sampled_rows():
    w = S.TORUS_3D_DG_Q3
    O = OracleProblem.from_workload(w)
    P = G.Problem.from_workload(w)
    x = S.random_vector(w.seed, O.n_dofs, w.dist)
    y = P.apply_f64(torch.from_numpy(x).cuda()).cpu().numpy()
    rng = np.random.default_rng(1)
    rows = rng.choice(O.n_dofs, 20000, replace=False)
    ref = O.apply_rows(x, rows)
    assert np.abs(y[rows] - ref).max() <= TOL * np.abs(ref).max()


DIAG_CASES = [S.DISK_2D_Q2, S.SPHERE_3D_Q4.resized(10), S.ELLIPSOID_3D_Q6.resized(8),
              S.TORUS_3D_DG_Q3.resized(12), DG_CASES[3]]


@pytest.mark.parametrize("w", DIAG_CASES, ids=lambda w: w.name)
def test_diagonal_matches_oracle(w):
    O = OracleProblem.from_workload(w)
    P = G.Problem.from_workload(w)
    d = P.diagonal().cpu().numpy()
    ref = O.diagonal()
    assert _rel(d, ref) <= TOL


F32_CASES = [S.DISK_2D_Q2, S.SPHERE_3D_Q4.resized(12), S.ELLIPSOID_3D_Q6.resized(9),
             S.TORUS_3D_DG_Q3.resized(14)]


@pytest.mark.parametrize("w", F32_CASES, ids=lambda w: w.name)
def test_f32_apply_error_vs_oracle(w):
    """FP32 apply: relative max-norm error against the FP64 oracle is at the
    FP32 rounding level amplified by the extrapolation at shifted points
    (measured on a GB300: 4e-8 .. 1.5e-7 for p = 1..6, 2D and 3D; bound
    5e-7, about 3x the largest)."""
    O = OracleProblem.from_workload(w)
    P = G.Problem.from_workload(w)
    x = S.random_vector(w.seed, O.n_dofs, w.dist)
    y = P.apply_f32(torch.from_numpy(x).float().cuda()).double().cpu().numpy()
    ref = O.apply(x.astype(np.float32).astype(np.float64))
    err = _rel(y, ref)
    print(f"{w.name}: fp32 rel err {err:.3e}")
    assert err <= 5e-7


@pytest.mark.parametrize("w", [w for w in DG_CASES if w.dim == 3], ids=lambda w: w.name)
def test_f32_dg_apply_error_vs_oracle(w):
    """The FP32 line operators of the 3D DG apply, to test_f32_apply_error_vs_oracle's bound."""
    O = OracleProblem.from_workload(w)
    P = G.Problem.from_workload(w)
    x = S.random_vector(w.seed, O.n_dofs, w.dist)
    y = P.apply_f32(torch.from_numpy(x).float().cuda()).double().cpu().numpy()
    ref = O.apply(x.astype(np.float32).astype(np.float64))
    assert _rel(y, ref) <= 5e-7


@pytest.mark.parametrize("cells", [5, 23, 40])
@pytest.mark.parametrize("p", range(1, 7))
def test_register_kernels_equal_chunk_kernels_bitwise(p, cells):
    """FP32 applies by one or n threads per cell (shape 0, at p = 4, 5 from 9 000
    and 16 000 cells on, here 40^3; shape 2 at every size up to p = 4) against
    the chunks without staged runs (shape 3) and, where built, with
    colour-ordered stores: mesh rows of 1 to 33 active cells, so chunks of
    every length and blocks that end anywhere."""
    w = S._wl("ball", 3, p, cells, S.ball(3, (0.02, 0.01, -0.03), 0.81), seed=7)
    P = G.Problem.from_workload(w)
    x = torch.from_numpy(S.random_vector(7, P.n_dofs, "uniform")).float().cuda()
    G.sbm_set_tile_shape(P.handle, 0, 0)
    y = P.apply_f32(x)
    for shape in (3, 2) if p <= 4 else (3,):
        G.sbm_set_tile_shape(P.handle, 0, shape)
        assert torch.equal(P.apply_f32(x), y)
    G.sbm_set_tile_shape(P.handle, 0, 0)
    try:
        G.sbm_set_ordered_stores(P.handle, -1, 1)
    except G.SbmError:
        return
    assert torch.equal(P.apply_f32(x), y)
