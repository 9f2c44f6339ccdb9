"""Kernels chosen by size, at the edges of their ranges.

* Coarse blocks inverted by panels: 257 to 511 rows (FP32: step by step), 512 to 1024 (an odd and an even number of
  32-wide panels), above 1024 (16-wide panels, four rows a thread), and the same blocks in FP64, through the coarse
  solve.
* The matrix-free residual and FP64 operator (3D; order 4 in FP32): cell columns that fill the 31 owned lanes of a
  row, one less and one more, cell counts that are and are not multiples of 32, with and without Newton's term.
* Bases of up to 4, up to 8 and more vectors in the orthogonalisation.
"""
import numpy as np
import pytest

import stg_inputs as si
from oracle import assemble, mesh, newton

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

OUT2 = si.FACE_XLO | si.FACE_YLO | si.FACE_YHI
OUT3 = si.ALL3 & ~si.FACE_XHI
NU, TAU = 1e-3, 0.01
EPS = np.finfo(float).eps


def _spec(cells, levels, order=2):
    hi = tuple(c / max(cells) for c in cells)
    return si.MeshSpec(len(cells), cells, (0.0,) * len(cells), hi, levels, OUT2 if len(cells) == 2 else OUT3, (), order)


def _w(spec, k):
    """A smooth w that differs from Radau node to Radau node."""
    w = si.fourier_w(spec, k) * (1.0 + 0.1 * np.arange(k + 1))[:, None]
    return w


def _solver(spec, k, w, newton=True, **opt):
    from paper_2210_02690_gb300 import Solver
    return Solver(spec, k, NU, TAU, torch.from_numpy(np.ascontiguousarray(w).ravel()).cuda(),
                  linearisation="newton" if newton else "oseen", nu1=2, nu2=2, **opt)


def _operator(spec, level, k, w, newton):
    lev = mesh.Level(spec, level, k)
    return lev, assemble.jacobian(lev, w, NU, TAU, newton).tocsr()


# coarsest cells, k: rows of an interior block (r - 1) pn NV + cells NP - nt
BLOCKS = [((2, 16), 2), ((2, 16), 3), ((2, 15), 4), ((2, 16), 4), ((2, 5, 5), 1), ((2, 5, 5), 2)]  # 339 452 530 565 924 1386


@pytest.mark.parametrize("form", ["f32", "f64"])
@pytest.mark.parametrize("cells,k", BLOCKS)
def test_coarse_solve_at_panel_sizes(cells, k, form):
    """Residual of J_0 x = b with the oracle's J_0: an LU-like 1e-12 in FP64 (one refinement), 1e-5 for FP32 factors
    (at most 1e-3 unrefined, a factor of 100 for the refinement step)."""
    spec = _spec(tuple(2 * c for c in cells), 2)
    w = _w(spec, k)
    s = _solver(spec, k, w, vcycle_prec=form, factor_prec=form)
    lev0 = mesh.Level(spec, 0, k)
    fine = mesh.Level(spec, 1, k)
    from oracle import multigrid
    _, J = _operator(spec, 0, k, multigrid.inject_w(w, fine, lev0), True)
    b = J @ si.random_vector(lev0.N, 5)
    x = s.coarse_solve(torch.from_numpy(b).cuda()).cpu().numpy()
    assert np.linalg.norm(b - J @ x) <= (1e-12 if form == "f64" else 1e-5) * np.linalg.norm(b)
    s.close()


MF_CASES = [((60, 4), 0, 4), ((62, 2), 1, 4), ((64, 6), 2, 4),
            ((4, 2, 6), 0, 2), ((8, 4, 2), 1, 2), ((34, 2, 2), 1, 2), ((4, 4, 2), 2, 2)]


@pytest.mark.parametrize("newton_term", [True, False])
@pytest.mark.parametrize("cells,k,order", MF_CASES)
def test_matrix_free_residual(cells, k, order, newton_term):
    """Two FP32 sweeps from a given x against the FP64 form's (its own operator and factors): 1e-4, the bar of
    the FP32 form's V-cycle."""
    spec = _spec(cells, 2, order)
    w = _w(spec, k)
    s32 = _solver(spec, k, w, newton_term, vcycle_prec="f32", factor_prec="f32")
    s64 = _solver(spec, k, w, newton_term)
    n = si.n_dofs(spec.dim, spec.n, k, order)
    b, x = (torch.from_numpy(si.random_vector(n, seed)).cuda() for seed in (3, 4))
    y32, y64 = s32.smooth(1, 2, b, x), s64.smooth(1, 2, b, x)
    assert torch.linalg.norm(y32 - y64) <= 1e-4 * torch.linalg.norm(y64)
    s32.close()
    s64.close()


@pytest.mark.parametrize("newton_term", [True, False])
@pytest.mark.parametrize("cells,k", [(c, k) for c, k, o in MF_CASES if o == 2])
def test_matrix_free_operator(cells, k, newton_term):
    """J x in 3D against the oracle's assembled J: the forward-error bound of the other operator tests."""
    spec = _spec(cells, 2)
    w = _w(spec, k)
    s = _solver(spec, k, w, newton_term)
    lev, J = _operator(spec, 1, k, w, newton_term)
    x = si.random_vector(lev.N, 6)
    y, ref = s.apply_jacobian(torch.from_numpy(x).cuda()).cpu().numpy(), J @ x
    assert np.linalg.norm(y - ref) <= 64 * EPS * np.linalg.norm(abs(J) @ np.abs(x))
    s.close()


def test_newton_residual_and_operator_in_3d():
    """newton_slab without a step: the residual at X0 is the oracle's, and the finest operator is then the Oseen
    Jacobian at X0; a re-linearisation brings Newton's back."""
    spec, k = _spec((4, 2, 2), 2), 1
    w = _w(spec, k)
    s = _solver(spec, k, w)
    lev = mesh.Level(spec, 1, k)
    X0 = si.random_vector(lev.N, 8)
    v0 = si.random_vector(lev.R, 9)
    b = newton.rhs_nodal(lev, None, None, v0, NU, TAU)
    ref = np.linalg.norm(newton.residual(lev, X0, b, NU, TAU))
    _, steps, _, res, _ = s.newton_slab(torch.from_numpy(X0).cuda(), v_prev=torch.from_numpy(v0).cuda(), maxit=0)
    assert steps == 0 and abs(res - ref) <= 1e-12 * ref
    vel = X0.reshape(k + 1, -1)[:, :lev.R]
    x = si.random_vector(lev.N, 10)
    for wj, newton_term in ((vel, False), (w, True)):
        if newton_term:
            s.update_linearisation(torch.from_numpy(np.ascontiguousarray(w).ravel()).cuda())
        _, J = _operator(spec, 1, k, wj, newton_term)
        y = s.apply_jacobian(torch.from_numpy(x).cuda()).cpu().numpy()
        assert np.linalg.norm(y - J @ x) <= 64 * EPS * np.linalg.norm(abs(J) @ np.abs(x))
    s.close()


@pytest.mark.parametrize("iters", [3, 7, 12])
def test_orthogonalisation_of_short_and_long_bases(iters):
    """FGMRES stopped after `iters` steps: the residual norm of the Arnoldi relation is the true one to 1e-10, which
    an orthonormal basis gives for the fused passes (up to 8 vectors) and the separate ones alike."""
    spec, k = _spec((16, 8), 3), 1
    s = _solver(spec, k, _w(spec, k), gmres_maxit=iters, gmres_rtol=1e-30, omega=0.3)
    n = si.n_dofs(2, spec.n, k)
    b = torch.from_numpy(si.random_vector(n, 12)).cuda()
    x, its, rel, ok = s.gmres_solve(b)
    assert its == iters and not ok
    true = float(torch.linalg.norm(b - s.apply_jacobian(x)) / torch.linalg.norm(b))
    assert abs(rel - true) <= 1e-10 * true
    prev = _solver(spec, k, _w(spec, k), gmres_maxit=iters - 1, gmres_rtol=1e-30, omega=0.3)
    assert rel <= prev.gmres_solve(b)[2] * (1 + 1e-10)   # the residual of a growing basis does not grow
    s.close()
    prev.close()
