"""One finest-level operator behind every entry point, after each call that changes it, assembled or not.

newton_slab leaves the Oseen Jacobian of its final iterate on the finest level (in 3D without assembling it); a
re-linearisation brings the option's back, which is assembled or not by the size of the level.  In the FP64 form J x
and the smoother's b - J x run the same operations, so b = J x leaves a residual of exactly zero, and a V-cycle
captured before the change has to take the new operator as an uncaptured one does.
"""
import numpy as np
import pytest

import stg_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NU, TAU = 1e-3, 0.01
# cells, levels, k: the last one has a matrix-free finest level (10000 cells of dG(2) and more)
CASES = [((8, 4), 2, 1), ((4, 2, 2), 2, 0), ((4, 2, 2), 2, 1), ((4, 2, 2), 2, 2), ((24, 24, 20), 3, 2)]


def _spec(cells, levels):
    dim = len(cells)
    faces = (si.FACE_XLO | si.FACE_YLO | si.FACE_YHI) if dim == 2 else si.ALL3 & ~si.FACE_XHI
    hi = tuple(w * c / max(cells) for w, c in zip((1.0, 0.7, 0.45), cells))
    return si.MeshSpec(dim, cells, (0.0,) * dim, hi, levels, faces)


def _vector(spec, k, seed):
    return torch.from_numpy(si.random_vector(si.n_dofs(spec.dim, spec.n, k), seed)).cuda()


@pytest.mark.parametrize("cells,levels,k", CASES)
def test_smoother_and_vcycle_follow_the_newton_iterate(cells, levels, k):
    from paper_2210_02690_gb300 import Solver
    spec = _spec(cells, levels)
    w = torch.from_numpy(np.ascontiguousarray(si.fourier_w(spec, k)).ravel()).cuda()
    captured, plain = (Solver(spec, k, NU, TAU, w, nu1=1, nu2=1, use_graph=g, gmres_restart=1) for g in (1, 0))
    X0, x, b = (_vector(spec, k, seed) for seed in (1, 2, 3))
    first = captured.vcycle(b)
    for change in (lambda s: s.newton_slab(X0, maxit=0), lambda s: s.update_linearisation(w)):
        change(captured)
        change(plain)
        r = captured.level_residual(levels - 1, captured.apply_jacobian(x), x)
        assert torch.count_nonzero(r) == 0
        assert torch.equal(captured.vcycle(b), plain.vcycle(b))
    assert torch.equal(captured.vcycle(b), first)
    captured.close()
    plain.close()


@pytest.mark.parametrize("cells,levels,k", CASES)
def test_newton_jacobian_is_the_derivative_of_the_oseen_form(cells, levels, k):
    """X -> J_Oseen(v(X)) X is quadratic, so its central difference is its derivative, the Newton Jacobian at v(X): the
    assembled (or, on the largest level, matrix-free) one against the matrix-free Oseen form of the iterates."""
    from paper_2210_02690_gb300 import Solver
    spec = _spec(cells, levels)
    X, x = _vector(spec, k, 4), _vector(spec, k, 5)
    R = spec.dim * int(np.prod([2 * c + 1 for c in cells]))
    w = X.view(k + 1, -1)[:, :R].reshape(-1).contiguous()
    s = Solver(spec, k, NU, TAU, w, vcycle_prec="f32", factor_prec="f32", gmres_restart=1)
    jx = s.apply_jacobian(x)
    y = []
    for sign in (1.0, -1.0):
        s.newton_slab(X + sign * x, maxit=0)
        y.append(s.apply_jacobian(X + sign * x))
    s.close()
    error = torch.linalg.norm(jx - 0.5 * (y[0] - y[1]))
    assert error <= 1e-13 * (torch.linalg.norm(y[0]) + torch.linalg.norm(y[1]))
