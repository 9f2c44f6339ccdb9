"""One finest-level operator behind every entry point, after each call that changes it.

newton_slab leaves the Oseen Jacobian of its final iterate on the finest level; a re-linearisation brings the
option's back.  In the FP64 form J x and the smoother's b - J x run the same operations, so b = J x leaves a
residual of exactly zero, and a V-cycle captured before the change has to take the new operator as an uncaptured one
does.
"""
import numpy as np
import pytest

import stg_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NU, TAU = 1e-3, 0.01


@pytest.mark.parametrize("cells,k", [((4, 2, 2), 1), ((8, 4), 1)])
def test_smoother_and_vcycle_follow_the_newton_iterate(cells, k):
    from paper_2210_02690_gb300 import Solver
    dim = len(cells)
    faces = (si.FACE_XLO | si.FACE_YLO | si.FACE_YHI) if dim == 2 else si.ALL3 & ~si.FACE_XHI
    spec = si.MeshSpec(dim, cells, (0.0,) * dim, tuple(c / max(cells) for c in cells), 2, faces)
    w = torch.from_numpy(np.ascontiguousarray(si.fourier_w(spec, k)).ravel()).cuda()
    captured, plain = (Solver(spec, k, NU, TAU, w, nu1=2, nu2=2, use_graph=g) for g in (1, 0))
    n = si.n_dofs(dim, spec.n, k)
    X0, x, b = (torch.from_numpy(si.random_vector(n, seed)).cuda() for seed in (1, 2, 3))
    first = captured.vcycle(b)
    for change in (lambda s: s.newton_slab(X0, maxit=0), lambda s: s.update_linearisation(w)):
        change(captured)
        change(plain)
        r = captured.level_residual(1, captured.apply_jacobian(x), x)
        assert torch.count_nonzero(r) == 0
        assert torch.equal(captured.vcycle(b), plain.vcycle(b))
    assert torch.equal(captured.vcycle(b), first)
    captured.close()
    plain.close()
