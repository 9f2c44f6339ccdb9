"""3D cells with a different width in every direction, against the oracle.

Every scale factor of the 3D kernels (1D Jacobians, penalties, face weights) has one value per direction; on cubes
of cells an exchanged one would not show.
"""
import numpy as np
import pytest

import oracle
import stg_inputs as si
from oracle import vanka

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NU, TAU = 1e-3, 0.01
EPS = {"f64": np.finfo(np.float64).eps, "f32": np.finfo(np.float32).eps}
SPEC = si.MeshSpec(3, (4, 2, 2), (0.0,) * 3, (1.0, 0.35, 0.225), 2, si.ALL3 & ~si.FACE_XHI)


@pytest.mark.parametrize("form", ["f64", "f32"])
@pytest.mark.parametrize("k,newton", [(0, False), (0, True), (1, True), (2, True)])
def test_operator_inverses_and_vcycle(k, newton, form):
    """J x within the forward-error bound of the other operator tests; local inverses within 50 cond eps of their
    form; V-cycles at the bars of the forms, 1e-10 and 1e-4."""
    from paper_2210_02690_gb300 import Solver
    w = si.fourier_w(SPEC, k) * (1.0 + 0.1 * np.arange(k + 1))[:, None]
    s = Solver(SPEC, k, NU, TAU, torch.from_numpy(np.ascontiguousarray(w).ravel()).cuda(),
               linearisation="newton" if newton else "oseen", nu1=2, nu2=2, vcycle_prec=form, factor_prec=form)
    ref = oracle.Hierarchy(SPEC, k, NU, TAU, w, newton=newton, nu1=2, nu2=2)
    for level, lev in enumerate(ref.levels):
        x = si.random_vector(lev.N, 21 + level)
        y, exact = s.apply_jacobian(torch.from_numpy(x).cuda(), level=level).cpu().numpy(), ref.J[level] @ x
        assert np.linalg.norm(y - exact) <= 64 * EPS["f64"] * np.linalg.norm(abs(ref.J[level]) @ np.abs(x))
    local = vanka.local_matrices(ref.J[1], ref.levels[1])
    for cell in range(ref.levels[1].n_cells):
        inv, err = ref.jinv[1][cell], np.linalg.norm(s.local_inverse(1, cell) - ref.jinv[1][cell])
        assert err <= 50 * np.linalg.cond(local[cell]) * EPS[form] * np.linalg.norm(inv)
    b = ref.apply(si.reference_solution(SPEC, k, seed=5))
    v, exact = s.vcycle(torch.from_numpy(b).cuda()).cpu().numpy(), ref.vcycle(b)
    assert np.linalg.norm(v - exact) <= (1e-10 if form == "f64" else 1e-4) * np.linalg.norm(exact)
    s.close()
