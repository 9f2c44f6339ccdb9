"""Coarse blocks of every size that the direct solver accepts.

A 2D coarsest mesh of 1 x n cells has one interior block of (k + 1)(7 n + 1) unknowns and two planes of
(k + 1)(4 n + 3): sizes on and beside the lines at which the inversion changes its panels (512, 1024, 2048, 4608,
9216), and the largest that FP32 factors take.  A misplaced row, pivot or panel gives an error of order 1; explicit
inverses of 10^4 rows keep a few digits in FP32, squared by the step of refinement: 1e-3, and 1e-10 in FP64.
"""
import numpy as np
import pytest

import stg_inputs as si
from oracle import assemble, mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NU, TAU = 1e-3, 0.01
FACES = si.FACE_XLO | si.FACE_YLO | si.FACE_YHI


def _spec(n):
    return si.MeshSpec(2, (1, n), (0.0, 0.0), (1.0 / n, 1.0), 1, FACES)


# n, k: interior 505 512 519 1023 1024 1030 2048 2052 4608 4622
SIZES = [(72, 0), (73, 0), (74, 0), (146, 0), (73, 1), (147, 0), (73, 3), (293, 0), (329, 1), (330, 1)]
# 9216 9244 9665
LARGEST = [(329, 3), (330, 3), (276, 4)]


@pytest.mark.parametrize("form,n,k", [("f32", n, k) for n, k in SIZES + LARGEST] + [("f64", n, k) for n, k in SIZES])
def test_coarse_solve_at_every_block_size(form, n, k):
    from paper_2210_02690_gb300 import Solver
    spec = _spec(n)
    w = si.fourier_w(spec, k)
    s = Solver(spec, k, NU, TAU, torch.from_numpy(np.ascontiguousarray(w).ravel()).cuda(), vcycle_prec=form,
               factor_prec=form, gmres_restart=1)
    lev = mesh.Level(spec, 0, k)
    J = assemble.jacobian(lev, w, NU, TAU, True).tocsr()
    b = J @ si.random_vector(lev.N, 7)
    x = s.coarse_solve(torch.from_numpy(b).cuda()).cpu().numpy()
    s.close()
    assert np.linalg.norm(b - J @ x) <= (1e-3 if form == "f32" else 1e-10) * np.linalg.norm(b)


@pytest.mark.parametrize("form,n,k", [("f32", 278, 4), ("f64", 330, 3)])
def test_larger_blocks_are_refused_at_set_up(form, n, k):
    """9735 and 9244 unknowns."""
    from paper_2210_02690_gb300 import Solver, StgError
    spec = _spec(n)
    w = torch.from_numpy(np.ascontiguousarray(si.fourier_w(spec, k)).ravel()).cuda()
    with pytest.raises(StgError) as e:
        Solver(spec, k, NU, TAU, w, vcycle_prec=form, factor_prec=form)
    assert e.value.status == 1 and "coarsest level" in str(e.value)


def test_inversion_scratch_is_paid_for_only_where_it_is_used():
    """FP32 blocks of 253 rows are inverted on chip, blocks of 260 by panels into a second copy that an array of the
    factorisation lends (W); neither size allocates a copy of its blocks.  The memory per unknown of order 2's arrays,
    counted from their sizes, is the bound."""
    from paper_2210_02690_gb300 import Solver
    for ny in (36, 37):
        nx, nsv = 512, 513
        spec = si.MeshSpec(2, (nx, ny), (0.0, 0.0), (float(nx) / ny, 1.0), 1, FACES)
        mI, mV = 7 * ny + 1, 4 * ny + 3
        # A_II, A_IV, A_VI, W, C; D, L, U, GL, GU; per level PL, PR and new L, U of every even plane
        levels = sum(4 * len(range(0, nsv, 2 * s)) for s in (2 ** i for i in range(10)))
        arrays = 4 * (nx * (mI * mI + 6 * mI * mV + 4 * mV * mV) + (5 * nsv + levels) * mV * mV)
        w = torch.from_numpy(np.ascontiguousarray(si.fourier_w(spec, 0)).ravel()).cuda()
        used = []
        for form in ("f32", "f64"):
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            s = Solver(spec, 0, NU, TAU, w, vcycle_prec="f32", factor_prec="f32", coarse_prec=form, gmres_restart=1)
            used.append(free - torch.cuda.mem_get_info()[0])
            s.close()
        # the two forms differ by 4 bytes a value of the arrays, and by the panels (2% here)
        assert used[1] - used[0] <= 1.06 * arrays
