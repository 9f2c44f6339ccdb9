"""Rounding error of the FP32 V-cycle's residual, row type by row type.

The residual may be computed without a matrix, but no less accurately than from the operator's entries, integrated
in 64 bits and rounded once to FP32: that product is formed here in numpy, one FP32 multiply-add at a time, and the
root mean square of |error| / (|J| |x|) over the velocity rows and over the pressure rows is the bar (5% for
another order of the sums).  The cells have a different width in every direction, so that an exchanged one in any
scale factor shows as an error of order 1.
"""
import numpy as np
import pytest

import stg_inputs as si
from oracle import assemble, mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NU, TAU = 1e-3, 0.01
OUT2 = si.FACE_XLO | si.FACE_YLO | si.FACE_YHI
OUT3 = si.ALL3 & ~si.FACE_XHI
WIDTHS = (1.0, 0.7, 0.45)


def _spec(cells, order):
    hi = tuple(w * c / max(cells) for w, c in zip(WIDTHS, cells))
    return si.MeshSpec(len(cells), cells, (0.0,) * len(cells), hi, 2, OUT2 if len(cells) == 2 else OUT3, (), order)


def _product_fp32(J, x):
    """J x with the entries of J rounded to FP32 and FP32 fused multiply-adds along each row."""
    data, xf = J.data.astype(np.float32).astype(np.float64), x.astype(np.float32).astype(np.float64)
    y, length = np.zeros(J.shape[0], np.float32), np.diff(J.indptr)
    for t in range(length.max()):
        rows = np.nonzero(length > t)[0]
        at = J.indptr[rows] + t
        y[rows] = (y[rows] + data[at] * xf[J.indices[at]]).astype(np.float32)
    return y.astype(np.float64)


CASES = [((16, 8), k, 4) for k in (0, 1, 2)] + [((6, 4, 8), k, 2) for k in (0, 1, 2)] + [((12, 6), 1, 2)]


@pytest.mark.parametrize("newton_term", [True, False])
@pytest.mark.parametrize("cells,k,order", CASES)
def test_residual_as_accurate_as_rounded_entries(cells, k, order, newton_term):
    from paper_2210_02690_gb300 import Solver
    spec = _spec(cells, order)
    w = si.fourier_w(spec, k) * (1.0 + 0.1 * np.arange(k + 1))[:, None]
    s = Solver(spec, k, NU, TAU, torch.from_numpy(np.ascontiguousarray(w).ravel()).cuda(),
               linearisation="newton" if newton_term else "oseen", vcycle_prec="f32", factor_prec="f32")
    lev = mesh.Level(spec, 1, k)
    J = assemble.jacobian(lev, w, NU, TAU, newton_term).tocsr()
    x = si.random_vector(lev.N, 4).astype(np.float32).astype(np.float64)
    b = torch.zeros(lev.N, dtype=torch.float64, device="cuda")
    y = -s.level_residual(1, b, torch.from_numpy(x).cuda()).cpu().numpy()
    s.close()
    exact, size = J @ x, abs(J) @ np.abs(x)

    def error(v, part):
        e = (np.abs(v - exact) / size).reshape(k + 1, -1)[:, part]
        return np.sqrt(np.mean(e * e))

    bar = _product_fp32(J, x)
    for part in (slice(0, lev.R), slice(lev.R, None)):
        assert error(y, part) <= 1.05 * error(bar, part)
