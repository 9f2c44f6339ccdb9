"""The patch kernel that a level starts with goes by the patches of one launch: all of a level's for the averaged
smoother, a colour's for the coloured one.

A sweep with the default variant is the sweep of the warp-per-patch form up to the order of its sums.
"""
import numpy as np
import pytest

import stg_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FEW_COLUMNS, WARP, STAGED, TWO_ROWS = 0, 3, 11, 15
# form, k, finest cells, smoother, default of the finest level
CASES = [("f64", 2, (32, 32), "coloured", STAGED), ("f64", 2, (32, 32), "averaged", STAGED),
         ("f64", 2, (64, 64), "averaged", WARP), ("f64", 2, (64, 64), "coloured", STAGED),
         ("f64", 2, (64, 32), "averaged", STAGED), ("f64", 2, (66, 32), "averaged", WARP),
         ("f64", 4, (16, 16), "coloured", STAGED), ("f64", 1, (64, 64), "averaged", STAGED),
         ("bf16", 1, (32, 16), "averaged", STAGED), ("bf16", 1, (32, 18), "averaged", TWO_ROWS),
         ("bf16", 1, (32, 18), "coloured", STAGED), ("f32", 1, (16, 16), "coloured", STAGED),
         ("f64", 2, (4, 4, 4), "coloured", FEW_COLUMNS), ("f64", 2, (4, 4, 4), "averaged", FEW_COLUMNS),
         ("f64", 1, (4, 4, 4), "coloured", WARP), ("f32", 2, (4, 4, 4), "coloured", WARP)]


@pytest.mark.parametrize("form,k,cells,smoother,variant", CASES)
def test_default_variant(form, k, cells, smoother, variant):
    from paper_2210_02690_gb300 import Solver
    dim = len(cells)
    spec = si.MeshSpec(dim, cells, (0.0,) * dim, tuple(c / max(cells) for c in cells), 2,
                       (si.ALL2 if dim == 2 else si.ALL3) & ~si.FACE_XHI)
    w = torch.from_numpy(np.ascontiguousarray(si.fourier_w(spec, k)).ravel()).cuda()
    s = Solver(spec, k, 1e-3, 0.01, w, smoother=smoother, gmres_restart=1, factor_prec=form,
               vcycle_prec="f64" if form == "f64" else "f32")
    assert s.colour_variants() == [variant]
    b, x = (torch.from_numpy(si.random_vector(si.n_dofs(dim, cells, k), seed)).cuda() for seed in (1, 2))
    y = s.smooth(1, 2, b, x)
    s.set_colour_variants([4])
    ref = s.smooth(1, 2, b, x)
    assert torch.linalg.norm(y - ref) <= (1e-12 if form == "f64" else 1e-4) * torch.linalg.norm(ref)
    s.autotune()   # times the coloured form's own kernels, and leaves the smoother's results alone
    again = s.smooth(1, 2, b, x)
    assert torch.linalg.norm(again - ref) <= (1e-12 if form == "f64" else 1e-4) * torch.linalg.norm(ref)
    s.close()
