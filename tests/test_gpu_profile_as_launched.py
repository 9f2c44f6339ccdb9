"""stg_profile as an ordinary sweep is launched: the sampled V-cycle launches what an unprofiled one does.

One launch per sampled sweep of the averaged smoother, 2^d of the coloured one, over every finest patch once, and
no other kernel count than with profiling off.
"""
import numpy as np
import pytest

import stg_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPEC = si.MeshSpec(2, (32, 16), (0.0, 0.0), (2.2, 0.41), 3, si.FACE_XLO | si.FACE_YLO | si.FACE_YHI)


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("smoother,launches", [("averaged", 1), ("coloured", 4)])
def test_sampled_sweep_is_an_ordinary_one(smoother, launches, use_graph):
    from paper_2210_02690_gb300 import Solver
    w = torch.from_numpy(np.ascontiguousarray(si.channel_w(SPEC, 1)).ravel()).cuda()
    s = Solver(SPEC, 1, 1e-3, 0.01, w, nu1=2, nu2=2, smoother=smoother, use_graph=use_graph, vcycle_prec="f32",
               factor_prec="f32")
    b = s.apply_jacobian(torch.from_numpy(si.reference_solution(SPEC, 1, seed=4)).cuda())

    def vcycle():
        before = s.kernel_launches()
        x = s.vcycle(b)
        return x, s.kernel_launches() - before

    x0, ordinary = vcycle()
    for n in (1, 2):
        s.profile(True, as_launched=True)
        for _ in range(n):
            x, count = vcycle()
            assert count == ordinary and torch.equal(x, x0)
        ms, timed, patches = s.profile_read()
        assert timed == n * launches and patches == n * SPEC.n[0] * SPEC.n[1] and ms > 0.0
    s.profile(False)
    s.close()
