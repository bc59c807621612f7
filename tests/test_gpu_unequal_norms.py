"""GPU test of the FP32 form's reliable updates on the tensor cores (Q = R C^-1 by split
products) for right-hand sides of very different norms."""
import numpy as np
import pytest

import hisq_inputs as hi
from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,N", [((16, 16, 16, 16), 8), ((16, 16, 16, 64), 16)])
def test_iterations_do_not_depend_on_the_norms(dims, N):
    """Scaling the columns of B scales those of every residual block and nothing else, so
    norms from 1 to 1e-12 take the iterations of equal norms (a tenth more or less: FP32
    roundings) and meet tol.  The first size updates from FP64 residuals alone, the second
    from double-float ones first (V_h N >= 2^21)."""
    mass, tol = 0.1, 1e-9
    s, _, _ = gh.make_solver(dims, mass, prec="mixed_f32", seed=61, max_rhs=N, max_iter=2000)
    b = hi.gaussian_sources(dims, N, seed=62)
    iters = []
    for decades in (0, 12):
        scale = 10.0 ** (-decades * np.arange(N) / (N - 1))
        X, info = s.solve(b * scale[:, None, None], tol=tol)
        assert info["status"] == 0 and max(info["true_rel_res"]) <= tol
        assert info["reliable_updates"] >= 3
        iters.append(info["iters"])
    assert abs(iters[1] - iters[0]) <= iters[0] // 10, iters
