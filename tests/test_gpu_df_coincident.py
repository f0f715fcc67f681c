"""Two points at the same place: the FP64 form gives them the infinities that the IEEE form gives, and
every other target its value (double-float bounds: 1e-12, 1e-11 for the gradient)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nvec", [1, 3, 16])
@pytest.mark.parametrize("opt", [dict(), dict(adaptive=True, leaf_target=16), dict(depth=0)])
def test_coincident_points(nvec, opt):
    import torch

    import paper_1902_08250_gb300 as lm

    x, y, q = workloads.uniform_strip(300, 0.0, 1.9, -0.9, -0.1, nvec=nvec, seed=3)
    x[7], y[7] = x[3], y[3]
    x, y, q = (torch.from_numpy(a).cuda() for a in (x, y, q))
    t, t64 = (lm.build_tree(lm.create_medium(*workloads.MEDIUM_A, p=20, m2l_fp64=f, **opt), x, y) for f in (False, True))
    for tol, a, b in ((1e-12, lm.apply(t, q), lm.apply(t64, q)), *((1e-11, *g) for g in zip(lm.apply_grad(t, q), lm.apply_grad(t64, q)))):
        a, b = (torch.view_as_real(v).cpu().numpy() for v in (a, b))
        fin = np.isfinite(b)
        assert not fin[:, [3, 7]].any() and fin.sum() == b.size - 4 * nvec
        assert np.array_equal(a[~fin], b[~fin], equal_nan=True)
        assert np.linalg.norm(a[fin] - b[fin]) <= tol * np.linalg.norm(b[fin])
