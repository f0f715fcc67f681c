"""Boxes of very different strength in one vector, where the contractions of the FP64 form are fixed-point
digits: strong sources at one end of a strip, 1e-10 of them elsewhere.  Potentials and gradients of every unit of
length, also of those whose own sources are the weak ones, against the IEEE form with the double-float form's
bound, 1e-12 (48 bits, about 100 dependent operations)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth, nvec", [(4, 1), (4, 16), (6, 2)])  # M2L; M2L, M2M and L2L by digits
def test_weak_boxes_beside_strong_ones(depth, nvec):
    import torch

    import paper_1902_08250_gb300 as lm

    x, y, q = workloads.uniform_strip(20_000, 0.0, 6.0, -0.95, -0.05, nvec=nvec, seed=depth)
    q = q * np.where(x < 0.1, 1.0, 1e-10)
    xd, yd, qd = (torch.from_numpy(a).cuda() for a in (x, y, q))
    out = []
    for f in (False, True):
        t = lm.build_tree(lm.create_medium(*workloads.MEDIUM_A, p=24, depth=depth, m2l_fp64=f), xd, yd)
        out.append([lm.apply(t, qd), *lm.apply_grad(t, qd)[1:]])
    for a, b in zip(*out):
        for lo in range(6):
            m = torch.from_numpy((x >= lo) & (x < lo + 1)).cuda()
            err = float(torch.linalg.norm((a - b)[:, m]) / torch.linalg.norm(b[:, m]))
            print(f"depth {depth} x {lo}: {err:.1e}")
            assert err <= 1e-12
