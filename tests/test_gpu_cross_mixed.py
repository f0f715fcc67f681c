"""Arithmetic of the mixed cross-layer operator: FP32 L2T values, near kernel values rounded to
FP32, FP32 multiply-adds.  Its results are FP32 numbers (cross_apply returns them as complex128),
and a vector's bits do not depend on the vectors applied with it."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("band", [(0.05, 0.95), (1e-5, 0.02)])  # few near pairs; nearly all of the sum is near
@pytest.mark.parametrize("nvec", [1, 3, 16, 17])
def test_mixed_results_are_fp32(band, nvec):
    import torch

    import paper_1902_08250_gb300 as lm

    rng = np.random.default_rng(nvec)
    pts = [torch.from_numpy(a).cuda() for a in (rng.uniform(0, 3, 401), rng.uniform(*band, 401),
                                                rng.uniform(0, 3, 333), -rng.uniform(*band, 333))]
    q = torch.from_numpy(rng.standard_normal((nvec, 401)) + 1j * rng.standard_normal((nvec, 401))).cuda()
    c, c64 = (lm.build_cross(lm.create_medium(*workloads.MEDIUM_A, p=p, depth=3, precision=pr), *pts)
              for p, pr in ((14, "mixed"), (22, "fp64")))
    u = c.apply(q)
    assert torch.equal(u, u.to(torch.complex64).to(torch.complex128))
    assert torch.equal(u[-1:], c.apply(q[-1:].contiguous()))
    ref = c64.apply(q)
    assert float(torch.linalg.norm(u - ref) / torch.linalg.norm(ref)) <= 1e-6  # the mixed form's bound
