"""Device memory of FP64 trees per point, from two trees of the same boxes: tree-order potentials and
double-float densities of 16 vectors (512 bytes), coordinates, their offsets and heights, permutation (56)."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opt", [dict(depth=4), dict(depth=4, m2l_fp64=True)])
def test_bytes_per_point(opt):
    import torch

    import paper_1902_08250_gb300 as lm

    med = lm.create_medium(*workloads.MEDIUM_A, p=20, **opt)
    used = []
    for n in (100_000, 300_000):
        x, y, q = (torch.from_numpy(a).cuda() for a in workloads.uniform_strip(n, 0.0, 3.0, -0.95, -0.05, nvec=1, seed=1))
        t = lm.build_tree(med, x, y)
        used.append(t.info["device_bytes"])
        assert bool(torch.isfinite(lm.apply(t, q)).all())
    assert (used[1] - used[0]) / 200_000 <= 600
