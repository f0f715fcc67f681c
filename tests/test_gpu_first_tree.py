"""Applies in a process whose first tree they are: a kernel's dynamic shared-memory limit belongs to
the process, so a launch that needs it raised must not count on a tree built earlier."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import torch, workloads
import paper_1902_08250_gb300 as lm
x, y, q = (torch.from_numpy(a).cuda() for a in workloads.uniform_strip(600, 0.0, 2.0, -0.99, -1e-4, nvec=16, seed=3))
u = [lm.apply(lm.build_tree(lm.create_medium(*{med}, p=20, adaptive={ad}, leaf_target=16, m2l_fp64=f, **{opt}), x, y), q)
     for f in (False, True)]
assert float(torch.linalg.norm(u[0] - u[1]) / torch.linalg.norm(u[1])) <= 1e-12
"""


# segments of 80 nodes (40960 bytes of coefficients at 16 vectors), of 77, 78 and 81, and a short one
@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("med, opt", [((1.0, 1.5, 1.2, 1.0), {}), ((1.0, 1.5, 1.5, 1.0), {"seg_order": 16}),
                                      ((1.0, 2.5, 1.2, 1.0), {"seg_order": 11}), ((1.0, 2.2, 1.2, 1.0), {"seg_order": 13}),
                                      ((1.0, 4.0, 1.0, 1.0), {"seg_order": 9}), ((0.4, 0.6, 0.5, 1.0), {})])
def test_first_fp64_apply_of_16_vectors(adaptive, med, opt):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE.format(med=med, ad=adaptive, opt=opt)], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
