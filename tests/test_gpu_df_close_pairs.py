"""Target gradient of close pairs in the FP64 form, beside the IEEE form.  Leaf-relative coordinates are good
to 2^-49 of the leaf, so a pair's offset from them to 2^-48 / s at s leaf widths: 2^-42 from s = 2^-6 on,
below which FP64 offsets are taken.  The kernel's derivative adds as much again (2^-48 an operation).
The errors are measured against the pair's own derivative, 1 / (2 pi s): other sources may cancel it."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opt", [dict(), dict(top_bc="dirichlet", bottom_bc="neumann")])
def test_gradient_of_close_pairs(opt):
    import torch

    import paper_1902_08250_gb300 as lm

    rng = np.random.default_rng(5)
    m = 40  # pairs in one leaf of width 1
    x, y, th = rng.uniform(0.1, 0.9, m), rng.uniform(-0.9, -0.1, m), rng.uniform(0.0, 2 * np.pi, m)
    q = torch.zeros(1, 2 * m, dtype=torch.complex128)
    q[0, :m] = 1.0
    for s in 2.0 ** np.array([-10.5, -9.9, -8.0, -6.1, -5.9, -4.5]):
        xy = [torch.from_numpy(np.concatenate(a)).cuda() for a in ((x, x + s * np.cos(th)), (y, y + s * np.sin(th)))]
        g = [torch.stack(lm.apply_grad(lm.build_tree(lm.create_medium(*workloads.MEDIUM_A, p=20, depth=0, m2l_fp64=f, **opt), *xy),
                                       q.cuda())[1:])[:, 0, m:] for f in (False, True)]
        err = float((g[0] - g[1]).abs().max()) * 2 * np.pi * s
        print(f"s 2^{np.log2(s):.1f}: {err:.1e}")
        assert err <= 2.0 ** -41
