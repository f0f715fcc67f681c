"""Vectors of very different size in one call of the FP64 form: each keeps its own exponent, so its
result has the accuracy and the bits that it has alone (the double-float form's bounds: 1e-12, 1e-11
for the gradient)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

A = workloads.MEDIUM_A
TREES = {
    # name: (n, x_hi, y band, options)
    "small": (700, 2.0, (-0.99, -1e-4), dict(p=20)),
    "digits": (9001, 4.9, (-0.99, -0.01), dict(p=20, depth=6)),  # M2L, M2M and L2L on the tensor cores
    "adaptive": (1500, 2.0, (-0.05, -1e-6), dict(p=20, adaptive=True, leaf_target=16)),
}


def _check(us, ref, alone, s, tol):
    s = s.reshape(-1, 1)
    us, ref = us / s, ref / s
    for v in range(len(s)):
        assert np.linalg.norm(us[v] - ref[v]) <= tol * np.linalg.norm(ref[v]), v
    assert np.array_equal(us[-1], alone[0] / s[-1])


@pytest.mark.parametrize("name", list(TREES))
@pytest.mark.parametrize("nvec", [2, 3, 16])
def test_small_vectors_beside_large_ones(name, nvec):
    import torch

    import paper_1902_08250_gb300 as lm

    n, x_hi, band, opt = TREES[name]
    x, y, q = workloads.uniform_strip(n, 0.0, x_hi, *band, nvec=nvec, seed=nvec)
    s = 10.0 ** np.linspace(0.0, -300.0, nvec)
    s[0] = 1e30
    x, y, q = (torch.from_numpy(a).cuda() for a in (x, y, q * s[:, None]))
    t, t64 = (lm.build_tree(lm.create_medium(*A, m2l_fp64=f, **opt), x, y) for f in (False, True))
    one = q[-1:].contiguous()
    _check(*(a.cpu().numpy() for a in (lm.apply(t, q), lm.apply(t64, q), lm.apply(t, one))), s, 1e-12)
    for a in zip(lm.apply_grad(t, q), lm.apply_grad(t64, q), lm.apply_grad(t, one)):
        _check(*(b.cpu().numpy() for b in a), s, 1e-11)


@pytest.mark.parametrize("nvec", [2, 3, 16])
def test_small_vectors_beside_large_ones_cross(nvec):
    import torch

    import paper_1902_08250_gb300 as lm

    rng = np.random.default_rng(nvec)
    pts = [torch.from_numpy(a).cuda() for a in (rng.uniform(0, 3, 400), rng.uniform(1e-4, 0.9, 400),
                                                rng.uniform(0, 3, 500), -rng.uniform(1e-4, 0.9, 500))]
    s = 10.0 ** np.linspace(0.0, -300.0, nvec)
    q = torch.from_numpy((rng.standard_normal((nvec, 400)) + 1j * rng.standard_normal((nvec, 400))) * s[:, None]).cuda()
    c, c64 = (lm.build_cross(lm.create_medium(*A, p=22, depth=3, m2l_fp64=f), *pts) for f in (False, True))
    _check(*(a.cpu().numpy() for a in (c.apply(q), c64.apply(q), c.apply(q[-1:].contiguous()))), s, 1e-12)
