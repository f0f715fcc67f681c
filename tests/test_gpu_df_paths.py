"""The double-float kernels of the FP64 form, the tensor-core M2L by digits and the
few-vector kernels of the mixed form at the sizes where they change path: edges of
their tiles, remainders, the smallest and largest of their ranges.  Each is compared
with the other path of the same tree: the FP64 form against IEEE FP64 (m2l_fp64), the
mixed form against the FP64 form.

Tolerances.  Double-float carries 48 bits; a kernel value or basis entry of about 100
dependent operations is good to 100 * 2^-48 = 4e-13 of the largest term, and the sums
round at 2^-48: 1e-12 relative l2, the bound of the double-float M2L test.  The mixed
form's bound is its own, 1e-6, met from p = 14 on."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for -m gpu tests")
    import paper_1902_08250_gb300 as lm

    return lm


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _tree(lm, med, x, y, **opt):
    import torch

    return lm.build_tree(lm.create_medium(*med, **opt), torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())


def _apply(lm, t, q, fn=None):
    import torch

    return (fn or lm.apply)(t, torch.from_numpy(np.ascontiguousarray(q)).cuda()).cpu().numpy()


A, B = workloads.MEDIUM_A, workloads.MEDIUM_B
NEAR = {
    # name: (medium, n, x_hi, y band, nvec, options)
    "one_point": (A, 1, 1.0, (-0.6, -0.4), 1, dict(p=20)),
    "two_points": (A, 2, 1.0, (-0.6, -0.4), 3, dict(p=20)),
    "one_root": (A, 60, 0.9, (-0.95, -0.05), 2, dict(p=20, depth=0)),           # every pair direct
    "far_series": (B, 200, 1.9, (-0.95, -0.05), 2, dict(p=24, depth=0)),        # k r up to 16: z > 1
    "short_series": (A, 3000, 3.0, (-0.95, -0.05), 5, dict(p=20, depth=4)),     # z <= 1/16
    "leaf_of_17": (A, 17, 0.9, (-0.9, -0.1), 16, dict(p=20, depth=0)),          # one past a pass of targets
    "leaf_of_65": (A, 65, 0.9, (-0.9, -0.1), 8, dict(p=20, depth=0)),           # one past a round of sources
    "wide_pass": (A, 100_000, 4.9, (-0.95, -0.05), 1, dict(p=20, depth=5)),     # 20 points a leaf, passes of 32
    "wide_pass_two": (A, 180_000, 4.9, (-0.95, -0.05), 2, dict(p=20, depth=5)), # 35 points: two passes
    "low_order": (A, 500, 2.0, (-0.9, -0.1), 4, dict(p=1, depth=2)),
    "high_order": (A, 500, 2.0, (-0.9, -0.1), 16, dict(p=48, depth=1)),
    "interface": (A, 1500, 2.0, (-0.02, -1e-7), 11, dict(p=20, depth=3)),
    "adaptive": (A, 1500, 2.0, (-0.02, -1e-7), 3, dict(p=20, adaptive=True, leaf_target=16)),
    "impedance": (A, 900, 2.0, (-0.99, -0.01), 3, dict(p=22, depth=2, top_bc="impedance", top_alpha=0.7,
                                                      bottom_bc="neumann")),
    "walls": (A, 900, 2.0, (-0.99, -0.01), 1, dict(p=22, depth=2, top_bc="dirichlet", bottom_bc="neumann")),
    "dg_dd": (A, 900, 2.0, (-0.9, -0.01), 2, dict(p=22, depth=2, kernel=1)),
}


@pytest.mark.parametrize("name", list(NEAR))
def test_double_float_form_matches_ieee(lm, name):
    med, n, x_hi, band, nvec, opt = NEAR[name]
    x, y, q = workloads.uniform_strip(n, 0.0, x_hi, *band, nvec=nvec, seed=len(name))
    a, b = (_tree(lm, med, x, y, m2l_fp64=f, **opt) for f in (False, True))
    ua, ub = _apply(lm, a, q), _apply(lm, b, q)
    if n == 1:  # the reflected self term alone
        assert abs(ua[0, 0] - ub[0, 0]) <= 1e-12 * abs(ub[0, 0])
        return
    assert _rel(ua, ub) <= 1e-12
    import torch

    qd = torch.from_numpy(q).cuda()
    # the y-derivative divides by the distance of the pair: a factor 10 beside the value's bound
    for ga, gb in zip(lm.apply_grad(a, qd), lm.apply_grad(b, qd)):
        assert _rel(ga.cpu().numpy(), gb.cpu().numpy()) <= 1e-11


def test_close_and_coincident_pairs_take_the_fp64_kernel(lm):
    """Points 1e-4 to 1e-18 apart (FP64 offsets below 2^-10 leaf widths, the FP64 functions below
    2^-45 / k), one source of each group active."""
    import torch

    x = np.concatenate([[0.3], 0.3 + 10.0 ** -np.arange(4.0, 17.0), [1e-18, 3e-18, 0.7]])
    y = np.full(x.size, -0.4)
    q = np.zeros((1, x.size), complex)
    q[0, -2] = q[0, 0] = 1.0
    a, b = (_tree(lm, A, x, y, p=20, depth=0, m2l_fp64=f) for f in (False, True))
    ua, ub = (lm.apply(t, torch.from_numpy(q).cuda()).cpu().numpy() for t in (a, b))
    assert np.all(np.isfinite(ua)) and np.max(np.abs(ua - ub)) <= 1e-12 * np.max(np.abs(ub))


@pytest.mark.parametrize("p", [7, 8, 20, 23, 24, 31, 32])  # 2(2p+1) against 16-wide K steps, 48-wide stages, 128 rows
@pytest.mark.parametrize("nvec", [1, 3, 16])
def test_digit_m2l_orders(lm, p, nvec):
    """Uniform tree with 3072 leaf boxes (3 roots: the last tile of a row is partly filled)."""
    x, y, q = workloads.uniform_strip(9001, 0.0, 2.9, -0.99, -0.01, nvec=nvec, seed=p)
    a, b = (_tree(lm, A, x, y, p=p, depth=5, m2l_fp64=f) for f in (False, True))
    assert _rel(_apply(lm, a, q), _apply(lm, b, q)) <= 1e-12


@pytest.mark.parametrize("nvec", [2, 5, 8, 9])
def test_digit_m2l_vector_forms_and_scales(lm, nvec):
    """Every slot count; vectors of very different size keep their own relative accuracy."""
    x, y, q = workloads.uniform_strip(20_000, 0.0, 4.0, -0.95, -0.05, nvec=nvec, seed=nvec)
    q *= 10.0 ** np.linspace(0.0, -20.0, nvec)[:, None]
    a, b = (_tree(lm, B, x, y, p=20, depth=5, m2l_fp64=f) for f in (False, True))
    ua, ub = _apply(lm, a, q), _apply(lm, b, q)
    for v in range(nvec):
        assert _rel(ua[v], ub[v]) <= 1e-12
    assert np.array_equal(ua[-1], _apply(lm, a, q[-1]))  # alone or among others: the same bits


@pytest.mark.parametrize("p", [7, 20, 24, 32])
@pytest.mark.parametrize("nvec", [1, 3, 8, 16])
def test_digit_shifts(lm, p, nvec):
    """M2M and L2L by digits on two levels (20480 and 5120 boxes, ragged tiles, most leaves empty)."""
    x, y, q = workloads.uniform_strip(9001, 0.0, 4.9, -0.99, -0.01, nvec=nvec, seed=p)
    a, b = (_tree(lm, A, x, y, p=p, depth=6, m2l_fp64=f) for f in (False, True))
    assert _rel(_apply(lm, a, q), _apply(lm, b, q)) <= 1e-12


FEW = {
    "one_point": (A, 1, 1.0, (-0.6, -0.4), dict(p=14)),
    "one_root": (A, 200, 0.9, (-0.95, -0.05), dict(p=16, depth=0)),
    "far_series": (B, 300, 1.9, (-0.95, -0.05), dict(p=24, depth=0)),
    "leaf_of_17": (A, 17, 0.9, (-0.9, -0.1), dict(p=14, depth=0)),
    "short_series": (A, 4000, 3.0, (-0.95, -0.05), dict(p=14, depth=4)),
    "wide_tiles": (A, 30000, 3.0, (-0.95, -0.05), dict(p=14, depth=4)),
    "wide_tiles_full_series": (A, 30000, 9.0, (-0.95, -0.05), dict(p=14, depth=3)),
    "interface": (A, 1500, 2.0, (-0.02, -1e-6), dict(p=14, depth=3)),
    "adaptive": (A, 1500, 2.0, (-0.02, -1e-6), dict(p=14, adaptive=True, leaf_target=16)),
    "adaptive_high": (A, 1500, 2.0, (-0.5, -1e-6), dict(p=24, adaptive=True, leaf_target=16)),
    "impedance": (A, 900, 2.0, (-0.95, -0.05), dict(p=16, depth=2, top_bc="impedance", top_alpha=0.7,
                                                    bottom_bc="neumann")),
}


@pytest.mark.parametrize("name", list(FEW))
@pytest.mark.parametrize("nvec", [1, 2, 3, 4])
def test_few_vector_mixed_kernels(lm, name, nvec):
    med, n, x_hi, band, opt = FEW[name]
    x, y, q = workloads.uniform_strip(n, 0.0, x_hi, *band, nvec=nvec, seed=len(name) + nvec)
    t = _tree(lm, med, x, y, precision="mixed", **opt)
    ref = _apply(lm, _tree(lm, med, x, y, **dict(opt, p=max(24, opt["p"]))), q)
    assert _rel(_apply(lm, t, q.astype(np.complex64)), ref) <= 1e-6


@pytest.mark.parametrize("n, p", [(20_000, 14), (20_000, 24), (250_000, 8)])
def test_adaptive_m2l_by_classes(lm, n, p):
    """One vector (V entries by class; one slice and several) against two (a block per target box)."""
    x, y, q = workloads.uniform_strip(n, 0.0, 9.9, -0.99, -0.01, nvec=2, seed=p)
    q = q.astype(np.complex64)
    t = _tree(lm, A, x, y, precision="mixed", p=p, adaptive=True, leaf_target=16)
    assert _rel(_apply(lm, t, q[:1])[0], _apply(lm, t, q)[0]) <= 1e-6


@pytest.mark.parametrize("n", [1, 40, 270, 1100, 2100, 4000])
@pytest.mark.parametrize("band", [(-0.95, -0.05), (-1.0 + 1e-6, -1e-6)])
def test_tensor_core_leaf_tiles(lm, n, band):
    """32 leaves of 0 to 150 points: target groups of 8, passes of 64, chunks of 64 sources, tails."""
    x, y, q = workloads.uniform_strip(n, 0.0, 1.9, *band, nvec=16, seed=n)
    t = _tree(lm, A, x, y, precision="mixed", p=14, depth=2)
    ref = _apply(lm, _tree(lm, A, x, y, p=24, depth=2), q)
    assert _rel(_apply(lm, t, q.astype(np.complex64)), ref) <= 1e-6


@pytest.mark.parametrize("nvec", [1, 2, 3, 5, 16])
@pytest.mark.parametrize("band", [(0.05, 0.95), (1e-6, 0.02)])
def test_cross_double_float_matches_ieee(lm, nvec, band):
    import torch

    rng = np.random.default_rng(7)
    pts = [torch.from_numpy(a).cuda() for a in (rng.uniform(0, 3, 400), rng.uniform(*band, 400),
                                                rng.uniform(0, 3, 500), -rng.uniform(*band, 500))]
    q = torch.from_numpy(rng.standard_normal((nvec, 400)) + 1j * rng.standard_normal((nvec, 400))).cuda()
    u = [lm.build_cross(lm.create_medium(*A, p=22, depth=3, m2l_fp64=f), *pts).apply(q).cpu().numpy() for f in (False, True)]
    assert _rel(*u) <= 1e-12
