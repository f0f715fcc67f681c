"""The digit contraction's accumulators at the largest sums that multipoles can ask of them: four boxes
whose 10-bit digits are all largest and match, sign by sign, the digits of a row of their tables (weight
1: first by second and second by first digits).  k1 = k2 = k3, so that the free-space tables set the
scales.  The tables and digits are restated here from the formulas (Rokhlin's translation scaled by
S(n) = (k w / 2)^n / n!).

Tolerance: the multipoles are sums of large, cancelling densities, each product good to 2^-48, a few
units: 2^-46 of the sum of the densities' magnitudes (|G| < 1/16 between the boxes)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K, D, DEPTH, P = 96.0, 1.0, 4, 10
W = D / 2 ** DEPTH
N = np.arange(-P, P + 1)
S = np.array([(K * W / 2) ** abs(n) / math.factorial(abs(n)) for n in N])


def _table(special, dc, dr):
    """Real-block table [2 np][2 np] of the offset (dc, dr) in boxes, rows and columns 2 order + re / im."""
    cx, cy = dc * W, -dr * W
    m = N[None, :] - N[:, None]
    t = 0.25j * special.hankel1(m, K * math.hypot(cx, cy)) * np.exp(1j * m * math.atan2(cy, cx)) * np.outer(S, S)
    a = np.empty((2 * N.size, 2 * N.size))
    a[0::2, 0::2] = a[1::2, 1::2] = t.real
    a[0::2, 1::2], a[1::2, 0::2] = -t.imag, t.imag
    return a


def test_digits_largest_and_aligned():
    special = pytest.importorskip("scipy.special")
    import torch

    import paper_1902_08250_gb300 as lm

    tab = {(c, r): _table(special, c, r) for c in range(-3, 4) for r in range(-3, 4) if max(abs(c), abs(r)) >= 2}
    ex = lambda v: np.floor(np.log2(v))
    mags = np.abs(np.array(list(tab.values())))  # [offset][row][column]; a scale per row: components below 1/2, row sums at most 4
    scale = 2.0 ** -np.maximum(ex(mags.max((0, 2))) + 2, ex(mags.sum(2).max(0)) - 1)[:, None]
    # the first entries of the list of a target box of even row and column: two rows up
    offs = [(2, 2), (1, 2), (0, 2), (-1, 2)]
    d0 = [np.rint(tab[o] * scale * 1024.0) for o in offs]
    d1 = [np.rint((tab[o] * scale * 1024.0 - d) * 1024.0) for o, d in zip(offs, d0)]
    row = int(np.argmax(sum(np.abs(a).sum(1) + np.abs(b).sum(1) for a, b in zip(d0, d1))))
    assert 512 * sum(np.abs(a[row]).sum() + np.abs(b[row]).sum() for a, b in zip(d0, d1)) > 1.5 * 2 ** 24
    ct, rt, rng = 8, 8, np.random.default_rng(1)
    x, y, q = [np.array([1e-3, 1.99])], [np.array([-0.9, -0.9])], [np.zeros(2)]  # two roots of the strip
    for o, a, b in zip(offs, d0, d1):
        sgn = lambda v: np.where(v[row] >= 0, 1.0, -1.0)
        comp = (sgn(b) * 511 + sgn(a) * 0.499) / 1024.0  # first digits 511 beside second ones, second 511 beside first
        u, side = rng.uniform(-0.49, 0.49, 160) * W, np.arange(160) % 4  # points along the box's edges
        px = np.where(side == 0, -0.49 * W, np.where(side == 1, 0.49 * W, u))
        py = np.where(side == 2, -0.49 * W, np.where(side == 3, 0.49 * W, u))
        th = np.arctan2(py, px)
        basis = special.jv(np.abs(N)[:, None], K * np.hypot(px, py)) / S[:, None] * np.where((N < 0) & (N % 2 == 1), -1.0, 1.0)[:, None]
        q.append(np.linalg.lstsq(basis * np.exp(-1j * np.outer(N, th)), comp[0::2] + 1j * comp[1::2], rcond=1e-14)[0])
        x.append((ct - o[0] + 0.5) * W + px)
        y.append(-(rt - o[1] + 0.5) * W + py)
    x.append((ct + rng.uniform(0.02, 0.98, 64)) * W)
    y.append(-(rt + rng.uniform(0.02, 0.98, 64)) * W)
    q.append(np.zeros(64))
    x, y, q = (torch.from_numpy(np.concatenate(v)).cuda() for v in (x, y, q))
    med = dict(p=P, depth=DEPTH)
    t, t64 = (lm.build_tree(lm.create_medium(K, K, K, D, m2l_fp64=f, **med), x, y) for f in (False, True))
    u, ref = (lm.apply(a, q.reshape(1, -1)).cpu().numpy()[0, -64:] for a in (t, t64))
    bound = 2.0 ** -46 * float(q.abs().sum())
    print(f"row {row}: {np.abs(u - ref).max():.1e}, bound {bound:.1e}, potentials {np.abs(ref).max():.1e}")
    assert np.abs(u - ref).max() <= bound
