"""The image tables' scales at high order and wide boxes (k2 w = 3400 at level 0): finite entries are built."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k2, p", [(3.4, 48), (8.0, 48), (3.4, 24)])
def test_wide_boxes_are_built(k2, p):
    import torch

    import paper_1902_08250_gb300 as lm

    rng = np.random.default_rng(1)
    x, y = (torch.from_numpy(a).cuda() for a in (rng.uniform(1, 999, 40), -rng.uniform(50, 950, 40)))
    t = lm.build_tree(lm.create_medium(1.0, k2, 2.0, 1000.0, p=p, depth=0), x, y)
    assert t.info["n"] == 40
