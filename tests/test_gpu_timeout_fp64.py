"""Failure path of the FP64 form's tensor-core M2L (no GPU fault is provoked): with the MMA issuer's
first operand wait limited to zero polls every CTA gives up, lets its copies land, frees its tensor
memory and returns; the applies until lm_sync_status are invalid, the next one is right again."""
import pytest

import workloads

pytestmark = pytest.mark.gpu

LM_ETIMEOUT = 4


@pytest.mark.parametrize("n, depth", [(3001, 4), (9001, 6)])  # M2L alone; M2L, M2M and L2L by digits
@pytest.mark.parametrize("nvec", [1, 16])
def test_fp64_wait_timeout_is_reported_and_recovers(n, depth, nvec):
    import torch

    import paper_1902_08250_gb300 as lm

    x, y, q = (torch.from_numpy(a).cuda() for a in workloads.uniform_strip(n, 0.0, 2.9, -0.99, -0.01, nvec=nvec, seed=4))
    t = lm.build_tree(lm.create_medium(*workloads.MEDIUM_A, p=20, depth=depth), x, y)
    ref = lm.apply(t, q)
    lm.sync_status(t)
    lm.set_poll_limit(t, 0)
    lm.apply(t, q)
    lm.apply(t, q)  # the flag stands: this one is invalid too
    with pytest.raises(lm.LMError) as e:
        lm.sync_status(t)
    assert e.value.status == LM_ETIMEOUT and "tensor-core kernel" in str(e.value)
    u = lm.apply(t, q)
    lm.sync_status(t)
    assert torch.equal(u, ref)
