"""New charges on a kept plan: non-finite ones are refused wherever they stand,
again and again, and a refusal does not stick to the next charges."""
import numpy as np
import pytest
import torch

from paper_2012_06925_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 256, 257, 1000])
def test_refused_then_accepted(n):
    rng = np.random.default_rng(n)
    pts = torch.from_numpy(rng.uniform(-1, 1, (3, n))).cuda()
    q = torch.from_numpy(rng.uniform(-1, 1, n)).cuda()
    kw = dict(n=3, theta=0.7, N0=50, M0=50, precision=B.FP64)
    with B.Plan(pts, pts, q, **kw) as fresh:
        want = fresh.compute()
    with B.Plan(pts, pts, torch.ones_like(q), **kw) as plan:
        for at in {0, n // 2, n - 1}:
            for value in (float("nan"), float("inf"), -float("inf")):
                bad = q.clone()
                bad[at] = value
                with pytest.raises(Exception, match="not finite"):
                    plan.set_charges(bad)
        plan.set_charges(q)
        assert torch.equal(plan.compute(), want)
