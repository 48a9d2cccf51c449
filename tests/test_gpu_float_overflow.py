"""Charges that a float cannot hold (finite in double, so a plan takes them) are
infinite in the FP32 kernels: every target but those at the charge's own point
gets an infinity, and those get the sum over the others, since a pair at distance
0 contributes nothing."""
import numpy as np
import pytest

import oracle as O
from paper_2012_06925_gb300 import binding as B
from _gpu_util import rel_l2, run_gpu

pytestmark = pytest.mark.gpu

KERNELS = [(B.COULOMB, 0.0), (B.YUKAWA, 0.7), (B.OSCILLATORY, 2.0), (B.REG_COULOMB, 0.005), (B.TEST_POLY, 0.0)]


@pytest.mark.parametrize("kernel,kappa", KERNELS)
@pytest.mark.parametrize("n,leaf", [(1, 10), (40, 100), (700, 100), (700, 1000)])
def test_own_target_of_a_charge_beyond_float(n, leaf, kernel, kappa):
    rng = np.random.default_rng(n + leaf)
    pts = rng.uniform(-1, 1, (3, n))
    q = rng.uniform(0.5, 1.5, n)
    at = n // 3
    q[at] = 1e39
    if n > 1:
        pts[:, at + 1] = pts[:, at]               # another target at the same point
    phi, plan = run_gpu(pts, pts, q, precision=B.FP32_BULK, kernel=kernel, kappa=kappa, n=2, theta=0.0, N0=leaf,
                        M0=leaf)
    plan.close()
    own = [at, at + 1] if n > 1 else [at]
    assert not np.any(np.isfinite(np.delete(phi, own)))
    rest = np.delete(np.arange(n), at)
    want = O.direct_sum(pts[:, own], pts[:, rest], q[rest], kernel, kappa)
    assert rel_l2(want, phi[own]) <= 1e-6
