"""The oscillatory and regularized kernels in packed FP32: pairs at distance 0
(targets among the sources, repeated points, a chunk of one repeated point) are
selected away, odd source counts leave half a pair record empty, and phases
that a float cannot hold stay bounded.  FP32 budget of the parity tests: 1e-6."""
import numpy as np
import pytest

import oracle as O
from paper_2012_06925_gb300 import binding as B
from paper_2012_06925_gb300 import workloads as W
from _gpu_util import rel_l2, run_gpu

pytestmark = pytest.mark.gpu

KERNELS = [(B.OSCILLATORY, float(np.pi)), (B.REG_COULOMB, 0.005)]


@pytest.mark.parametrize("kernel,kappa", KERNELS)
@pytest.mark.parametrize("n", [1, 2, 31, 255, 257, 513])
def test_direct_sum_with_pairs_at_distance_zero(n, kernel, kappa):
    rng = np.random.default_rng(n)
    src = rng.uniform(-1, 1, (3, n))
    src[:, n // 2:] = src[:, :1]                    # the second half is one repeated point
    tgt = np.concatenate([src, rng.uniform(-1, 1, (3, 130))], axis=1)
    q = rng.uniform(0.5, 1.5, n)
    ref = O.direct_sum(tgt, src, q, kernel, kappa)
    phi, plan = run_gpu(tgt, src, q, precision=B.FP32_BULK, kernel=kernel, kappa=kappa, n=2, theta=0.0,
                        N0=100, M0=100)
    plan.close()
    assert rel_l2(ref, phi) <= 1e-6


@pytest.mark.parametrize("kernel,kappa", KERNELS)
def test_tree_with_repeated_points(kernel, kappa):
    tgt, src, q = W.make_problem("sphere", 1800, seed=5)
    pts = np.concatenate([tgt, tgt[:, :700]], axis=1)
    q = np.concatenate([q, q[:700] + 0.25])
    kw = dict(kernel=kernel, kappa=kappa, n=4, theta=0.7, N0=50, M0=50)
    ref = O.bldtt(pts, pts, q, **kw).phi
    phi, plan = run_gpu(pts, pts, q, precision=B.FP32_BULK, **kw)
    plan.close()
    assert rel_l2(ref, phi) <= 1e-6


def test_phases_beyond_float_integers_stay_bounded():
    tgt, src, q = W.make_problem("uniform", 300, 280, seed=9)
    for kappa in (1e6, 1e9, 1e20):
        phi, plan = run_gpu(tgt, src, q, precision=B.FP32_BULK, kernel=B.OSCILLATORY, kappa=kappa, n=2, theta=0.0,
                            N0=100, M0=100)
        plan.close()
        bound = O.direct_sum(tgt, src, np.abs(q), O.COULOMB)
        assert np.all(np.abs(phi) <= 1.001 * bound)
