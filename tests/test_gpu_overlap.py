"""theta >= 1 lets overlapping clusters approximate each other, so a target (or a
target proxy) can lie at a source proxy: such a pair contributes nothing, as
anywhere.  Sources repeated at a corner of the targets' box: all their proxies
are that point, the targets' corner proxy among the targets' own, and a target
lies there too.  FP32 against the FP64 oracle, budget of the parity tests 1e-6
(2e-6 where every target's potential is one interpolation of the proxies')."""
import numpy as np
import pytest

import oracle as O
from paper_2012_06925_gb300 import binding as B
from _gpu_util import rel_l2, run_gpu

pytestmark = pytest.mark.gpu

KERNELS = [(B.COULOMB, 0.0), (B.YUKAWA, 0.7), (B.OSCILLATORY, 2.0), (B.REG_COULOMB, 0.01), (B.REG_COULOMB, 0.0)]


@pytest.mark.parametrize("kernel,kappa", KERNELS)
@pytest.mark.parametrize("precision", [B.FP64, B.FP32_BULK])
@pytest.mark.parametrize("m", [5, 100, 300])                # PC (targets as particles), CC, CC
def test_target_at_a_source_proxy(m, precision, kernel, kappa):
    rng = np.random.default_rng(m)
    tgt = rng.uniform(-1, 1, (3, m))
    tgt[:, 0] = tgt.max(axis=1)
    src = np.repeat(tgt[:, :1], 120, axis=1)
    q = rng.uniform(0.5, 1.5, 120)
    kw = dict(kernel=kernel, kappa=kappa, n=1, theta=2.5, N0=400, M0=400)
    ref = O.bldtt(tgt, src, q, **kw).phi
    phi, plan = run_gpu(tgt, src, q, precision=precision, **kw)
    pc, cc = len(plan.export_lists()[1][0]), len(plan.export_lists()[3][0])
    plan.close()
    assert (pc if m == 5 else cc) == 1
    assert rel_l2(ref, phi) <= (1e-12 if precision == B.FP64 else 2e-6)
