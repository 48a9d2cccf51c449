"""Executed evaluations of a plan as the header defines them: every 32-target row
group that holds a real target meets every real source; in FP32 the default
layout skips idle groups only where that saves 2 % of the evaluations, in FP64
they are always left out."""
import pytest

from paper_2012_06925_gb300 import binding as B
from paper_2012_06925_gb300 import workloads as W
from _gpu_util import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,rows32,rows64", [(7720, 7680 + 128, 7680 + 64), (7681, 7680 + 128, 7680 + 32),
                                             (40, 64, 64), (256, 256, 256)])
def test_executed_evaluations(m, rows32, rows64):
    n = 300
    tgt, src, q = W.make_problem("uniform", m, n, seed=1, sources_kind="plummer")
    for precision, rows in ((B.FP32_BULK, rows32), (B.FP64, rows64)):
        phi, plan = run_gpu(tgt, src, q, precision=precision, n=2, theta=0.0, N0=10000, M0=10000)
        st = plan.stats()
        plan.close()
        assert st["executed_evaluations"] == rows * n
