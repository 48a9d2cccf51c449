"""Work items split over their sources: an item's chunks are summed per
segment whatever tasks the segments are shared out as, so the potentials do
not depend on the split (BLDTT_TASK_CHUNKS, the chunks of a task) bit for bit,
with the default split, one chunk per task, three, and no split at all; and
they match the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2012_06925_gb300 import binding as B
from paper_2012_06925_gb300 import workloads as W
from _gpu_util import rel_l2, run_gpu

pytestmark = pytest.mark.gpu

CASES = [
    # targets, sources, leaf: one chunk per item; tile and chunk remainders; long items (many chunks a segment)
    (200, 256, 300), (257, 4097, 5000), (513, 1100, 400), (3000, 9000, 9000), (6000, 6000, 150),
]


@pytest.mark.parametrize("precision", [B.FP64, B.FP32_BULK])
@pytest.mark.parametrize("m,n,leaf", CASES)
def test_split_does_not_change_the_bits(m, n, leaf, precision, monkeypatch):
    tgt, src, q = W.make_problem("uniform", m, n, seed=m + n, sources_kind="plummer")
    kw = dict(kernel=B.YUKAWA if m % 2 else B.COULOMB, kappa=0.5, n=3, theta=0.7, N0=leaf, M0=leaf)
    out, items = [], []
    for chunks in (None, "1", "3", "1000000"):
        if chunks is None:
            monkeypatch.delenv("BLDTT_TASK_CHUNKS", raising=False)
        else:
            monkeypatch.setenv("BLDTT_TASK_CHUNKS", chunks)
        phi, plan = run_gpu(tgt, src, q, precision=precision, **kw)
        with plan:
            again = plan.compute().cpu().numpy()          # the finished-segment counts were reset
            items.append(plan.stats()["work_items"])
        assert np.array_equal(phi, again)
        out.append(phi)
    for other in out[1:]:
        assert np.array_equal(out[0], other)
    assert items[1] >= items[2] >= items[3]
    if n > 4096:
        assert items[1] > items[3]
    ref = O.bldtt(tgt, src, q, **kw).phi
    assert rel_l2(ref, out[0]) <= (1e-12 if precision == B.FP64 else 1e-6)
