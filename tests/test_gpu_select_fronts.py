"""The selector inside the traversal on fronts of every size (a warp takes 4 to
32 pairs, four networks at a time): each list entry's class is the one that the
network outputs of bldtt_mlp_forward on bldtt_pair_features decide."""
import numpy as np
import pytest
import torch

from paper_2012_06925_gb300 import binding as B
from paper_2012_06925_gb300 import workloads as W
from _gpu_util import to_dev
from test_gpu_learned import pack, random_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,leaf,degrees", [(90, 40, [4]), (3000, 30, [2, 3, 5]), (40000, 40, [2, 3, 4, 5, 6]),
                                                (60000, 30, [1, 2, 3, 4, 5, 6, 7, 8])])
def test_entries_are_the_networks_decisions(count, leaf, degrees):
    nout = 3 * len(degrees)
    p = random_params(nout, 3 + nout, scale=4.0)
    lo, hi = np.full(6, -100.0, np.float32), np.full(6, 100.0, np.float32)
    t, s, q = W.make_problem("uniform", count, seed=nout)
    sel = B.Selector(degrees, pack(p), lo, hi, log10_budget=-0.5)
    d = to_dev(t)
    with B.Plan.learned(d, d, to_dev(q), sel, theta=0.7, N0=leaf, M0=leaf, precision=B.FP32_BULK) as plan:
        size = np.diff(np.stack([plan.export_tree(0)["begin"], plan.export_tree(0)["end"]]), axis=0)[0].astype(np.int64)
        lists = plan.export_lists()
        pairs = np.concatenate([np.stack([a, b], axis=1) for a, b in lists]).astype(np.int32)
        cls = np.repeat(np.arange(len(lists)), [len(a) for a, _ in lists])
        f = B.pair_features(plan, torch.from_numpy(pairs).cuda())
        y = B.mlp_forward(torch.from_numpy(pack(p)).cuda(), nout, f.float().contiguous()).cpu().numpy()
        known = ~torch.isnan(f[:, 0]).cpu().numpy()
    ct, cs = size[pairs[:, 0]], size[pairs[:, 1]]
    cost = np.stack([c for n in degrees for np_ in [(n + 1) ** 3] for c in (ct * np_, np_ * cs, 0 * ct + np_ * np_)], 1)
    cost = np.where(y <= np.float32(-0.5), cost, np.iinfo(np.int64).max)
    best = np.argmin(cost, axis=1)                  # the first of equal costs
    least = cost[np.arange(len(best)), best]
    want = np.where(known & (least < ct * cs), best + 1, 0)
    assert np.array_equal(cls, want)
    assert count < 100 or len(np.unique(cls)) >= 2  # the smallest problem has no pair worth approximating
