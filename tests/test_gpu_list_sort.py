"""The interaction lists around the sizes where their sort changes its form (one
CTA up to 4096 entries, radix passes above): theta = 0 and one particle a leaf
give exactly (leaves)^2 particle-particle entries."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2012_06925_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("points", [1, 2, 3, 8, 31, 63, 64, 65, 91, 128])
@pytest.mark.parametrize("precision", [B.FP32_BULK, B.FP64])
def test_all_pairs_of_leaves(points, precision):
    rng = np.random.default_rng(points)
    cells = rng.permutation(512)[:points]           # distinct cells of an 8^3 lattice
    pts = np.stack([cells // 64, cells // 8 % 8, cells % 8]) / 8 + rng.uniform(0.01, 0.11, (3, points))
    q = rng.uniform(0.5, 1.5, points)
    d = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
    with B.Plan(d, d, torch.from_numpy(q).cuda(), n=2, theta=0.0, N0=1, M0=1, precision=precision) as plan:
        phi = plan.compute().cpu().numpy()
        tree, lists, st = plan.export_tree(0), plan.export_lists(), plan.stats()
    (t, s), rest = lists[0], lists[1:]
    assert st["list_entries"] == [points * points, 0, 0, 0] and all(len(a) == 0 for a, _ in rest)
    assert np.all(np.diff(t) >= 0)                  # by target cluster
    assert np.all(tree["end"][t] - tree["begin"][t] == 1) and np.all(tree["end"][s] - tree["begin"][s] == 1)
    assert len(np.unique(t.astype(np.int64) * len(tree["begin"]) + s)) == points * points
    ref = O.direct_sum(pts, pts, q, O.COULOMB)
    # every term to 1e-6 (the FP32 budget; FP64 far below), all of one sign
    np.testing.assert_allclose(phi, ref, rtol=1e-6 if precision == B.FP32_BULK else 1e-13)
