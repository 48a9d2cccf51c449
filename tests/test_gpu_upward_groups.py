"""Proxy charges of every cluster: leaves of one to a few chunks of 64 particles, and inner clusters with the children side by side in eight
groups (levels of few clusters) and in two (levels of more than 2048 / P): the
interpolation reproduces polynomials of degree n, so the moments
sum_k qhat_k s_k^m of a cluster are those of its particles, m <= n."""
import numpy as np
import pytest
import torch

from paper_2012_06925_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,count,leaf", [(1, 40, 3), (3, 3000, 2), (6, 3000, 4), (8, 1200, 5), (11, 700, 40),
                                          (16, 400, 60), (1, 700, 200), (2, 129, 150), (4, 900, 190), (5, 64, 80),
                                          (7, 1500, 260), (8, 700, 128)])
def test_moments_of_every_cluster(n, count, leaf):
    rng = np.random.default_rng(n)
    pts = rng.uniform(-1, 1, (3, count))
    q = rng.uniform(-1, 1, count)
    d = torch.from_numpy(pts).cuda()
    with B.Plan(d, d, torch.from_numpy(q).cuda(), n=n, theta=0.7, N0=leaf, M0=leaf, precision=B.FP64) as plan:
        plan.compute()
        tree = plan.export_tree(1)
        qhat = plan.proxy_charges()
    s = np.cos(np.pi * np.arange(n + 1) / n)
    x, w = pts[:, tree["perm"]], q[tree["perm"]]
    for c, (b, e) in enumerate(zip(tree["begin"], tree["end"])):
        mid, half = (tree["hi"][:, c] + tree["lo"][:, c]) / 2, (tree["hi"][:, c] - tree["lo"][:, c]) / 2
        scale = np.abs(w[b:e]).sum()
        assert abs(qhat[c].sum() - w[b:e].sum()) <= 1e-12 * scale
        for ax in range(3):
            if half[ax] == 0:
                continue
            other = tuple(a for a in range(3) if a != ax)
            u = (x[ax, b:e] - mid[ax]) / half[ax]
            for m in (1, n):
                got = (qhat[c].sum(axis=other) * s ** m).sum()
                # a few hundred roundings, each of up to the Lebesgue constant squared (about 5)
                assert abs(got - (w[b:e] * u ** m).sum()) <= 1e-11 * scale, (c, ax, m)
