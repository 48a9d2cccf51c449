"""Pairs at distance 0 are left out of the direct sum whatever their charge: a
charge that is infinite or NaN reaches every target but those at its own point.
In every form of the sum (FP64 expressions, fixed point, fixed-point
coordinates) and with one and several splits of the sources."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2012_06925_gb300 import binding as B
from _gpu_util import to_dev

pytestmark = pytest.mark.gpu

KERNELS = [(B.COULOMB, 0.0), (B.YUKAWA, 0.7), (B.OSCILLATORY, 2.0), (B.REG_COULOMB, 0.01), (B.REG_COULOMB, -0.01),
           (B.TEST_POLY, 0.0)]


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("kernel,kappa", KERNELS)
@pytest.mark.parametrize("m,n", [(7, 5), (40, 700), (300, 30011)])       # the last: fixed-point coordinates
def test_coincident_pair_with_a_charge_that_is_not_finite(m, n, kernel, kappa, bad):
    rng = np.random.default_rng(n)
    src = rng.uniform(-1, 1, (3, n))
    tgt = rng.uniform(-1, 1, (3, m))
    at = n // 2
    tgt[:, 1] = tgt[:, 4] = src[:, at]
    q = rng.uniform(0.5, 1.5, n)
    rest = np.delete(np.arange(n), at)
    q[at] = bad
    phi = B.direct_sum(to_dev(tgt), to_dev(src), to_dev(q), kernel, kappa).cpu().numpy()
    own = np.zeros(m, bool)
    own[[1, 4]] = True
    assert not np.any(np.isfinite(phi[~own])) and np.all(np.isfinite(phi[own]))
    want = O.direct_sum(tgt[:, own], src[:, rest], q[rest], kernel, kappa)
    # sum of |terms|: the terms have one sign, or the Coulomb terms bound them, or |G q| <= 32 in the test kernel
    size = {B.OSCILLATORY: O.direct_sum(tgt[:, own], src[:, rest], q[rest], O.COULOMB),
            B.TEST_POLY: 32.0 * n}.get(kernel, np.abs(want))
    assert np.all(np.abs(phi[own] - want) <= 2 * (n + 8) * 2.0 ** -53 * size)


def test_pairs_at_infinite_distance_keep_their_product():
    """exp(-kappa r)/r = 0 is a factor, not a pair left out: 0 times an infinite charge is NaN."""
    src = torch.tensor([[0.0, 5.0], [0.0, 0.0], [0.0, 0.0]], dtype=torch.float64, device="cuda")
    tgt = torch.tensor([[5.0, 1e200], [0.0, 0.0], [0.0, 0.0]], dtype=torch.float64, device="cuda")
    q = torch.tensor([2.0, np.inf], dtype=torch.float64, device="cuda")
    for kernel, kappa in ((B.COULOMB, 0.0), (B.YUKAWA, 0.5), (B.REG_COULOMB, 0.01)):
        phi = B.direct_sum(tgt, src, q, kernel, kappa).cpu().numpy()
        assert np.isfinite(phi[0]) and np.isnan(phi[1]), (kernel, phi)
