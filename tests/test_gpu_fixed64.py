"""The FP64 kernel functions in integer arithmetic on the device, pair by pair:
the direct sum of one unit charge at the origin is G itself, against extended
precision with the bounds of test_fixed64_cpu (the device's seed of the square
root differs from the host's, the bounds do not)."""
import numpy as np
import pytest
import torch

from paper_2012_06925_gb300 import binding as B
from test_fixed64_cpu import radius, vectors

pytestmark = pytest.mark.gpu


def single(d, kernel, kappa):
    tgt = torch.from_numpy(np.ascontiguousarray(d.T)).cuda()
    src = torch.zeros(3, 1, dtype=torch.float64, device="cuda")
    q = torch.ones(1, dtype=torch.float64, device="cuda")
    return B.direct_sum(tgt, src, q, kernel, kappa).cpu().numpy()


@pytest.mark.parametrize("kind", ["plain", "mixed", "scaled", "ulps"])
def test_inverse_distance(kind):
    d = vectors(kind)
    got = single(d, B.COULOMB, 0.0)
    assert np.max(np.abs(got.astype(np.longdouble) * radius(d) - 1)) <= 1.2e-16


@pytest.mark.parametrize("kind", ["plain", "mixed", "ulps"])
@pytest.mark.parametrize("kappa", [0.0, 1e-5, 0.5, 30.0, 400.0])
def test_screened(kind, kappa):
    d = vectors(kind)
    r = radius(d)
    want = np.exp(-np.longdouble(kappa) * r) / r
    got = single(d, B.YUKAWA, kappa)
    keep = want > 1e-300
    err = np.abs(got[keep].astype(np.longdouble) / want[keep] - 1)
    assert np.all(err <= 1.3e-16 + kappa * r[keep] * 1.45 * 2.0 ** -58)
    assert np.all(got[~keep] <= 1e-299) and np.all(got >= 0)


@pytest.mark.parametrize("kappa", [0.0, 0.005, 1.0])
def test_regularized(kappa):
    d = vectors("mixed")
    r = radius(d)
    got = single(d, B.REG_COULOMB, kappa)
    assert np.max(np.abs(got.astype(np.longdouble) * np.sqrt(r * r + np.longdouble(kappa) ** 2) - 1)) <= 1.2e-16


def test_ends_of_the_range():
    d = np.array([[0, 0, 0], [1e-170, 0, 0], [5e-324, 0, 1e-310], [1e200, 0, 0], [0, -1e300, 1e300]])
    for kernel, kappa in ((B.COULOMB, 0.0), (B.YUKAWA, 0.5), (B.REG_COULOMB, 0.005)):
        assert np.all(single(d, kernel, kappa) == 0.0), kernel
    one = np.array([[1.0, 0, 0], [0, -0.5, 0], [3.0, 0, 4.0], [2.0 ** -500, 0, 0]])
    assert np.array_equal(single(one, B.COULOMB, 0.0), [1.0, 2.0, 0.2, 2.0 ** 500])


@pytest.mark.parametrize("kernel,kappa", [(B.YUKAWA, -2.0), (B.REG_COULOMB, -0.5), (B.YUKAWA, np.inf),
                                          (B.REG_COULOMB, np.nan)])
def test_parameters_a_plan_refuses(kernel, kappa):
    """The direct sum takes any kappa; negative and non-finite ones are FP64 expressions."""
    d = np.random.default_rng(0).uniform(-1, 1, (64, 3))
    r = radius(d).astype(np.float64)
    want = np.exp(-kappa * r) / r if kernel == B.YUKAWA else 1 / np.sqrt(r * r + kappa * kappa)
    np.testing.assert_allclose(single(d, kernel, kappa), want, rtol=16 * 2.0 ** -53)


def test_plan_and_direct_sum_agree_to_rounding():
    """theta = 0: the FP64 plan and the direct sum add the same terms in other orders."""
    rng = np.random.default_rng(3)
    pts = torch.from_numpy(rng.uniform(-1, 1, (3, 700))).cuda()
    q = torch.from_numpy(rng.uniform(0.5, 1.5, 700)).cuda()
    for kernel, kappa in ((B.COULOMB, 0.0), (B.YUKAWA, 0.7), (B.REG_COULOMB, 0.01)):
        with B.Plan(pts, pts, q, kernel=kernel, kappa=kappa, n=2, theta=0.0, N0=64, M0=64, precision=B.FP64) as p:
            phi = p.compute()
        ref = B.direct_sum(pts, pts, q, kernel, kappa)
        assert torch.max(torch.abs(phi / ref - 1)).item() <= 700 * 2.0 ** -53


@pytest.mark.parametrize("kernel,kappa", [(B.COULOMB, 0.0), (B.YUKAWA, 0.7), (B.OSCILLATORY, 2.0)])
@pytest.mark.parametrize("m", [1, 31, 32, 33, 127, 128, 129, 160, 255, 256, 257, 300])
def test_partial_target_tiles(m, kernel, kappa):
    """Warps and target slots without a real row are left out; the rows that are there are not."""
    rng = np.random.default_rng(m)
    tgt = torch.from_numpy(rng.uniform(-1, 1, (3, m))).cuda()
    src = torch.from_numpy(rng.uniform(-1, 1, (3, 300))).cuda()
    q = torch.from_numpy(rng.uniform(0.5, 1.5, 300)).cuda()
    with B.Plan(tgt, src, q, kernel=kernel, kappa=kappa, n=2, theta=0.0, N0=512, M0=512,
                precision=B.FP64) as p:
        phi = p.compute()
    ref = B.direct_sum(tgt, src, q, kernel, kappa)
    scale = B.direct_sum(tgt, src, q, B.COULOMB, 0.0)       # bounds the sum of |terms|
    assert torch.max(torch.abs(phi - ref) / scale).item() <= 310 * 2.0 ** -53


@pytest.mark.parametrize("case", ["uniform", "shifted", "clustered", "one_point", "infinite"])
@pytest.mark.parametrize("kernel,kappa", [(B.COULOMB, 0.0), (B.YUKAWA, 0.6), (B.REG_COULOMB, 0.01)])
def test_direct_sum_in_fixed_coordinates(case, kernel, kappa):
    """A sum large enough for fixed-point coordinates against the same targets in calls that are
    not: terms to 2e-16 in each, tiles of 256 and their sums one after the other."""
    rng = np.random.default_rng(6)
    m, n = 300, 40000
    src, tgt = rng.uniform(-1, 1, (3, n)), rng.uniform(-1, 1, (3, m))
    if case == "shifted":
        src, tgt = src + 1e5, tgt + 1e5
    elif case == "clustered":                       # most pairs far closer than 1/64 of the extent
        src[:, 1:], tgt[:, 3:] = src[:, 1:] * 1e-4, tgt[:, 3:] * 1e-4
    elif case == "one_point":
        src[:], tgt[:] = 0.3, 0.3
    elif case == "infinite":
        tgt[1, 5], src[2, 7] = np.inf, -np.inf
    tgt[:, :100] = src[:, :100]                     # coincident pairs
    q = torch.from_numpy(rng.uniform(0.5, 1.5, n)).cuda()
    src, tgt = torch.from_numpy(src).cuda(), torch.from_numpy(np.ascontiguousarray(tgt)).cuda()
    whole = B.direct_sum(tgt, src, q, kernel, kappa)
    parts = torch.cat([B.direct_sum(tgt[:, i:i + 100].contiguous(), src, q, kernel, kappa)
                       for i in range(0, m, 100)])
    torch.testing.assert_close(whole, parts, rtol=4e-16 + 2 * (256 + n / 256) * 2.0 ** -53, atol=0)
