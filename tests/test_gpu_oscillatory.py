"""The FP32 oscillatory kernel's sine by itself: one unit charge at the origin and
targets at distances that are powers of two, where the kernel's 1/r is exact (the
Coulomb kernel shows it), so the potential is sin(kappa r)/r with the sine's own
error.  Many kappas in one plan, a problem each.

Bounds in units u = 2^-24.  For a phase below pi/2 nothing is rounded before the
sine if kappa is a float: one final rounding (u relative), the correction's (its
share of the sine is at most 0.37 on top, three roundings of it: 0.6 u), the
polynomial's 6.3e-9.  Otherwise kappa's own rounding scales the reduced phase by up to u,
and the reduction rounds a phase of at most pi/2 twice (u each, times |cos| < 0.6
where |f| >= 1 and half of u below it)."""
import numpy as np
import pytest
import torch

from paper_2012_06925_gb300 import binding as B

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
R = np.array([0.25, 1.0, 4.0])


def potentials(kernel, kappas):
    p = len(kappas)
    tgt = np.zeros((3, 3 * p))
    tgt[1] = np.tile(R, p)
    to = np.arange(p + 1) * 3
    so = np.arange(p + 1)
    src = torch.zeros(3, p, dtype=torch.float64, device="cuda")
    q = torch.ones(p, dtype=torch.float64, device="cuda")
    with B.Plan.batch(torch.from_numpy(tgt).cuda(), to, src, so, q, [kernel] * p, kappas, n=2, theta=0.0, N0=10,
                      M0=10, precision=B.FP32_BULK) as plan:
        return plan.compute().cpu().numpy().reshape(p, 3)


def test_reciprocal_distances_are_exact():
    assert np.array_equal(potentials(B.COULOMB, [0.0] * 3), np.tile(1 / R, (3, 1)))


@pytest.mark.parametrize("is_float", [True, False])
def test_small_phases(is_float):
    kappas = np.random.default_rng(1).uniform(0.001, 0.39, 3000)         # phases to 1.56
    if is_float:
        kappas = kappas.astype(np.float32).astype(np.float64)
    phase = kappas[:, None] * R
    err = potentials(B.OSCILLATORY, kappas) * R / np.sin(phase) - 1
    assert np.max(np.abs(err)) <= (1.6 * U if is_float else 2.6 * U) + 6.3e-9
    assert abs(np.mean(err)) <= 0.1 * U                                  # no bias


@pytest.mark.parametrize("top", [6.0, 100.0, 5000.0])
def test_large_phases(top):
    kappas = np.random.default_rng(2).uniform(0.4, top / 4, 3000)
    err = potentials(B.OSCILLATORY, kappas) * R - np.sin(kappas[:, None] * R)
    # reduction 2 x 0.6 u, kappa's rounding 0.6 u (f cos f), final and correction 1.6 u of at most 1, and the
    # rest of pi: n pi 3e-4 to a float
    assert np.max(np.abs(err)) <= 3.4 * U + 6.3e-9 + top * 3.1e-4 * U
    assert abs(np.mean(err)) <= 0.1 * U


def test_kappa_zero():
    assert np.array_equal(potentials(B.OSCILLATORY, [0.0] * 3), np.zeros((3, 3)))
