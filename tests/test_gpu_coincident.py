"""Targets that coincide with sources, in every kernel and consumer layout: the
guard stands in the near chunks' path only, so a chunk's box and near distance
must catch every coincident pair - also chunks of one point or of one repeated
point (extent 0, exactly representable in float or not) and targets on the
faces of a chunk's box.  FP32 budget of the parity tests: 1e-6."""
import numpy as np
import pytest

import oracle as O
from paper_2012_06925_gb300 import binding as B
from _gpu_util import rel_l2, run_gpu

pytestmark = pytest.mark.gpu

KERNELS = [(B.COULOMB, 0.0), (B.YUKAWA, 0.7), (B.OSCILLATORY, 2.0), (B.REG_COULOMB, 0.005)]
POINTS = {"float": (0.5, 0.25, -0.125), "double": (0.1, -0.7, 0.3)}


def check(tgt, src, kernel, kappa, leaf=100):
    q = np.random.default_rng(7).uniform(0.5, 1.5, src.shape[1])
    ref = O.direct_sum(tgt, src, q, kernel, kappa)
    phi, plan = run_gpu(tgt, src, q, precision=B.FP32_BULK, kernel=kernel, kappa=kappa, n=2, theta=0.0,
                        N0=leaf, M0=leaf)
    plan.close()
    assert rel_l2(ref, phi) <= 1e-6


@pytest.mark.parametrize("kernel,kappa", KERNELS)
@pytest.mark.parametrize("point", sorted(POINTS))
@pytest.mark.parametrize("n", [1, 40, 255, 256])
def test_chunk_of_one_point(n, point, kernel, kappa):
    p = np.array(POINTS[point])[:, None]
    tgt = np.concatenate([p, p + 1e-3, np.random.default_rng(n).uniform(-1, 1, (3, 70))], axis=1)
    check(tgt, np.repeat(p, n, axis=1), kernel, kappa, leaf=300)


@pytest.mark.parametrize("kernel,kappa", KERNELS)
@pytest.mark.parametrize("layout", ["0", "1", "2", "3", "4", "5"])
def test_faces_and_interior_of_chunk_boxes(layout, kernel, kappa, monkeypatch):
    monkeypatch.setenv("BLDTT_INTERACT_LAYOUT", layout)
    rng = np.random.default_rng(3)
    src = rng.uniform(-1, 1, (3, 600))
    src[0, ::3] = np.sign(src[0, ::3])              # a third on two faces of the domain
    tgt = np.concatenate([src, rng.uniform(-1, 1, (3, 333))], axis=1)
    check(tgt, src, kernel, kappa)


@pytest.mark.parametrize("kernel,kappa", KERNELS[:2])
@pytest.mark.parametrize("n", [2, 31, 255, 257, 513])
def test_repeated_points(n, kernel, kappa):
    rng = np.random.default_rng(n)
    src = rng.uniform(-1, 1, (3, n))
    src[:, n // 2:] = src[:, :1]
    check(np.concatenate([src, rng.uniform(-1, 1, (3, 130))], axis=1), src, kernel, kappa)
