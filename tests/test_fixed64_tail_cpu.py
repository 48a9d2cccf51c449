"""exp(-kappa r)/r below the normal range of double (csrc/fixed64.cuh, compiled
for the host): subnormal values, as FP64 expressions give them, down to 0; and the
same kappa r at distances so small that the value is a normal number.  The
value is rounded once to the subnormal spacing 2^-1074 (half of it) after the
relative error of the normal range (test_fixed64_cpu)."""
import numpy as np
import pytest

from test_fixed64_cpu import call, lib, radius      # noqa: F401  (lib is the fixture)

TINY = np.longdouble(2.0) ** -1074


@pytest.mark.parametrize("kappa", [0.7, 30.0, 700.0, 1e5, 0.7 * 2.0 ** 400])
def test_screened_below_the_normal_range(lib, kappa):      # noqa: F811
    rng = np.random.default_rng(len(str(kappa)))
    # kappa r from 690 to 760: from 1e-300 through the subnormals (1e-308 .. 5e-324) to 0
    d = rng.uniform(-1, 1, (20000, 3))
    d *= (rng.uniform(690, 760, 20000) / kappa / radius(d).astype(float))[:, None]
    r = radius(d)
    want = np.exp(-np.longdouble(kappa) * r) / r
    got = call(lib, "scr", d, kappa).astype(np.longdouble)
    rel = 1.3e-16 + kappa * r * 1.45 * 2.0 ** -58
    assert np.all(np.abs(got - want) <= want * rel + TINY / 2 * (1 + 1e-9))
    assert np.all(got[want > 0.51 * TINY] > 0) and np.all(got[want < 0.49 * TINY] == 0)
    if kappa < 1e6:
        assert ((want < 2.2e-308) & (want > TINY)).sum() > 1000 and np.any(want < 0.49 * TINY)


def test_one_value(lib):      # noqa: F811
    assert call(lib, "scr", [[1.02, 0, 0]], 700.0)[0] == pytest.approx(np.exp(-700 * 1.02) / 1.02, rel=1e-12)
