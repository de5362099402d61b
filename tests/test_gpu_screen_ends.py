"""The screened Creutz trial where its difference A - t (2 - t) is extreme: the
smallest and largest words, t beyond 2 (a0 clamped to -1), the largest and
smallest 1/(beta k), the Haar branch and values that are not numbers.  A
decided trial has the exact test's verdict, everything else is undecided."""
import numpy as np
import pytest

from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ibk", [1e6, 40.0, 2.0, 0.1, 1.0 / 43.0, 1e-18, 0.0, np.nan])
def test_ends_of_the_screen(ibk):
    bk = 1.0 / ibk if ibk > 0.0 else 0.0
    e = np.exp(-2.0 * bk) if 0.0 < bk <= 21.0 else 0.0
    r1 = np.concatenate([2.0 ** -33 + 2.0 ** -32 * np.arange(64.0), 2.0 ** -np.arange(1.0, 33.0),
                         1.0 - 2.0 ** -24 * np.arange(64.0)])
    r2 = np.concatenate([2.0 ** -24 * np.arange(1.0, 65.0), 2.0 ** -np.arange(1.0, 24.0), 1.0 - 2.0 ** -24 * np.arange(64.0)])
    a, b = (g.ravel() for g in np.meshgrid(r1, r2))
    q = np.stack([a, b, np.full_like(a, ibk), np.full_like(a, e)], axis=1).astype(np.float32)
    screen, exact = su2.su2_selftest_math(4, q)
    decided = screen != 2.0
    assert np.array_equal(screen[decided], exact[decided])
    if not ibk > 0.0:  # Haar branch, not a number
        assert not decided.any()
    else:  # decided wherever the difference in binary64 is beyond twice the slack (its estimate is within a third of it)
        e32 = np.float32(e)
        x = (q[:, 0].astype(np.float64) * np.float64(np.float32(1.0) - e32) + e32).astype(np.float32).astype(np.float64)
        t = -np.log(x) * np.float32(ibk)
        diff = q[:, 1].astype(np.float64) ** 2 - t * (2.0 - t)
        assert decided[np.abs(diff) > 2.0 * (2e-6 + 4e-6 * ibk + 2e-5 * t)].all()
