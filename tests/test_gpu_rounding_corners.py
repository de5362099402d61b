"""The quotient of the draws next to the middle of two binary32 numbers, and at
the largest couplings, where it falls below the range in which it is correctly
rounded."""
import numpy as np
import pytest

from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu


def test_quotients_next_to_a_midpoint():
    """Numerators a with a 2^s = M B + d: the quotient a / B is d / 2^s B away
    from the middle M 2^-s of two binary32 numbers (M odd, 25 bits)."""
    rng = np.random.default_rng(3)
    B = rng.integers(1 << 23, 1 << 24, 1 << 20, dtype=np.uint64) | np.uint64(1)
    inverse = B.copy()
    for _ in range(5):
        inverse = inverse * (np.uint64(2) - B * inverse)
    tops, bottoms = [], []
    for s in (24, 25):
        for d in (-7, -5, -3, -2, -1, 1, 2, 3, 5, 7):
            m = (np.uint64((-d) % (1 << 64)) * inverse) & np.uint64((1 << s) - 1)
            if s == 24:
                m += np.uint64(1 << 24)
            a = (m * B + np.uint64(d % (1 << 64))) >> np.uint64(s)
            ok = (m >= 1 << 24) & (m % np.uint64(2) == 1) & (a >= 1 << 23) & (a < 1 << 24) & ((a >= B) == (s == 24))
            tops.append(a[ok])
            bottoms.append(B[ok])
    a, b = np.concatenate(tops).astype(np.float32), np.concatenate(bottoms).astype(np.float32)
    assert a.size > 1 << 20
    y, want = su2.su2_selftest_rounding(3, a * np.float32(2.0 ** -40), b)
    assert np.array_equal(y.view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("eb", [23, 40, 61])
@pytest.mark.parametrize("ea", [-67, -60, -25, 5])
def test_tiny_quotients_give_the_same_trial(ea, eb):
    """A trial takes 1 - 2 l and 1 - l of its quotient l.  Below 2^-90 the
    refined quotient may differ from the correctly rounded one, and both vanish
    beside 1."""
    mantissa = np.linspace(1.0, 2.0, 1 << 16, endpoint=False).astype(np.float32)
    a, b = mantissa * np.float32(2.0 ** ea), mantissa[::-1] * np.float32(2.0 ** eb)
    y, want = su2.su2_selftest_rounding(3, a, b)
    one = np.float32(1.0)
    assert np.array_equal(one - np.float32(2.0) * y, one - np.float32(2.0) * want)
    assert np.array_equal(one - y, one - want)
    exact = a.astype(np.float64) / b
    assert np.all(np.abs(y - exact) <= np.maximum(2.0 ** -24 * exact, 2.0 ** -148))
    inside = exact >= 2.0 ** -90
    assert np.array_equal(y[inside].view(np.uint32), want[inside].view(np.uint32))
