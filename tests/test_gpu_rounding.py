"""The range-limited reciprocal, square root, quotient and logarithm of the
draws equal the correctly rounded operations bit for bit: every mantissa at
several exponents of their ranges; and couplings whose beta k leaves those
ranges (drawn by the checked operations) follow the oracle link for link."""
import numpy as np
import pytest

import oracle
from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu
MANTISSAS = np.arange(1 << 23, dtype=np.uint32)


def _floats(exponent):
    """All binary32 numbers in [2^exponent, 2^(exponent + 1))."""
    return (MANTISSAS | np.uint32((exponent + 127) << 23)).view(np.float32)


def _same(pair):
    assert np.array_equal(pair[0].view(np.uint32), pair[1].view(np.uint32))


@pytest.mark.parametrize("exponent", [-100, -31, 0, 3, 61, 99])
def test_reciprocal(exponent):
    _same(su2.su2_selftest_rounding(0, _floats(exponent)))


@pytest.mark.parametrize("exponent", [-70, -69, -1, 0, 1, 5, 98, 99])
def test_square_root(exponent):
    _same(su2.su2_selftest_rounding(1, _floats(exponent)))


@pytest.mark.parametrize("exponent", [-26, -25, -24, -13, -2, -1])
def test_square_root_up_to_one(exponent):
    _same(su2.su2_selftest_rounding(2, _floats(exponent)))
    _same(su2.su2_selftest_rounding(2, np.array([0.0, 1.0], dtype=np.float32)))


def test_square_root_below_its_range_is_small_or_nan():
    x = np.concatenate([np.array([0.0, np.inf], dtype=np.float32), np.float32(2.0) ** -np.arange(71, 150, dtype=np.float32)])
    y, _ = su2.su2_selftest_rounding(1, x.astype(np.float32))
    assert np.all(np.isnan(y) | (y <= 2.0 ** -34))


@pytest.mark.parametrize("eb,ea", [(2, 0), (2, -80), (5, 5), (61, 5), (3, -24), (6, -45)])
def test_quotient(eb, ea):
    rng = np.random.default_rng(eb + 100 * ea % 97)
    a, b = _floats(ea), _floats(eb)
    _same(su2.su2_selftest_rounding(3, a[rng.permutation(a.size)], b))
    # divisors and numerators next to a power of two
    a, b = np.meshgrid(np.concatenate([a[:500], a[-500:]]), np.concatenate([b[:500], b[-500:]]))
    _same(su2.su2_selftest_rounding(3, a.ravel(), b.ravel()))


def test_logarithm_every_mantissa():
    x = _floats(0)
    assert np.array_equal(su2.su2_selftest_math(0, x).view(np.uint32), oracle.logf(x).view(np.uint32))


@pytest.mark.parametrize("beta", [1e-12, 3e9, 1e13, 1e25, 3e35])
def test_extreme_couplings(beta):
    ns, nt, seed = 4, 4, 9
    kp = su2.su2_create(ns, nt, beta, seed, su2.SU2_HOT)
    b = su2.su2_batch_create([ns], [nt], [beta], [seed], su2.SU2_HOT)
    try:
        su2.su2_set_sampler(kp, su2.SU2_SAMPLER_KP)
        su2.su2_batch_set_sampler(b, su2.SU2_SAMPLER_KP)
        su2.su2_heatbath_sweep(kp, 1)
        su2.su2_batch_sweep(b, 1)
        ref = oracle.hot_start(ns, nt, seed)
        oracle.heatbath_sweep_kp(ns, nt, beta, seed, 0, ref)
        assert np.array_equal(su2.su2_get_links(kp, ns, nt), ref)
        assert np.array_equal(su2.su2_batch_get_links(b, 0, ns, nt), ref)
    finally:
        su2.su2_destroy(kp)
        su2.su2_batch_destroy(b)


@pytest.mark.parametrize("ns,nt,sampler,overrelax", [(32, 34, 0, 1), (36, 36, 0, 1), (40, 38, 0, 1), (28, 50, 1, 0)])
def test_rounds_per_warp_either_side_of_the_peeled_last_round(ns, nt, sampler, overrelax):
    """One to about ten rounds per warp, where the kernels change between the
    peeled and the plain loop."""
    h = su2.su2_create(ns, nt, 2.4, 5, su2.SU2_HOT)
    try:
        su2.su2_set_sampler(h, sampler)
        su2.su2_set_overrelax(h, overrelax)
        su2.su2_heatbath_sweep(h, 1)
        got = su2.su2_get_links(h, ns, nt)
    finally:
        su2.su2_destroy(h)
    ref = oracle.hot_start(ns, nt, 5)
    sweep = oracle.heatbath_sweep_kp if sampler else oracle.heatbath_sweep
    sweep(ns, nt, 2.4, 5, 0, ref, nthreads=oracle.max_threads())
    for _ in range(overrelax):
        oracle.overrelax_sweep(ns, nt, ref, nthreads=oracle.max_threads())
    assert np.array_equal(got, ref)
