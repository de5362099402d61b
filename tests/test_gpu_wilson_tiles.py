"""The tiled Wilson-loop kernel at the edges of its tiles: ragged tiles in
space and time, several chunks of R and of T, lattices smaller than a warp,
and links that are not unit (which the binary64 path takes).  The binary32
loops are the oracle's; the fixed-point sum is within 2^-44 of the exact one
per loop and the oracle's binary64 sum within N 2^-53 of it (N < 2e6 loops)."""
import os

import numpy as np
import pytest

import oracle
from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu
TOL = 2.0 ** -44 + 2e6 * 2.0 ** -53


def _links(ns, nt, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    u = rng.normal(size=(ns ** 3 * nt, 4, 4)) * 0.3
    u[..., 0] += 1.0
    return (scale * u / np.linalg.norm(u, axis=-1, keepdims=True)).astype(np.float32)


def _both(ns, nt, rmax, tmax, links):
    h = su2.su2_create(ns, nt, 2.3, 1, su2.SU2_COLD)
    try:
        su2.su2_set_links(h, links)
        got = su2.su2_wilson_loops(h, rmax, tmax)
        again = su2.su2_wilson_loops(h, rmax, tmax)
    finally:
        su2.su2_destroy(h)
    assert np.array_equal(got, again, equal_nan=True)
    return got, oracle.wilson_loops(ns, nt, links, rmax, tmax, nthreads=min(16, os.cpu_count() or 1))


@pytest.mark.parametrize("ns,nt,rmax,tmax", [(2, 2, 1, 1), (2, 40, 2, 40), (10, 6, 10, 6), (12, 22, 12, 9),
                                             (16, 10, 9, 10), (18, 8, 16, 8), (66, 2, 16, 2), (4, 66, 4, 64)])
def test_ragged_tiles_and_chunks(ns, nt, rmax, tmax):
    got, want = _both(ns, nt, rmax, tmax, _links(ns, nt, ns + nt))
    assert np.abs(got - want).max() <= TOL


def test_links_beyond_the_fixed_point_range():
    # loops reach 1.5^(2 (R + T)): every value still comes out, to binary64 sums
    got, want = _both(6, 4, 4, 3, _links(6, 4, 3, scale=1.5))
    assert np.abs(want).max() > 2.0 and np.all(np.abs(got - want) <= 1e-12 * np.abs(want).max())


def test_not_a_number_link_reaches_the_result():
    links = _links(4, 4, 4)
    links[100, 3, 2] = np.nan
    got, want = _both(4, 4, 4, 4, links)
    assert np.isnan(want).all() and np.isnan(got).all()
