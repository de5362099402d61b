"""su2_wilson_loops takes the walks for few small loops and the tiles for the
rest.  Either side of that line: the same values (binary32 loops, sums to
2^-44 per loop), and a few loops never at the price of many."""
import time

import numpy as np
import pytest

from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu
TOL = 2.0 ** -44 + 2e6 * 2.0 ** -53


@pytest.mark.parametrize("ns,nt", [(4, 4), (16, 64), (24, 24), (36, 36), (34, 8), (66, 16), (128, 2)])
def test_every_form_agrees_with_the_whole_call(ns, nt):
    h = su2.su2_create(ns, nt, 2.3, 7, su2.SU2_HOT)
    try:
        su2.su2_set_sampler(h, su2.SU2_SAMPLER_KP)
        su2.su2_heatbath_sweep(h, 3)
        whole = su2.su2_wilson_loops(h, min(ns, 12), min(nt, 9))
        for r, t in [(1, 1), (2, 1), (1, 2), (2, 2), (3, 2), (4, 1), (1, 4), (4, 4), (8, 1), (9, 1), (9, 2), (12, 1)]:
            if r <= ns and t <= nt:
                got = su2.su2_wilson_loops(h, r, t)
                # the walks add up to 10^7 loops in binary64
                assert np.abs(got - whole[:r, :t]).max() <= TOL + 1e7 * 2.0 ** -53, (r, t)
    finally:
        su2.su2_destroy(h)


@pytest.mark.parametrize("ns,nt", [(40, 40), (66, 16)])
def test_one_loop_costs_a_fraction_of_sixty_four(ns, nt):
    h = su2.su2_create(ns, nt, 2.3, 7, su2.SU2_HOT)
    try:
        def us(r, t):
            took = []
            for _ in range(8):
                start = time.perf_counter()
                su2.su2_wilson_loops(h, r, t)
                took.append(time.perf_counter() - start)
            return min(took) * 1e6

        # 40^4: 117 of 1700 us (490 on the tiles once), 66^3 x 16: 190 of 3800 (2570 of 8500)
        assert us(1, 1) < 0.2 * us(8, 8)
    finally:
        su2.su2_destroy(h)
