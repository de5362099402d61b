"""The Kennedy-Pendleton phase with and without its peeled last round: either
side of the couplings and rounds per warp where the launch changes, against the
oracle, and what a phase costs where most links pass through the retry queue."""
import time

import numpy as np
import pytest

import oracle
from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu
KP = su2.SU2_SAMPLER_KP


# 32^3 x 26 has 3.65 rounds of 32 links per warp, 32^3 x 28 3.93: the line is 3.7 up to beta = 1
@pytest.mark.parametrize("ns,nt,beta", [(32, 26, 0.7), (32, 28, 0.7), (32, 28, 0.44), (32, 28, 0.46), (32, 28, 1.1),
                                        (32, 28, 1.2), (36, 24, 1.3)])
def test_sweep_equals_the_oracle(ns, nt, beta):
    h = su2.su2_create(ns, nt, beta, 5, su2.SU2_HOT)
    try:
        su2.su2_set_sampler(h, KP)
        plaq, _, st = su2.su2_generate(h, 1, 1, 0)
        got = su2.su2_get_links(h, ns, nt)
        separate = su2.su2_plaquette(h)
    finally:
        su2.su2_destroy(h)
    ref = oracle.hot_start(ns, nt, 5)
    trials = oracle.heatbath_sweep_kp(ns, nt, beta, 5, 0, ref, nthreads=oracle.max_threads())
    assert np.array_equal(got, ref)
    assert list(st["trials"]) == [int(t) for t in trials]
    assert abs(plaq[0] - separate) < 1e-6


def test_phase_where_most_links_wait_in_the_queue():
    """40^4: 62 us per phase at beta = 1 and 39 at beta = 6 (70 with the last
    round peeled)."""
    def us(beta):
        h = su2.su2_create(40, 40, beta, 5, su2.SU2_HOT)
        try:
            su2.su2_set_sampler(h, KP)
            su2.su2_heatbath_sweep(h, 10)
            su2.su2_sync(h)
            took = []
            for _ in range(12):
                start = time.perf_counter()
                su2.su2_heatbath_sweep(h, 5)
                su2.su2_sync(h)
                took.append((time.perf_counter() - start) * 1e6 / 40)
            return min(took)
        finally:
            su2.su2_destroy(h)

    assert us(1.0) < 1.69 * us(6.0)
