"""The plaquette kernel's walk along t at the edges of its split, and the
page-locked result pages under more threads than there are pages."""
import threading

import numpy as np
import pytest

import oracle
from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,nt", [(2, 2), (2, 40), (4, 6), (10, 6), (10, 18), (28, 2), (28, 6), (36, 4), (56, 2)])
def test_plaquette_is_the_mean_of_its_sites(ns, nt):
    """Blocks of 384 pairs, ragged in space and time, one to many chunks of t:
    the oracle's binary32 site values, summed in binary64 on both sides."""
    h = su2.su2_create(ns, nt, 2.3, 5 + ns, su2.SU2_HOT)
    try:
        got = su2.su2_plaquette(h)
        links = su2.su2_get_links(h, ns, nt)
    finally:
        su2.su2_destroy(h)
    sites = oracle.site_plaquettes(ns, nt, links).astype(np.float64)
    # |site| <= 6 over 6 V; N binary64 additions in another order
    assert abs(got - sites.sum() / (6.0 * sites.size)) <= sites.size * 2.0 ** -53


def test_many_threads_read_their_own_results():
    n = 24
    lats = [su2.su2_create(4, 4, 2.0, 100 + i, su2.SU2_HOT) for i in range(n)]
    try:
        want = [(su2.su2_plaquette(h), su2.su2_polyakov(h)) for h in lats]
        bad = []

        def work(i):
            for _ in range(50):
                if (su2.su2_plaquette(lats[i]), su2.su2_polyakov(lats[i])) != want[i] or su2.su2_check_links(lats[i]) != (0, 0):
                    bad.append(i)

        threads = [threading.Thread(target=work, args=(i,)) for i in range(n)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not bad and len(set(want)) == n
    finally:
        for h in lats:
            su2.su2_destroy(h)
    # the pages went with the last handle; new ones work
    h = su2.su2_create(4, 4, 2.0, 100, su2.SU2_HOT)
    try:
        assert (su2.su2_plaquette(h), su2.su2_polyakov(h)) == want[0]
        p, q, _ = su2.su2_generate(h, 6000, 1, 0)  # more values than a page holds
        assert p.size == 6000 and np.all(np.isfinite(p)) and np.all(np.isfinite(q)) and np.all(p != 0)
    finally:
        su2.su2_destroy(h)
