"""The page-locked result pages under more threads than there are pages."""
import threading

import numpy as np
import pytest

from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu


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
