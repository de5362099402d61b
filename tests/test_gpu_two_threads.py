"""Two threads with a lattice each: a kernel's shared-memory limit belongs to the
kernel, not to the handle, so one thread's small launch must not take the limit
from under the other's large one."""
import threading

import numpy as np
import pytest

from paper_1010_1486_gb300 import learn, su2

pytestmark = pytest.mark.gpu


def _both(*calls, n=400):
    """Each of the calls n times in a thread of its own; what they returned."""
    out, errors = [[] for _ in calls], []
    start = threading.Barrier(len(calls))

    def work(i):
        try:
            start.wait()
            for _ in range(n):
                out[i].append(calls[i]())
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    return out


def test_wilson_loops_of_a_small_and_a_larger_lattice():
    torch = pytest.importorskip("torch")
    small = su2.su2_create(4, 4, 2.3, 1, su2.SU2_HOT, stream=torch.cuda.Stream())
    large = su2.su2_create(24, 24, 2.3, 2, su2.SU2_HOT, stream=torch.cuda.Stream())
    try:
        want = [su2.su2_wilson_loops(small, 4, 4), su2.su2_wilson_loops(large, 4, 4)]
        out = _both(lambda: su2.su2_wilson_loops(small, 4, 4), lambda: su2.su2_wilson_loops(large, 4, 4), n=4000)
        for w, got in zip(want, out):
            assert all(np.array_equal(w, g) for g in got)
    finally:
        su2.su2_destroy(small)
        su2.su2_destroy(large)


def test_learned_sweeps_with_a_small_and_a_large_table():
    torch = pytest.importorskip("torch")
    lats = [su2.su2_create(4, 4, 3.0, 3, su2.SU2_HOT, stream=torch.cuda.Stream()) for _ in range(2)]
    try:
        w = learn.initial_weights(1, 10.0, 0.2)
        for h, rows in zip(lats, (2, 400)):
            su2.su2_set_proposal(h, w, -2.0, 2.0, rows)
            su2.su2_set_timing(h, True)  # launches of its own in every call, no graph
        out = _both(*[lambda h=h: su2.su2_learned_generate(h, 1, 0, 0.0)[2]["learned_sweeps"] for h in lats], n=200)
        assert out == [[1] * 200, [1] * 200]
    finally:
        for h in lats:
            su2.su2_destroy(h)
