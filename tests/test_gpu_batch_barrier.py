"""The grid barrier of the batched sweeps, through the function that the sweep
kernel calls: barriers that complete order the blocks' writes, and a wait that
nothing completes gives up in every block and leaves its mark in the error word."""
import numpy as np
import pytest

from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks,barriers", [(1, 0), (1, 9), (2, 1), (8, 9), (152, 100), (1024, 9)])
def test_barriers_complete_and_the_last_wait_gives_up(blocks, barriers):
    assert su2.su2_selftest_barrier(blocks, barriers, 20_000_000) == [blocks, 0, 1]


def test_barrier_self_test_arguments():
    for blocks, barriers, ns in ((0, 1, 1), (1025, 1, 1), (8, -1, 1), (8, 1001, 1), (8, 1, 5_000_000_001)):
        with pytest.raises(su2.SU2Error):
            su2.su2_selftest_barrier(blocks, barriers, ns)


@pytest.mark.parametrize("stream", [False, True])
@pytest.mark.parametrize("sweeps,every", [(1, 0), (5, 0), (6, 2)])
def test_a_sweep_that_was_given_up_is_reported(stream, sweeps, every):
    """The error word outlives the launches queued behind the one that set it,
    these leave links and counters alone, and the next call starts clean."""
    torch = pytest.importorskip("torch")
    shapes = ([4, 6], [4, 2], [2.1, 2.4], [3, 4])
    b = su2.su2_batch_create(*shapes, su2.SU2_HOT, stream=torch.cuda.Stream() if stream else None)
    ref = su2.su2_batch_create(*shapes, su2.SU2_HOT)
    try:
        for h in (b, ref):
            su2.su2_batch_generate(h, 2, 3, 1)
        with pytest.raises(su2.SU2Error) as err:
            su2.su2_selftest_batch_stopped(b, sweeps, every)
        assert err.value.status == 5  # SU2_E_DEVICE_TIMEOUT
        assert su2.su2_batch_info(b)["sweep"] == 3
        pb, lb, sb = su2.su2_batch_generate(b, 2, 4, 1)
        pr, lr, sr = su2.su2_batch_generate(ref, 2, 4, 1)
        assert np.array_equal(pb, pr) and np.array_equal(lb, lr) and sb["trials"] == sr["trials"]
        assert np.array_equal(su2.su2_batch_plaquette(b, 2), su2.su2_batch_plaquette(ref, 2))
        for i, (ns, nt) in enumerate(zip(*shapes[:2])):
            assert np.array_equal(su2.su2_batch_get_links(b, i, ns, nt), su2.su2_batch_get_links(ref, i, ns, nt))
    finally:
        su2.su2_batch_destroy(b)
        su2.su2_batch_destroy(ref)
