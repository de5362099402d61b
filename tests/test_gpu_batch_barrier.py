"""The grid barrier of the batched sweeps, through the function that the sweep
kernel calls: barriers that complete order the blocks' writes, and a wait that
nothing completes gives up in every block and leaves its mark in the error word."""
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
