"""The pool of page-locked result pages, compiled for the host over a fake of
the runtime calls that it makes."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1010_1486_gb300", "csrc")


@pytest.fixture(scope="module")
def scenario(tmp_path_factory):
    from paper_1010_1486_gb300 import _build

    try:
        cuda = os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc())))
    except RuntimeError:
        pytest.skip("CUDA headers not available")
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("pages") / "host_pages_fake")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "host_pages_fake.cpp"), "-o", exe], check=True)
    return lambda name: [int(v) for v in subprocess.run([exe, name], capture_output=True, text=True,
                                                        check=True).stdout.split()]


def test_a_call_that_returns_early_waits_for_its_stream(scenario):
    # no wait after settled(); one on the page's own stream without; the pool
    # holds 16 pages, and a call without a page has nothing to wait for
    assert scenario("settle") == [0, 1, 1, 1, 16, 16]


def test_one_page_stays_when_the_last_handle_goes(scenario):
    """Five turns of a handle with three pages: the first makes three, the
    others two each, and two go back at the end of each.  A page that a device
    reset took away is forgotten, not freed, and a new one made."""
    assert scenario("turns") == [3 + 4 * 2, 5 * 2, 1, 12, 10, 10, 1]
