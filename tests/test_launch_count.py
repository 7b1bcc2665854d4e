"""The number of kernels in a captured line search is a difference of one thread's count: launches of other
threads meanwhile belong to the total only (CPU)."""
import ctypes as ct
import threading

import pytest


@pytest.fixture(scope="module")
def counters():
    from paper_1312_1549_gb300 import _native, build
    lib = ct.CDLL(build.build())
    counted = lib._ZN3omm16launches_countedEv      # omm::launches_counted()
    counted.restype = ct.c_ulonglong
    launch = lib._ZN3omm12count_launchEv           # omm::count_launch()
    add = lib._ZN3omm14count_launchesEl            # omm::count_launches(long)
    add.argtypes = [ct.c_long]
    return counted, launch, add, _native.lib().omm_launch_count


def test_other_threads_do_not_count(counters):
    counted, launch, add, total = counters
    before, all_before = counted(), total()
    launch()
    other = threading.Thread(target=lambda: [launch() for _ in range(7)])
    other.start()
    other.join()
    launch()
    assert counted() - before == 2
    assert total() - all_before == 9
    add(-2)  # the end of a capture
    assert counted() == before and total() - all_before == 7
