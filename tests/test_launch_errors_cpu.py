"""A launch that fails is reported by the call that made it, whatever the calls after it did."""
import ctypes

import pytest


@pytest.mark.parametrize("results,last,want", [([0, 0], 0, 0), ([0, 1, 0], 0, 1), ([1, 9], 0, 1), ([0], 700, 700), ([9, 0], 700, 9), ([], 0, 0)])
def test_the_first_launch_error_of_a_call_is_reported_once(results, last, want):
    from paper_2002_07627_gb300 import build
    build.build()
    r = (ctypes.c_int * max(len(results), 1))(*results)
    nxt = ctypes.c_int(-1)
    assert ctypes.CDLL(build.HOSTLIB).imf_host_launch_errors(r, len(results), last, ctypes.byref(nxt)) == want
    assert nxt.value == 0
