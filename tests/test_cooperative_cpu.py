"""How many blocks a cooperative kernel gets where the stream owns fewer SMs than the device has."""
import ctypes

import pytest

TOO_LARGE = 720      # cudaErrorCooperativeLaunchTooLarge


@pytest.mark.parametrize("want,room", [(1216, 1216), (1216, 64), (1216, 63), (5, 4), (3, 1), (1, 1), (0, 1), (257, 16)])
def test_a_launch_that_does_not_fit_is_made_with_fewer_blocks(want, room):
    from paper_2002_07627_gb300 import build
    build.build()
    L = ctypes.CDLL(build.HOSTLIB)
    tries = ctypes.c_int()
    n = L.imf_host_launch_fitting(ctypes.c_long(want), ctypes.c_long(room), 0, ctypes.byref(tries))
    assert 1 <= n <= room and tries.value <= 12
    assert n == max(want, 1) if want <= room else 2 * n > room or room == 1
    # another error is the launch's result, at once; where not one block fits, so is this one
    assert L.imf_host_launch_fitting(ctypes.c_long(1), ctypes.c_long(1), 9, ctypes.byref(tries)) == -9 and tries.value == 1
    assert L.imf_host_launch_fitting(ctypes.c_long(want), ctypes.c_long(0), 0, ctypes.byref(tries)) == -TOO_LARGE


def test_a_solve_in_which_a_block_gave_up_is_not_taken():
    """A block that gives up at the last barrier leaves without its share of the compliance, while the others pass
    the barrier and report that the iteration converged."""
    from paper_2002_07627_gb300 import build
    build.build()
    taken = lambda done, err: ctypes.CDLL(build.HOSTLIB).imf_host_mg_converged(ctypes.c_double(done), ctypes.c_uint(err))
    assert taken(1.0, 0) == 1 and taken(1.0, 1) == 0 and taken(0.0, 0) == 0 and taken(0.0, 1) == 0


def test_a_large_hierarchy_takes_a_sixteenth_of_the_free_memory_at_most():
    from paper_2002_07627_gb300 import build
    build.build()
    L = ctypes.CDLL(build.HOSTLIB)
    ok = lambda b, room: L.imf_host_mg_affordable(ctypes.c_ulonglong(b), ctypes.c_ulonglong(room))
    G = 1 << 30
    assert ok(256 << 20, 0) == 1 and ok((256 << 20) + 1, 4 * G) == 0 and ok((256 << 20) + 1, 5 * G) == 1
    assert ok(16 * G, 256 * G) == 1 and ok(16 * G + 1, 256 * G) == 0 and ok(142 * G, 250 * G) == 0
