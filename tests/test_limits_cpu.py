"""Launch limits of the C-ABI that the host checks before any buffer."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def libgk():
    from paper_2103_14978_gb300 import build, gk

    build.build()
    return gk


def test_more_pairs_than_a_grid_has_blocks_for(libgk):
    """2^38 pairs in blocks of 128 threads are 2^31 blocks, one more than a
    grid holds; one pair fewer passes on to the check of the buffers."""
    L = libgk.lib()
    handle = ctypes.create_string_buffer(256)  # not looked into before these checks
    ref = ctypes.cast(handle, ctypes.c_void_p)
    calls = [lambda n: L.gk_filter(ref, None, 4, 1, None, 100, None, None, None, 2, n, 0, 0, None, None, None, None),
             lambda n: L.gk_filter_sweep(ref, None, 4, 1, None, 100, None, None, 0, 5, n, 0, 0, None, None, n, None,
                                         None),
             lambda n: L.gk_filter_ascii(ref, None, 100, 1, 100, None, None, None, 2, n, 0, 0, None, None, None, None)]
    for call in calls:
        assert call(1 << 38) == libgk.GK_ERANGE
        assert call((1 << 38) - 128) == libgk.GK_EINVAL
