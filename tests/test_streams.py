"""Launches are chained (a kernel may start while the one before it drains) only
while all grids of the process work on one stream: the count of the grids'
streams, on the CPU."""
import ctypes
import gc

import pytest

import paper_2510_09081_gb300 as vrt


@pytest.fixture
def streams():
    lib = vrt.load()
    fns = [getattr(lib, f"_ZN3vrt12stream_{what}EP11CUstream_st") for what in ("enter", "leave", "alone")]
    for f in fns:
        f.argtypes, f.restype = [ctypes.c_void_p], None
    fns[2].restype = ctypes.c_bool
    gc.collect()
    if not fns[2](0x1000):
        pytest.skip("grids of other tests are alive in this process")
    return fns


def test_only_the_streams_of_live_grids_count(streams):
    enter, leave, alone = streams
    a, b = 0x1000, 0x2000
    assert alone(a) and alone(None)        # no grid anywhere
    enter(a)
    enter(a)                               # two grids on one stream
    assert alone(a) and not alone(b) and not alone(None)
    enter(b)
    assert not alone(a) and not alone(b)
    leave(a)
    assert not alone(a) and not alone(b)   # one grid is still on a
    leave(a)
    assert alone(b) and not alone(a)
    leave(b)
    leave(b)                               # a stream nobody is on
    assert alone(a) and alone(b)
    enter(None)                            # the default stream is a stream like others
    assert alone(None) and not alone(a)
    leave(None)
