"""The context's side stream is optional: when one of the three objects cannot
be created there is no stream, nothing is leaked, and no error stays behind
for the next call's launch check to report."""
import ctypes as C

import pytest

import host


@pytest.mark.parametrize("call", [0, 1, 2, 3])
def test_failed_creation_leaves_nothing(call):
    out = (C.c_int * 4)()
    host.load("side_stream_host").side_with_failure(call, out)
    exists, live, live_after, error = out
    assert exists == (call == 0) and live == (3 if call == 0 else 0)
    assert live_after == 0 and error == 0
