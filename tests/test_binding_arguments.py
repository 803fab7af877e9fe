"""Arguments of the hot entry points (csrc/fastcall.c): what a ctypes prototype takes they take, and a call that names its stream
needs neither torch nor a device to report a bad argument."""
import ctypes
import subprocess
import sys

import pytest

from paper_2608_16308_b200 import binding as B


class Wrapped:
    def __init__(self, v):
        self._as_parameter_ = v


def status(f, *args, **kw):
    with pytest.raises(B.DbSpmspvError) as e:
        f(*args, **kw)
    return e.value.status


HANDLES = [None, ctypes.c_void_p(), 4096, ctypes.c_void_p(4096), Wrapped(4096), Wrapped(ctypes.c_void_p(4096)), -4096, 1 << 70]


@pytest.mark.parametrize("h", HANDLES, ids=str)
@pytest.mark.parametrize("stream", [0, ctypes.c_void_p(0), ctypes.c_void_p(), Wrapped(0)], ids=["int", "zero", "null", "wrapped"])
def test_handles_and_streams(h, stream):
    """(a negative length is refused before the handle is looked at)"""
    for n in (-1, ctypes.c_int32(-1), (1 << 40) - 1):
        assert status(B.dbspmspv_run, h, None, None, n, B.PLUS_TIMES, None, None, 0, None, stream) == B.ERR_INVALID_ARG
    assert status(B.dbspmspv_run_masked, h, None, None, -1, B.OR_AND, None, 0, None, None, ctypes.c_int64(0), None, stream=stream) == B.ERR_INVALID_ARG
    assert status(B.dbspmspv_decode, h, None, None, stream=stream) == B.ERR_INVALID_ARG
    assert status(B.dbspmspv_decode_batch, h, None, 0, None, 1 << 64, 0, stream) == B.ERR_INVALID_ARG
    assert status(B.db_bfs, h, 0, None, stream) == B.ERR_INVALID_ARG
    assert status(B.db_sssp, h, 0, None, stream) == B.ERR_INVALID_ARG


@pytest.mark.parametrize("bad", ["4096", 1.0, ctypes.c_float(1.0), object()], ids=["text", "float", "c_float", "object"])
def test_other_types_are_refused(bad):
    with pytest.raises(TypeError):
        B.db_bfs(bad, 0, None, 0)
    with pytest.raises(TypeError):
        B.db_bfs(None, bad, None, 0)
    with pytest.raises(TypeError):
        B.db_bfs(None, 0, None, bad)


def test_a_named_stream_needs_no_torch():
    code = ("import sys; from paper_2608_16308_b200 import binding as B\n"
            "try: B.db_bfs(None, 0, None, 0)\n"
            "except B.DbSpmspvError as e: print(e.status, 'torch' in sys.modules)")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.stdout.split() == [str(B.ERR_INVALID_ARG), "False"], r.stdout + r.stderr
