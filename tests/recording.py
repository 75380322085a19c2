"""The library's host code over a recording stand-in for the CUDA runtime
(recording_runtime.cpp): which calls are made in what order, with how much memory.
No GPU and no kernel runs."""
import contextlib
import ctypes as C
import os
import shutil
import subprocess

import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
STREAM = 4711   # a stream that the legacy default stream does not wait for


@pytest.fixture(scope="session")
def recorder(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    B.build()
    objs = [os.path.join(B.BUILD, u.replace(".cu", ".o")) for u in B.UNITS]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    out = str(tmp_path_factory.mktemp("recording") / "librecording.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    subprocess.run([gxx, "-shared", "-fPIC", "-O1", "-std=c++17", "-I", inc, os.path.join(HERE, "recording_runtime.cpp"),
                    *objs, "-Wl,-Bsymbolic", "-o", out], check=True)
    return Recorder(out)


class Recorder:
    def __init__(self, path):
        own, P._lib = P._lib, None
        try:
            self.lib = P.load(path)
        finally:
            P._lib = own
        self.lib.rec_log.restype = C.c_char_p
        self.lib.rec_held.restype = C.c_size_t
        self.lib.rec_limit.argtypes = [C.c_size_t]

    @contextlib.contextmanager
    def in_place(self, limit=2 ** 64 - 1):
        """The package's calls go to the recorded library; `limit` bytes can be allocated."""
        own, P._lib = P._lib, self.lib
        self.lib.rec_clear()
        self.lib.rec_limit(limit)
        try:
            yield self
        finally:
            P._lib = own

    def calls(self):
        return [l.split() for l in self.lib.rec_log().decode().splitlines()]

    def held(self):
        return self.lib.rec_held()


def unordered(calls):
    """Calls on another stream than the legacy one that may run before an earlier legacy copy from
    pageable memory or clear is done.  A legacy copy waits for what was queued there before it; one to
    the device may return, and end, later."""
    bad, pending = [], None
    for c in calls:
        if c[0] == "sync" and c[1] in ("0", "all"):
            pending = None
        elif c[0] in ("memset", "copy") and c[1] == "0":
            pending = None if c[0] == "copy" and c[2] == "2" else c
        elif c[0] in ("memset", "copy", "launch") and pending:
            bad.append((pending, c))
    return bad
