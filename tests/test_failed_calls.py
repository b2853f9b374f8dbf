"""Calls of the CUDA runtime that fail, on CPU: each case runs in a child process with
the runtime's calls replaced (fake_cudart.c), makes one of them fail, and checks that
the library reports it and that the calls after it are answered as if it had not been."""
import os
import subprocess
import sys
import textwrap

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes
from paper_2606_22423_gb300 import gbscan

rt = ctypes.CDLL(None)
rt.fake_copy_bytes.restype = ctypes.c_size_t
rt.fake_symbols.restype = ctypes.c_void_p
INVALID, NO_MEMORY = 1, 2

def fail(name, after=0, code=INVALID):
    rt.fake_fail(name.encode(), after, code)

def status_of(f, *args):
    try:
        f(*args)
    except gbscan.ScanError as e:
        assert rt.fake_pending() == 0
        return e.status
    return gbscan.SCAN_OK

def column(n=5000, b=8):
    return gbscan.Column.from_packed(4096, n, b)   # an address: no kernel runs
"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    import __graft_entry__

    __graft_entry__.build()
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run(["gcc", "-O1", "-Wall", "-shared", "-fPIC", os.path.join(HERE, "fake_cudart.c"), "-o", so], check=True)

    def run(code):
        env = dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT)
        p = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(code)], env=env, capture_output=True, text=True,
                           timeout=120)
        assert p.returncode == 0, p.stdout + p.stderr

    return run


def test_a_scan_whose_kernel_cannot_be_set_up_is_an_error(child):
    """The first launch of a kernel sets its shared memory; if that fails nothing is
    launched, and the call must not return an older result as its own."""
    child("""
        for strategy in ("branchfree", "branchy"):
            for b in (8, 20):
                c = column(b=b)
                fail("cudaFuncSetAttribute", code=NO_MEMORY)
                assert status_of(c.run, 1, 5, strategy) == gbscan.SCAN_ENOMEM, (strategy, b)
                assert status_of(c.run, 1, 5, strategy) == gbscan.SCAN_OK
    """)
