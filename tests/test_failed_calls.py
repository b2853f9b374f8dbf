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
rt.fake_symbols.restype = rt.fake_block.restype = ctypes.c_void_p
rt.fake_block.argtypes = [ctypes.c_size_t]
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

memory = ctypes.create_string_buffer(1 << 16)      # kernels do nothing: only copied and set
x = (ctypes.addressof(memory) + 255) & ~255

def column(n=5000, b=8):
    return gbscan.Column.from_packed(x, n, b)
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


@pytest.mark.parametrize("name", ["launch", "cudaFuncSetAttribute", "cudaMalloc", "cudaMemsetAsync"])
def test_a_failed_call_is_not_reported_again_by_the_next_one(child, name):
    """Launch checks read cudaGetLastError; an error that an earlier call has reported
    must be gone from it."""
    child(f"""
        name = {name!r}
        c = column(n=5000, b=8)
        c.zonemap_build()                      # launches once, so that its kernel is set up
        net = gbscan.Planner(4)
        failing = {{
            "launch": [lambda: c.run(1, 5), lambda: c.run(1, 5, "zone_bf"), lambda: c.select(1, 5),
                       lambda: gbscan.scan_conj([c, c], [(1, 5), (1, 5)], c),
                       lambda: gbscan.scan_run_packed_noalloc(x, 5000, 8, 0, 1, 5, x, x),
                       lambda: net.forward(x, 16, x)],
            "cudaFuncSetAttribute": [lambda: c.run(1, 5, "branchy"), lambda: column(b=9).select(1, 5),
                                     lambda: gbscan.scan_conj([column(b=9)], [(1, 5)])],
            "cudaMalloc": [lambda: column(), lambda: gbscan.Planner(4),
                           lambda: gbscan.Batch([c], tiles_per_pop=1), lambda: c.autotune(1, 5)],
            "cudaMemsetAsync": [lambda: c.select_async(9, 9, x, x, capacity=1),
                                lambda: gbscan.scan_run_packed_noalloc(x, 5000, 8, 0, 1, 5, x, x)],
        }}[name]
        for i, f in enumerate(failing):
            skipped = 1 if name == "launch" and i == 1 else 0    # the filter's launch, then the scan's
            fail(name, skipped)
            assert status_of(f) == gbscan.SCAN_ECUDA, i
            assert rt.cudaGetLastError() == 0, i
    """)


def test_a_zone_scan_that_fails_behind_its_filter_leaves_no_candidates(child):
    """The filter counts the surviving blocks for the scan, which resets the count; if the
    scan is not launched, the next filter must not append to that list (it holds one entry
    per block, so a second list would run past its end)."""
    child("""
        c = column(n=5000, b=8)
        qctl = (ctypes.c_uint64 * 8).from_address(rt.fake_block(128 + 16 * 1024) + 64)   # in the column's workspace
        c.zonemap_build()

        def check(strategy):
            qctl[0], qctl[3], qctl[4] = 4, 1024, 77                 # as the filter leaves them
            assert status_of(c.run, 1, 5, strategy) == gbscan.SCAN_ECUDA
            assert list(qctl) == [0] * 8, strategy

        for strategy in ("zone_bf", "zone_br"):
            fail("cudaFuncSetAttribute")
            check(strategy)
        for strategy in ("zone_bf", "zone_br", "zone_agg_bf", "zone_agg_br"):
            fail("launch", 1)                                       # the filter's is the first
            check(strategy)
    """)


def test_an_encode_that_failed_leaves_no_error_for_the_next(child):
    """A device encode reads its range error from one of a set of words; a call that fails
    before it has read or cleared its word must not leave the error to a later call."""
    child("""
        word = ctypes.c_uint32.from_address(rt.fake_symbols())
        encode = lambda: gbscan.scan_encode_device(x, 1000, 8, 0, x)
        for name in ("cudaMemcpyAsync", "cudaStreamSynchronize", "cudaMemsetAsync"):   # read, wait, reset
            word.value = 2                      # as the kernel sets it for a value out of range
            fail(name)
            assert status_of(encode) == gbscan.SCAN_ECUDA, name
            assert word.value == 2
            for _ in range(2):
                assert status_of(encode) == gbscan.SCAN_OK, name
        word.value = 2
        assert status_of(encode) == gbscan.SCAN_EINVAL and word.value == 0
        assert status_of(encode) == gbscan.SCAN_OK
    """)
