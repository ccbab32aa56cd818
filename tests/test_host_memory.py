"""Host memory that runs out while a graph is built or loaded is a status, not an
exception across the C ABI (which would end the process).  The calls run in a
child process whose address space has no room for their working arrays."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = """
import ctypes, resource
import numpy as np
import __graft_entry__ as g
g.build()
from paper_2502_10579_gb300 import svv

def used():
    return int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()

def limited(call, room):
    soft, hard = resource.getrlimit(resource.RLIMIT_AS)
    resource.setrlimit(resource.RLIMIT_AS, (used() + room, hard))
    try:
        return call()
    finally:
        resource.setrlimit(resource.RLIMIT_AS, (soft, hard))

V = 1 << 25  # one 64-bit word per vertex: 256 MB
row_ptr = np.zeros(V + 1, np.uint64)
E = ctypes.c_uint64(7)
"""

BUILD = """
L = svv.lib()
print("status", limited(lambda: L.svv_build_versioned_csr(V, 8, 0, *[None] * 5, svv._ptr(row_ptr), None, None, None,
                                                          ctypes.byref(E)), 64 << 20))
"""

LOAD = """
import torch
from workloads import small_rmat
import oracle
log = small_rmat()
want = oracle.query(log, 0, 0, 0, log.S)
ctx = svv.Context(0)
ctx.load_log(log)
assert (svv.to_u32(ctx.query(0, 0, 0, log.S)) == want).all()
no = np.zeros(1, np.uint32)
print("status", limited(lambda: svv.lib().svv_load(ctx.h, V, 0, 8, svv._ptr(row_ptr), svv._ptr(no), svv._ptr(no),
                                                   svv._ptr(no), 0), 64 << 20))
assert (svv.to_u32(ctx.query(0, 0, 0, log.S)) == want).all()  # the graph loaded before is still there
ctx.close()
"""


def child(code):
    r = subprocess.run([sys.executable, "-c", COMMON + code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.split()[-2:]


def test_builder_out_of_host_memory():
    assert child(BUILD) == ["status", "2"]


@pytest.mark.gpu
def test_load_out_of_host_memory():
    assert child(LOAD) == ["status", "2"]
