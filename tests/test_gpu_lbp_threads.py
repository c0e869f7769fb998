"""cnf_lbp where no host thread can be started (every new thread asks for an impossible stack): the same
results. In a child process, which a thrown C++ exception would end."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes, sys
import numpy as np
import nmc_inputs as W
import paper_2111_13628_gb300 as nmc

n, S = 3000, 64
lits = W.random_ksat(n, 4.0, 3, 5)
x = (W.splitmix64(6, S * n) & np.uint64(1)).astype(np.uint8).reshape(S, n)
with nmc.Context(0) as ctx:
    inst = ctx.load_ksat(lits, n)
    run = lambda: ctx.cnf_lbp(inst, x, 1.0, [0.3], 1e-8, 5)
    want = run()
    assert want["marg"].nbytes >= 1 << 20
    libc, attr, old = ctypes.CDLL(None), ctypes.create_string_buffer(256), ctypes.create_string_buffer(256)
    assert libc.pthread_getattr_default_np(old) == 0
    assert libc.pthread_attr_init(attr) == 0
    assert libc.pthread_attr_setstacksize(attr, ctypes.c_size_t(1 << 60)) == 0
    assert libc.pthread_setattr_default_np(attr) == 0
    tid, entry = ctypes.c_ulong(), ctypes.cast(libc.getpid, ctypes.c_void_p)
    assert libc.pthread_create(ctypes.byref(tid), None, entry, None) != 0  # none to be had
    got = run()
    assert libc.pthread_setattr_default_np(old) == 0
for key in want:
    assert np.array_equal(got[key], want[key]), key
print("same")
"""


def test_without_host_threads():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "same", out.stderr[-2000:]
