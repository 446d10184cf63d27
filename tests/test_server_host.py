"""The server's sizing of queued jobs, which runs on its callers' threads and
needs no GPU."""
from __future__ import annotations

import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# the library's own symbol (C++ linkage, no header): n, m, k, graphs
SIZES = r"""
import ctypes, sys
sys.path.insert(0, {root!r})
from paper_2308_15494_gb300 import build
lib = ctypes.CDLL(build.build())
f = lib._Z17upr_ctx_footprintllii
f.restype, f.argtypes = ctypes.c_size_t, [ctypes.c_int64, ctypes.c_int64, ctypes.c_int32, ctypes.c_int32]
last = 0
for n in (0, 2048, 65536, 65537, 1 << 20, 1 << 24):
    size = f(n, 16 * n, 64, 1)
    assert size > last and size >= n * 64 * 4 + 16 * n * 4, (n, size)
    last = size
assert f(70000, 70000, 8, 100) > f(70000, 70000, 8, 1)
print("ok")
"""


def test_job_sizes_without_a_device():
    """A job's device bytes are arithmetic: no CUDA call, which could fail (and
    throw through the C entry points) on a thread or process without a device."""
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")
    r = subprocess.run([sys.executable, "-c", SIZES.format(root=ROOT)], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.returncode, r.stderr[-1000:])
