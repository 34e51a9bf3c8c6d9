"""gmg_setup on a host that is out of memory: a status, not an exception through
the C ABI (which ends the process).  The set-up's first host buffer is wanted
before any device call, so this runs without a GPU, in a process of its own
whose address space is limited."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes, resource, sys
import numpy as np
sys.path.insert(0, {root!r})
import paper_2307_04886_gb300 as g
lib = g.load_library()
n = 16_000_000  # the validation's cursors take 128 MB
rp, ci, va = np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), np.ones(n)
csr = g.gmg_csr(n, rp.ctypes.data, ci.ctypes.data, va.ctypes.data)
h = ctypes.c_void_p()
now = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (now + (32 << 20), resource.RLIM_INFINITY))
st = lib.gmg_setup(ctypes.byref(h), ctypes.byref(csr), 0, (g.gmg_prolong * 1)(), None, None, None)
print(st, h.value, lib.gmg_last_error().decode())
"""


def test_out_of_host_memory_is_a_status():
    import paper_2307_04886_gb300 as g

    try:
        g.build_library()
    except Exception as e:  # pragma: no cover - nvcc missing
        pytest.skip(f"cannot build libgmg: {e}")
    p = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT)], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    status, handle, message = p.stdout.split(maxsplit=2)
    assert int(status) == g.GMG_ERR_OOM and handle == "None" and message.startswith("gmg_setup: ")
