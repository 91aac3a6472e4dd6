"""Host memory of the set-up: a C entry that runs out of it returns an error code,
and what a worker thread keeps for itself does not grow with the mesh."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# felbm_init's host tables under an address-space limit a little above what the
# process holds.  The workspace pointer is never used: the limits are far below
# what the tables need, so every call fails before its first upload.
STARVED = r"""
import ctypes, resource, sys
import numpy as np
from paper_1708_04678_gb300 import felbm as F, inputs as I
w = I.small_sessile(nx=800, ny=400, R=100.0)
mesh = F.Mesh.from_dict(w["mesh"])
lib = F.lib()
rcs = []
for precision in (F.FP64, F.FP32_DEV):
    params = F.params_derive(w["phys"], precision=precision)
    nbytes = mesh.workspace_bytes(params)
    C0 = np.ascontiguousarray(w["C0"])
    for spare in (1, 4, 8, 16):
        out = ctypes.c_void_p()
        kb = next(int(l.split()[1]) for l in open("/proc/self/status") if l.startswith("VmSize"))
        resource.setrlimit(resource.RLIMIT_AS, ((kb << 10) + (spare << 20), resource.RLIM_INFINITY))
        rc = lib.felbm_init(mesh.handle, ctypes.byref(params), C0.ctypes.data, None, None, 1 << 40, nbytes, None,
                            ctypes.byref(out))
        resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
        rcs.append((rc, lib.felbm_last_error().decode(), out.value))
print(rcs)
sys.exit(0 if all(rc == -1 and "felbm_init" in msg and p is None for rc, msg, p in rcs) else 3)
"""


@pytest.mark.skipif(torch.cuda.is_available(), reason="the workspace pointer is not a device's")
def test_init_returns_an_error_when_host_memory_runs_out():
    r = subprocess.run([sys.executable, "-c", STARVED], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr[-2000:])
