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


# The other entries that make tables, in the same way.
STARVED_OTHERS = r"""
import ctypes, resource, sys
import numpy as np
from paper_1708_04678_gb300 import felbm as F, felbm3d as F3, inputs as I, inputs3d as I3

def starved(call, spare):
    kb = next(int(l.split()[1]) for l in open("/proc/self/status") if l.startswith("VmSize"))
    resource.setrlimit(resource.RLIMIT_AS, ((kb << 10) + (spare << 20), resource.RLIM_INFINITY))
    rc = call()
    resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
    return rc, F.lib().felbm_last_error().decode()

rcs = []
w = I3.small_sessile_3d(n=40, nz=40)
mesh = F3.Mesh3D.from_dict(w["mesh"])
params = F.params_derive(w["phys"])
C0, out = np.ascontiguousarray(w["C0"]), ctypes.c_void_p()
args = (mesh.handle, ctypes.byref(params), C0.ctypes.data, 1 << 40, mesh.workspace_bytes(params), None, ctypes.byref(out))
rcs.append(starved(lambda: F3.lib().felbm3d_init(*args), 1))
m = I.small_sessile(nx=1500, ny=700, R=100.0)["mesh"]
xy, tri = np.ascontiguousarray(m["xy"], dtype=np.float64), np.ascontiguousarray(m["tri"], dtype=np.int32)
we, wid = np.ascontiguousarray(m["wall_edges"], dtype=np.int32), np.ascontiguousarray(m["wall_id"], dtype=np.int32)
d = (F.MeshDesc * 1)()
d[0].xy, d[0].n_nodes, d[0].tri, d[0].n_tri = xy.ctypes.data, len(xy), tri.ctypes.data, len(tri)
d[0].wall_edges, d[0].wall_id, d[0].n_wall_edges = we.ctypes.data, wid.ctypes.data, len(we)
d[0].period_x = float(m["period"][0])
for spare in (0, 8, 16, 32):
    rcs.append(starved(lambda: F.lib().felbm_mesh_create_batch(1, d, ctypes.byref(out)), spare))
print(rcs)
sys.exit(0 if all(rc == -1 and "felbm" in msg and not out.value for rc, msg in rcs) else 3)
"""


@pytest.mark.skipif(torch.cuda.is_available(), reason="the workspace pointer is not a device's")
def test_other_entries_return_an_error_when_host_memory_runs_out():
    # large blocks straight from the system, so that none comes from freed memory
    r = subprocess.run([sys.executable, "-c", STARVED_OTHERS], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, MALLOC_MMAP_THRESHOLD_="65536"))
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr[-2000:])


# Largest block of memory that a worker thread of the set-up asks for, with the
# threads that a host of many cores would start: a preloaded library answers
# std::thread::hardware_concurrency and watches operator new.  felbm_init stops at
# its first upload (no device here).
WATCH = r"""
#include <atomic>
#include <cstdlib>
#include <new>
#include <thread>
#include <unistd.h>
static std::atomic<size_t> biggest{0}, workers{0};
unsigned std::thread::hardware_concurrency() noexcept { return 16; }
void* operator new(size_t n) {
    static thread_local bool seen = false;
    if (gettid() != getpid()) {
        if (!seen) workers++;
        seen = true;
        size_t b = biggest;
        while (n > b && !biggest.compare_exchange_weak(b, n)) {}
    }
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }
extern "C" size_t biggest_of_workers() { return biggest.exchange(0); }
extern "C" size_t workers_seen() { return workers.exchange(0); }
"""

SET_UP = r"""
import ctypes, sys
import numpy as np
from paper_1708_04678_gb300 import felbm as F, inputs as I
watch = ctypes.CDLL(sys.argv[1])
watch.biggest_of_workers.restype = watch.workers_seen.restype = ctypes.c_size_t
w = I.small_sessile(nx=500, ny=250, R=60.0)
F.lib()
watch.biggest_of_workers(), watch.workers_seen()
mesh = F.Mesh.from_dict(w["mesh"])
print(watch.workers_seen(), watch.biggest_of_workers())
params = F.params_derive(w["phys"], precision=F.FP32_DEV)
out, C0 = ctypes.c_void_p(), np.ascontiguousarray(w["C0"])
rc = F.lib().felbm_init(mesh.handle, ctypes.byref(params), C0.ctypes.data, None, None, 1 << 40,
                        mesh.workspace_bytes(params), None, ctypes.byref(out))
assert rc == -3, rc
print(watch.workers_seen(), watch.biggest_of_workers())
"""


@pytest.mark.skipif(torch.cuda.is_available(), reason="the workspace pointer is not a device's")
def test_scratch_of_the_threads_does_not_grow_with_the_mesh(tmp_path):
    src, lib = tmp_path / "watch.cpp", tmp_path / "watch.so"
    src.write_text(WATCH)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", str(src), "-o", str(lib)], check=True)
    r = subprocess.run([sys.executable, "-c", SET_UP, str(lib)], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=str(lib)))
    assert r.returncode == 0, r.stderr[-2000:]
    for line in r.stdout.splitlines():
        workers, biggest = (int(v) for v in line.split())
        # a word per node would be 502 KB; a block has at most 1,024 nodes and 1,400 triangles
        assert workers > 0 and biggest < 64 * 1024, r.stdout
